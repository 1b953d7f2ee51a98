"""A step budget counts finished paths: no more paths are begun than the budget's
worth of finished ones and one per lane group, however short the FP32 phases are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc as mod
    return mod


@pytest.mark.parametrize("fp32_steps", [1, 10000])
def test_paths_begun_under_a_budget(hc, fp32_steps):
    import torch
    from paper_2112_03444_gb300 import inputs
    n, count, budget = 6, 4096, 150_000
    base, coefs = inputs.dense_batch(n, 2, [950])
    rng = np.random.default_rng(950)
    coefs = rng.standard_normal((count, coefs.shape[1])) + 1j * rng.standard_normal(
        (count, coefs.shape[1]))
    pr = hc.Problem(base, gamma=inputs.unit_gamma(950),
                    settings=dict(max_steps_fp32=fp32_steps, escalate=0))
    b = pr.track(n_instances=count, coef=coefs, step_budget=budget)
    assert b.poll(-1) == hc.HC_ERR_TIMEOUT
    steps = b.steps[..., :2].sum(-1)
    begun = b.status != 0
    assert np.array_equal(begun, steps != 0)
    assert b.result["untracked"] == int((~begun).sum())
    assert b.result["steps_total"] == int(steps.sum()) >= budget
    # 2048 threads per SM in groups of 8 lanes; the paths that make up the budget
    # took at least the fewest steps of any
    groups = torch.cuda.get_device_properties(0).multi_processor_count * 2048 // 8
    assert int(begun.sum()) <= groups + budget // int(steps[begun].min()) + 1
