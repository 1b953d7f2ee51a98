"""The mixed batch kernels track a path in two loops (FP32 phase, then the
rest) and hand it over between them; a resident launch (hc_stream) tracks it in
one.  Both do the same arithmetic in the same order, so every result agrees bit
for bit, whatever ends the FP32 phase: t_endgame, t = 1 itself, the FP32 step
limit, steps below dt_min_fp32, the step limit of the path, or divergence."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STARTS = os.path.join(ROOT, "paper_2112_03444_gb300", "startsets")
SETTINGS = [dict(), dict(t_endgame=1.0), dict(t_endgame=0.3), dict(max_steps_fp32=7),
            dict(dt_min_fp32=0.02), dict(max_steps=20), dict(r_inf=1.5), dict(grow_after=1)]


@pytest.fixture(scope="module")
def hc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc as mod
    return mod


def _bits(a):
    return np.ascontiguousarray(a).view(np.uint8)


def _compare(hc, pr, key, data):
    ref = pr.track(n_instances=len(data), **{key: data}).wait()
    s = hc.Stream(pr, slots=len(data), idle_us=5000)
    try:
        tickets = [s.submit(**{key: row}) for row in data]
        for j, tk in enumerate(tickets):
            x, st, steps, be = s.poll(tk)
            assert np.array_equal(st, ref.status[j])
            assert np.array_equal(steps, ref.steps[j])
            assert np.array_equal(_bits(x), _bits(ref.x[j]))
            assert np.array_equal(_bits(be), _bits(ref.be[j]))
    finally:
        s.close()


@pytest.mark.parametrize("settings", SETTINGS, ids=lambda s: "-".join(s) or "default")
@pytest.mark.parametrize("n,d", [(1, 2), (1, 3), (2, 2), (4, 2), (5, 3), (7, 2), (9, 2)])
def test_two_loops_match_one_dense(hc, n, d, settings):
    from paper_2112_03444_gb300 import inputs
    base, coefs = inputs.dense_batch(n, d, [900 + n, 901 + n, 902 + n])
    pr = hc.Problem(base, gamma=inputs.unit_gamma(900 + n), settings=settings)
    _compare(hc, pr, "coef", coefs)


@pytest.mark.parametrize("settings", SETTINGS[:5], ids=lambda s: "-".join(s) or "default")
@pytest.mark.parametrize("name", ["p3p", "triangulation2", "pose5_depth"])
def test_two_loops_match_one_family(hc, name, settings):
    from paper_2112_03444_gb300 import inputs
    fam, scene = {"p3p": (inputs.p3p_family(), inputs.p3p_scene),
                  "triangulation2": (inputs.triangulation_family(2),
                                     lambda s: inputs.triangulation_scene(s, views=2)),
                  "pose5_depth": (inputs.pose5_depth_family(), inputs.pose5_scene)}[name]
    z = np.load(os.path.join(STARTS, f"{name}.npz"))
    pr = hc.Problem(fam.system, kind=hc.HC_PARAMETER, p0=z["p0"], start=z["start"],
                    settings=settings)
    _compare(hc, pr, "p1", np.array([scene(s)[0] for s in (81, 82, 83)]))


def test_hand_over_under_a_step_budget(hc):
    """The budget stops new paths; every started one ends, and the steps
    counted against it are those of the tracked paths."""
    from paper_2112_03444_gb300 import inputs
    base, coefs = inputs.dense_batch(8, 2, list(range(940, 980)))
    pr = hc.Problem(base, gamma=inputs.unit_gamma(940), settings=dict(escalate=0))
    full = pr.track(n_instances=len(coefs), coef=coefs).wait()
    b = pr.track(n_instances=len(coefs), coef=coefs, step_budget=1)
    b.poll(-1)
    started = b.status != 0
    assert np.array_equal(b.status[started], full.status[started])
    assert np.array_equal(b.steps[started], full.steps[started])
    assert b.result["untracked"] == int((~started).sum())
    assert b.result["steps_total"] == int(b.steps[started][:, :2].sum())
