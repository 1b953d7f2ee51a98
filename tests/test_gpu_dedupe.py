"""Duplicate endpoints: exactly the paths whose FP32 endpoint copies collide in
their instance (and those that failed) are re-tracked, over instances smaller and
larger than the check's block and tile, with a step test loose enough that many
paths jump."""
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


@pytest.mark.parametrize("n,d,count", [(2, 2, 40), (3, 3, 11), (5, 2, 9), (7, 3, 1), (11, 2, 3),
                                       (12, 2, 1)])
def test_colliding_endpoints_are_retracked(hc, n, d, count):
    from paper_2112_03444_gb300 import inputs
    base, coefs = inputs.dense_batch(n, d, list(range(620, 620 + count)))
    loose = dict(max_first_corr_fp32=50.0, newton_tol_fp32=1e-2, dt_init=0.05)
    runs = []
    for escalate in (0, 1):
        pr = hc.Problem(base, gamma=inputs.unit_gamma(620), settings=dict(loose, escalate=escalate))
        runs.append(pr.track(n_instances=count, coef=coefs).wait())
    plain, full = runs
    total = 0
    for i in range(count):
        st = plain.status[i] & 0x7F
        ok = (st == 1) | (st == 6)
        x = plain.x[i].astype(np.complex64)
        v = np.concatenate([x.real, x.imag], axis=1)
        thr = np.float32(1e-6) * np.maximum(np.float32(1), np.abs(v).max(axis=1))
        dup = np.zeros(len(x), bool)
        for a in np.nonzero(ok)[0]:
            near = ok & (np.abs(v - v[a]) <= thr[a]).all(axis=1)
            near[a] = False
            dup[a] = near.any()
        again = dup | (st != 1)
        changed = (full.steps[i] != plain.steps[i]).any(axis=1)
        assert np.array_equal(changed & ~again, np.zeros(len(x), bool)), i
        assert np.array_equal(full.x[i][~again], plain.x[i][~again])
        assert changed[dup & (st == 1)].all()
        total += int(dup.sum())
    if n >= 7:
        assert total > 0
