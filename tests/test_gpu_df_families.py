"""Double-float tracking of parameter families (precision DF) over the sizes at
which its kernel changes: warps per path (n = 4 / 5, 8 / 9), rows per replica of
the solve (4, 8, 16, 32 lanes), rounds of terms per thread, most factors per
term, up to the largest n -- against the FP64 oracle path by path."""
import numpy as np
import pytest

import oracle
from oracle import KIND_COEFFICIENT, KIND_PARAMETER, OracleProblem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc as mod
    return mod


def _ring_family(n, extra, seed):
    """F_i = x_i^2 - p_i + q_i x_i x_(i+1) + `extra` terms of up to 6 factors,
    small in q; at q = 0, p = 1 the roots are sign vectors."""
    from paper_2112_03444_gb300.inputs import TermSystem
    rng = np.random.default_rng([seed, n])
    eq, cf, ex, pa = [], [], [], []

    def term(i, c, xs, ps):
        e = np.zeros(n, np.uint8)
        for x in xs:
            e[x % n] += 1
        eq.append(i)
        cf.append(c)
        ex.append(e)
        pa.append(list(ps) + [-1] * (2 - len(ps)))
    for i in range(n):
        term(i, 1.0, [i, i], [])
        term(i, -1.0, [], [i])
        term(i, 1.0, [i, i + 1], [n + i])
        for k in range(extra):
            term(i, 0.1, rng.integers(0, n, 1 + k % 4), [n + i, n + (i + k) % n])
    system = TermSystem(n=n, term_eq=np.array(eq), term_coef=np.array(cf, np.complex128),
                        term_exp=np.array(ex), term_param=np.array(pa, np.int32), n_params=2 * n,
                        name="ring")
    p0 = np.concatenate([np.ones(n), np.zeros(n)]).astype(np.complex128)
    z = rng.standard_normal(4 * n)
    p1 = np.concatenate([1.0 + 0.5 * (z[:n] + 1j * z[n:2 * n]),
                         0.2 * (z[2 * n:3 * n] + 1j * z[3 * n:])])
    start = rng.choice([-1.0, 1.0], size=(12, n)).astype(np.complex128)
    return system, p0, p1, np.unique(start, axis=0)


@pytest.mark.parametrize("kind", ["parameter", "coefficient"])
@pytest.mark.parametrize("n,extra", [(1, 0), (2, 5), (4, 12), (5, 1), (8, 9), (9, 0), (16, 3),
                                     (17, 6), (24, 8)])
def test_df_families_match_oracle(hc, n, extra, kind):
    system, p0, p1, start = _ring_family(n, extra, 3)
    k = hc.HC_PARAMETER if kind == "parameter" else hc.HC_COEFFICIENT
    pr = hc.Problem(system, kind=k, p0=p0, start=start, settings=dict(precision=hc.HC_PREC_DF))
    b = pr.track(n_instances=2, p1=np.array([p1, p1 * np.exp(0.1j)])).wait()
    ok = KIND_PARAMETER if kind == "parameter" else KIND_COEFFICIENT
    for s, q in enumerate((p1, p1 * np.exp(0.1j))):
        ref = OracleProblem(system, kind=ok, p0=p0, p1=q).track(start=start)
        assert np.array_equal(b.status[s] & 0x7F, ref["status"] & 0x7F)
        fin = (ref["status"] & 0x7F) == oracle.FINITE
        assert fin.sum() >= 1
        d = np.abs(b.x[s][fin] - ref["x"][fin]).max(axis=1)
        assert (d <= 1e-8 * np.maximum(1.0, np.abs(ref["x"][fin]).max(axis=1))).all()
