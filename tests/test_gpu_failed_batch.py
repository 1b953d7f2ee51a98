"""A batch that cannot be set up returns its error without waiting for work of
other streams: a resident launch (hc_stream) ends only after its idle time."""
import time

import pytest

pytestmark = pytest.mark.gpu


def test_out_of_memory_beside_a_resident_launch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc, inputs
    base, coefs = inputs.dense_batch(6, 2, [960])
    pr = hc.Problem(base, gamma=inputs.unit_gamma(960))
    small = torch.zeros(1024, dtype=torch.complex128, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()

    def too_large():  # terabytes of tables: refused at the first allocation
        t0 = time.perf_counter()
        with pytest.raises(hc.HCError) as e:
            pr.track(n_instances=2 ** 31 - 1, coef=small, x_out=small, status_out=small,
                     steps_out=small, be_out=small, device=True, stream=side.cuda_stream)
        assert e.value.code == hc.HC_ERR_OOM
        return time.perf_counter() - t0

    idle_s = 4.0
    s = hc.Stream(pr, slots=2, idle_us=int(idle_s * 1e6))
    try:
        assert s.poll(s.submit(coef=coefs[0])) is not None
        ticket = s.submit(coef=coefs[0])  # the launch is resident until this is polled
        took = too_large()
        assert took < idle_s / 4, took
        assert s.poll(ticket) is not None
    finally:
        s.close()


def test_a_failed_batch_leaves_no_error_behind():
    import numpy as np
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc, inputs
    base, coefs = inputs.dense_batch(6, 2, [961])
    pr = hc.Problem(base, gamma=inputs.unit_gamma(961))
    small = torch.zeros(1024, dtype=torch.complex128, device="cuda")
    x = np.ones((3, 6), np.complex128)
    want = pr.evaluate(x, 0.5, coef=coefs)
    s = hc.Stream(pr, slots=2, idle_us=20000)
    try:
        for after in (lambda: s.poll(s.submit(coef=coefs[0])), lambda: (small + 1).sum().item(),
                      lambda: pr.evaluate(x, 0.5, coef=coefs),
                      lambda: pr.track(n_instances=1, coef=coefs).wait()):
            with pytest.raises(hc.HCError):
                pr.track(n_instances=2 ** 31 - 1, coef=small, x_out=small, status_out=small,
                         steps_out=small, be_out=small, device=True)
            assert after() is not None
        got = pr.evaluate(x, 0.5, coef=coefs)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
    finally:
        s.close()
