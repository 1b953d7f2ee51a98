"""The batched solve takes several rows per lane for double-precision batches
that fill the chip and one row per lane below: the same operations per entry, so
a system's solution has the same bits in a small batch and in a large one, whose
last block is ragged; singular systems are marked in both."""
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


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 12, 13, 16, 17, 20, 24, 25, 32])
def test_rows_per_lane_same_bits(hc, n):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lanes = 4 if n <= 4 else 8 if n <= 8 else 16 if n <= 16 else 32
    big = 16 * sms * (32 // lanes) + 3
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((big, n, n), dtype=torch.complex128, device="cuda", generator=g)
    b = torch.randn((big, n), dtype=torch.complex128, device="cuda", generator=g)
    A[4] = 0.0          # singular
    if n > 1:
        A[big - 2, -1] = A[big - 2, 0]
        A[6] = torch.diag(torch.arange(1, n + 1, device="cuda").to(torch.complex128)).flip(0)
    x = torch.empty_like(b)
    info = torch.full((big,), 7, dtype=torch.int32, device="cuda")
    assert hc.batched_solve(A, b, x, info) == 0
    for part in (slice(0, 9), slice(big - 5, big)):
        xs = torch.empty_like(b[part])
        infos = torch.full((xs.shape[0],), 7, dtype=torch.int32, device="cuda")
        assert hc.batched_solve(A[part].contiguous(), b[part].contiguous(), xs, infos) == 0
        torch.cuda.synchronize()
        assert torch.equal(infos, info[part])
        assert np.array_equal(xs.cpu().numpy().view(np.uint8), x[part].cpu().numpy().view(np.uint8))
    assert int(info[4]) == 1
    ok = (info == 0)
    assert int((~ok).sum()) <= 2
    ref = torch.linalg.solve(A[ok].cpu()[:64], b[ok].cpu()[:64])
    got = x[ok].cpu()[:64]
    # backward stable: residual of the size of the rounding, n ulps of |A| |x|
    r = (torch.einsum("kij,kj->ki", A[ok].cpu()[:64], got) - b[ok].cpu()[:64]).abs().amax(1)
    s = (torch.einsum("kij,kj->ki", A[ok].cpu()[:64].abs(), got.abs())).amax(1)
    assert bool((r <= 64 * n * 2.3e-16 * s).all())
    assert got.shape == ref.shape
