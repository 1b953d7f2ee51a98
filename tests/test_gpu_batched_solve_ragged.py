"""Batches of the batched solve whose last block is ragged: what lies past the
end costs next to nothing, and the systems before it keep their bits, residuals
and singularity marks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_03444_gb300 import hc
    return torch, hc


def _per_block(n):
    """Systems of a block of 128 threads with one row per lane."""
    return 128 // (4 if n <= 4 else 8 if n <= 8 else 16 if n <= 16 else 32)


def _systems(torch, n, batch, dtype):
    g = torch.Generator(device="cuda").manual_seed(100 * n + batch)
    A = torch.randn((batch, n, n), dtype=dtype, device="cuda", generator=g)
    b = torch.randn((batch, n), dtype=dtype, device="cuda", generator=g)
    return A, b, torch.zeros_like(b), torch.full((batch,), 7, dtype=torch.int32, device="cuda")


def _device_us(env, n, batch, dtype):
    """Device time of one call: the least of 9 replays of 20 captured calls."""
    torch, hc = env
    A, b, x, info = _systems(torch, n, batch, dtype)
    assert hc.batched_solve(A, b, x, info) == hc.HC_OK
    torch.cuda.synchronize()
    graph, best = torch.cuda.CUDAGraph(), float("inf")
    with torch.cuda.graph(graph):
        st = torch.cuda.current_stream().cuda_stream
        for _ in range(20):
            assert hc.batched_solve(A, b, x, info, st) == hc.HC_OK
    for _ in range(9):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) * 50.0)
    return best


@pytest.mark.parametrize("n", [9, 13, 16, 20])
def test_one_system_more_than_a_block_per_sm(env, n):
    """One SM gets a second block with one system, a quarter of a block's warps:
    at most a quarter more of the FP64 pipe's time, and some latency.  (All of
    the block's groups eliminating would take half to three quarters more.)"""
    torch, _ = env
    full = _per_block(n) * torch.cuda.get_device_properties(0).multi_processor_count
    t0 = _device_us(env, n, full, torch.complex128)
    t1 = _device_us(env, n, full + 1, torch.complex128)
    assert t1 <= 1.45 * t0, (t0, t1)


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 9, 13, 16, 17, 24, 31, 32])
def test_ragged_last_block(env, n, dtype):
    torch, hc = env
    dt = getattr(torch, dtype)
    G = _per_block(n)
    A, b, x, info = _systems(torch, n, 3 * G, dt)
    A[0, :, n - 1] = 0.0  # a zero column: an exact zero pivot
    assert hc.batched_solve(A, b, x, info) == hc.HC_OK
    for batch in sorted({1, 2, G - 1, G, G + 1, 2 * G - 1, 2 * G + 1}):
        if batch < 1:
            continue
        part = slice(0, batch)
        xs = torch.zeros_like(b[part])
        infos = torch.full((batch + 1,), 7, dtype=torch.int32, device="cuda")
        assert hc.batched_solve(A[part], b[part], xs, infos) == hc.HC_OK
        torch.cuda.synchronize()
        assert int(infos[batch]) == 7  # nothing is written behind the batch
        assert torch.equal(infos[:batch], info[part]), batch
        same = xs[1:].cpu().numpy().view(np.uint8) == x[1:batch].cpu().numpy().view(np.uint8)
        assert same.all(), batch
    assert int(info[0]) == 1 and int(info[1:].abs().sum()) == 0
    # forward error of a backward stable elimination
    wide = torch.complex128
    A64, b64 = A[1:].to(wide).cpu().numpy(), b[1:].to(wide).cpu().numpy()
    want = np.linalg.solve(A64, b64[..., None])[..., 0]
    err = np.abs(x[1:].to(wide).cpu().numpy() - want).max(1) / np.abs(want).max(1)
    u = 2.0 ** -24 if dtype == "complex64" else 2.0 ** -53
    assert (err <= 64 * n * np.linalg.cond(A64) * u).all()


@pytest.mark.parametrize("n", [8, 13, 16])
def test_one_fp32_system_is_no_slower_than_two(env, n):
    """One system has no company to keep in step with: the maximum over its own
    lanes, not the butterfly that the groups of a warp share."""
    torch, _ = env
    t1 = _device_us(env, n, 1, torch.complex64)
    t2 = _device_us(env, n, 2, torch.complex64)
    assert t1 <= 0.97 * t2, (t1, t2)


@pytest.mark.parametrize("n", [20, 24])
def test_six_rounds_of_blocks(env, n):
    """Six blocks per SM, three with two rows per lane (of which some SM would get
    four): half again as long as four blocks per SM, and a fifth for the rounds."""
    torch, _ = env
    per_round = _per_block(n) * torch.cuda.get_device_properties(0).multi_processor_count
    t4 = _device_us(env, n, 4 * per_round, torch.complex128)
    t6 = _device_us(env, n, 6 * per_round, torch.complex128)
    assert t6 <= 1.8 * t4, (t4, t6)


@pytest.mark.parametrize("n", [2, 4, 8, 12, 16, 20, 24])
def test_same_bits_on_both_sides_of_the_choice(env, n):
    """Batches of 1 to 9 rounds take one row per lane or several: the same bits."""
    torch, hc = env
    per_round = _per_block(n) * torch.cuda.get_device_properties(0).multi_processor_count
    A, b, x, info = _systems(torch, n, 9 * per_round, torch.complex128)
    assert hc.batched_solve(A, b, x, info) == hc.HC_OK
    for batch in [per_round * r + k for r in range(1, 9) for k in (-1, 0, 1, per_round // 2)]:
        xs = torch.zeros_like(b[:batch])
        infos = torch.full((batch,), 7, dtype=torch.int32, device="cuda")
        assert hc.batched_solve(A[:batch], b[:batch], xs, infos) == hc.HC_OK
        assert torch.equal(torch.view_as_real(xs), torch.view_as_real(x[:batch])), batch
        assert torch.equal(infos, info[:batch]), batch
