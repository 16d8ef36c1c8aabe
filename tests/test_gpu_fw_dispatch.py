"""The single-graph kernels at the sizes where their dispatch changes or a tile
is ragged, bit for bit against the oracle's blocked FW at the library's block
size on real weights (one rounded sum per candidate, ascending k)."""
import numpy as np
import pytest
import torch

import graphgen
import oracle
import paper_2105_07298_gb300 as apsp
from paper_2105_07298_gb300 import batched

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _expect(n, p, seed, dtype=np.float32):
    W = graphgen.dense_graph(n, p, seed, weights="real", lo=0.5, hi=2.0, dtype=dtype)
    return W, *oracle.bfw(W, 128)


# One quad of the diagonal block; a block less one; two blocks, the last one
# vertex wide; the last size with two lines a warp in the panels and the first
# with four; the first past the 32-row pieces; one well past it.
@pytest.mark.parametrize("n", [1, 3, 5, 127, 129, 258, 2305, 2433, 2689, 5121])
def test_real_weights_bitwise_at_dispatch_limits(n):
    W, Db, Pb = _expect(n, 0.3 if n < 300 else 0.05, 900 + n)
    D, P = torch.from_numpy(W).to(DEV), torch.full((n, n), 77, dtype=torch.int32, device=DEV)
    apsp.apsp_fw(D, P)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    np.testing.assert_array_equal(P.cpu().numpy(), Pb)
    D = torch.from_numpy(W).to(DEV)
    apsp.apsp_fw(D)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    assert apsp.device_status() == apsp.APSP_OK


# The same edges in FP64; the first size with four phase-4 CTAs per SM.
@pytest.mark.parametrize("n", [1, 3, 5, 127, 129, 258, 3073])
def test_real_weights_f64_bitwise_at_dispatch_limits(n):
    W, Db, Pb = _expect(n, 0.3 if n < 300 else 0.05, 700 + n, np.float64)
    assert apsp.block_size(torch.float64) == 128
    D, P = torch.from_numpy(W).to(DEV), torch.full((n, n), 77, dtype=torch.int32, device=DEV)
    apsp.apsp_fw(D, P)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    np.testing.assert_array_equal(P.cpu().numpy(), Pb)
    D = torch.from_numpy(W).to(DEV)
    apsp.apsp_fw(D)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    assert apsp.device_status() == apsp.APSP_OK


def test_f64_sums_within_a_float_step():
    """Weights 1 + j 2^-40 + i 2^-52: every sum shares one float, so candidates can
    only be told apart in FP64, and many tie exactly (the first k wins)."""
    n = 200
    rng = np.random.default_rng(4)
    W = 1.0 + rng.integers(0, 3, (n, n)) * 2.0 ** -40 + rng.integers(0, 3, (n, n)) * 2.0 ** -52
    W[rng.random((n, n)) >= 0.1] = np.inf
    np.fill_diagonal(W, 0)
    Db, Pb = oracle.bfw(W, 128)
    D, P = torch.from_numpy(W).to(DEV), torch.empty((n, n), dtype=torch.int32, device=DEV)
    apsp.apsp_fw(D, P)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    np.testing.assert_array_equal(P.cpu().numpy(), Pb)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("ld,d_off,p_off", [(263, 0, 0), (264, 1, 0), (264, 0, 1), (264, 3, 2)])
def test_unaligned_rows_and_buffers(ld, d_off, p_off, dtype):
    """Odd leading dimensions and buffers that start off a 16-byte boundary, D
    and P apart; the columns past n stay as they are."""
    n = 261
    W, Db, Pb = _expect(n, 0.3, 5, np.float32 if dtype == torch.float32 else np.float64)
    dbuf = torch.full((n * ld + 4,), -3.0, dtype=dtype, device=DEV)
    pbuf = torch.full((n * ld + 4,), -9, dtype=torch.int32, device=DEV)
    D = dbuf[d_off:d_off + n * ld].view(n, ld)
    P = pbuf[p_off:p_off + n * ld].view(n, ld)
    D[:, :n].copy_(torch.from_numpy(W))
    apsp.apsp_fw(D[:, :n], P[:, :n])
    np.testing.assert_array_equal(D[:, :n].cpu().numpy(), Db)
    np.testing.assert_array_equal(P[:, :n].cpu().numpy(), Pb)
    assert bool((D[:, n:] == -3.0).all()) and bool((P[:, n:] == -9).all())


@pytest.mark.parametrize("with_path", [True, False])
@pytest.mark.parametrize("d_off", [0, 1])
def test_batched_blocks_at_quad_and_tile_edges(d_off, with_path):
    """Batched sizes around the quads of the closure, the eight rows of a warp
    and the 64-blocks, even and odd, from a buffer on and off an 8-byte boundary."""
    sizes = [1, 2, 3, 4, 5, 8, 9, 31, 33, 63, 64, 65, 66, 72, 73, 127, 128, 129, 130, 194]
    off = batched.packed_offsets(sizes)
    mats = [graphgen.dense_graph(n, 0.3, 40 + n) for n in sizes]
    total = batched.packed_numel(sizes)
    buf = torch.zeros(total + 1, device=DEV)[d_off:d_off + total]
    for m, n, o in zip(mats, sizes, off):
        buf[int(o):int(o) + n * n] = torch.from_numpy(m.reshape(-1)).to(DEV)
    P = torch.full((total,), -7, dtype=torch.int32, device=DEV) if with_path else None
    apsp.apsp_fw_batched(buf, sizes, off, P)
    for m, n, o in zip(mats, sizes, off):
        D = buf[int(o):int(o) + n * n].view(n, n).cpu().numpy()
        np.testing.assert_array_equal(D, oracle.fw(m)[0])
        if with_path:
            assert oracle.check_paths(m, D, P[int(o):int(o) + n * n].view(n, n).cpu().numpy()) == 0


def _screened_graph(kind, n):
    """Weights for the screened rounds (FP32: from 22 blocks a side and round 8 on; FP64: 32, 16)."""
    rng = np.random.default_rng(3)
    if kind == "integers":
        return graphgen.dense_graph(n, 0.1, 21)
    if kind == "halves":
        return graphgen.dense_graph(n, 0.1, 22) * np.float32(0.5)
    if kind == "beyond 2^22":  # integers, but not all of them below 2^22
        return graphgen.dense_graph(n, 0.02, 23, lo=1, hi=9_000_000)
    if kind == "sparse":  # most pairs far apart, some unreachable; diagonal blocks nearly empty
        return graphgen.dense_graph(n, 0.001, 24, weights="real", lo=0.5, hi=2.0)
    if kind == "no edges":
        return graphgen.dense_graph(n, 0.0, 25)
    if kind == "most improve":  # rounds between two probes go without the screen
        return graphgen.dense_graph(n, 0.4, 28, weights="real", lo=0.0, hi=1.0)
    W = graphgen.dense_graph(n, 0.05, 26, weights="real", lo=0.5, hi=2.0)
    if kind == "negative":  # shifted by potentials: negative edges, no negative cycle but by rounding
        h = rng.integers(-64, 65, n).astype(np.float32)
        W = graphgen.dense_graph(n, 0.05, 26, lo=1, hi=100) + h[:, None] - h[None, :]
    if kind == "clusters":  # distances within a cluster near 1e-3, between clusters near 1e6
        c = np.arange(n) % 3
        W = np.where(c[:, None] == c[None, :], W * np.float32(1e-3), W + np.float32(1e6)).astype(np.float32)
    if kind == "huge":  # far above the diagonal blocks' spread: in its units the weights overflow
        c = np.arange(n) // 128
        near = rng.uniform(0.005, 0.02, (n, n)).astype(np.float32)
        far = graphgen.dense_graph(n, 1e-4, 27, weights="real", lo=0.5, hi=2.0) * np.float32(5e37)
        W = np.where(c[:, None] == c[None, :], near, far)
    np.fill_diagonal(W, 0)
    return W


@pytest.mark.parametrize("kind", ["integers", "halves", "beyond 2^22", "sparse", "no edges", "real", "negative",
                                  "clusters", "huge", "most improve"])
def test_screened_rounds_bitwise(kind):
    n = 2900
    W = _screened_graph(kind, n)
    Db, Pb = oracle.bfw(W, 128)
    ld = n + 1 if kind in ("real", "integers") else n  # rows off 16-byte boundaries too
    D = torch.empty((n, ld), device=DEV)[:, :n]
    P = torch.empty((n, ld), dtype=torch.int32, device=DEV)[:, :n]
    D.copy_(torch.from_numpy(W))
    apsp.apsp_fw(D, P)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    np.testing.assert_array_equal(P.cpu().numpy(), Pb)
    D.copy_(torch.from_numpy(W))
    apsp.apsp_fw(D)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    assert apsp.device_status() == apsp.APSP_OK


def _screened_graph_f64(kind, n):
    rng = np.random.default_rng(5)
    if kind == "real":
        return graphgen.dense_graph(n, 0.05, 31, weights="real", lo=0.5, hi=2.0, dtype=np.float64)
    if kind == "one float":  # all sums within a float step of each other
        W = 1.0 + rng.integers(0, 3, (n, n)) * 2.0 ** -40 + rng.integers(0, 3, (n, n)) * 2.0 ** -52
        W[rng.random((n, n)) >= 0.05] = np.inf
    elif kind == "beyond the floats":  # edges of either sign, exact sums
        h = rng.integers(-64, 65, n) * 2.0 ** 1000
        W = graphgen.dense_graph(n, 0.02, 32, lo=1, hi=100).astype(np.float64) * 2.0 ** 1000 + h[:, None] - h[None, :]
    else:
        return _screened_graph(kind, n).astype(np.float64)
    np.fill_diagonal(W, 0)
    return W


@pytest.mark.parametrize("kind", ["real", "one float", "beyond the floats", "integers", "beyond 2^22", "sparse",
                                  "negative", "clusters", "huge", "most improve"])
def test_screened_rounds_f64_bitwise(kind):
    n = 4000
    W = _screened_graph_f64(kind, n)
    Db, Pb = oracle.bfw(W, 128)
    ld = n + 1 if kind in ("real", "integers") else n  # rows off 16-byte boundaries too
    D = torch.empty((n, ld), device=DEV, dtype=torch.float64)[:, :n]
    P = torch.empty((n, ld), dtype=torch.int32, device=DEV)[:, :n]
    D.copy_(torch.from_numpy(W))
    apsp.apsp_fw(D, P)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    np.testing.assert_array_equal(P.cpu().numpy(), Pb)
    D.copy_(torch.from_numpy(W))
    apsp.apsp_fw(D)
    np.testing.assert_array_equal(D.cpu().numpy(), Db)
    assert apsp.device_status() == apsp.APSP_OK


def test_bounded_wait_ends_within_seconds():
    """As many polls as the kernels' waits for their copies make (csrc/bulk.cuh): a wait that runs
    out must not hold the GPU for long."""
    apsp.wait_timeout_selftest(1 << 10)
    assert apsp.device_status() == apsp.APSP_ETIMEOUT
    t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    t0.record()
    apsp.wait_timeout_selftest(1 << 18)
    t1.record()
    assert apsp.device_status() == apsp.APSP_ETIMEOUT
    assert t0.elapsed_time(t1) < 3000.0
