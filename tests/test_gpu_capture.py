"""Calls while a stream is being captured into a CUDA graph, and from several streams at once."""
from concurrent.futures import ThreadPoolExecutor

import pytest
import torch

import graphgen
import paper_2105_07298_gb300 as apsp

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_one_shot_batches_refuse_graph_capture():
    """Also through the packed autograd function; nothing is enqueued and the capture goes on."""
    sizes = [5, 8]
    W = torch.ones(64 + 28, device=DEV)
    apsp.apsp_fw_batched(W.clone(), sizes)  # the kernels are loaded
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(apsp.ApspError):
            apsp.apsp_fw_batched(W, sizes)
        with pytest.raises(apsp.ApspError):
            apsp.shortest_path_distances_packed(W, sizes)
        out = W + 1
    g.replay()
    torch.cuda.synchronize()
    assert bool((out == 2).all()) and bool((W == 1).all())


def _weights(n, lo, dtype):
    """Integers (few outputs improve late), or reals down to `lo` = 0, which keep improving: the
    probes then leave screens out, and take samples."""
    W = graphgen.dense_graph(n, 0.1, 21) if lo else graphgen.dense_graph(n, 0.4, 28, weights="real", lo=0.0, hi=1.0)
    return torch.from_numpy(W).to(DEV, dtype)


# Past the first size whose later rounds are screened, with a ragged last block.
SCREENED = [(2900, torch.float32), (4000, torch.float64)]


@pytest.mark.parametrize("n,dtype", SCREENED)
@pytest.mark.parametrize("lo", [1, 0])
def test_screened_solve_captured_in_cuda_graph(n, dtype, lo):
    """One stream, all blocks of phase 4 in one launch, lists and probes of these; replayed
    on restored inputs, bit for bit the direct call."""
    W = _weights(n, lo, dtype)
    Dd, Pd = W.clone(), torch.empty((n, n), dtype=torch.int32, device=DEV)
    apsp.apsp_fw(Dd, Pd)
    D, P = W.clone(), torch.empty_like(Pd)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        apsp.apsp_fw(D, P)
    for _ in range(2):
        D.copy_(W)
        P.fill_(77)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(D, Dd) and torch.equal(P, Pd)
    assert apsp.device_status() == apsp.APSP_OK


@pytest.mark.parametrize("n,dtype", SCREENED)
def test_solves_on_two_streams_at_once(n, dtype):
    """Each with its own scratch from the one pool, again and again, from two host threads."""
    cases = []
    for lo in (1, 0):
        W = _weights(n, lo, dtype)
        Dd, Pd = W.clone(), torch.empty((n, n), dtype=torch.int32, device=DEV)
        apsp.apsp_fw(Dd, Pd)
        cases.append((W, Dd, Pd, torch.cuda.Stream()))
    torch.cuda.synchronize()

    def solve(case):
        W, Dd, Pd, s = case
        same = True
        with torch.cuda.stream(s):
            for _ in range(3):
                D, P = W.clone(), torch.full_like(Pd, 77)
                apsp.apsp_fw(D, P)
                same = same and torch.equal(D, Dd) and torch.equal(P, Pd)
        return same

    with ThreadPoolExecutor(2) as pool:
        assert list(pool.map(solve, cases)) == [True, True]
    assert apsp.device_status() == apsp.APSP_OK
