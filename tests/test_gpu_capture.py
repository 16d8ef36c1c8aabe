"""Calls while a stream is being captured into a CUDA graph."""
import pytest
import torch

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
