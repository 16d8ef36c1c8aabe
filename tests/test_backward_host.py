"""Host logic of the autograd wrapper, without a GPU."""
import pytest
import torch

import paper_2105_07298_gb300 as apsp
from paper_2105_07298_gb300 import backward


def test_stacked_solve_refuses_graph_capture(monkeypatch):
    """Its work list is uploaded from memory of the call, which a replay would not find."""
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    for n in (8, 7):  # in place, and through the aligned copy
        with pytest.raises(apsp.ApspError):
            backward._solve_stack(torch.zeros(2, n, n), torch.zeros(2, n, n, dtype=torch.int32))
