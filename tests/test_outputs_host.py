"""The output tensors of a call are ordinary views (no device needed)."""
import types

import pytest
import torch

import paper_2504_17987_gb300 as rp


@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("k", [0, 1, 2])
def test_outputs_take_in_place_work_of_a_graph(n, k):
    grid = types.SimpleNamespace(nx=5, ny=4, _dev=torch.device("cpu"))
    x = torch.ones(4, 5, requires_grad=True)
    out = rp.Engine.empty_outputs(grid, n)[k]
    out.zero_()
    out.add_(x)
    out.sum().backward()
    assert torch.equal(x.grad, torch.full((4, 5), float(n)))
