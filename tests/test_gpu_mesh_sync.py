"""The neighbour list is complete when the call returns: built on one
non-blocking stream, read at once on another."""
import ctypes

import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["pd_build_neighbours", "pd_build_neighbours_noalloc"])
def test_list_is_complete_on_return(built_lib, entry):
    pd = built_lib
    g = W.Grid(140, 40, 40, 1e-3, 6.0)  # 224,000 nodes, a fill of some hundred us
    row, col = pd.build_neighbours(g)
    torch.cuda.synchronize()
    build, read = torch.cuda.Stream(), torch.cuda.Stream()
    G, nb = pd.grid_struct(g), ctypes.c_int64(0)
    for _ in range(3):
        r, c = torch.full_like(row, -1), torch.full_like(col, -1)
        torch.cuda.synchronize()
        rc = getattr(pd.lib(), entry)(ctypes.byref(G), pd._ptr(r), pd._ptr(c), c.numel(), ctypes.byref(nb), pd._stream(build))
        with torch.cuda.stream(read):
            tail = c[-1000000:].clone()  # (the rows written last)
            got, got_row = c.clone(), r.clone()
        torch.cuda.synchronize()
        assert rc == pd.PD_OK and nb.value == col.numel()
        assert torch.equal(tail, col[-1000000:]) and torch.equal(got, col) and torch.equal(got_row, row)
