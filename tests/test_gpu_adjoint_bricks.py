"""An adjoint whose checkpoints do not fit in whole bricks (a body two nodes thick
in bricks of 16 layers) but do in CSR order: the general adjoint takes it, with
the gradients of the run that had the room.

Tolerance: both sum a node's FP32 terms over its row in the same groups; 1e-4 of
the largest, as between the two precisions."""
import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu


def test_general_path_where_the_bricks_do_not_fit(built_lib):
    pd = built_lib
    w = W.tiny_beam(64, 64, 2)
    g, B, T = w.grid, 8, 6
    row, col = pd.build_neighbours(g)
    st = pd.State(g, row, col, w.mat, w.bc, batch=B, schedule=(2, 16, 1))
    s0 = torch.tensor(W.lognormal_like_field(g.n_nodes, B, 3), device="cuda") * 1e-3
    wts = torch.ones((B, 2), dtype=torch.float64, device="cuda")
    # four checkpoints of 8 x 64 x 64 x 16 x 128 words: 1.07 GB; in CSR order 0.14 GB, and 0.2 GB of trajectory
    st.reset(s0)
    want = st.adjoint(T, [3, 5], wts, s0, None, ckpt_every=2)
    shuffled = col.clone()
    shuffled[:2] = col[:2].flip(0)  # (loads the general path's kernels)
    other = pd.State(g, row, shuffled, w.mat, w.bc, batch=B, schedule=(2, 16, 1))
    other.reset(s0)
    other.adjoint(T, [3, 5], wts, s0, None, ckpt_every=2)
    other.close()
    st.reset(s0)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.empty(torch.cuda.mem_get_info()[0] - (700 << 20), dtype=torch.uint8, device="cuda")
    got = st.adjoint(T, [3, 5], wts, s0, None, ckpt_every=2)
    del room
    torch.cuda.empty_cache()
    after = st.store()
    st.reset(s0)
    st.step(T)
    assert all(torch.equal(a, b) for a, b in zip(after, st.store()))
    st.close()
    assert torch.equal(got[2], want[2]) and want[1].abs().max() > 0
    for a, b in zip(got[:2], want[:2]):
        assert (a - b).abs().max() <= 1e-4 * b.abs().max()
