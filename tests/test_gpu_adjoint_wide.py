"""The adjoint of a state whose damage words do not fit 31 or 32 bits: flat bodies
in bricks that reach far past them (8 x 2 x 16 of a body two nodes thick), so a
few million nodes have more than 2^31, or 2^32, words a sample. The load line
lies along the last rows, whose words come last. Its surroundings do not feel
the other end within the steps taken, so a short body with the same end has the
same gradients there, bit for bit."""
import dataclasses

import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu

TOP = 30  # rows compared (6 steps reach 18 rows from the load line)


def _gradients(pd, nx, ny, descending=False):
    w = W.tiny_beam(nx, ny, 2, notch=False)
    w = dataclasses.replace(w, mat=dataclasses.replace(w.mat, s_ratio=1e4))
    g = w.grid
    row, col = pd.build_neighbours(g)
    if descending:
        r = row.long()
        col = col[torch.repeat_interleave(r[:-1] + r[1:] - 1, r.diff()) - torch.arange(col.numel(), device="cuda")]
    st = pd.State(g, row, col, w.mat, w.bc, batch=1, schedule=(2, 16, 1))
    del row, col
    s0 = torch.full((1, g.n_nodes), 1e-7, device="cuda")
    st.reset(s0)
    wts = torch.ones((1, 2), dtype=torch.float64, device="cuda")
    gs, gk, R = st.adjoint(6, [3, 5], wts, s0, None, ckpt_every=6)
    st.close()
    top = lambda a: a.view(2, ny, nx)[:, -TOP:].cpu()
    return top(gs), top(gk), R.cpu()


@pytest.mark.parametrize("nx,ny,bits", [(1032, 1040, 31), (2040, 1040, 32)])
def test_words_past_31_and_32_bits(built_lib, nx, ny, bits):
    words = nx * ny * 16 * 128
    last = nx * (ny - 10) * 16 * 128  # where the tenth row from the end begins
    assert words < 2 ** (bits + 1) and last > 2 ** bits and torch.cuda.mem_get_info()[0] > 20 * words
    big, small = _gradients(built_lib, nx, ny), _gradients(built_lib, nx, 40)
    assert small[0].abs().max() > 0 and small[0][:, -3:].abs().max() > 0
    for a, b in zip(big[:2], small[:2]):
        assert torch.equal(a, b)
    assert torch.allclose(big[2], small[2], rtol=1e-12, atol=0.0)
    torch.cuda.empty_cache()
