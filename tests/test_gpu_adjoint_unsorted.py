"""The adjoint of mixed states on the compile-time stencil whose neighbour lists
have rows in another order (which keep the general adjoint) against the same
run with ascending rows.

Tolerance: the forward run and its branches are the same bits (the step does not
read the list's order); the gradients' FP32 terms are summed in another order,
8 at a time: 1e-4 of the largest, as between the two precisions."""
import numpy as np
import pytest
import torch

import pd_workloads as W
from test_gpu_adjoint_wide import TOP, _gradients

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), device="cuda")


def _close(a, b):
    return bool((a - b).abs().max() <= 1e-4 * b.abs().max())


@pytest.mark.parametrize("shape,sched", [((16, 6, 4), None), ((13, 7, 5), (4, 2, 2)), ((9, 11, 13), (4, 4, 1))])
def test_shuffled_rows(built_lib, shape, sched):
    pd = built_lib
    w = W.tiny_beam(*shape)
    g, B, T = w.grid, 2, 9
    row, col = pd.build_neighbours(g)
    rp, c = row.cpu().numpy(), col.cpu().numpy().copy()
    d = W.pair_damage(np.repeat(np.arange(g.n_nodes), np.diff(rp)), c, 5, B).astype(np.float32).astype(np.float64)
    perm, rng = np.arange(len(c)), np.random.default_rng(4)
    for i in range(g.n_nodes):
        rng.shuffle(perm[rp[i]:rp[i + 1]])
    u, v = W.random_state(g.n_nodes, B, 9, u_scale=1e-7)
    s0, kap = _dev(W.lognormal_like_field(g.n_nodes, B, 3)), _dev(W.lognormal_like_field(g.n_nodes, B, 4, mean=1.0))
    wts = _dev(np.random.default_rng(1).standard_normal((B, 2)))
    out = []
    for cc, dd in ((col, d), (_dev(c[perm]), d[:, perm])):
        st = pd.State(g, row, cc, w.mat, w.bc, batch=B, schedule=sched)
        st.reset(s0, kap)
        st.load(_dev(u), _dev(v), _dev(dd), step=3)
        out.append(st.adjoint(T, [4, 8], wts, s0, kap, ckpt_every=4))
        st.close()
    (gs, gk, R), (fs, fk, fR) = out
    assert torch.equal(R, fR) and gs.abs().max() > 0
    for b in range(B):
        assert _close(fs[b], gs[b]) and _close(fk[b], gk[b])


def test_words_past_31_bits(built_lib):
    """Rows in descending order, more than 2^31 damage words (test_gpu_adjoint_wide.py)."""
    big, small = _gradients(built_lib, 1032, 1040, descending=True), _gradients(built_lib, 1032, 40)
    assert small[0].shape == (2, TOP, 1032)
    for a, b in zip(big, small):
        assert _close(a, b)
    torch.cuda.empty_cache()
