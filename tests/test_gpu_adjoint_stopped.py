"""The adjoint from a state whose samples pd_run_to_peak stopped at different
steps: each sample goes on from its own displacements, velocities and damage at
sample 0's step index, bit for bit as from a state that was loaded with them."""
import dataclasses

import numpy as np
import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 6, 4), (16, 8, 1)])
def test_each_sample_from_its_own_content(built_lib, shape):
    pd = built_lib
    w = W.tiny_beam(*shape, n_steps=1500)
    w = dataclasses.replace(w, bc=dataclasses.replace(w.bc, u_max=3.0e-5))
    if shape[2] == 1:
        w = dataclasses.replace(w, grid=dataclasses.replace(w.grid, m_ratio=np.pi),
                                mat=dataclasses.replace(w.mat, model=W.MODEL_PLANE_STRESS, thickness=0.05))
    g, B = w.grid, 8
    scale = np.linspace(0.4, 1.1, B)[:, None]
    s0 = torch.tensor((W.lognormal_like_field(g.n_nodes, B, 3) * scale).astype(np.float32), device="cuda")
    row, col = pd.build_neighbours(g)
    st = pd.State(g, row, col, w.mat, w.bc, batch=B)
    st.reset(s0)
    nd = st.run_to_peak(w.n_steps)[2].cpu().numpy()
    assert len({int(n) & 1 for n in nd}) == 2, "the case needs stops of both parities"
    at = st.store()
    obs, wts = [2, 6], torch.tensor(np.random.default_rng(2).standard_normal((B, 2)), device="cuda")
    got = st.adjoint(9, obs, wts, s0, None, ckpt_every=4)
    after = st.store()
    st.reset(s0)
    st.load(*at, step=int(nd[0]))
    want = st.adjoint(9, obs, wts, s0, None, ckpt_every=4)
    for a, b in zip(got + after, want + st.store()):
        assert torch.equal(a, b)
    assert all(want[1][b].abs().max() > 0 for b in range(B))
    st.close()
