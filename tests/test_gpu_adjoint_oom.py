"""An adjoint whose trajectory of growing damage does not fit (its size is known
only after the forward run) fails with PD_ERR_OOM and leaves the state as it
was: content, step, stopped samples."""
import dataclasses

import numpy as np
import pytest
import torch

import pd_workloads as W

pytestmark = pytest.mark.gpu


def test_state_is_as_before_when_the_trajectory_does_not_fit(built_lib):
    pd = built_lib
    w = W.tiny_beam(40, 16, 16)
    w = dataclasses.replace(w, mat=dataclasses.replace(w.mat, s_ratio=1e4))  # damage that goes on growing
    g, B, T = w.grid, 4, 64
    row, col = pd.build_neighbours(g)
    s0 = torch.full((B, g.n_nodes), 1e-7, device="cuda")
    v = torch.tensor(np.random.default_rng(5).normal(0.0, 1e-2, (B, g.n_nodes, 3)), device="cuda")
    wts = torch.ones((B, 1), dtype=torch.float64, device="cuda")
    st, twin = (pd.State(g, row, col, w.mat, w.bc, batch=B) for _ in range(2))
    for s in (st, twin):
        s.reset(s0)
        s.load(torch.zeros_like(v), v, None, step=0)
        s.run_to_peak(3)  # every sample is marked done at step 3
    d = st.store()[2]
    st.adjoint(T, [T - 1], wts, s0, None, ckpt_every=T)  # (fits; loads every kernel)
    grown = int((st.store()[2] > d).sum())
    del d
    # checkpoints, records and sums take less than 150 MB; 260 bytes a growing bond
    assert grown * 4 * T > 400 << 20
    st.reset(s0)
    st.load(torch.zeros_like(v), v, None, step=0)
    st.run_to_peak(3)
    before = st.store()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device="cuda")
    with pytest.raises(pd.PdError) as e:
        st.adjoint(T, [T - 1], wts, s0, None, ckpt_every=T)
    del room
    torch.cuda.empty_cache()
    assert e.value.code == pd.PD_ERR_OOM
    for a, b in zip(before, st.store()):
        assert torch.equal(a, b)
    st.step(2)  # stopped samples do not move
    for a, b in zip(before, st.store()):
        assert torch.equal(a, b)
    # and run on like a state that never met the failure
    for s in (st, twin):
        s.out = s.run_to_peak(40), s.adjoint(6, [5], wts, s0, None, ckpt_every=3), s.store()
    for a, b in zip(st.out, twin.out):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    st.close()
    twin.close()
