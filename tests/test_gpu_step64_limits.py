"""The FP64 step at the ends of the bond law, against the oracle: elastic limits
of zero and below the normal range, both laws, with the critical stretch from
the ratio and from the fracture energy; and bonds compressed to a small part of
their length.

Tolerance: the damage law's slope is at most k / (s_c - s0) = 25 / 0.025 (nodes
of 0 and 0.05, ratio 2) on stretches off by at most 10 x 2^-53, so damage agrees
to 1.2e-12: 2e-12. That error enters the force of each of a node's at most 122
bonds, none of them more than a fifth of the largest node force: 3e-11."""
import dataclasses

import numpy as np
import pytest
import torch

import pd_workloads as W
from oracle import core

pytestmark = pytest.mark.gpu


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("least", [0.0, 3e-310])
@pytest.mark.parametrize("G_F", [0.0, 5e6])
@pytest.mark.parametrize("law", [W.LAW_BILINEAR, W.LAW_EXPLINEAR])
def test_elastic_limit_of_zero(built_lib, law, G_F, least):
    """Half of the nodes without an elastic limit: bonds between two of them soften under any tension (G_F: the
    critical stretch is infinite, and the exponential law breaks them)."""
    pd = built_lib
    w = W.tiny_beam()
    g = W.Grid(13, 7, 5, 2.5e-3, 3.01)
    w = dataclasses.replace(w, grid=g, mat=dataclasses.replace(w.mat, law=law, s_ratio=2.0, G_F=G_F),
                            bc=dataclasses.replace(w.bc, support_x2=(1, 2 * g.nx - 1), load_x2=g.nx))
    rng = np.random.default_rng(17)
    u = rng.normal(0.0, 0.1 * g.dx, (1, g.n_nodes, 3))
    s0 = np.where(rng.random((1, g.n_nodes)) < 0.5, least, rng.uniform(0.05, 0.15, (1, g.n_nodes)))
    orow, ocol = core.neighbours(g)
    row, col = pd.build_neighbours(g)
    st = pd.State(g, row, col, w.mat, w.bc, batch=1, precision=pd.PREC_FP64)
    st.reset_f64(_dev(s0))
    st.load(_dev(u), _dev(np.zeros_like(u)), None, step=0)
    F, d = st.force().cpu().numpy()[0], st.store()[2].cpu().numpy()[0]
    st.close()
    Fo, do, _ = core.Model(w, orow, ocol, s0=s0[0]).force(u[0], np.zeros(len(ocol)))
    i = np.repeat(np.arange(g.n_nodes), np.diff(orow))
    both = (s0[0][i] == least) & (s0[0][ocol] == least)
    assert both.sum() > 100 and ((do > 0) & (do < 1)).any()
    if law == W.LAW_EXPLINEAR or G_F == 0.0:
        assert (do[both] == 1.0).sum() > 100
    assert np.abs(d - do).max() <= 2e-12
    assert np.abs(F - Fo).max() <= 3e-11 * np.abs(Fo).max()


@pytest.mark.parametrize("shrink", [0.5, 2.0 ** -4, 2.0 ** -10, 2.0 ** -30])
def test_compressed_bonds(built_lib, shrink):
    """A body shrunk to `shrink` of its size, its nodes a tenth of the shrunk spacing off. Positions, displacements and
    their differences are exact (multiples of 2^-56 below 2^-4), so both sides hold the same bond vectors and a bond
    force is at most 20 roundings off: 20 x 122 x 2^-53 of the largest, below 1e-12."""
    pd = built_lib
    w = W.tiny_beam()
    g = W.Grid(9, 6, 5, 2.0 ** -9, 3.01)
    w = dataclasses.replace(w, grid=g, bc=dataclasses.replace(w.bc, support_x2=(1, 2 * g.nx - 1), load_x2=g.nx))
    n = np.arange(g.n_nodes)
    X = (np.stack([n % g.nx, n // g.nx % g.ny, n // (g.nx * g.ny)], 1) + 0.5) * g.dx
    noise = np.random.default_rng(3).uniform(-0.1, 0.1, X.shape) * shrink * g.dx
    u = (shrink - 1.0) * X + np.rint(noise * 2.0 ** 56) * 2.0 ** -56
    orow, ocol = core.neighbours(g)
    i = np.repeat(n, np.diff(orow))
    eta = u[ocol] - u[i]
    assert np.array_equal(u[i] + eta, u[ocol]) and np.array_equal(X[ocol] - X[i] + eta - eta, X[ocol] - X[i])
    row, col = pd.build_neighbours(g)
    st = pd.State(g, row, col, w.mat, w.bc, batch=1, precision=pd.PREC_FP64)
    st.reset(torch.full((1, g.n_nodes), 1e-4, device="cuda"))
    st.load(_dev(u[None]), _dev(np.zeros_like(u[None])), None, step=0)
    F = st.force().cpu().numpy()[0]
    st.close()
    Fo, do, _ = core.Model(w, orow, ocol).force(u, np.zeros(len(ocol)))
    assert not do.any() and np.isfinite(Fo).all()
    assert np.abs(F - Fo).max() <= 1e-12 * np.abs(Fo).max()


def test_bonds_of_undefined_damage_carry_no_force(built_lib):
    """Damage that is not a number, of either sign, is not below 1: such a bond counts as broken, as in the oracle."""
    pd = built_lib
    w = W.tiny_beam()
    g = w.grid
    orow, ocol = core.neighbours(g)
    rng = np.random.default_rng(6)
    d = np.where(rng.random(len(ocol)) < 0.2, rng.random(len(ocol)), 0.0)
    d[::5], d[1::7], d[2::9] = np.nan, -np.float64(np.nan), 1.0
    assert np.signbit(d).any() and np.isnan(d[0]) and not np.signbit(d[0])
    u, _ = W.random_state(g.n_nodes, 1, 9)
    row, col = pd.build_neighbours(g)
    st = pd.State(g, row, col, w.mat, w.bc, batch=1, precision=pd.PREC_FP64)
    st.reset(torch.full((1, g.n_nodes), 1e-4, device="cuda"))
    st.load(_dev(u), _dev(np.zeros_like(u)), _dev(d[None]), step=0)
    F = st.force().cpu().numpy()[0]
    st.close()
    Fo, _, _ = core.Model(w, orow, ocol).force(u[0], d.copy())
    assert np.isfinite(Fo).all() and np.abs(Fo).max() > 0
    assert np.abs(F - Fo).max() <= 1e-10 * np.abs(Fo).max()  # (stretches of 1e-5: the oracle's (|y| - |xi|) / |xi| cancels)
