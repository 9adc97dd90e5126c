"""The chain rule to the KL coefficients on a grid whose blocks take several tiles
of nodes (the last one fewer) and a batch taken in groups of samples: values, a
sample's independence of its batch, and the scratch, which stays at 64 MB (one
partial sum per tile, mode and sample would be 230 MB here).

Tolerance: as in test_gpu_field_grad.py (FP32 basis, lognormal marginal)."""
import numpy as np
import pytest
import torch

import pd_workloads as W
from oracle import field

pytestmark = pytest.mark.gpu


def test_many_tiles_and_samples_in_bounded_scratch(built_lib):
    pd = built_lib
    K, B = 256, 100
    g = W.Grid(40, 30, 30, 2.5e-3, 3.01)  # 36,000 nodes: 1,125 tiles of 32
    cfg = W.FieldCfg(W.COV_SQEXP, 5e-3, K, 0, 1e-4, 0.1)
    rng = np.random.default_rng(8)
    xi, dj = rng.standard_normal((B, K)), rng.standard_normal((B, g.n_nodes)) * 1e6
    xd, dd = torch.tensor(xi, device="cuda"), torch.tensor(dj, device="cuda")
    fld = pd.Field(g, 1, cfg)
    some = {b: fld.adjoint(0, xd[b:b + 1], dd[b:b + 1]) for b in (0, 47, 48, 99)}
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.empty(torch.cuda.mem_get_info()[0] - (150 << 20), dtype=torch.uint8, device="cuda")
    got = fld.adjoint(0, xd, dd)
    del room
    torch.cuda.empty_cache()
    for b, v in some.items():
        assert torch.equal(got[b:b + 1], v)
    fld.close()
    Phi, lam = field.kl_separable(g, cfg.length, K)
    psi = Phi * np.sqrt(np.maximum(lam, 0.0))
    s2 = np.log(1.01)
    w = dj * np.sqrt(s2) * 1e-4 * np.exp(-0.5 * s2 + np.sqrt(s2) * (xi @ psi.T))
    tol = 2.0 ** -24 * (1 + 0.0998 * np.linalg.norm(xi, axis=1))[:, None] * (np.abs(w) @ np.abs(psi))
    assert np.all(np.abs(got.cpu().numpy() - w @ psi) <= tol + 1e-12 * np.abs(w) @ np.abs(psi))
