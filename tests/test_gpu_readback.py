"""Read-back of rho, u, the state and the diagnostic sums against numpy sums of the state that was
set: deviations spanning many decades inside a node, FP32 subnormals and zeros, odd sizes, all
lattices and both precisions.  The bound on a sum of Q deviations is a few units of 2^-53 of
Q max |g| (FP64 rounding of the sum and of its division by rho)."""
import numpy as np
import pytest

import workloads as W
from oracle.lattice import lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_19171_gb300 import build
    build.build()
    import paper_2509_19171_gb300 as pkg
    return pkg


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("lat,N", [("D2Q9", 5), ("D3Q19", 3), ("D3Q27", 7)])
def test_moments_and_state(P, lat, N, prec):
    dim = 2 if lat == "D2Q9" else 3
    mesh = W.box_mesh((3, 2, 1)[:dim], (0.0,) * dim, (1.0, 0.7, 0.4)[:dim], (False,) * dim, walls={0: 1},
                      wall_velocity=[[0.0] * dim])
    s = P.SELBM(mesh, lat, N, 1e-2, precision=prec)
    e, t, _ = lattice(lat)
    rng = np.random.default_rng(N)
    l2 = s.node_coords().reshape(-1, dim).round(9)
    _, first, inv = np.unique(l2, axis=0, return_index=True, return_inverse=True)
    n = len(first)
    g = rng.standard_normal((len(t), n)) * 10.0 ** rng.uniform(-12, -2, (len(t), n))
    g[:, :3] = 0.0
    g[1, 3:6] = 1e-40
    f = (t[:, None] + g)[:, inv.ravel()].reshape(len(t), s.E, s.Np)
    s.set_state(np.ascontiguousarray(f))
    dev = f - t[:, None, None]
    if prec == 1:
        dev = dev.astype(np.float32).astype(np.float64)
    assert np.array_equal(s.get_state(), dev + t[:, None, None])
    rho, u = s.moments()
    drho, j = dev.sum(0), np.einsum("ak,aep->epk", e.astype(float), dev)
    bound = 8 * 2.0 ** -53 * (1 + len(t) * np.abs(dev).max())
    assert np.abs(rho - (1 + drho)).max() <= bound
    assert np.abs(u - j / (1 + drho)[..., None]).max() <= bound
    d = s.diagnostics()
    assert abs(d[0] - 0.7 ** (dim > 1) * 0.4 ** (dim > 2)) < 0.05 and np.isfinite(d).all()
    dev[2] = np.nan                                  # every copy: set_state takes a node from its first
    s.set_state(np.ascontiguousarray(dev + t[:, None, None]))
    with pytest.raises(P.SelbmError):
        s.diagnostics()
