"""The diagnostic sums (mass, momentum, kinetic energy) against numpy sums over the unique nodes with the
oracle's assembled masses, for states with deviations over many decades.  A sum of G products in
blocks and trees of FP64 additions is within 2^-53 (4 + additions in a row, at most G / 155648 + 8 + 16 of
them: 64) of the sum of the magnitudes; mesh masses agree to 1e-13."""
import numpy as np
import pytest

import workloads as W
from oracle.selbm import OracleSELBM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("lat,N,shape", [("D2Q9", 5, (3, 2)), ("D2Q9", 14, (31, 7)), ("D3Q19", 3, (3, 2, 1)), ("D3Q27", 7, (5, 4, 3))])
def test_sums(lat, N, shape, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_19171_gb300 as P
    dim = len(shape)
    mesh = W.box_mesh(shape, (0.0,) * dim, (1.0, 0.7, 0.4)[:dim], (True,) + (False,) * (dim - 1), walls={2: 1, 3: 1}, wall_velocity=[[0.0] * dim])
    o = OracleSELBM(mesh, lat, N, 1e-2)
    s = P.SELBM(mesh, lat, N, 1e-2, precision=prec)
    rng = np.random.default_rng(N)
    g = o.t[:, None] * rng.standard_normal((o.Q, o.G)) * 10.0 ** rng.uniform(-9, -1, (o.Q, o.G))
    f = o.t[:, None] + g
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    g = f - o.t[:, None]
    if prec == 1:
        g = g.astype(np.float32).astype(np.float64)
    rho, j = 1 + g.sum(0), np.asarray(o.e, float).T @ g
    uu = ((j / rho) ** 2).sum(0)
    d = s.diagnostics()
    eps = 64 * 2.0 ** -53 + 1e-13
    assert abs(d[0] - (o.mass * rho).sum()) <= eps * (o.mass * rho).sum()
    for k in range(3):
        want, size = ((o.mass * j[k]).sum(), (o.mass * np.abs(g).sum(0)).sum()) if k < dim else (0.0, 0.0)
        assert abs(d[1 + k] - want) <= eps * size
    assert abs(d[4] - 0.5 * (o.mass * uu).sum()) <= eps * (o.mass * uu).sum()
    s.close()
