"""Device memory of a handle against the arrays that its form needs: metrics once, no array beside the
staging buffer for a read-back."""
import numpy as np
import pytest

import workloads as W

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


def free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("lat,N,prec", [("D3Q19", 7, 1), ("D3Q19", 6, 1), ("D3Q27", 7, 0)])
def test_metrics_are_held_once(P, lat, N, prec):
    small = P.SELBM(W.pipe_mesh(n_core=1, n_radial=1, n_axial=2), lat, N, 1e-2, precision=prec)      # loads the kernels
    before = free()
    s = P.SELBM(W.pipe_mesh(n_core=6, n_radial=4, n_axial=24), lat, N, 1e-2, precision=prec)
    held = before - free()
    E, Np, Q, G, r = s.E, s.Np, s.Q, s.G, 4 if prec else 8
    nb = Np - (N - 1) ** 3
    # four states, the shares, rho and the control's node moments; ten metric values a local node; numbering
    # and owners; mass and first copies; copies of shared nodes (index, 1 / mass, offsets); 32 MB of granularity
    need = ((4 * Q + 3) * G + Q * E * nb + 10 * E * Np) * r + 5 * E * Np + 12 * G + 24 * E * nb + 2 ** 25
    assert held <= need, (held, need)
    s.close()
    small.close()


@pytest.mark.parametrize("lat,N,prec", [("D2Q9", 8, 1), ("D2Q9", 8, 0), ("D3Q19", 7, 1)])
def test_read_back_allocates_its_staging_alone(P, lat, N, prec):
    mesh = [W.box_mesh((k,) * 2, (0, 0), (1, 1), (True, True)) if lat == "D2Q9" else W.box_mesh((k,) * 3, (0,) * 3, (1,) * 3, (True,) * 3)
            for k in ((2, 160) if lat == "D2Q9" else (2, 14))]
    for m in mesh:                                       # the small one loads the kernels
        s = P.SELBM(m, lat, N, 1e-2, precision=prec)
        x = s.node_coords()
        u = np.ascontiguousarray(0.01 * np.sin(6.28 * x))
        before = free()
        s.init(np.ones((s.E, s.Np)), u)
        s.step(1)
        s.moments()
        s.diagnostics()
        s.radial_profile([0, 0, 0], [1, 0, 0], 1.0, 8)
        held = before - free()
        fields, coords = (1 + s.dim) * s.E * s.Np * 8, s.dim * s.G * 8
        # staging of fields (+ sums per element), node coordinates of the profile, granularity
        assert held <= fields + 8 * (s.E + 1) + coords + 2 ** 23, (held, fields, coords)
        assert np.isfinite(s.moments()[0]).all()
        s.close()
