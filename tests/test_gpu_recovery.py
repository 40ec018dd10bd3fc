"""A handle that held NaN gives the results of a fresh one once a finite state is set: nothing of the
broken state stays in its buffers."""
import numpy as np
import pytest

import workloads as W
from oracle import learned as Lr

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


@pytest.mark.parametrize("lat,N,prec,timed", [
    ("D2Q9", 5, 0, False), ("D2Q9", 5, 1, False), ("D2Q9", 5, 0, True),      # timers on: the several-kernel form
    ("D3Q19", 7, 0, False), ("D3Q19", 7, 1, False), ("D3Q27", 6, 0, False), ("D3Q27", 6, 1, False)])
@pytest.mark.parametrize("learned", [True, False])
def test_finite_state_after_nan(P, lat, N, prec, timed, learned):
    dim = 2 if lat == "D2Q9" else 3
    mesh = W.box_mesh((3, 2, 2)[:dim], (0.0,) * dim, (1.0, 0.8, 0.7)[:dim], (True, False, True)[:dim], walls={2: 1},
                      wall_velocity=[[0.0] * dim])
    nin = 2 * (N + 1)
    params = np.float64(np.float32(Lr.init_params(nin, seed=11) * 1.5))
    rng = np.random.default_rng(5)
    out = []
    for broken in (False, True):
        s = P.SELBM(mesh, lat, N, 1e-2, precision=prec, filt={"shape": 0, "gamma": 0.1, "kc": float(N - 2)})
        s.timers(timed)
        if learned:
            s.set_learned_filter(params, np.full(nin, -35.0), np.full(nin, 5.0), mass_bound=1e9)
        if not out:
            x = s.node_coords()
            k = rng.integers(1, 3, (dim, dim))
            u = np.ascontiguousarray(0.02 * np.sin(x @ k) * (x[..., 1:2] * (0.8 - x[..., 1:2])))
            rho = 1 + 1e-3 * np.cos(x @ k[0])
        if broken:
            bad = np.full((s.Q, s.E, s.Np), np.nan)
            s.set_state(bad)
            s.step(2)
            assert np.isnan(s.get_state()).all()         # read with the filter pending
            with pytest.raises(P.SelbmError):
                s.diagnostics()
        s.init(rho, u)
        first = s.moments()[0]
        assert np.isfinite(first).all()
        s.step(2)
        out.append([s.get_state(), *s.moments()])
        s.set_filter({"shape": 0, "gamma": 0.2, "kc": float(N - 2)})    # applies the pending filter to the state
        s.step(1)
        out[-1].append(s.get_state())
        s.close()
    for a, b in zip(*out):
        assert np.isfinite(b).all() and np.array_equal(a, b)
