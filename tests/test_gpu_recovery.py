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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("learned", [False, True])
def test_exchange_that_gives_up(P, monkeypatch, prec, learned):
    """A wait of the resident 2D step that runs out (a share that nobody writes; it gives up after seconds)
    is reported by every call that would hand on the lost state, until a new state is set."""
    N, nin = 5, 12
    monkeypatch.setenv("SELBM_FLOW_STALL", "1")
    mesh = W.box_mesh((20, 16), (0, 0), (1, 1), (True, False), walls={2: 1, 3: 1}, wall_velocity=[[0.0, 0.0]])
    filt = {"shape": 0, "gamma": 0.1, "kc": 3.0}
    s = P.SELBM(mesh, "D2Q9", N, 1e-2, precision=prec, filt=filt)
    params = np.float64(np.float32(Lr.init_params(nin, seed=11)))
    if learned:
        s.set_learned_filter(params, np.full(nin, -35.0), np.full(nin, 5.0), mass_bound=1e9)
    x = s.node_coords()
    rho, u = 1 + 1e-3 * np.cos(6 * x[..., 0]), np.ascontiguousarray(0.01 * np.sin(3 * x) * x[..., 1:2] * (1 - x[..., 1:2]))
    s.init(rho, u)
    want = s.get_state()
    s.step(20)
    calls = [s.sync, s.get_state, s.moments, s.stress, s.diagnostics, s.features, s.element_sigma, s.learned_status,
             lambda: s.wall_stress([1, 0]), lambda: s.radial_profile([0, 0], [1, 0], 1.0, 4), lambda: s.step(1),
             lambda: s.set_filter(filt), lambda: s.set_learned_filter(params, np.full(nin, -35.0), np.full(nin, 5.0))]
    if learned:
        calls.append(s.clear_learned_filter)
    for call in calls:
        with pytest.raises(P.SelbmError) as ei:
            call()
        assert ei.value.code == -5
    s.init(rho, u)
    assert s.sync() == 0 and np.array_equal(s.get_state(), want)
    s.step(20)
    with pytest.raises(P.SelbmError):
        s.sync()
    s.set_state(want)
    assert np.array_equal(s.get_state(), want)
    s.set_filter({"shape": 0, "gamma": 0.2, "kc": 3.0})
    s.close()
