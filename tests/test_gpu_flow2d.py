"""The resident 2D step (one cooperative launch for any number of steps) against the FP64 oracle:
every order, walls and body force, both filter shapes, curved node-form meshes with turned element
frames, meshes of fewer and more elements than the GPU has SMs, and its independence of how the
steps are split into calls.  Tolerances: 1e-12 (FP64) and 1e-6 (FP32) of max |f| per step.
"""
import math

import numpy as np
import pytest

import workloads as W
from oracle import gll
from oracle import learned as Lr
from oracle.selbm import OracleSELBM

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


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def rough_state(o, amp, seed):
    rng = np.random.default_rng(seed)
    rho = 1 + 0.01 * rng.standard_normal(o.G)
    f = o.initial_state(rho, amp * rng.standard_normal((o.G, o.dim)))
    return f + 1e-3 * o.t[:, None] * rng.standard_normal((o.Q, o.G))


def compare(P, mesh, N, prec, filt, g=(0.0, 0.0), steps=3):
    o = OracleSELBM(mesh, "D2Q9", N, 1e-2, filt=filt, body_accel=g)
    s = P.SELBM(mesh, "D2Q9", N, 1e-2, precision=prec, filt=filt, body_accel=g)
    f = rough_state(o, 0.02, N)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(steps):
        f = o.step(f)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= (1e-12 if prec == P.FP64 else 1e-6)
    s.close()


def channel(nx, ny):
    return W.box_mesh((nx, ny), (0, 0), (1, 0.8), (True, False), walls={2: 1, 3: 2}, wall_velocity=[[0, 0], [0.02, 0]])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", range(2, 15))
def test_channel_every_order(P, N, prec):
    filt = {"shape": N % 2, "gamma": 0.2, "kc": float(max(1, N - 3)), "p": 8.0} if N > 2 else None
    compare(P, channel(3, 2), N, prec, filt, (2e-4, 1e-4))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shape,N", [((1, 1), 4), ((19, 9), 3), ((20, 17), 5)])
def test_more_and_fewer_elements_than_ctas(P, shape, N, prec):
    mesh = W.box_mesh(shape, (0, 0), (1, 1), (True, True))
    compare(P, mesh, N, prec, {"shape": 0, "gamma": 0.3, "kc": float(N - 2)}, steps=2)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", [4, 7, 12])
def test_curved_turned_elements(P, N, prec):
    box = W.box_mesh((3, 3), (0, 0), (1, 1), (True, False), walls={2: 1, 3: 1}, wall_velocity=[[0.01, 0]])
    nm = W.node_mesh(box, gll.gll_nodes(4), deform=lambda x: x + 0.02 * np.stack(
        [np.sin(2 * math.pi * x[:, 0]) * np.sin(math.pi * x[:, 1]), np.sin(math.pi * x[:, 1]) * np.cos(2 * math.pi * x[:, 0])], 1),
        rotate=(1, 5, 6))
    compare(P, nm, N, prec, {"shape": 1, "gamma": 0.1, "kc": float(N - 2), "p": 6.0}, (1e-4, 0.0))


@pytest.mark.parametrize("prec", [0, 1])
def test_step_split_and_mixed_forms(P, prec):
    """Seven steps in one call, one by one and with the per-kernel timers on for some of them (the
    several-kernel form): the first two bit for bit, the third within the step's tolerance."""
    filt = {"shape": 0, "gamma": 0.1, "kc": 4.0}
    out = []
    for mode in range(3):
        s = P.SELBM(channel(6, 5), "D2Q9", 6, 1e-3, precision=prec, filt=filt, body_accel=(1e-4, 0.0, 0.0))
        s.init_from(W.shear_layer_init(U0=0.02, kappa=5.0))
        if mode == 0:
            s.step(7)
        else:
            for k in range(7):
                s.timers(mode == 2 and k in (2, 3))
                s.step(1)
        assert s.steps == 7
        out.append(s.get_state())
        s.close()
    assert np.array_equal(out[0], out[1])
    assert rel(out[2], out[0]) <= (1e-12 if prec == 0 else 1e-6)


def test_nonfinite_state(P):
    s = P.SELBM(channel(4, 3), "D2Q9", 5, 1e-2)
    f = np.ones((9, s.E, s.Np)) / 9
    f[3, 2, 14] = np.nan
    s.set_state(f)
    s.step(2)
    g = s.get_state()
    assert np.isnan(g).any() and np.isfinite(g).any()
    with pytest.raises(P.SelbmError):
        s.diagnostics()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N", [4, 7, 11, 14])
def test_learned_control(P, N, prec):
    """The learned control inside the resident step, one call per step and all steps in one call, then
    the drift fallback (a negative mass bound trips at the second pass) and the transfer functions."""
    mesh = channel(5, 4)
    filt = {"shape": 0, "gamma": 0.1, "kc": float(N - 2)}
    nin = 2 * (N + 1)
    lo, hi = np.full(nin, -35.0), np.full(nin, 5.0)
    params = np.float64(np.float32(Lr.init_params(nin, seed=11) * 1.5))
    tol = 1e-10 if prec == 0 else 1e-6
    o = OracleSELBM(mesh, "D2Q9", N, 1e-2, filt=filt)
    f = f0 = rough_state(o, 0.02, 3)
    one, many, drift = (P.SELBM(mesh, "D2Q9", N, 1e-2, filt=filt, precision=prec) for _ in range(3))
    for s, bound in ((one, 1.0), (many, 1.0), (drift, -1.0)):
        s.set_learned_filter(params, lo, hi, mass_bound=bound, ke_bound=0.0)
        s.set_state(np.ascontiguousarray(o.to_local(f0)))
    for k in range(4):
        sig, _, _ = o.learned_sigma(o.stream(*o.collide(f)), params, lo, hi)
        f = o.step_learned(f, params, lo, hi)
        one.step(1)
        assert rel(one.get_state(), o.to_local(f)) <= tol
        assert np.abs(one.element_sigma() - sig).max() <= (1e-9 if prec == 0 else 1e-4)
    assert one.learned_status()["fixed_element_steps"] == 0
    many.step(4)
    assert np.array_equal(many.get_state(), one.get_state())
    g = o.step_learned(o.step_learned(f0, params, lo, hi), params, lo, hi)
    g = o.step(o.step(g))
    drift.step(4)
    assert rel(drift.get_state(), o.to_local(g)) <= tol
    st = drift.learned_status()
    assert st["fallback_flag"] == 1 and st["fixed_element_steps"] == mesh.nelem
