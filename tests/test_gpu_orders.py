"""The any-order element kernels (one thread per line, FP64 lines in 64-bit fixed point)
against the FP64 oracle at every order they are compiled for: affine boxes with walls on every
face and curved pipes, both lattices, with and without a pending filter, learned control, and
states with NaN, infinities or a large dynamic range.  Tolerances are those of the step's other
parity tests: 1e-12 (FP64) and 1e-6 (FP32) of max |f| per step.
"""
import math

import numpy as np
import pytest

import workloads as W
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


def filt_of(N):
    return {"shape": 0, "gamma": 0.3, "kc": max(1.0, float(N - 3))} if N > 2 else None


def walled_box():
    return W.box_mesh((2, 1, 2), (0, 0, 0), (1, 0.6, 1.1), (False, False, False),
                      walls={0: 1, 1: 1, 2: 1, 3: 2, 4: 1, 5: 1}, wall_velocity=[[0, 0, 0], [0.02, 0, 0.01]])


def compare(P, mesh, lat, N, prec, filt, g=(0.0, 0.0, 0.0), steps=2):
    o = OracleSELBM(mesh, lat, N, 1e-2, filt=filt, body_accel=g)
    s = P.SELBM(mesh, lat, N, 1e-2, precision=prec, filt=filt, body_accel=g)
    f = rough_state(o, 0.02, N)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(steps):
        f = o.step(f)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= (1e-12 if prec == P.FP64 else 1e-6)
    s.close()


@pytest.mark.parametrize("N", range(2, 12))
def test_affine_walls_fp32(P, N):
    compare(P, walled_box(), "D3Q19" if N % 2 else "D3Q27", N, P.FP32DEV, filt_of(N))


@pytest.mark.parametrize("N", range(2, 10))
def test_affine_walls_fp64(P, N):
    compare(P, walled_box(), "D3Q27" if N % 2 else "D3Q19", N, P.FP64, filt_of(N))


@pytest.mark.parametrize("N", [2, 3, 5, 6, 8, 11])
def test_curved_pipe_fp32(P, N):
    mesh = W.pipe_mesh(n_core=1, n_radial=1, n_axial=2, length=1.0)
    compare(P, mesh, "D3Q19" if N % 2 else "D3Q27", N, P.FP32DEV, filt_of(N), (0.0, 0.0, 2e-4))


@pytest.mark.parametrize("N", [2, 3, 4, 6, 7, 9])
def test_curved_pipe_fp64(P, N):
    mesh = W.pipe_mesh(n_core=1, n_radial=1, n_axial=2, length=1.0)
    compare(P, mesh, "D3Q27" if N % 2 else "D3Q19", N, P.FP64, filt_of(N), (0.0, 0.0, 2e-4))


@pytest.mark.parametrize("prec,N,lat", [(0, 7, "D3Q27"), (0, 6, "D3Q19"), (1, 8, "D3Q19"), (1, 5, "D3Q27")])
def test_learned_control(P, prec, N, lat):
    mesh = W.box_mesh((2, 2, 1), (0, 0, 0), (2 * math.pi, 2 * math.pi, 3.0), (True, True, True))
    filt = {"shape": 0, "gamma": 0.1, "kc": float(N - 2)}
    o = OracleSELBM(mesh, lat, N, 1e-3, filt=filt)
    s = P.SELBM(mesh, lat, N, 1e-3, filt=filt, precision=prec)
    nin = 2 * (N + 1)
    lo, hi = np.full(nin, -35.0), np.full(nin, 5.0)
    params = np.float64(np.float32(Lr.init_params(nin, seed=11) * 1.5))
    s.set_learned_filter(params, lo, hi, mass_bound=1.0, ke_bound=1.0)
    f = rough_state(o, 0.02, 3)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(2):
        f = o.step_learned(f, params, lo, hi)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= (1e-10 if prec == 0 else 1e-6)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_state_spreads_as_in_the_whole_element_form(P, monkeypatch, bad):
    """A NaN or infinity at one node of an FP64 state: the same entries are non-finite after a
    step in the split form as in the generic kernels, and the finite ones agree."""
    mesh, out = walled_box(), []
    for generic in (False, True):
        if generic:
            monkeypatch.setenv("SELBM_GENERIC_KERNEL", "1")
        o = OracleSELBM(mesh, "D3Q19", 6, 1e-2)
        s = P.SELBM(mesh, "D3Q19", 6, 1e-2)
        f = o.to_local(rough_state(o, 0.02, 1)).copy()
        q = 3 * 49 + 3 * 7 + 2                       # an element-interior node
        f[4, 1, q] = bad
        s.set_state(np.ascontiguousarray(f))
        s.step(1)
        out.append(s.get_state())
        with pytest.raises(P.SelbmError):
            s.diagnostics()
    fin = np.isfinite(out[0])
    assert np.array_equal(fin, np.isfinite(out[1])) and fin.any() and not fin.all()
    assert rel(out[0][fin], out[1][fin]) <= 1e-12


def test_large_dynamic_range(P):
    """Populations whose values span many decades inside an element (an FP64 state of small
    deviations with one large pulse): within 1e-12 of the oracle."""
    mesh = walled_box()
    o = OracleSELBM(mesh, "D3Q19", 6, 1e-2)
    s = P.SELBM(mesh, "D3Q19", 6, 1e-2)
    rng = np.random.default_rng(2)
    f = o.initial_state(np.ones(o.G), 1e-9 * rng.standard_normal((o.G, 3)))
    f[:, rng.integers(0, o.G, 5)] += 0.3 * o.t[:, None]
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(2):
        f = o.step(f)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= 1e-12
