"""2D steps beside the plain resident one: meshes that the SMs cannot hold (several-kernel form).
Tolerances of the step's other parity tests: 1e-12 (FP64) and 1e-6 (FP32) of max |f| per step."""
import numpy as np
import pytest

import workloads as W
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


@pytest.mark.parametrize("prec", [0, 1])
def test_mesh_beyond_the_sms(P, prec):
    # 227 KB hold 9 elements of this order in FP64 and 18 in FP32; 56 x 56 quads are 21 to an SM
    mesh = W.box_mesh((56, 56), (0, 0), (1, 1), (True, False), walls={2: 1, 3: 1}, wall_velocity=[[0.01, 0]])
    filt = {"shape": 0, "gamma": 0.2, "kc": 6.0}
    o = OracleSELBM(mesh, "D2Q9", 8, 1e-2, filt=filt)
    s = P.SELBM(mesh, "D2Q9", 8, 1e-2, precision=prec, filt=filt)
    f = rough_state(o, 0.02, 8)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(2):
        f = o.step(f)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= (1e-12 if prec == P.FP64 else 1e-6)


def channel():
    return W.box_mesh((6, 5), (0, 0), (1, 0.8), (True, False), walls={2: 1, 3: 2}, wall_velocity=[[0, 0], [0.02, 0]])


@pytest.mark.parametrize("prec", [0, 1])
def test_refused_cooperative_launch(P, monkeypatch, prec):
    """A device that refuses the cooperative launch (here: its error code) steps in the several-kernel form."""
    filt = {"shape": 0, "gamma": 0.1, "kc": 4.0}
    out = []
    for refuse in (False, True):
        if refuse:
            monkeypatch.setenv("SELBM_FLOW_REFUSE", "1")
        s = P.SELBM(channel(), "D2Q9", 6, 1e-3, precision=prec, filt=filt, body_accel=(1e-4, 0.0, 0.0))
        s.init_from(W.shear_layer_init(U0=0.02, kappa=5.0))
        s.step(3)
        s.step(2)
        assert s.steps == 5
        out.append(s.get_state())
        s.close()
    assert 0 < rel(out[1], out[0]) <= (1e-12 if prec == 0 else 1e-6)


@pytest.mark.parametrize("prec", [0, 1])
def test_captured_by_the_caller(P, monkeypatch, prec):
    """Steps that the caller captures into a graph of its own and replays."""
    import torch
    monkeypatch.setenv("SELBM_NO_GRAPH", "1")
    filt = {"shape": 0, "gamma": 0.1, "kc": 4.0}
    stream = torch.cuda.Stream()
    a, b = (P.SELBM(channel(), "D2Q9", 6, 1e-3, precision=prec, filt=filt, stream=stream.cuda_stream) for _ in range(2))
    for s in (a, b):
        s.timers(True)                                    # the kernels of the several-kernel form are loaded
        s.init_from(W.shear_layer_init(U0=0.02, kappa=5.0))
        s.step(2)
        s.timers(False)
        s.step(2)
        s.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(3)
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
    b.step(9)
    assert rel(a.get_state(), b.get_state()) <= 9 * (1e-12 if prec == 0 else 1e-6)
    a.step(2)                                             # the resident step goes on from there
    b.step(2)
    assert rel(a.get_state(), b.get_state()) <= 11 * (1e-12 if prec == 0 else 1e-6)
