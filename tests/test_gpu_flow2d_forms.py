"""2D steps beside the plain resident one: meshes that the SMs cannot hold, refused launches and captured
steps (several-kernel form), the FP64 line form of CTAs with many elements, nodes of many elements.
Tolerances of the step's other parity tests: 1e-12 (FP64) and 1e-6 (FP32) of max |f| per step."""
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


def check(P, mesh, N, prec, filt, g, steps=2):
    o = OracleSELBM(mesh, "D2Q9", N, 1e-2, filt=filt, body_accel=g)
    s = P.SELBM(mesh, "D2Q9", N, 1e-2, precision=prec, filt=filt, body_accel=g)
    f = rough_state(o, 0.02, N)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(steps):
        f = o.step(f)
        s.step(1)
        assert rel(s.get_state(), o.to_local(f)) <= (1e-12 if prec == P.FP64 else 1e-6)
    s.close()


# above 3000 (population, node) tasks a CTA the FP64 form takes lines, not nodes: 6 elements at N = 7
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("curved", [False, True])
def test_many_elements_a_cta(P, prec, curved):
    mesh = W.box_mesh((30, 28), (0, 0), (1, 1), (True, False), walls={2: 1, 3: 1}, wall_velocity=[[0.01, 0]])
    if curved:
        mesh = W.node_mesh(mesh, gll.gll_nodes(3), deform=lambda x: x + 0.004 * np.stack(
            [np.sin(2 * np.pi * x[:, 0]) * np.sin(np.pi * x[:, 1]), np.sin(np.pi * x[:, 1]) * np.cos(2 * np.pi * x[:, 0])], 1),
            rotate=(1, 70, 500))
    check(P, mesh, 7, prec, {"shape": 0, "gamma": 0.2, "kc": 5.0}, (2e-4, 1e-4))


def fans(valence, count):
    """`count` discs of `valence` quads around one vertex each (walls outside), in node form."""
    E = valence * count
    th = 2 * np.pi * np.arange(valence + 1) / valence
    spoke = np.stack([np.cos(th), np.sin(th)], 1)
    xyz, nbr, face = np.zeros((E, 2, 4)), np.full((E, 4), -1, np.int32), np.zeros((E, 4), np.int8)
    for d in range(count):
        for q in range(valence):
            e = d * valence + q
            a, b = spoke[q], spoke[q + 1]
            out = (a + b) / np.linalg.norm(a + b) * 1.3
            xyz[e] = (np.stack([0 * a, a, b, out]) + [3.0 * d, 0]).T
            nbr[e, 0], face[e, 0] = d * valence + (q + 1) % valence, 2      # along the next spoke
            nbr[e, 2], face[e, 2] = d * valence + (q - 1) % valence, 0
    bc = np.zeros((E, 4), np.int32)
    bc[:, 1] = bc[:, 3] = 1
    return W.NodeMeshSpec(2, 1, xyz, nbr, face, np.zeros((E, 4), np.int8), bc, np.array([[0.01, 0.0]]))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("valence,count,N", [(5, 1, 4), (6, 1, 7), (9, 1, 5), (5, 70, 5)])
def test_vertex_of_many_elements(P, valence, count, N, prec):
    """A node with more copies than the kernel keeps in shared memory (four): on CTAs of one element and of several."""
    check(P, fans(valence, count), N, prec, {"shape": 0, "gamma": 0.2, "kc": float(N - 2)}, (1e-4, 0.0))


@pytest.mark.parametrize("prec", [0, 1])
def test_vertex_of_many_elements_learned(P, prec):
    N, nin = 5, 12
    mesh, filt = fans(7, 1), {"shape": 0, "gamma": 0.1, "kc": 3.0}
    params = np.float64(np.float32(Lr.init_params(nin, seed=11) * 1.5))
    lo, hi = np.full(nin, -35.0), np.full(nin, 5.0)
    o = OracleSELBM(mesh, "D2Q9", N, 1e-2, filt=filt)
    s = P.SELBM(mesh, "D2Q9", N, 1e-2, filt=filt, precision=prec)
    s.set_learned_filter(params, lo, hi, mass_bound=1.0)
    f = rough_state(o, 0.02, 3)
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    s.step(3)
    for _ in range(3):
        f = o.step_learned(f, params, lo, hi)
    assert rel(s.get_state(), o.to_local(f)) <= 3 * (1e-10 if prec == 0 else 1e-6)
    s.close()
