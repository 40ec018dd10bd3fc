"""Handles stepped from several host threads: a thread with a small mesh does not take away the shared
memory that another thread's larger mesh of the same order needs."""
import threading

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


def in_thread(fn):
    out = []

    def body():
        try:
            out.append(fn())
        except Exception as ex:                          # handed to the test
            out.append(ex)
    t = threading.Thread(target=body)
    t.start()
    t.join()
    if isinstance(out[0], Exception):
        raise out[0]
    return out[0]


def square(n):
    return W.box_mesh((n, n), (0, 0), (1, 1), (True, True))


def box(walls):
    return W.box_mesh((1, 1, 2), (0, 0, 0), (1, 1, 2), (not walls, not walls, True),
                      walls={0: 1, 1: 1, 2: 1, 3: 1} if walls else {}, wall_velocity=[[0.0] * 3] if walls else None)


# what is larger: the elements of a CTA (2D), the wall nodes of an element (3D)
@pytest.mark.parametrize("lat,N,prec,form", [("D2Q9", 8, 0, ""), ("D2Q9", 8, 1, ""), ("D3Q19", 9, 0, ""), ("D3Q19", 11, 1, ""),
                                              ("D3Q27", 7, 1, ""), ("D3Q19", 7, 1, "SELBM_SPLIT"), ("D2Q9", 8, 0, "SELBM_GENERIC_KERNEL")])
def test_small_mesh_in_another_thread(P, monkeypatch, lat, N, prec, form):
    monkeypatch.setenv("SELBM_NO_GRAPH", "1")
    if form:
        monkeypatch.setenv(form, "0" if form == "SELBM_SPLIT" else "1")
    big, small = (square(20), square(2)) if lat == "D2Q9" else (box(True), box(False))
    a = P.SELBM(big, lat, N, 1e-2, precision=prec, stream=0)
    rho, u = np.ones((a.E, a.Np)), np.zeros((a.E, a.Np, a.dim))
    u[..., 0] = 0.01
    a.init(rho, u)
    a.step(2)

    def other():
        b = P.SELBM(small, lat, N, 1e-2, precision=prec, stream=0)
        b.init(np.ones((b.E, b.Np)), np.zeros((b.E, b.Np, b.dim)))
        b.step(2)
        b.sync()
    in_thread(other)
    a.step(2)                                            # same thread, larger launches of the same kernels
    a.sync()
    f = a.get_state()
    a.init(rho, u)
    a.step(4)
    assert np.array_equal(f, a.get_state())
    a.close()
