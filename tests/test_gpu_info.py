"""The step form that selbm_info reports is the one whose kernels run (the timers' prologue launches tell
them apart)."""
import math

import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,N,prec,env,split", [
    ("D3Q19", 7, 1, None, True), ("D3Q19", 8, 1, None, True), ("D3Q27", 6, 1, None, True), ("D3Q19", 11, 1, None, True),
    ("D3Q19", 12, 1, None, False), ("D3Q19", 6, 0, None, True), ("D3Q27", 5, 0, None, True), ("D3Q19", 9, 0, None, True),
    ("D3Q19", 8, 1, "SELBM_SPLIT", False), ("D2Q9", 6, 0, None, False)])
def test_step_form(monkeypatch, lat, N, prec, env, split):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_19171_gb300 as P
    if env:
        monkeypatch.setenv(env, "0")
    dim = 2 if lat == "D2Q9" else 3
    mesh = W.box_mesh((2, 1, 2)[:dim], (0,) * dim, (2 * math.pi,) * dim, (True,) * dim)
    s = P.SELBM(mesh, lat, N, 1e-3, precision=prec)
    assert s.split == split
    s.init_from(W.tgv3d_init(0.05) if dim == 3 else W.shear_layer_init(U0=0.02, kappa=5.0))
    s.timers(True)
    s.step(2)
    n = {k: v[1] for k, v in s.timers_read().items()}
    assert n["prologue"] == (2 if split else 0) and n["stage1"] == 2 and n["stage23"] == 4 and n["assembly"] == 6
    s.close()
