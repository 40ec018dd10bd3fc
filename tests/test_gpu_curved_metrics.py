"""The FP32 split stage on curved elements, whose metrics are read by component: the compiled
orders of both lattices, swizzled (N = 7, 16-byte copies) and plain tiles, with walls and a body
force, against the FP64 oracle.  Tolerance of the FP32 step parity: 1e-6 of max |f| per step.
"""
import numpy as np
import pytest

import workloads as W
from oracle.selbm import OracleSELBM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,N", [("D3Q19", 4), ("D3Q27", 5), ("D3Q19", 7), ("D3Q27", 7)])
def test_curved_split_stage_fp32(lat, N):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_19171_gb300 as P
    mesh = W.pipe_mesh(n_core=1, n_radial=1, n_axial=2, length=1.0)
    filt, g = {"shape": 0, "gamma": 0.3, "kc": float(N - 3)}, (0.0, 0.0, 2e-4)
    o = OracleSELBM(mesh, lat, N, 1e-2, filt=filt, body_accel=g)
    s = P.SELBM(mesh, lat, N, 1e-2, precision=P.FP32DEV, filt=filt, body_accel=g)
    assert s.split
    rng = np.random.default_rng(N)
    f = o.initial_state(1 + 0.01 * rng.standard_normal(o.G), 0.02 * rng.standard_normal((o.G, 3)))
    s.set_state(np.ascontiguousarray(o.to_local(f)))
    for _ in range(2):
        f = o.step(f)
        s.step(1)
        ref = o.to_local(f)
        assert np.abs(s.get_state() - ref).max() <= 1e-6 * np.abs(ref).max()
    s.close()
