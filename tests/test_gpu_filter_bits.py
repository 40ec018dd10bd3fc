"""Rounding of the FP64 filter in fixed point.  Two handles take the same step, one without a filter;
the other's state is the filter of it.  With gamma = 1e-6 the correction is small (its matrices' rounding
is below the bits looked at) and what is left is the arithmetic's own rounding: half a unit in the last
place of the value, and in each of the three passes half a unit of the tile's integers, 2^(e - 56) for a
largest value below 2^e.  Values small next to the tile's largest are not pulled towards zero: over M
values the mean of the units' errors, uniform in [-1/2, 1/2] a pass, is below 6 sqrt(3 / 12 M)."""
import numpy as np
import pytest

import workloads as W
from oracle import gll

pytestmark = pytest.mark.gpu


def modal(N):
    from numpy.polynomial import legendre as L
    xi, V = np.asarray(gll.gll_nodes(N)), np.zeros((N + 1, N + 1))
    for k in range(N + 1):
        c = np.zeros(k + 1)
        c[k] = 1
        if k >= 2:
            c[k - 2] = -1
        V[:, k] = L.legval(xi, c)
    return V, np.linalg.inv(V)


@pytest.mark.parametrize("lat,N", [("D3Q19", 4), ("D3Q27", 7), ("D3Q19", 9)])
def test_filter_rounds_to_nearest(lat, N):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_19171_gb300 as P
    mesh = W.box_mesh((4, 3, 4), (0, 0, 0), (1, 0.8, 1.1), (True, True, True))
    gamma, kc, n = 1e-6, float(N - 2), N + 1
    out = []
    for g in (0.0, gamma):
        # rho0 = 0 up to the smallest numbers: the state array is the stored deviation, bit for bit
        s = P.SELBM(mesh, lat, N, 1e-2, rho0=1e-300, filt={"shape": 0, "gamma": g, "kc": kc})
        e, t, _ = s.lattice_table()
        x = s.node_coords()
        rng = np.random.default_rng(N)
        f = np.empty((s.Q, s.E, s.Np))
        for a in range(s.Q):
            ph = rng.uniform(0, 6.28, 3)
            f[a] = t[a] * (1 + 3 * np.sin(2 * np.pi * x / [1, 0.8, 1.1] + ph).sum(-1))
        s.set_state(f)
        s.step(1)
        out.append(s.get_state())
        s.close()
    ld = np.longdouble
    v = out[0].astype(ld).reshape(-1, n, n, n)
    k = np.arange(n)
    V, Vi = modal(N)
    r = np.clip((k - kc) / (N - kc), 0, None)
    F = (V * ((1.0 - gamma * r * r) - 1.0)) @ Vi          # sigma is an FP64 number
    F[0] = F[-1] = 0
    F = F.astype(ld)
    ref = v + np.einsum("ij,eabj->eabi", F, v)
    ref = ref + np.einsum("ij,eajb->eaib", F, ref)
    ref = ref + np.einsum("ij,ejab->eiab", F, ref)
    got = out[1].reshape(v.shape)
    top = np.abs(out[0].reshape(v.shape)).max((1, 2, 3), keepdims=True)
    unit = np.exp2(np.floor(np.log2(top)) + 1 - 57).astype(ld)
    err = ((got - ref) / unit).astype(float)
    own = (np.spacing(np.abs(got)) / 2 / unit).astype(float)
    # element-interior nodes: a shared node comes from its owner's tile, at that tile's unit
    inner = (slice(None),) + (slice(1, -1),) * 3
    err, own, got = err[inner], own[inner], got[inner]
    # F's own rounding: gamma n 2^-52 of the largest value
    assert (np.abs(err) <= 1.5 + own + gamma * n * 2.0 ** -52 * 2 ** 57).all()
    small = np.abs(got) < top / 64
    m = int(small.sum())
    assert m > 200
    bound = 6 * np.sqrt(3 / 12 / m) + gamma * n * 2.0 ** -52 * 2 ** 57
    assert abs((err * np.sign(got))[small].mean()) <= bound
    assert abs(err[small].mean()) <= bound
