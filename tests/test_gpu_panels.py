"""Break points, node search and point split of the response at the sizes where
they change: no history, one node, nodes at a_init, a full table of 256 nodes
(more points than one step of the ten warps of a bin), ragged bin counts."""
import numpy as np
import pytest

from oracle import pm_oracle as O
from paper_1209_0461_gb300 import nupm, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nh,nk,a,quad", [(0, 5, 0.1, 8), (1, 33, 0.021, 8), (2, 7, 1.0, 16), (31, 12, 0.3, 8),
                                          (33, 9, 0.05, 12), (256, 6, 0.9, 8)])
def test_response_and_features(nh, nk, a, quad):
    import torch
    w = synth.Workload("w", 32, 32, 1000.0, 0.3, 3, max(nh, 1), nk, "fp64")
    kb = synth.surrogate_kbins(nk)
    pi, ti = synth.nu_initial_at(kb, w)
    p = np.sqrt(synth.linear_power(kb, w))
    a_hist = w.a_init * (a / w.a_init) ** (np.arange(nh) / max(nh, 1))
    D = np.array([synth.growth(x, w.omega_m)[0] for x in a_hist])
    hist = np.ascontiguousarray(D[:, None] * p[None, :])
    cur = p * synth.growth(a, w.omega_m)[0]
    pm = nupm.PM(32, 8, w.box, w.omega_cdm, w.omega_nu, w.h, w.m_nu_total, w.n_species, a_init=w.a_init, n_kbins=nk,
                 n_hist_max=256, precision="fp64", quad_nodes=quad, sqrtPnu_init=pi, theta_over_delta_init=ti)
    count = np.ones(nk)
    if nk > 8:
        count[3] = 0.0                                    # an empty bin: outputs and features 0
    pm.set_power(count, kb * count, cur ** 2 * 32.0 ** 6 / w.box ** 3 * count)
    R = torch.full((nk,), -1.0, dtype=torch.float64, device="cuda")
    ht = torch.from_numpy(hist).cuda() if nh else None
    pm.nu_response(a, a_hist, ht, ratio=R)
    X = pm.response_features(a, a_hist, ht).cpu().numpy()
    pm.check()
    pm.close()
    R = R.cpu().numpy()
    ok = count > 0
    assert np.all(R[~ok] == 0) and np.all(X[~ok] == 0)
    cos = O.Cosmo(w.omega_cdm, w.omega_nu, w.h, w.masses, w.a_init)
    ref = O.nu_response(kb[ok], cur[ok], a, cos, a_hist, hist[:, ok], pi[:, ok], ti[:, ok])["R"]
    # Gauss-Legendre panels against the adaptive integral: 1e-7 over the surrogate's range
    assert np.max(np.abs(R[ok] / ref - 1)) < 1e-6
    u = np.log(w.a_init) + 0.5 * (np.cos(np.pi * (np.arange(8) + 0.5) / 8) + 1) * np.log(a / w.a_init)
    nodes = np.append(np.log(a_hist), np.log(a))
    for b in np.flatnonzero(ok):
        h = np.interp(u, nodes, np.append(hist[:, b], cur[b]))
        c = [0.25 * np.sum(np.log(h / cur[b]) * np.cos(j * np.pi * (np.arange(8) + 0.5) / 8)) for j in range(8)]
        np.testing.assert_allclose(X[b], np.array([np.log(kb[b]), np.log(a), 0.3, w.omega_nu] + c, np.float32),
                                   rtol=2e-6, atol=2e-7)
