"""The table of the whole history intervals' quadrature points (2048 bins x
nodes and more): against the same bins answered without it (fewer bins a call;
bins do not depend on each other), against the oracle's adaptive integral, and
in the batched kick beside boxes that do not use it."""
import numpy as np
import pytest

from oracle import pm_oracle as O
from paper_1209_0461_gb300 import batch, nupm, synth

pytestmark = pytest.mark.gpu


def _problem(nk, nh, a, first):
    w = synth.Workload("w", 32, 32, 1000.0, 0.3, 3, max(nh, 1), nk, "fp64")
    kb = synth.surrogate_kbins(nk)
    pi, ti = synth.nu_initial_at(kb, w)
    p = np.sqrt(synth.linear_power(kb, w))
    a0 = w.a_init * first
    a_hist = a0 * (a / a0) ** (np.arange(nh) / nh)
    eps = 1.0 + 0.05 * np.sin(3.0 * np.arange(nh) / nh)[:, None] * np.tanh(np.log(kb / 0.1))[None, :]
    hist = np.ascontiguousarray(synth.growth_interp(a_hist, w.omega_m)[:, None] * p[None, :] * eps)
    return w, kb, pi, ti, a_hist, hist, p * float(synth.growth_interp(a, w.omega_m))


def _ratio(w, kb, pi, ti, a_hist, hist, cur, a, sel, **kw):
    import torch
    nk = len(sel)
    pm = nupm.PM(32, 8, w.box, w.omega_cdm, w.omega_nu, w.h, w.m_nu_total, w.n_species, a_init=w.a_init, n_kbins=nk,
                 n_hist_max=256, precision="fp64", sqrtPnu_init=np.ascontiguousarray(pi[:, sel]),
                 theta_over_delta_init=np.ascontiguousarray(ti[:, sel]), **kw)
    pm.set_power(np.ones(nk), kb[sel], cur[sel] ** 2 * 32.0 ** 6 / w.box ** 3)
    R = torch.full((nk,), -1.0, dtype=torch.float64, device="cuda")
    pm.nu_response(a, a_hist, torch.from_numpy(np.ascontiguousarray(hist[:, sel])).cuda(), ratio=R)
    pm.check()
    pm.close()
    return R.cpu().numpy()


@pytest.mark.parametrize("flags", [0, nupm.PM_RELATIVISTIC, nupm.PM_I_FIT, nupm.PM_IC_MULTIPOLE])
@pytest.mark.parametrize("nk,nh,a,first,quad", [(16, 128, 0.5, 1.0, 8), (9, 256, 0.9, 1.0, 12), (64, 32, 0.05, 1.5, 16),
                                                (64, 33, 1.0, 1.0, 8), (1024, 2, 0.3, 1.0, 8), (40, 256, 0.021, 1.01, 2)])
def test_table_against_its_absence(nk, nh, a, first, quad, flags):
    pr = _problem(nk, nh, a, first)
    assert nk * nh >= 2048
    part = max(1, 2047 // nh)
    got = _ratio(*pr, a, np.arange(nk), quad_nodes=quad, flags=flags)
    ref = np.concatenate([_ratio(*pr, a, np.arange(i, min(i + part, nk)), quad_nodes=quad, flags=flags)
                          for i in (range(0, nk, part) if nk < 1024 else (0, 500))])
    if nk >= 1024:
        got = np.concatenate([got[0:part], got[500:min(500 + part, nk)]])
    # the same points: ln a to 2^-52 of 4 against intervals of 1e-4 and more, sums of up to 4e3 terms in another order
    assert np.all(np.isfinite(ref)) and np.max(np.abs(got / ref - 1)) < 1e-10


@pytest.mark.parametrize("nk,nh,a,rel", [(16, 128, 0.5, False), (64, 32, 0.9, True), (9, 256, 0.1, False)])
def test_table_against_the_oracle(nk, nh, a, rel):
    pr = _problem(nk, nh, a, 1.0)
    w, kb, pi, ti, a_hist, hist, cur = pr
    got = _ratio(*pr, a, np.arange(nk), flags=nupm.PM_RELATIVISTIC if rel else 0)
    sel = np.unique(np.linspace(0, nk - 1, 2 if rel else 6).astype(int))   # (the oracle takes long with the relativistic background)
    cos = O.Cosmo(w.omega_cdm, w.omega_nu, w.h, w.masses, w.a_init, relativistic=rel)
    ref = O.nu_response(kb[sel], cur[sel], a, cos, a_hist, hist[:, sel], pi[:, sel], ti[:, sel])["R"]
    assert np.max(np.abs(got[sel] / ref - 1)) < 1e-6     # as the response's other oracle tests


def test_batched_boxes_with_and_without_the_table():
    # 64 bins on 32, 40, 8 and 31 nodes: the table for the first two only
    boxes = [synth.with_(b, n_hist=nh, m_nu_total=0.3) for b, nh in zip(synth.batched_boxes(10, n_hist=8, n_kbins=64)[::3], (32, 40, 8, 31))]
    assert {b.ngrid for b in boxes} == {64} and len(boxes) == 4
    res = []
    for kw in (dict(n_streams=1, autotune=False), dict(persistent=True, split=1)):
        b = batch.Batch(boxes, **kw)
        b.eager_step()
        b.check()
        res.append([(it["vel"] - it["vel0"]).cpu().numpy() for it in b.items])
        b.close()
    for d0, d1 in zip(*res):
        assert np.abs(d1 - d0).max() <= 1e-5 * np.abs(d0).max()
        assert np.sqrt(((d1 - d0) ** 2).mean()) <= 1e-6 * np.sqrt((d0 ** 2).mean())
