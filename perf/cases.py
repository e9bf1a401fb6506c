"""The work a user of the particle-mesh kick library has it do, as cases to measure.

A case is a plain dict; ``listed`` gives the fixed ones, ``draw`` one more of
the same ranges, ``prepare`` what a simulation holds before the call (contexts,
particles, stored history, network), ``run`` one pass through the public
binding, ``work`` its compulsory bytes and operations, and ``exact`` the same
outputs in 64 bits from plain torch and numpy.

Kinds:
  kick      nu_prepare, deposit, nu_response (or nu_response_mlp), kick of one box
  step      two leapfrog steps from a snapshot (pm_step), FP64
  batch     boxes of one grid size kicked together by persistent kernels
  graph     boxes of several grid sizes, their kicks captured in one CUDA graph
  response  the exact response and the surrogate's features on given spectra
            (one training scenario of the surrogate)
  mlp_grad  loss gradient of the surrogate network on one minibatch
  mlp_fwd   the surrogate network on a set of feature rows
"""
import math

import numpy as np
import torch

from paper_1209_0461_gb300 import nupm, synth

A_INIT, A_KICK, H0, OMEGA_M, N_SPECIES = 0.02, 0.1, 0.7, 0.3, 3
T_NU0 = 1.68e-4          # eV
C_OVER_H0 = 2997.92458   # Mpc/h
ZETA3 = 1.2020569031595942


# ------------------------------------------------------------------ the cases
def _kick(name, ngrid, npart, precision, box, m_nu, n_kbins, n_hist, clustered=False, tuned=False,
          response="exact", acc=False, deconv=False):
    return {"name": name, "kind": "kick", "ngrid": ngrid, "npart": npart, "precision": precision, "box": box,
            "m_nu": m_nu, "n_kbins": n_kbins, "n_hist": n_hist, "clustered": clustered, "tuned": tuned,
            "response": response, "acc": acc, "deconv": deconv}


def listed():
    return [
        # the smallest simulation box: a test or teaching run; launches and latency count
        _kick("kick_32_fp64", 32, 32 ** 3, "fp64", 256.0, 0.3, 32, 16, acc=True),
        # a radix-3 grid with a thinned, odd particle count and the learned response
        _kick("kick_192_fp32_odd_mlp", 192, 6_999_999, "fp32", 350.0, 0.3, 64, 32, response="mlp"),
        # an ordinary production box in FP32, built-in tile choices, forces written out
        _kick("kick_256_fp32", 256, 256 ** 3, "fp32", 512.0, 0.3, 128, 64, acc=True),
        # the same box in full FP64, the form the FP32 one is checked against
        _kick("kick_256_fp64", 256, 256 ** 3, "fp64", 512.0, 0.15, 128, 64),
        # late times: clustered particles far from their storage order, tuned as a long run would be
        _kick("kick_512_fp32_clustered", 512, 512 ** 3, "fp32", 500.0, 0.3, 256, 128, clustered=True, tuned=True),
        # the largest box, tuned: the headline workload
        _kick("kick_1024_fp32", 1024, 512 ** 3, "fp32", 1000.0, 0.06, 256, 128, tuned=True),
        # leapfrog steps of a small FP64 run restarted from a snapshot: kicks, stored history and drifts
        {"name": "step_128_fp64", "kind": "step", "ngrid": 128, "npart": 128 ** 3, "precision": "fp64", "box": 256.0,
         "m_nu": 0.3, "n_kbins": 64, "n_hist": 32},
        # an ensemble of equal grids with different seeds and neutrino masses (emulator runs)
        {"name": "batch_128", "kind": "batch", "ngrid": 128, "nbox": 12, "n_kbins": 64, "n_hist": 32},
        # an ensemble of mixed grids replayed as one captured graph
        {"name": "graph_mixed", "kind": "graph", "nbox": 9, "n_kbins": 64, "n_hist": 32},
        # one scenario of the surrogate's training set: exact response and features on given spectra
        {"name": "response_256", "kind": "response", "n_kbins": 256, "n_hist": 128, "m_nu": 0.2, "a": 0.5},
        # one minibatch of the surrogate's training
        {"name": "mlp_grad_4096", "kind": "mlp_grad", "rows": 4096},
        # the trained network over a validation set (a ragged row count)
        {"name": "mlp_fwd_500k", "kind": "mlp_fwd", "rows": 500_001},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("kick", "step", "batch", "graph", "response", "mlp_grad", "mlp_fwd"),
                       (8, 1, 2, 1, 2, 1, 1))[0]
    nk = int(_log(rng, 12, 300))
    nh = int(_log(rng, 1, 129)) - (1 if rng.random() < 0.1 else 0)
    m_nu = rng.choice((0.06, 0.15, 0.3, 0.6, round(rng.uniform(0.05, 0.6), 4)))
    if kind == "kick":
        fp64 = rng.random() < 0.3
        n = rng.choice((16, 32, 64, 128, 192, 256) if fp64 else (16, 32, 64, 128, 192, 256, 256, 512, 512, 1024))
        most = min(n ** 3, 100_000_000)
        np_ = int(_log(rng, max(64, most // 12), most)) | 1
        clustered = n <= 512 and rng.random() < 0.25
        return {"kind": "kick", "ngrid": n, "npart": min(np_, most), "precision": "fp64" if fp64 else "fp32",
                "box": round(n * rng.uniform(0.9, 2.5), 3), "m_nu": rng.choice((0.0, m_nu, m_nu, m_nu)),
                "n_kbins": nk, "n_hist": nh, "clustered": clustered, "tuned": rng.random() < 0.4,
                "response": "mlp" if rng.random() < 0.15 else "exact", "acc": rng.random() < 0.3,
                "deconv": rng.random() < 0.2}
    if kind == "step":
        n = rng.choice((16, 32, 64, 128))
        return {"kind": "step", "ngrid": n, "npart": int(_log(rng, n ** 3 // 8, n ** 3)) | 1, "precision": "fp64",
                "box": round(n * rng.uniform(0.9, 2.5), 3), "m_nu": m_nu, "n_kbins": nk, "n_hist": nh}
    if kind == "batch":
        n = rng.choice((32, 64, 128, 192))
        return {"kind": "batch", "ngrid": n, "nbox": rng.randint(1, 24 if n <= 64 else 12 if n <= 128 else 4),
                "n_kbins": nk, "n_hist": nh}
    if kind == "graph":
        return {"kind": "graph", "nbox": rng.randint(1, 12), "n_kbins": nk, "n_hist": nh}
    if kind == "response":
        return {"kind": "response", "n_kbins": nk, "n_hist": nh, "m_nu": m_nu, "a": round(_log(rng, 0.04, 1.0), 5)}
    if kind == "mlp_grad":
        return {"kind": "mlp_grad", "rows": int(_log(rng, 40, 60_000))}
    return {"kind": "mlp_fwd", "rows": int(_log(rng, 40, 1_000_000))}


# ------------------------------------------------------------------ inputs
def _workload(case, ngrid, npart, box, m_nu, precision="fp32", clustered=False):
    side = max(2, math.ceil(round(npart ** (1.0 / 3.0), 9)))
    while side ** 3 < npart:
        side += 1
    return synth.Workload("case", ngrid, side, box, m_nu, N_SPECIES, max(case["n_hist"], 0), case["n_kbins"],
                          precision, A_INIT, A_KICK, clustered=clustered)


def _particles(w, npart, seed):
    """Zel'dovich particles of a seeded Gaussian field (power of ``synth``) on
    the GPU: FP64 positions [3, npart] in [0, L) and velocities [3, npart]."""
    n, dev = w.npart_side, torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 17)
    wk = torch.fft.rfftn(torch.randn((n, n, n), dtype=torch.float64, device=dev, generator=gen))
    kf = 2 * math.pi / w.box
    f = torch.fft.fftfreq(n, d=1.0 / n, device=dev, dtype=torch.float64).round().long()
    x = torch.arange(n // 2 + 1, device=dev)
    n2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + x[None, None, :] ** 2
    t = np.arange(3 * (n // 2) ** 2 + 3 * n + 1, dtype=np.float64)
    amp = np.zeros_like(t)
    amp[1:] = np.sqrt(synth.linear_power(kf * np.sqrt(t[1:]), w) * n ** 3 / w.box ** 3) / (kf * t[1:])
    wk *= torch.from_numpy(amp).to(dev)[n2]
    del n2
    D, _ = synth.growth(1.0 if w.clustered else w.a_kick, w.omega_m)
    Dv, fv = synth.growth(w.a_kick, w.omega_m)
    uv = w.a_kick ** 2 * float(synth.hubble(w.a_kick, w.omega_m)) * fv * Dv
    keep = None
    if npart < n ** 3:   # a thinned sample, in storage order
        keep = torch.randperm(n ** 3, device=dev, generator=gen)[:npart].sort().values
    site = (torch.arange(n, device=dev, dtype=torch.float64) + 0.5) * (w.box / n)
    pos = torch.empty((3, npart), dtype=torch.float64, device=dev)
    vel = torch.empty((3, npart), dtype=torch.float64, device=dev)
    for d in range(3):
        shape = [1, 1, 1]
        shape[2 - d] = -1
        k = (x if d == 0 else f).double()
        k = torch.where(k.abs() * 2 == n, torch.zeros_like(k), k).reshape(shape)
        psi = torch.fft.irfftn(1j * k * wk, s=(n, n, n))
        q = (site.reshape(shape) + D * psi).reshape(-1)
        psi = psi.reshape(-1)
        if keep is not None:
            q, psi = q[keep], psi[keep]
        q = torch.remainder(q, w.box)
        pos[d] = torch.where(q >= w.box, torch.zeros_like(q), q)
        vel[d] = uv * psi
        del psi, q
    return pos, vel


def _cell_offset(pos, box, ngrid):
    """FP64 positions -> int32 [6, np]: cells, then FP32 offset bits."""
    out = torch.empty((6, pos.shape[1]), dtype=torch.int32, device=pos.device)
    for d in range(3):
        u = pos[d] / (box / ngrid)
        c = torch.floor(u)
        off = (u - c).float()
        bump = off >= 1.0
        out[3 + d] = torch.where(bump, torch.zeros_like(off), off).view(torch.int32)
        out[d] = torch.remainder(c.long() + bump, ngrid).int()
    return out


def _tables(w):
    a_hist, hist = synth.history(w)
    pi, ti = synth.nu_initial(w)
    return np.ascontiguousarray(a_hist[:w.n_hist]), np.ascontiguousarray(hist[:w.n_hist]), pi, ti


def _mlp_numbers(seed):
    """Parameters (Xavier) and normalisation of a surrogate network, host FP32."""
    rng = np.random.default_rng(int(seed) + 5)

    def xavier(o, i):
        return rng.uniform(-1, 1, size=(o, i)) * math.sqrt(6.0 / (i + o))

    W = nupm.MLP_WIDTH
    theta = np.concatenate([xavier(W, nupm.MLP_FEATURES).ravel(), 0.1 * rng.standard_normal(W), xavier(W, W).ravel(),
                            0.1 * rng.standard_normal(W), xavier(1, W).ravel(), [0.05]]).astype(np.float32)
    mu = np.array([-1.6, -1.6, 0.3, 0.01, -0.6, 1.4, -0.2, 0.1, 0.0, 0.0, 0.0, 0.0], np.float32)
    sig = np.array([2.6, 0.9, 0.18, 0.005, 0.4, 0.5, 0.2, 0.1, 0.05, 0.05, 0.05, 0.05], np.float32)
    return theta, mu, sig, np.float32(-2.0), np.float32(0.8)


def _mlp(seed, stream=None):
    theta, mu, sig, ym, ys = _mlp_numbers(seed)
    mlp = nupm.MLP(stream=stream)
    mlp.set_params(theta)
    mlp.set_norm(mu, sig, float(ym), float(ys))
    return mlp


def _mlp_rows(case, seed):
    """Feature rows spread as the normalisation says, and smooth targets."""
    _, mu, sig, ym, ys = _mlp_numbers(seed)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 99)
    z = torch.randn((case["rows"], nupm.MLP_FEATURES), device=dev, generator=gen).clamp_(-3, 3)
    X = z * torch.from_numpy(sig).to(dev) + torch.from_numpy(mu).to(dev)
    y = float(ym) + float(ys) * (torch.tanh(z[:, 0] - 0.5 * z[:, 1]) + 0.3 * z[:, 2] * z[:, 4])
    return X.contiguous(), y.contiguous()


def _box(case, w, npart, seed, stream, flags=0):
    """One simulation box as a program holds it."""
    pos64, vel64 = _particles(w, npart, seed)
    a_hist, hist, pi, ti = _tables(w)
    fp64 = w.precision == "fp64"
    pos = pos64 if fp64 else _cell_offset(pos64, w.box, w.ngrid)
    vel = vel64 if fp64 else vel64.float()
    hist_d = torch.from_numpy(hist).cuda() if len(a_hist) else None
    torch.cuda.synchronize()   # the inputs are ready before another stream reads them
    pm = nupm.PM(w.ngrid, npart, w.box, w.omega_cdm, w.omega_nu, w.h, w.m_nu_total, w.n_species, a_init=w.a_init,
                 n_kbins=w.n_kbins, n_hist_max=max(w.n_hist, 1) + 4, precision=w.precision, flags=flags,
                 sqrtPnu_init=pi, theta_over_delta_init=ti, stream=stream)
    a = w.a_kick
    return {"w": w, "pm": pm, "pos": pos, "vel": vel, "a": a, "K": pm.kick_factor(a, 1.01 * a), "a_hist": a_hist,
            "hist": hist_d, "stream": stream}


_ENSEMBLE = (128, 64, 192)


def _members(case):
    """(ngrid, box side, M_nu) of an ensemble's boxes."""
    nb = case["nbox"]
    return [(case["ngrid"] if case["kind"] == "batch" else _ENSEMBLE[b % 3], 200.0 + 300.0 * b / 31.0,
             synth.BATCH_M_NU[b % 5]) for b in range(nb)]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("mlp_grad", "mlp_fwd"):
        X, y = _mlp_rows(case, seed)
        return {"kind": kind, "mlp": _mlp(seed), "X": X, "y": y}
    if kind == "response":
        w, kb, power, a_hist, hist, (pi, ti) = _scenario(case, seed)
        pm = nupm.PM(w.ngrid, 8, w.box, w.omega_cdm, w.omega_nu, w.h, w.m_nu_total, w.n_species, a_init=w.a_init,
                     n_kbins=w.n_kbins, n_hist_max=max(len(a_hist), 1), precision="fp64", sqrtPnu_init=pi,
                     theta_over_delta_init=ti)
        unit = float(w.ngrid) ** 6 / w.box ** 3
        out = [torch.empty(w.n_kbins, dtype=torch.float64, device="cuda") for _ in range(3)]
        return {"kind": kind, "pm": pm, "count": np.ones(w.n_kbins), "kb": kb, "psum": power * unit, "a": case["a"],
                "a_hist": a_hist, "hist": torch.from_numpy(hist).cuda() if len(a_hist) else None, "out": out}
    if kind in ("batch", "graph"):
        cur = torch.cuda.current_stream()
        streams = [cur] if kind == "batch" else [torch.cuda.Stream() for _ in range(4)]
        boxes = []
        for b, (n, L, m_nu) in enumerate(_members(case)):
            w = _workload(case, n, n ** 3, L, m_nu)
            boxes.append(_box(case, w, n ** 3, 1000 * int(seed) + b, streams[b % len(streams)]))
        st = {"kind": kind, "boxes": boxes}
        if kind == "batch":
            st["batch"] = nupm.BatchPM([b["pm"] for b in boxes], cur)
            return st
        main = torch.cuda.Stream()

        def body():
            fork = torch.cuda.Event()
            fork.record(main)
            for s in streams:
                s.wait_event(fork)
            for b in boxes:
                _kick_once(b, 0.0 if warm else b["K"])
            for s in streams:
                ev = torch.cuda.Event()
                ev.record(s)
                main.wait_event(ev)

        warm = True     # an uncaptured round first (kernel attributes, tables); it leaves the velocities alone
        body()
        torch.cuda.synchronize()
        warm = False
        st["graph"], st["streams"] = nupm.Graph.capture(main, body), (main, streams)
        torch.cuda.synchronize()
        return st
    w = _workload(case, case["ngrid"], case["npart"], case["box"], case["m_nu"], case["precision"],
                  case.get("clustered", False))
    flags = nupm.PM_DECONV_CIC if case.get("deconv") else 0
    b = _box(case, w, case["npart"], seed, torch.cuda.current_stream(), flags)
    b["kind"] = kind
    if kind == "step":
        pm = b["pm"]
        a0, a1, a2 = A_KICK, 1.01 * A_KICK, 1.01 ** 2 * A_KICK
        b["pos0"], b["vel0"] = b["pos"].clone(), b["vel"].clone()
        h = math.sqrt(1.01)
        b["steps"] = [(a0, pm.kick_factor(a0 / h, a0 * h), pm.drift_factor(a0, a1)),
                      (a1, pm.kick_factor(a1 / h, a1 * h), pm.drift_factor(a1, a2))]
        return b
    if case["tuned"]:
        b["pm"].autotune(b["pos"], b["vel"], b["a"], b["a_hist"], b["hist"])
    b["mlp"] = _mlp(seed) if case["response"] == "mlp" and case["m_nu"] > 0 else None
    b["acc"] = torch.empty_like(b["vel"]) if case["acc"] else None
    if case["precision"] == "fp64":
        b["ratio"] = torch.empty(case["n_kbins"], dtype=torch.float64, device="cuda")
        b["sqrtPM"] = torch.empty(case["n_kbins"], dtype=torch.float64, device="cuda")
    return b


# ------------------------------------------------------------------ one pass
def _kick_once(b, K):
    pm = b["pm"]
    mlp = b.get("mlp")
    if mlp is None:
        pm.nu_prepare(b["a"], b["a_hist"], b["hist"])
    pm.deposit(b["pos"])
    if mlp is None:
        pm.nu_response(b["a"], b["a_hist"], b["hist"], ratio=b.get("ratio"), sqrtPM=b.get("sqrtPM"))
    else:
        pm.nu_response_mlp(mlp, b["a"], b["a_hist"], b["hist"], ratio=b.get("ratio"), sqrtPM=b.get("sqrtPM"))
    pm.kick(b["pos"], b["vel"], b["a"], K, acc_out=b.get("acc"))


def run(state):
    kind = state["kind"]
    if kind == "mlp_grad":
        g, loss = state["mlp"].grad(state["X"], state["y"])
        return {"grad": g, "loss": loss}
    if kind == "mlp_fwd":
        return {"lnR": state["mlp"].forward(state["X"])}
    if kind == "response":
        pm, (R, pnu, pmm) = state["pm"], state["out"]
        pm.set_power(state["count"], state["kb"], state["psum"])
        pm.nu_response(state["a"], state["a_hist"], state["hist"], ratio=R, sqrtPnu=pnu, sqrtPM=pmm)
        X = pm.response_features(state["a"], state["a_hist"], state["hist"])
        return {"ratio": R, "sqrtPnu": pnu, "sqrtPM": pmm, "X": X}
    if kind == "batch":
        bs = state["boxes"]
        has = len(bs[0]["a_hist"]) > 0
        state["batch"].kick([b["pos"] for b in bs], [b["vel"] for b in bs], [b["a"] for b in bs],
                            [b["K"] for b in bs], [b["a_hist"] for b in bs] if has else None,
                            [b["hist"] for b in bs] if has else None)
        return {"vel%d" % i: b["vel"] for i, b in enumerate(bs)}
    if kind == "graph":
        state["graph"].launch(torch.cuda.current_stream())
        return {"vel%d" % i: b["vel"] for i, b in enumerate(state["boxes"])}
    if kind == "step":
        # restart from the snapshot, then two steps
        state["pos"].copy_(state["pos0"])
        state["vel"].copy_(state["vel0"])
        pm = state["pm"]
        pm.history_set(state["a_hist"], state["hist"])
        for a, K, ds in state["steps"]:
            pm.step(state["pos"], state["vel"], a, K, ds)
        return {"pos": state["pos"], "vel": state["vel"]}
    _kick_once(state, state["K"])
    out = {"vel": state["vel"]}
    for k in ("acc", "ratio", "sqrtPM"):
        if state.get(k) is not None:
            out[k] = state[k]
    return out


# ------------------------------------------------------------------ compulsory work
def _kick_work(n, npart, fp64, nk, nh):
    word = 8 if fp64 else 4
    pos = 24 * npart
    fft = 2 * 2.5 * n ** 3 * 3 * math.log2(n)
    return pos + 6 * word * npart + 8.0 * nk * nh, fft + 200.0 * npart + 600.0 * nk * (nh + 12)


def work(case):
    kind = case["kind"]
    P = 128 * (12 + 1) + 128 * 129 + 129
    if kind == "mlp_grad":
        return {"bytes": 4.0 * (13 * case["rows"] + 2 * P), "flops": 6.0 * case["rows"] * P}
    if kind == "mlp_fwd":
        return {"bytes": 4.0 * (13 * case["rows"] + P), "flops": 2.0 * case["rows"] * P}
    if kind == "response":
        return {"bytes": 8.0 * case["n_kbins"] * (case["n_hist"] + 8), "flops": 600.0 * case["n_kbins"] *
                (case["n_hist"] + 12)}
    if kind in ("batch", "graph"):
        ws = [_kick_work(n, n ** 3, False, case["n_kbins"], case["n_hist"]) for n, _, _ in _members(case)]
        return {"bytes": float(sum(b for b, _ in ws)), "flops": float(sum(f for _, f in ws))}
    b, f = _kick_work(case["ngrid"], case["npart"], case["precision"] == "fp64", case["n_kbins"], case["n_hist"])
    if kind == "step":   # a copy of the snapshot and two kicks and drifts, positions and velocities in FP64
        return {"bytes": float(2 * b + 48 * case["npart"] * 2), "flops": 2.0 * f + 12.0 * case["npart"]}
    if case["acc"]:
        b += (24 if case["precision"] == "fp64" else 12) * case["npart"]
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64-bit values
_GX, _GW = np.polynomial.legendre.leggauss(16)


def _hubble(a, om):
    return np.sqrt(om / a ** 3 + 1.0 - om)


def _integral(f, u0, u1, panels):
    """int_{u0}^{u1} f(u) du, vectorised over u0, u1 (16-point panels)."""
    u0, u1 = np.broadcast_arrays(np.asarray(u0, float), np.asarray(u1, float))
    h = (u1 - u0) / panels
    s = np.zeros(u0.shape)
    for p in range(panels):
        lo = u0 + p * h
        for x, wt in zip(_GX, _GW):
            s += 0.5 * h * wt * f(lo + 0.5 * h * (x + 1))
    return s


def _free_streaming(x):
    """I(x) = 4 / (3 zeta(3)) sum_n (-1)^{n+1} n / (n^2 + x^2)^2: the first terms,
    then Boole's summation of the alternating tail."""
    x = np.maximum(np.abs(np.asarray(x, float)), 1e-8)
    N, s = 40, np.zeros(x.shape)
    for n in range(N - 1, 0, -1):
        s += (1.0 if n & 1 else -1.0) * n / (n * n + x * x) ** 2
    r, th = np.hypot(N, x), np.arctan2(x, N)

    def d(k):   # k-th derivative of n / (n^2 + x^2)^2 at N
        return 0.5 * (-1) ** k * math.factorial(k + 1) * r ** -(k + 2.0) * np.sin((k + 2) * th) / x

    tail = 0.5 * (d(0) - d(1) / 2 + d(3) / 24 - d(5) / 240 + 17 * d(7) / 40320)
    return 4.0 / (3.0 * ZETA3) * (s + (1.0 if N & 1 else -1.0) * tail)


def _response(kb, pcdm, a, m_nu, om, onu, a_hist, hist, pi, ti, prev=None):
    """R, P_nu^{1/2}, P_M^{1/2} of bins with wavenumbers kb (hist, pi, ti on the
    same bins), one implicit iteration; degenerate species."""
    f_nu = onu / om
    if m_nu <= 0:
        return np.zeros_like(kb), np.zeros_like(kb), (1.0 - f_nu) * pcdm
    kap_s = C_OVER_H0 * T_NU0 / (m_nu / N_SPECIES)
    ue, ui = math.log(a), math.log(A_INIT)
    dsdu = lambda u: 1.0 / (np.exp(2 * u) * _hubble(np.exp(u), om))  # noqa: E731
    s_end = float(_integral(dsdu, ui, ue, 16))
    lu, nh = np.log(np.asarray(a_hist, float)), len(a_hist)
    pnu = np.empty_like(kb)
    for i, k in enumerate(kb):
        kap = k * kap_s
        ell = a * a * float(_hubble(a, om)) / kap
        cuts = [ui, ue] + [u for u in lu if ui < u < ue]
        g = ell * 0.25
        while ue - g > ui:
            cuts.append(ue - g)
            g *= 1.7
        cuts = np.unique(cuts)
        lo, hi = cuts[:-1], cuts[1:]
        half = 0.5 * (hi - lo)
        u = (lo[:, None] + half[:, None] * (_GX[None, :] + 1)).ravel()
        wq = (half[:, None] * _GW[None, :]).ravel()
        ds = _integral(dsdu, u, ue, 4)
        ap = np.exp(u)
        base = 1.5 * om * wq * _free_streaming(kap * ds) * ds / (ap * _hubble(ap, om))
        if nh:
            j = np.clip(np.searchsorted(lu, u, side="right") - 1, -1, nh - 1)
            u0, u1 = lu[np.maximum(j, 0)], np.append(lu, ue)[np.maximum(j, 0) + 1]
            h0 = hist[np.maximum(j, 0), i]
            last = j == nh - 1
            h1 = np.where(last, 0.0, hist[np.minimum(np.maximum(j, 0) + 1, nh - 1), i])
            tau = np.where(j < 0, 0.0, (u - u0) / (u1 - u0))
            jh = float(np.sum(base * (h0 * (1 - tau) + h1 * tau)))
            wc = float(np.sum(np.where(last, base * tau, 0.0)))
        else:
            jh, wc = 0.0, float(np.sum(base))
        ic = float(_free_streaming(kap * s_end)) * pi[0, i] * (1.0 - s_end * A_INIT * ti[0, i])
        guess = pi[0, i] if prev is None else prev[i]
        pnu[i] = ic + jh + ((1 - f_nu) * pcdm[i] + f_nu * guess) * wc
    return pnu / pcdm, pnu, (1 - f_nu) * pcdm + f_nu * pnu


def _features(kb, pcdm, a, m_nu, onu, a_hist, hist):
    ue, ui, nh = math.log(a), math.log(A_INIT), len(a_hist)
    m = np.arange(8)
    u = ui + 0.5 * (np.cos(np.pi * (m + 0.5) / 8) + 1) * (ue - ui)
    h = np.tile(pcdm[:, None], (1, 8))
    if nh:
        nodes = np.append(np.log(np.asarray(a_hist, float)), ue)
        h = np.stack([np.interp(u, nodes, np.append(hist[:, b], pcdm[b])) for b in range(len(kb))])
    g = np.log(h / pcdm[:, None])
    X = np.empty((len(kb), 12))
    X[:, 0], X[:, 1], X[:, 2], X[:, 3] = np.log(kb), ue, m_nu, onu
    for j in range(8):
        X[:, 4 + j] = 0.25 * (g * np.cos(j * np.pi * (m + 0.5) / 8)[None, :]).sum(1)
    return X


def _net(theta, norm, X, dev):
    """(parameters as leaves, out) of the network in FP64 with BF16 weight matrices."""
    W, n = nupm.MLP_WIDTH, nupm.MLP_FEATURES
    mu, sig, ym, ys = norm
    t = torch.from_numpy(theta).to(dev)
    cut = np.cumsum([0, W * n, W, W * W, W, W, 1])
    p = [t[cut[i]:cut[i + 1]] for i in range(6)]
    p = [(q.bfloat16() if i in (0, 2, 4) else q).double().requires_grad_(True) for i, q in enumerate(p)]
    xh = (X.double() - torch.from_numpy(mu).to(dev).double()) / torch.from_numpy(sig).to(dev).double()
    h1 = torch.tanh(xh @ p[0].reshape(W, n).T + p[1])
    h2 = torch.tanh(h1 @ p[2].reshape(W, W).T + p[3])
    return p, h2 @ p[4] + p[5]


def _scenario(case, seed):
    """Spectra of one training scenario of the surrogate (as ``synth.surrogate_group``)."""
    rng = np.random.default_rng(30_000 + int(seed))
    nk, nh, a = case["n_kbins"], case["n_hist"], case["a"]
    w = synth.Workload("scenario", 32, 32, 1000.0, case["m_nu"], N_SPECIES, nh, nk, "fp64")
    kb = synth.surrogate_kbins(nk)
    p = np.sqrt(synth.linear_power(kb, w))
    a_hist = A_INIT * (a / A_INIT) ** (np.arange(nh) / max(nh, 1))
    v = (np.log(a_hist) - math.log(A_INIT)) / (math.log(a) - math.log(A_INIT))
    e0, e1 = rng.uniform(-0.08, 0.08, size=2)
    D = np.array([synth.growth(x, w.omega_m)[0] for x in a_hist])
    eps = e0 + e1 * np.tanh(np.log(kb / 0.1))
    hist = np.ascontiguousarray(D[:, None] * p[None, :] * (1.0 + eps[None, :] * np.sin(np.pi * v)[:, None]))
    cur = p * synth.growth(a, w.omega_m)[0] * (1.0 + 0.02 * rng.normal(size=nk))
    return w, kb, cur ** 2, a_hist, hist, synth.nu_initial_at(kb, w)


def _exact_kick(b, case, seed, prev=None):
    """(acc [3, np] FP64, R, P_nu^{1/2}, P_M^{1/2}) of the box at its positions."""
    w, dev = b["w"], b["pos"].device
    n, L, np_, nk = w.ngrid, w.box, b["pos"].shape[1], w.n_kbins
    if w.precision == "fp64":
        def cells(d):
            u = b["pos"][d] / (L / n)
            c = torch.floor(u)
            return torch.remainder(c.long(), n), torch.floor((u - c) * 65536.0).long()
    else:
        def cells(d):
            return torch.remainder(b["pos"][d].long(), n), torch.floor(b["pos"][3 + d].view(torch.float32) * 65536.0).long()
    F = torch.zeros(n ** 3, dtype=torch.int64, device=dev)
    step = 1 << 24

    def corners(lo, hi, fn):
        cw = [(c[lo:hi], q[lo:hi]) for c, q in axes]
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    idx = torch.zeros_like(cw[0][0])
                    wt = torch.ones_like(idx)
                    for (c, q), d in zip(cw[::-1], (dz, dy, dx)):
                        idx = idx * n + torch.where(c + d == n, torch.zeros_like(c), c + d)
                        wt = wt * (q if d else 65536 - q)
                    fn(idx, wt)

    axes = [cells(d) for d in range(3)]
    if np_ > step:
        axes = [(c.int(), q.int()) for c, q in axes]
    for lo in range(0, np_, step):
        hi = min(np_, lo + step)
        axes_l = axes
        axes = [(c[lo:hi].long(), q[lo:hi].long()) for c, q in axes_l]
        corners(0, hi - lo, lambda i, t: F.index_add_(0, i, t))
        axes = axes_l
    delta = F.double().mul_(n ** 3 / (np_ * 2.0 ** 48)).sub_(1.0).reshape(n, n, n)
    del F
    dk = torch.fft.rfftn(delta)
    del delta
    # bins by integer n^2
    f = torch.fft.fftfreq(n, d=1.0 / n, device=dev, dtype=torch.float64).round().long()
    x = torch.arange(n // 2 + 1, device=dev)
    n2max = 3 * (n // 2) ** 2
    r = math.sqrt(3.0) * n / 2.0 * (1.0 + 1e-12)
    thr = np.array([math.ceil(r ** (2.0 * i / nk)) for i in range(nk + 1)])
    hp = torch.zeros(n2max + 1, dtype=torch.float64, device=dev)
    hc = torch.zeros_like(hp)
    wx = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device=dev)
    wx[0] = wx[-1] = 1.0
    plane = (f[:, None] ** 2 + x[None, :] ** 2).reshape(-1)
    wxy = wx[None, :].expand(n, -1).reshape(-1)
    for z in range(n):
        i = plane + f[z] ** 2
        d = torch.view_as_real(dk[z]).square().sum(-1).reshape(-1)
        hp.index_add_(0, i, wxy * d)
        hc.index_add_(0, i, wxy)
    hp, hc = hp.cpu().numpy(), hc.cpu().numpy()
    kf = 2 * math.pi / L
    n2 = np.arange(n2max + 1, dtype=np.float64)
    which = np.searchsorted(thr, np.arange(n2max + 1), side="right") - 1
    ok = (which >= 0) & (which < nk) & (n2 > 0)
    cnt, ks, ps = (np.bincount(which[ok], weights=v[ok], minlength=nk)[:nk] for v in (hc, hc * kf * np.sqrt(n2), hp))
    ne = cnt > 0
    kb, pcdm = ks[ne] / cnt[ne], np.sqrt(ps[ne] / cnt[ne] * L ** 3 / float(n) ** 6)
    pi, ti = b["tables"][2][:, ne], b["tables"][3][:, ne]
    a_hist, hist = b["tables"][0], b["tables"][1][:, ne]
    if case.get("response") == "mlp" and w.m_nu_total > 0:
        theta, mu, sig, ym, ys = _mlp_numbers(seed)
        X = torch.from_numpy(_features(kb, pcdm, b["a"], w.m_nu_total, w.omega_nu, a_hist, hist)).to(dev)
        _, out = _net(theta, (mu, sig, ym, ys), X, dev)
        R = np.exp(float(ym) + float(ys) * out.detach().cpu().numpy())
        f_nu = w.omega_nu / w.omega_m
        res = (R, R * pcdm, (1 - f_nu) * pcdm + f_nu * R * pcdm)
    else:
        res = _response(kb, pcdm, b["a"], w.m_nu_total, w.omega_m, w.omega_nu, a_hist, hist, pi, ti,
                        None if prev is None else prev[ne])
    full = [np.zeros(nk) for _ in range(3)]
    for v, q in zip(full, res):
        v[ne] = q
    # Poisson with the neutrino factor, R linear in ln k between non-empty bins
    f_nu = w.omega_nu / w.omega_m
    with np.errstate(divide="ignore"):
        lk = np.log(kf * np.sqrt(n2))
    fac = np.full(n2max + 1, 1 - f_nu)
    if w.m_nu_total > 0:
        fac += f_nu * np.interp(lk, np.log(kb), res[0])
    G = np.zeros(n2max + 1)
    G[1:] = -1.5 * w.omega_m / (b["a"] * kf * kf) * fac[1:] / n2[1:]
    G = torch.from_numpy(G).to(dev)
    win = torch.ones(n, dtype=torch.float64, device=dev)
    if case.get("deconv"):
        win = torch.special.sinc(f.double() / n) ** -4
    wp = (win[:, None] * win[:n // 2 + 1][None, :]).reshape(n, -1)
    for z in range(n):
        dk[z] *= G[plane + f[z] ** 2].reshape(n, -1) * wp * win[z]
    phi = torch.fft.irfftn(dk, s=(n, n, n))
    del dk
    acc = torch.empty((3, np_), dtype=torch.float64, device=dev)
    for d in range(3):
        ax = 2 - d
        g = torch.roll(phi, 1, ax).sub_(torch.roll(phi, -1, ax)).mul_(8.0)
        g += torch.roll(phi, -2, ax)
        g -= torch.roll(phi, 2, ax)
        g = g.mul_(1.0 / (12.0 * L / n)).reshape(-1)      # -S phi
        for lo in range(0, np_, step):
            hi = min(np_, lo + step)
            axes_l = axes
            axes = [(c[lo:hi].long(), q[lo:hi].long()) for c, q in axes_l]
            s = torch.zeros(hi - lo, dtype=torch.float64, device=dev)
            corners(0, hi - lo, lambda i, t: s.add_(g[i] * (t.double() * 2.0 ** -48)))
            acc[d, lo:hi] = s
            axes = axes_l
    return acc, full


def _exact_box(case, w, npart, seed):
    pos64, vel64 = _particles(w, npart, seed)
    fp64 = w.precision == "fp64"
    return {"w": w, "pos": pos64 if fp64 else _cell_offset(pos64, w.box, w.ngrid),
            "vel": vel64 if fp64 else vel64.float().double(), "a": w.a_kick, "tables": _tables(w)}


def _factor(a0, a1, om, power):
    return float(_integral(lambda u: np.exp(power * u) / _hubble(np.exp(u), om), math.log(a0), math.log(a1), 4))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mlp_grad", "mlp_fwd"):
        X, y = _mlp_rows(case, seed)
        theta, mu, sig, ym, ys = _mlp_numbers(seed)
        p, out = _net(theta, (mu, sig, ym, ys), X, X.device)
        if kind == "mlp_fwd":
            return {"lnR": float(ym) + float(ys) * out.detach()}
        loss = (out - (y.double() - float(ym)) / float(ys)).square().mean()
        return {"grad": torch.cat(torch.autograd.grad(loss, p)), "loss": loss.detach().reshape(1)}
    if kind == "response":
        w, kb, power, a_hist, hist, (pi, ti) = _scenario(case, seed)
        pcdm = np.sqrt(power)
        R, pnu, pmm = _response(kb, pcdm, case["a"], w.m_nu_total, w.omega_m, w.omega_nu, a_hist, hist, pi, ti)
        X = _features(kb, pcdm, case["a"], w.m_nu_total, w.omega_nu, a_hist, hist)
        return {"ratio": R, "sqrtPnu": pnu, "sqrtPM": pmm, "X": X}
    if kind in ("batch", "graph"):
        out = {}
        for i, (n, L, m_nu) in enumerate(_members(case)):
            w = _workload(case, n, n ** 3, L, m_nu)
            b = _exact_box(case, w, n ** 3, 1000 * int(seed) + i)
            acc, _ = _exact_kick(b, case, seed)
            out["vel%d" % i] = b["vel"] + acc * _factor(A_KICK, 1.01 * A_KICK, w.omega_m, 0)
        return out
    w = _workload(case, case["ngrid"], case["npart"], case["box"], case["m_nu"], case["precision"],
                  case.get("clustered", False))
    b = _exact_box(case, w, case["npart"], seed)
    if kind == "step":
        a0, h, prev = A_KICK, math.sqrt(1.01), None
        a_hist, hist, pi, ti = b["tables"]
        for a in (a0, 1.01 * a0):
            b["a"], b["tables"] = a, (a_hist, hist, pi, ti)
            acc, (R, pnu, pmm) = _exact_kick(b, case, seed, prev)
            b["vel"] = b["vel"] + acc * _factor(a / h, a * h, w.omega_m, 0)
            q = torch.remainder(b["pos"] + b["vel"] * _factor(a, 1.01 * a, w.omega_m, -2), w.box)
            b["pos"] = torch.where(q >= w.box, torch.zeros_like(q), q)
            a_hist, hist, prev = np.append(a_hist, a), np.vstack([hist, pmm[None, :]]), pnu
        return {"pos": b["pos"], "vel": b["vel"]}
    acc, (R, pnu, pmm) = _exact_kick(b, case, seed)
    out = {"vel": b["vel"] + acc * _factor(A_KICK, 1.01 * A_KICK, w.omega_m, 0)}
    if case["acc"]:
        out["acc"] = acc
    if case["precision"] == "fp64":
        out["ratio"], out["sqrtPM"] = R, pmm
    return out
