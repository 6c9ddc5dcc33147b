"""The workloads whose speed this library is measured by: ensembles of orbits taken
through the public entry points, from initial conditions in hand to the state and the
indicators a user reads, and the early-stop surrogate's decision and training step.

Every case is one kind of call sequence with its sizes.  `prepare` makes what a program
holds before the call (system handles, initial conditions, buffers), `run` is one pass,
`exact` is the same pass in plain float64 torch.

Two quantities are left out of the compared outputs because they are differences at
rounding level, of which no digits can be compared: `dh_max` (|H - H0|, about 1e-10 of H)
and, for adaptive runs, the proposal for the step after t_final.  For the FP32 frame the
frame itself is compared (float32), and labels, not SALI/GALI widened to float64."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_00622_gb300 import chs
from paper_2507_00622_gb300.surrogate import Surrogate

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)

# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------


def listed():
    return [
        # the library's main workload: a Henon-Heiles section grid at the escape energy with
        # SALI, GALI_2..4 and LD indicators per cell (RK4, FP64); one stretch of the long run
        dict(name="hh_grid_1024_k4_ld", kind="grid", E=1 / 6, ny=1024, npy=1024, k=4, ld=True, integrator="rk4",
             dt=0.01, steps=200, launch="batch"),
        # the smallest call: the 32 x 32 grid at E = 1/8 with two vectors and the LD, to t = 20;
        # the ensemble is far below the GPU's width, so the time of one step counts
        dict(name="hh_grid_32_k2_ld", kind="grid", E=1 / 8, ny=32, npy=32, k=2, ld=True, integrator="rk4",
             dt=0.01, steps=2000, launch="batch"),
        # the classification form: FP32 vector frame, early exit on, compacted chunks (CUDA graph)
        dict(name="hh_grid_512_frame32", kind="frame", model="hh", E=1 / 8, ny=512, npy=512, k=2, ld=True,
             dt=0.01, steps=500, chunk=250),
        # quartic oscillators on energy shells, GALI_2..6, FP32 frame, uneven end steps
        dict(name="quartic_k6_frame32", kind="frame", model="quartic", n=262144, k=6, ld=False, dt=0.01, steps=300,
             chunk=150),
        # FPUT Lyapunov spectra of five chain lengths in one call, QR every 10 steps
        dict(name="fput_lyap_mixed", kind="fput_lyap", Ns="4,8,16,32,64", n=1024, integrator="rk4", dt=0.05,
             steps=100, qr=10),
        # the FPU experiment: GALI_4 of 1e3 chains with adaptive DOP 8(5) at tolerance 1e-8
        dict(name="fput_gali4_adaptive_N32", kind="fput_adaptive", N=32, n=1000, k=4, tol=1e-8, t_final=50.0),
        # the saturation experiment: SALI of a Henon-Heiles grid with adaptive DOP 8(5)
        dict(name="hh_sali_adaptive_64", kind="hh_adaptive", E=1 / 8, ny=64, npy=64, k=2, tol=1e-8, t_final=60.0),
        # fixed-step DOP 8 on a section grid, GALI_2..4 and LD
        dict(name="hh_grid_256_dop853", kind="grid", E=1 / 8, ny=256, npy=256, k=4, ld=True, integrator="dop853",
             dt=0.1, steps=60, launch="batch"),
        # FPUT Lyapunov spectra with DOP 8 (ragged orbit count)
        dict(name="fput_lyap_dop853_N16", kind="fput_lyap", Ns="16", n=2047, integrator="dop853", dt=0.05, steps=40,
             qr=10),
        # Lyapunov spectra over a Henon-Heiles grid
        dict(name="hh_lyap_128", kind="hh_lyap", E=1 / 8, ny=128, npy=128, integrator="rk4", dt=0.01, steps=500, qr=10),
        # the surrogate's decision for the orbits of a large grid
        dict(name="surrogate_decide_512k", kind="decide", n=524288),
        # one training step of the surrogate at its usual batch size
        dict(name="surrogate_train_4096", kind="train", n=4096),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (sizes over their logarithm, odd ones among them)."""
    kind = rng.choice(["grid", "grid", "grid", "frame", "frame", "fput_lyap", "fput_lyap", "fput_adaptive",
                       "hh_adaptive", "hh_lyap", "decide", "train"])
    E = round(rng.uniform(0.10, 0.166), 4)
    if kind == "grid":
        dop = rng.random() < 0.4
        ny, npy = _logint(rng, 20, 400 if dop else 1000), _logint(rng, 20, 400 if dop else 1000)
        steps = min(_logint(rng, 20, 120) if dop else _logint(rng, 100, 2000),
                    max(10, int((6e6 if dop else 1.2e8) / (ny * npy))))
        return dict(kind="grid", E=E, ny=ny, npy=npy, k=rng.choice([2, 2, 3, 4]), ld=rng.random() < 0.6,
                    integrator="dop853" if dop else "rk4", dt=0.1 if dop else 0.01, steps=steps,
                    launch=rng.choice(["batch", "batch", "compacted", "persistent"]))
    if kind == "frame":
        if rng.random() < 0.5:
            ny, npy = _logint(rng, 64, 768), _logint(rng, 64, 768)
            steps = min(_logint(rng, 100, 600), max(50, int(1.2e8 / (ny * npy))))
            return dict(kind="frame", model="hh", E=E, ny=ny, npy=npy, k=rng.choice([2, 2, 3, 4]),
                        ld=rng.random() < 0.7, dt=0.01, steps=steps, chunk=rng.choice([100, 250, 500]))
        n = _logint(rng, 3000, 300000)
        return dict(kind="frame", model="quartic", n=n, k=rng.choice([3, 4, 5, 6]), ld=False, dt=0.01,
                    steps=min(_logint(rng, 100, 400), max(50, int(6e7 / n))), chunk=rng.choice([100, 150]))
    if kind == "fput_lyap":
        Ns = rng.choice(["4", "8", "16", "32", "64", "4,16", "8,32", "16,64"])
        big = max(int(v) for v in Ns.split(","))
        dop = "," not in Ns and rng.random() < 0.4
        n = _logint(rng, 60, min(4096, 400000 // big ** 2 * (1 if dop else 4)))
        return dict(kind="fput_lyap", Ns=Ns, n=n, integrator="dop853" if dop else "rk4", dt=0.05,
                    steps=_logint(rng, 20, 40 if dop else 100), qr=rng.choice([5, 10, 20]))
    if kind == "fput_adaptive":
        N = rng.choice([4, 8, 16, 32, 64])
        return dict(kind="fput_adaptive", N=N, n=_logint(rng, 100, 1100), k=rng.choice([2, 3, 4, 5]), tol=1e-8,
                    t_final=round(rng.uniform(15.0, 50.0 if N < 64 else 25.0), 2))
    if kind == "hh_adaptive":
        return dict(kind="hh_adaptive", E=E, ny=_logint(rng, 10, 72), npy=_logint(rng, 10, 72), k=rng.choice([2, 2, 4]),
                    tol=1e-8, t_final=round(rng.uniform(20.0, 60.0), 2))
    if kind == "hh_lyap":
        dop = rng.random() < 0.3
        return dict(kind="hh_lyap", E=E, ny=_logint(rng, 16, 160), npy=_logint(rng, 16, 160),
                    integrator="dop853" if dop else "rk4", dt=0.1 if dop else 0.01,
                    steps=_logint(rng, 30, 60) if dop else _logint(rng, 100, 600), qr=rng.choice([5, 10, 20]))
    if kind == "decide":
        return dict(kind="decide", n=_logint(rng, 1000, 1000000))
    return dict(kind="train", n=_logint(rng, 500, 16384))


# ----------------------------------------------------------------------------
# inputs, from the seed alone
# ----------------------------------------------------------------------------


def _section(case, seed):
    """Initial conditions on the x = 0 section: cell-centred ny x npy grid, p_x from the
    energy; cells without one are FORBIDDEN (1).  The energy moves a little with the seed."""
    E = case["E"] - 1e-3 * np.random.default_rng(seed).random()
    r = np.roots([-1 / 3, 0.5, 0.0, -E])
    r = np.sort(r[np.abs(r.imag) < 1e-9].real)
    y0, y1, pm = r[r < 0].max(), r[r > 0].min(), math.sqrt(2 * E)
    ny, npy = case["ny"], case["npy"]
    y = (y0 + (torch.arange(ny, **F64) + 0.5) * ((y1 - y0) / ny)).repeat_interleave(npy)
    p = (-pm + (torch.arange(npy, **F64) + 0.5) * (2 * pm / npy)).repeat(ny)
    rad = 2 * E - p * p - y * y + 2 * y ** 3 / 3
    ics = torch.stack([torch.zeros_like(y), y, rad.clamp(min=0).sqrt(), p])
    bad = rad < 0
    ics[:, bad] = float("nan")
    return ics.contiguous(), bad.to(torch.int32)


def _shell(case, seed):
    """Quartic-3 states on shells E in [1, 10] (eps = 0.1), radially scaled directions."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]
    u = torch.randn((6, n), generator=g, **F64)
    E = 1 + 9 * torch.rand(n, generator=g, **F64)
    u /= u.norm(dim=0)
    s = u[:3] ** 2
    h2, h4 = 0.5 * (u * u).sum(0), 0.1 * (s[0] * s[1] + s[1] * s[2] + s[0] * s[2])
    return (u * (2 * E / (h2 + (h2 * h2 + 4 * h4 * E).sqrt())).sqrt()).contiguous()


def _chain(N, n, seed):
    """FPUT-beta chains: random normal modes scaled to energy density 0.1."""
    g = torch.Generator(device=DEV).manual_seed(seed * 131 + N)
    i = torch.arange(1, N + 1, **F64)
    S = math.sqrt(2 / (N + 1)) * torch.sin(i[:, None] * i[None, :] * (math.pi / (N + 1)))
    q, p = (S @ torch.randn((N, n), generator=g, **F64) for _ in range(2))
    z = torch.zeros((1, n), **F64)
    r = torch.diff(torch.cat([z, q, z]), dim=0)
    h2, h4, E = 0.5 * (p * p).sum(0) + 0.5 * (r * r).sum(0), 0.25 * (r ** 4).sum(0), 0.1 * N
    return (torch.cat([q, p]) * (2 * E / (h2 + (h2 * h2 + 4 * h4 * E).sqrt())).sqrt()).contiguous()


def _early_samples(n, seed):
    """SALI samples, LD and energies of orbits at t = 500: regular ones keep SALI of order
    one, chaotic ones lose it exponentially from some time on."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    t = torch.arange(1, 11, **F64)[:, None] * 50.0
    chaotic = torch.rand(n, generator=g, **F64) < 0.45
    onset = 500 * torch.rand(n, generator=g, **F64)
    rate = 0.02 + 0.08 * torch.rand(n, generator=g, **F64)
    base = torch.log10(0.02 + 1.38 * torch.rand((10, n), generator=g, **F64))
    series = 10.0 ** (base - torch.where(chaotic, rate * (t - onset).clamp(min=0), 0.3 * torch.log10(t)))
    E = 0.10 + 0.066 * torch.rand(n, generator=g, **F64)
    ld = 500.0 * (1.55 + 2.0 * (E - 0.13) + 0.05 * torch.randn(n, generator=g, **F64))
    return series.contiguous(), ld, E, chaotic


def _train_batch(n, seed):
    """A training batch: standardised features, labels and final log10(SALI) / 8, and Adam moments of
    a run that is under way."""
    series, ld, E, chaotic = _early_samples(n, seed)
    X = torch.cat([series.clamp(min=1e-20).log10() / 8, (ld / 500 - 1)[None], ((E - 0.133) / 0.033)[None]])
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    P = 34946
    m = 1e-3 * torch.randn(P, generator=g, device=DEV)
    v = 1e-6 * (0.5 + torch.rand(P, generator=g, device=DEV))
    target = torch.where(chaotic, -1.5 + 0.3 * torch.rand(n, generator=g, **F64), X[9]).float()
    return X.float().contiguous(), chaotic.float(), target, m, v


# ----------------------------------------------------------------------------
# prepare
# ----------------------------------------------------------------------------

_INTEG = {"rk4": chs.RK4, "dop853": chs.DOP853}


def _seed_of(seed):
    return (seed * 2654435761 + 1) % (1 << 62)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("grid", "hh_adaptive", "hh_lyap") or case.get("model") == "hh":
        s["sys"] = chs.System(chs.HENON_HEILES, 2)
        s["ics"], s["st"] = _section(case, seed)
    elif kind == "frame":
        s["sys"] = chs.System(chs.QUARTIC3, 3, (0.1,))
        s["ics"], s["st"] = _shell(case, seed), None
    elif kind == "fput_adaptive":
        s["sys"] = chs.System(chs.FPUT, case["N"], (1.0, 0.0, 1.0))
        s["ics"], s["st"] = _chain(case["N"], case["n"], seed), None

    if kind in ("grid", "frame", "hh_adaptive", "fput_adaptive"):
        d, n, k = s["ics"].shape[0], s["ics"].shape[1], case["k"]
        frame, ld = kind == "frame", case.get("ld", False)
        s["ens"] = chs.DeviceEnsemble.empty(n, d, k, vec_fp32=frame)
        s["label"] = torch.empty(n, dtype=torch.int8, device=DEV)
        s["par"] = dict(n_dev=k, ld_p=0.5 if ld else 0.0, escape_r2=4.0 if d == 4 else 0.0, seed=_seed_of(seed),
                        sali_threshold=1e-8)
        t_end = None
        if frame:
            s["par"].update(vec_precision=chs.VEC_FP32, early_exit=True)
            if case["model"] == "quartic":
                g = torch.Generator(device=DEV).manual_seed(seed + 2)
                t_end = torch.randint(case["steps"] // 2, 2 * case["steps"], (n,), generator=g, device=DEV)
        else:
            s["sali"] = torch.empty(n, **F64)
            s["gali"] = torch.empty((k - 1, n), **F64)
            if kind == "grid" and ld:
                s["ldi"] = torch.empty((2, n), **F64)
        s["t_end"] = t_end
        s["abi"] = s["ens"].abi(with_ld=ld, t_end=t_end)
        if frame or case.get("launch") in ("compacted", "persistent"):
            s["work"] = chs.compact_work(n)
    if kind in ("hh_adaptive", "fput_adaptive"):
        s["par"]["integrator"] = chs.DOP853
        s["t"], s["h"] = torch.empty(n, **F64), torch.empty(n, **F64)
        s["rej"] = torch.empty(n, dtype=torch.int64, device=DEV)
    if kind == "hh_lyap":
        n = s["ics"].shape[1]
        s["lam"], s["sto"] = torch.empty((4, n), **F64), torch.empty(n, dtype=torch.int32, device=DEV)
    if kind == "fput_lyap":
        s["jobs"] = []
        for N in (int(v) for v in case["Ns"].split(",")):
            S = chs.System(chs.FPUT, N, (1.0, 0.0, 1.0))
            ics = _chain(N, case["n"], seed)
            lam = torch.empty((2 * N, case["n"]), **F64)
            sto = torch.empty(case["n"], dtype=torch.int32, device=DEV)
            s["jobs"].append((S, chs.params(case["dt"], case["steps"], qr_every=case["qr"],
                                            integrator=_INTEG[case["integrator"]]), ics, lam, sto))
    if kind == "decide":
        s["net"] = Surrogate.load()
        s["series"], s["ldv"], s["Ev"], _ = _early_samples(case["n"], seed)
        s["st0"] = (torch.rand(case["n"], generator=torch.Generator(device=DEV).manual_seed(seed + 3), device=DEV)
                    < 0.3).to(torch.int32) * chs.ORBIT_EARLY_CHAOTIC
        s["status"] = torch.empty_like(s["st0"])
        s["prob"] = torch.empty(case["n"], device=DEV)
    if kind == "train":
        n = case["n"]
        s["net"] = Surrogate.load()
        s["X"], s["lab"], s["tgt"], s["m"], s["v"] = _train_batch(n, seed)
        s["Y"], s["dY"] = torch.empty((2, n), device=DEV), torch.empty((2, n), device=DEV)
        s["act"] = torch.empty((3, 128, n), dtype=torch.bfloat16, device=DEV)
        s["loss"], s["delta"] = torch.empty(1, device=DEV), torch.empty((3, 128, n), device=DEV)
        s["G"] = torch.empty(34946, device=DEV)
    return s


# ----------------------------------------------------------------------------
# run
# ----------------------------------------------------------------------------


def run(s):
    return _RUN[s["case"]["kind"]](s, s["case"])


def _run_grid(s, c):
    h, ens, abi = s["sys"].h, s["ens"], s["abi"]
    prm = chs.params(c["dt"], c["steps"], integrator=_INTEG[c["integrator"]], **s["par"])
    chs.chs_ensemble_init(h, prm, abi, s["ics"], s["st"])
    if c["launch"] == "compacted":
        chs.chs_integrate_compacted(h, prm, abi, 100, s["work"])
    elif c["launch"] == "persistent":
        chs.chs_integrate_persistent(h, prm, abi, s["work"])
    else:
        chs.chs_integrate_batch(h, prm, abi)
    ldi = s.get("ldi")
    chs.chs_indicators(h, prm, abi, c["ny"] if ldi is not None else 0, c["npy"] if ldi is not None else 0, s["sali"],
                       s["gali"], ldi, s["label"])
    out = dict(x=ens.x, w=ens.w, status=ens.status, n_exec=ens.n_exec, sali=s["sali"], gali=s["gali"],
               label=s["label"])
    if ldi is not None:
        out.update(ld=ens.ld, ldi=ldi)
    return out


def _run_frame(s, c):
    h, ens, abi = s["sys"].h, s["ens"], s["abi"]
    prm = chs.params(c["dt"], c["steps"], **s["par"])
    chs.chs_ensemble_init(h, prm, abi, s["ics"], s["st"])
    chs.chs_integrate_compacted(h, prm, abi, c["chunk"], s["work"])
    chs.chs_indicators(h, prm, abi, label=s["label"])
    out = dict(x=ens.x, w=ens.w, status=ens.status, n_exec=ens.n_exec, label=s["label"])
    if c["ld"]:
        out["ld"] = ens.ld
    return out


def _run_adaptive(s, c):
    h, ens, abi = s["sys"].h, s["ens"], s["abi"]
    prm = chs.params(0.05, 1_000_000, **s["par"])
    chs.chs_ensemble_init(h, prm, abi, s["ics"], s["st"])
    s["t"].zero_()
    s["h"].fill_(0.05)
    s["rej"].zero_()
    chs.chs_integrate_adaptive(h, prm, chs.Adaptive(c["t_final"], c["tol"], c["tol"], 0.0), abi, s["t"], s["h"],
                               n_rejected=s["rej"])
    chs.chs_indicators(h, prm, abi, 0, 0, s["sali"], s["gali"], None, s["label"])
    return dict(x=ens.x, w=ens.w, status=ens.status, n_exec=ens.n_exec, n_rejected=s["rej"], t=s["t"], sali=s["sali"],
                gali=s["gali"], label=s["label"])


def _run_hh_lyap(s, c):
    prm = chs.params(c["dt"], c["steps"], qr_every=c["qr"], integrator=_INTEG[c["integrator"]])
    chs.chs_lyapunov_spectrum(s["sys"].h, prm, s["ics"].shape[1], s["ics"], s["st"], s["lam"], s["sto"])
    return dict(lam=s["lam"], status=s["sto"])


def _run_fput_lyap(s, c):
    jobs = s["jobs"]
    if len(jobs) == 1:
        S, prm, ics, lam, sto = jobs[0]
        chs.chs_lyapunov_spectrum(S.h, prm, c["n"], ics, None, lam, sto)
    else:
        chs.chs_lyapunov_batch([(S.h, prm, c["n"], ics, None, lam, sto) for S, prm, ics, lam, sto in jobs])
    return [dict(lam=lam, status=sto) for _, _, _, lam, sto in jobs]


def _run_decide(s, c):
    s["status"].copy_(s["st0"])
    chs.chs_surrogate_decide(s["net"].params, s["series"], 10, s["ldv"], 500.0, s["Ev"], 0.95, c["n"], s["status"],
                             s["prob"])
    return dict(status=s["status"], prob=s["prob"])


def _run_train(s, c):
    net, n = s["net"], c["n"]
    chs.chs_mlp_forward(net.params, s["X"], n, s["Y"], s["act"])
    chs.chs_mlp_loss_grad(s["Y"], s["lab"], s["tgt"], n, 0.25, s["dY"], s["loss"])
    chs.chs_mlp_backward(net.params, s["X"], s["act"], s["dY"], n, s["delta"], s["G"])
    chs.chs_mlp_adam(net.master, s["m"], s["v"], s["G"], 1e-3, 0.9, 0.999, 1e-8, 500, net.params)
    return dict(Y=s["Y"], loss=s["loss"], grad=s["G"], master=net.master, m=s["m"], v=s["v"], params=net.params)


_RUN = dict(grid=_run_grid, frame=_run_frame, fput_adaptive=_run_adaptive, hh_adaptive=_run_adaptive,
            hh_lyap=_run_hh_lyap, fput_lyap=_run_fput_lyap, decide=_run_decide, train=_run_train)


# ----------------------------------------------------------------------------
# work: what the path cannot do without
# ----------------------------------------------------------------------------


def _step_flops(N, k, stages, hess, force, ld):
    """A step of an s-stage method on orbit, k vectors and LD: per stage the force, k Hessian products
    and the LD's 2N roots, and a stage update of every component."""
    return stages * (force + k * hess + (4 * N if ld else 0)) + (1 + k) * 2 * N * 4 * stages


def work(case):
    kind = case["kind"]
    if kind in ("decide", "train"):
        n, mac = case["n"], 12 * 128 + 2 * 128 * 128 + 256
        if kind == "decide":
            return {"bytes": n * (10 * 8 + 16 + 12) + 70e3, "flops": 2.0 * mac * n}
        return {"bytes": n * (12 * 4 + 8 + 8) + 34946 * 30, "flops": 6.0 * mac * n}
    n = case["n"] if "n" in case else case["ny"] * case["npy"]
    stages = 12 if case.get("integrator") == "dop853" or "adaptive" in kind else 4
    if kind == "fput_lyap":
        b = f = 0.0
        for N in (int(v) for v in case["Ns"].split(",")):
            d = 2 * N
            b += n * (16.0 * d + 4)
            f += n * case["steps"] * (_step_flops(N, d, stages, 5 * N, 10 * N, False) + 2.0 * d * d * d / case["qr"])
        return {"bytes": b, "flops": f}
    N = case["N"] if "N" in case else 3 if case.get("model") == "quartic" else 2
    valid = n if N != 2 else 0.75 * n  # about a quarter of a section grid is FORBIDDEN
    hess, force = (5 * N, 10 * N) if N > 3 else (2 * N * N, 12 if N == 3 else 7)
    if kind == "hh_lyap":
        return {"bytes": n * (64.0 + 8), "flops": valid * case["steps"] * (_step_flops(2, 4, stages, hess, force, False)
                                                                           + 128 / case["qr"])}
    k = case["k"]
    steps = case["steps"] if "steps" in case else case["t_final"] / (0.25 if N > 3 else 0.6)
    vec = 4 * (2 * N * k + k * (k + 1) / 2) if kind == "frame" else 16 * N * k
    out = 16 * N + vec + 13 + (8 if case.get("ld") else 0) + (8 * k if kind != "frame" else 0)
    return {"bytes": n * (16.0 * N + out), "flops": valid * steps * _step_flops(N, k, stages, hess, force,
                                                                               case.get("ld", False))}


# ----------------------------------------------------------------------------
# exact: the same in plain float64 torch
# ----------------------------------------------------------------------------

_RK4 = ([[], [0.5], [0, 0.5], [0, 0, 1.0]], [1 / 6, 1 / 3, 1 / 3, 1 / 6], None, None)
# DOP853, Hairer, Norsett & Wanner, Solving ODEs I, 2nd ed., Sec. II.10
_DOP = (
    [[], [5.26001519587677318785587544488e-2], [1.97250569845378994544595329183e-2, 5.91751709536136983633785987549e-2],
     [2.95875854768068491816892993775e-2, 0, 8.87627564304205475450678981324e-2],
     [2.41365134159266685502369798665e-1, 0, -8.84549479328286085344864962717e-1, 9.24834003261792003115737966543e-1],
     [3.7037037037037037037037037037e-2, 0, 0, 1.70828608729473871279604482173e-1, 1.25467687566822425016691814123e-1],
     [3.7109375e-2, 0, 0, 1.70252211019544039314978060272e-1, 6.02165389804559606850219397283e-2, -1.7578125e-2],
     [3.70920001185047927108779319836e-2, 0, 0, 1.70383925712239993810214054705e-1, 1.07262030446373284651809199168e-1,
      -1.53194377486244017527936158236e-2, 8.27378916381402288758473766002e-3],
     [6.24110958716075717114429577812e-1, 0, 0, -3.36089262944694129406857109825e0, -8.68219346841726006818189891453e-1,
      2.75920996994467083049415600797e1, 2.01540675504778934086186788979e1, -4.34898841810699588477366255144e1],
     [4.77662536438264365890433908527e-1, 0, 0, -2.48811461997166764192642586468e0, -5.90290826836842996371446475743e-1,
      2.12300514481811942347288949897e1, 1.52792336328824235832596922938e1, -3.32882109689848629194453265587e1,
      -2.03312017085086261358222928593e-2],
     [-9.3714243008598732571704021658e-1, 0, 0, 5.18637242884406370830023853209e0, 1.09143734899672957818500254654e0,
      -8.14978701074692612513997267357e0, -1.85200656599969598641566180701e1, 2.27394870993505042818970056734e1,
      2.49360555267965238987089396762e0, -3.0467644718982195003823669022e0],
     [2.27331014751653820792359768449e0, 0, 0, -1.05344954667372501984066689879e1, -2.00087205822486249909675718444e0,
      -1.79589318631187989172765950534e1, 2.79488845294199600508499808837e1, -2.85899827713502369474065508674e0,
      -8.87285693353062954433549289258e0, 1.23605671757943030647266201528e1, 6.43392746015763530355970484046e-1]],
    [5.42937341165687622380535766363e-2, 0, 0, 0, 0, 4.45031289275240888144113950566e0, 1.89151789931450038304281599044e0,
     -5.8012039600105847814672114227e0, 3.1116436695781989440891606237e-1, -1.52160949662516078556178806805e-1,
     2.01365400804030348374776537501e-1, 4.47106157277725905176885569043e-2],
    [1.312004499419488073250102996e-2, 0, 0, 0, 0, -1.225156446376204440720569753e0, -4.957589496572501915214079952e-1,
     1.664377182454986536961530415e0, -3.503288487499736816886487290e-1, 3.341791187130174790297318841e-1,
     8.192320648511571246570742613e-2, -2.235530786388629525884427845e-2],
    [2.44094488188976377952755905512e-1, 0, 0, 0, 0, 0, 0, 0, 7.33846688281611857341361741547e-1, 0, 0,
     2.20588235294117647058823529412e-2])


def _force(model, q):
    if model == "hh":
        return torch.stack([-q[0] * (1 + 2 * q[1]), -q[1] - q[0] * q[0] + q[1] * q[1]])
    if model == "quartic":
        s = q * q
        return -q * (1 + 0.2 * (s.sum(0) - s))
    z = torch.zeros_like(q[:1])
    r = torch.diff(torch.cat([z, q, z]), dim=0)
    return torch.diff(r + r ** 3, dim=0)


def _minus_hess(model, q, u):
    """-Hess V(q) u for vectors u [k, N, n]."""
    if model == "hh":
        return torch.stack([-(1 + 2 * q[1]) * u[:, 0] - 2 * q[0] * u[:, 1],
                            -2 * q[0] * u[:, 0] - (1 - 2 * q[1]) * u[:, 1]], 1)
    if model == "quartic":
        s, qu = q * q, (q[None] * u).sum(1, keepdim=True)
        return -(1 + 0.2 * (s.sum(0) - s))[None] * u - 0.4 * q[None] * (qu - q[None] * u)
    z, zu = torch.zeros_like(q[:1]), torch.zeros_like(u[:, :1])
    r = torch.diff(torch.cat([z, q, z]), dim=0)
    return torch.diff((1 + 3 * r * r)[None] * torch.diff(torch.cat([zu, u, zu], 1), dim=1), dim=1)


def _comb(coef, K):
    acc = None
    for c, v in zip(coef, K):
        if c != 0:
            acc = c * v if acc is None else acc.add_(v, alpha=c)
    return acc


def _step(model, tab, x, W, h, ld=False):
    """One Runge-Kutta step of orbit x [2N, n] and vectors W [k, 2N, n] with step h (a number or [n]):
    new x, new W, LD increment, stage derivatives of the orbit."""
    N = x.shape[0] // 2
    Kx, KW, g = [], [], 0.0
    for row, b in zip(tab[0], tab[1]):
        xs = x if not row else x + h * _comb(row, Kx)
        Ws = W if not row else W + h * _comb(row, KW)
        Kx.append(torch.cat([xs[N:], _force(model, xs[:N])]))
        KW.append(torch.cat([Ws[:, N:], _minus_hess(model, xs[:N], Ws[:, :N])], 1))
        if ld and b != 0:
            g = g + b * Kx[-1].abs().sqrt().sum(0)
    return x + h * _comb(tab[1], Kx), W + h * _comb(tab[1], KW), (h * g if ld else None), Kx


def _unit(W):
    return W / W.norm(dim=1, keepdim=True)


def _seeded(seed, n, k, d):
    """Deviation vectors [k, d, n]: output m = (o k + j) d + c + 1 of the SplitMix64 stream of `seed`,
    top 53 bits to [-1, 1), normalised."""
    def shr(z, b):
        return (z >> b) & ((1 << (64 - b)) - 1)

    def mul(z, c):
        return z * (c - (1 << 64) if c >= 1 << 63 else c)

    o = torch.arange(n, device=DEV)[None, None, :]
    m = (o * k + torch.arange(k, device=DEV)[:, None, None]) * d + torch.arange(d, device=DEV)[None, :, None] + 1
    z = mul(m, 0x9E3779B97F4A7C15) + seed
    z = mul(z ^ shr(z, 30), 0xBF58476D1CE4E5B9)
    z = mul(z ^ shr(z, 27), 0x94D049BB133111EB)
    z = z ^ shr(z, 31)
    return _unit(shr(z, 11).double() * 2.0 ** -52 - 1.0)


def _gram_schmidt(W):
    """Q [k, d, n] and R (list of rows of tensors) of W = Q R, R_jj > 0."""
    Q, R = [], []
    for j in range(W.shape[0]):
        v, r = W[j], []
        for q in Q:
            a = (q * v).sum(0)
            r.append(a)
            v = v - a * q
        nr = v.norm(dim=0)
        R.append(r + [nr])
        Q.append(v / nr)
    return Q, R


def _indicators(W, bad):
    sali = torch.minimum((W[0] + W[1]).norm(dim=0), (W[0] - W[1]).norm(dim=0))
    R = _gram_schmidt(W)[1]
    g, prod = [], R[0][0]
    for j in range(1, len(R)):
        prod = prod * R[j][j]
        g.append(prod)
    sali, gali = sali.clone(), torch.stack(g)
    if bad is not None:
        sali[bad], gali[:, bad] = float("nan"), float("nan")
    return sali, gali


def _ld_indicators(ld, bad, ny, npy):
    L = torch.where(bad, torch.nan, ld).reshape(ny, npy)
    out = torch.full((2, ny, npy), float("nan"), **F64)
    c, u, d, l, r = L[1:-1, 1:-1], L[2:, 1:-1], L[:-2, 1:-1], L[1:-1, :-2], L[1:-1, 2:]
    out[0, 1:-1, 1:-1] = 0.25 * ((u - d).abs() + (r - l).abs()) / c
    out[1, 1:-1, 1:-1] = 0.5 * ((2 - (u + d) / c).abs() + (2 - (r + l) / c).abs())
    return out.reshape(2, -1)


def _start(case, seed, ics, bad):
    k, d, n = case["k"], ics.shape[0], ics.shape[1]
    x = ics if bad is None else torch.where(bad, 0.0, ics)
    return x, _seeded(_seed_of(seed), n, k, d)


def _put_back(x, W, x0, W0, bad):
    if bad is None:
        return x, W
    return torch.where(bad, x0, x), torch.where(bad, W0, W)


def _exact_grid(case, seed):
    ics, st = _section(case, seed)
    bad = st != 0
    x, W = _start(case, seed, ics, bad)
    W0, L = W, torch.zeros(ics.shape[1], **F64)
    tab = _RK4 if case["integrator"] == "rk4" else _DOP
    for _ in range(case["steps"]):
        x, W, dl, _ = _step("hh", tab, x, W, case["dt"], case["ld"])
        W = _unit(W)
        if case["ld"]:
            L = L + dl
    x, W = _put_back(x, W, ics, W0, bad)
    sali, gali = _indicators(W, bad)
    out = dict(x=x, w=W.reshape(-1, W.shape[2]), status=None, n_exec=None, sali=sali, gali=gali, label=None)
    if case["ld"]:
        L = torch.where(bad, 0.0, L)
        out.update(ld=L, ldi=_ld_indicators(L, bad, case["ny"], case["npy"]))
    return out


def _exact_frame(case, seed):
    hh = case["model"] == "hh"
    model = "hh" if hh else "quartic"
    if hh:
        ics, st = _section(case, seed)
        bad = st != 0
    else:
        ics, bad = _shell(case, seed), None
    x, W = _start(case, seed, ics, bad)
    W0, n = W, ics.shape[1]
    L, left = torch.zeros(n, **F64), None
    if not hh:
        g = torch.Generator(device=DEV).manual_seed(seed + 2)
        left = torch.randint(case["steps"] // 2, 2 * case["steps"], (n,), generator=g, device=DEV)
    for i in range(case["steps"]):
        xn, Wn, dl, _ = _step(model, _RK4, x, W, case["dt"], case["ld"])
        Wn = _unit(Wn)
        if left is not None:
            go = left > i
            xn, Wn = torch.where(go, xn, x), torch.where(go, Wn, W)
        x, W = xn, Wn
        if case["ld"]:
            L = L + dl
    x, W = _put_back(x, W, ics, W0, bad)
    Q, R = _gram_schmidt(W)
    w = torch.cat([torch.cat(Q), torch.stack([r for col in R for r in col])])
    out = dict(x=x, w=w, status=None, n_exec=None, label=None)
    if case["ld"]:
        out["ld"] = L if bad is None else torch.where(bad, 0.0, L)
    return out


def _exact_adaptive(case, seed):
    hh = case["kind"] == "hh_adaptive"
    if hh:
        ics, st = _section(case, seed)
        bad = st != 0
    else:
        ics, bad = _chain(case["N"], case["n"], seed), None
    model, T, tol = ("hh" if hh else "fput"), case["t_final"], case["tol"]
    x, W = _start(case, seed, ics, bad)
    W0, (d, n) = W, ics.shape
    t, h = torch.zeros(n, **F64), torch.full((n,), 0.05, **F64)
    rejected = torch.zeros(n, dtype=torch.bool, device=DEV)
    e3c = [b - c for b, c in zip(_DOP[1], _DOP[3])]
    for i in range(100000):
        act = t < T
        if i % 16 == 0 and not bool(act.any()):
            break
        tn = torch.clamp(t + h, max=T)
        hh_ = torch.where(act, tn - t, 0.0)
        xn, Wn, _, K = _step(model, _DOP, x, W, hh_)
        sc = tol + tol * torch.maximum(x.abs(), xn.abs())
        E5, E3 = ((_comb(_DOP[2], K) / sc) ** 2).sum(0), ((_comb(e3c, K) / sc) ** 2).sum(0)
        err = hh_ * E5 / (d * (E5 + 0.01 * E3)).sqrt()
        r8 = err ** -0.125
        ok = act & (err < 1)
        grow = torch.clamp(0.9 * r8, max=10.0)
        grow = torch.where(rejected, grow.clamp(max=1.0), grow)
        h = torch.where(act, hh_ * torch.where(ok, grow, (0.9 * r8).clamp(min=0.2)), h)
        x, W, t = torch.where(ok, xn, x), torch.where(ok, _unit(Wn), W), torch.where(ok, tn, t)
        rejected = act & ~ok
    x, W = _put_back(x, W, ics, W0, bad)
    if bad is not None:
        t = torch.where(bad, 0.0, t)
    sali, gali = _indicators(W, bad)
    return dict(x=x, w=W.reshape(-1, n), status=None, n_exec=None, n_rejected=None, t=t, sali=sali, gali=gali, label=None)


def _exact_lyap(model, tab, x, steps, dt, qr):
    d, n = x.shape
    W = torch.eye(d, **F64)[:, :, None].repeat(1, 1, n)
    S = torch.zeros((n, d), **F64)
    for i in range(1, steps + 1):
        x, W, _, _ = _step(model, tab, x, W, dt)
        if i % qr == 0 or i == steps:
            A = W.permute(2, 1, 0)
            C = torch.linalg.cholesky(A.transpose(1, 2) @ A)
            S += C.diagonal(dim1=1, dim2=2).log()
            W = torch.linalg.solve_triangular(C, A.transpose(1, 2), upper=False).permute(1, 2, 0).contiguous()
    return (S / (steps * dt)).t().contiguous()


def _exact_hh_lyap(case, seed):
    ics, st = _section(case, seed)
    bad = st != 0
    lam = _exact_lyap("hh", _RK4 if case["integrator"] == "rk4" else _DOP, torch.where(bad, 0.0, ics), case["steps"],
                      case["dt"], case["qr"])
    lam[:, bad] = float("nan")
    return dict(lam=lam, status=None)


def _exact_fput_lyap(case, seed):
    tab, out = _RK4 if case["integrator"] == "rk4" else _DOP, []
    for N in (int(v) for v in case["Ns"].split(",")):
        x = _chain(N, case["n"], seed)
        part = max(1, int(2e7) // (4 * N * N))  # orbits at a time
        out.append(dict(lam=torch.cat([_exact_lyap("fput", tab, x[:, i:i + part], case["steps"], case["dt"], case["qr"])
                                       for i in range(0, case["n"], part)], 1), status=None))
    return out


def _layers(p):
    o, W = 0, []
    for u, k in ((128, 12), (128, 128), (128, 128), (2, 128)):
        W.append((p[o:o + u * k].reshape(u, k), p[o + u * k:o + u * k + u]))
        o += u * k + u
    return W


def _exact_forward(p, X):
    a = [X]
    for i, (W, b) in enumerate(_layers(p)):
        y = W @ a[-1] + b[:, None]
        a.append(y.clamp(min=0).to(torch.bfloat16).double() if i < 3 else y)
    return a


def _exact_decide(case, seed):
    series, ld, E, _ = _early_samples(case["n"], seed)
    X = torch.cat([series.clamp(min=1e-20).log10() / 8, (ld / 500 - 1)[None], ((E - 0.133) / 0.033)[None]])
    p = _weights().to(torch.bfloat16).double()
    y = _exact_forward(p, X.float().double())[-1]
    return dict(status=None, prob=torch.sigmoid(y[0]))


def _weights():
    import os
    import paper_2507_00622_gb300 as pkg
    with np.load(os.path.join(os.path.dirname(pkg.__file__), "surrogate_weights.npz")) as z:
        return torch.from_numpy(np.asarray(z["params"], dtype=np.float32)).cuda()


def _exact_train(case, seed):
    n = case["n"]
    X, lab, tgt, m, v = (t.double() for t in _train_batch(n, seed))
    master = _weights()
    p = master.to(torch.bfloat16).double()
    a = _exact_forward(p, X)
    y = a[-1]
    loss = (y[0].clamp(min=0) - y[0] * lab + torch.log1p(torch.exp(-y[0].abs())) + 0.25 * (y[1] - tgt) ** 2).mean()
    d = torch.stack([torch.sigmoid(y[0]) - lab, 0.5 * (y[1] - tgt)]) / n
    L, parts = _layers(p), []
    for i in (3, 2, 1, 0):
        parts = [(d @ a[i].t()).reshape(-1), d.sum(1)] + parts
        if i:
            d = (L[i][0].t() @ d) * (a[i] > 0)
    G = torch.cat(parts)
    b1, b2, lr, eps = (float(np.float32(q)) for q in (0.9, 0.999, 1e-3, 1e-8))
    m, v = b1 * m + (1 - b1) * G, b2 * v + (1 - b2) * G * G
    w = master.double() - lr * (m / (1 - b1 ** 500)) / ((v / (1 - b2 ** 500)).sqrt() + eps)
    return dict(Y=y, loss=loss.reshape(1), grad=G, master=w, m=m, v=v, params=w)


_EXACT = dict(grid=_exact_grid, frame=_exact_frame, fput_adaptive=_exact_adaptive, hh_adaptive=_exact_adaptive,
              hh_lyap=_exact_hh_lyap, fput_lyap=_exact_fput_lyap, decide=_exact_decide, train=_exact_train)


def exact(case, seed):
    return _EXACT[case["kind"]](case, seed)
