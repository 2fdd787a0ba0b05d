"""Workloads whose speed is measured: what a user of the simulator has it do, through its
public entry points, from one small instance to the large batched ones.

A case is a dict of plain values.  Its "use" says how the library is called:

  solo     one context: integrate from seeds held on the device, then the Ising energies
  scan     the whole call on host arrays: integrate, energies, figures of merit
  batch    several contexts integrated as one batch
  packed   small graphs packed into the blocks of one context, energies per graph
  xy       the XY machine (D = 2, no annealing) with its best-axis readout
  learned  the learned early exit: snapshot, features, logits, decision pass, gradient

Couplings: "sk" is +-1 on every pair, "gauss" N(0, 1/N), "ladder" the Moebius ladder with
-1 bonds, "sparse" +-1 on a fraction 0.2 of the pairs.  The feedback strength follows from
the couplings' largest eigenvalue in the large-N limit (2 sqrt(N) for "sk", 2 for "gauss").
"""
import math

import numpy as np
import torch

from paper_2308_02329_gb300 import chym, packing

DT, SIGMA, INIT_STD, GAMMA, KAPPA = 0.01, 1e-3, 0.1, 25.0, 0.1
PRECS = {"fp64": chym.PREC_FP64, "fp32": chym.PREC_FP32, "bf16x2": chym.PREC_BF16X2,
         "fp8": chym.PREC_FP8}


def listed():
    return [
        # a first look at one small instance: few runs, few steps, one launch that matters
        dict(name="sk20_short", use="solo", J="sk", N=20, D=3, n_h=8, reps=8, prec="bf16x2", steps=64),
        # the plain method in the oracle-comparison mode: 256 runs of an exactly solvable size
        dict(name="sk20_fp64", use="solo", J="sk", N=20, D=3, n_h=8, reps=32, prec="fp64", steps=1000),
        # the call of the README: one SK instance, a pump scan, energies and figures of merit
        dict(name="sk100_scan", use="scan", J="sk", N=100, D=3, n_h=32, reps=128, prec="bf16x2", steps=2000),
        # the default workload of the benchmark: ladder and SK at D = 2, 3, 4 in one batch
        dict(name="n100_batch", use="batch", J="ladder+sk", N=100, N2=100, n_ctx=6, dims="2,3,4", n_h=32,
             reps=128, prec="bf16x2", steps=1000),
        # the size-scaling study: graphs of N = 10..100 packed, hyperspin machine, energies per graph
        dict(name="scaling_packed", use="packed", J="sparse", N=10, N2=100, n_ctx=30, D=2, n_h=21, reps=32,
             prec="bf16x2", steps=500),
        # a single mid-size instance with real couplings, too few tiles to fill the chip
        dict(name="gauss250", use="solo", J="gauss", N=250, D=3, n_h=16, reps=64, prec="bf16x2", steps=200),
        # large dense instances: +-1 couplings with the FP8 low half, Gaussian ones in BF16 halves
        dict(name="n1000_pair", use="batch", J="sk+gauss", N=1000, N2=1000, n_ctx=2, dims="4", n_h=32, reps=256,
             prec="fp8", steps=64),
        # many uneven instances with few runs each, as one batch
        dict(name="uneven_batch", use="batch", J="sk", N=50, N2=2000, n_ctx=32, dims="2,3,4,8", n_h=16, reps=4,
             prec="fp8", steps=100),
        # the plain FP32 form that the mixed precision is held against
        dict(name="sk100_plain", use="solo", J="sk", N=100, D=4, n_h=32, reps=128, prec="fp32", steps=300),
        # sparse couplings: a long ladder, coupling summed over the nonzeros
        dict(name="ladder2048", use="solo", J="ladder", N=2048, D=3, n_h=32, reps=64, prec="bf16x2", steps=250),
        # the XY machine and its best-axis readout
        dict(name="xy100", use="xy", J="sparse", N=100, D=2, n_h=16, reps=64, prec="bf16x2", steps=200),
        # one chunk of continuous operation with the learned exit, and a training gradient
        dict(name="exit_chunk", use="learned", J="sk", N=100, D=3, n_h=32, reps=128, prec="bf16x2", steps=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["solo", "solo", "solo", "scan", "batch", "batch", "packed", "xy", "learned"])
    n_h = _log(rng, 2, 32)
    reps = _log(rng, 2, 128)
    if use == "packed":
        return dict(use=use, J="sparse", N=rng.randint(8, 30), N2=rng.randint(31, 100), n_ctx=rng.randint(2, 30),
                    D=rng.choice([1, 2]), n_h=n_h, reps=rng.randint(8, 32), prec="bf16x2",
                    steps=_log(rng, 50, 500))
    if use == "xy":
        return dict(use=use, J=rng.choice(["sk", "sparse"]), N=_log(rng, 20, 200), D=2, n_h=n_h, reps=reps,
                    prec=rng.choice(["bf16x2", "fp32"]), steps=_log(rng, 20, 200))
    if use == "learned":
        return dict(use=use, J=rng.choice(["sk", "gauss"]), N=_log(rng, 20, 400), D=rng.choice([2, 3, 4]), n_h=n_h,
                    reps=reps, prec="bf16x2", steps=_log(rng, 20, 200))
    if use == "batch" and rng.random() < 0.5:   # small contexts
        lo = _log(rng, 16, 100)
        return dict(use=use, J=rng.choice(["sk", "sk+gauss", "ladder+sk"]), N=lo + lo % 2, N2=lo + lo % 2,
                    n_ctx=rng.randint(2, 8), dims=rng.choice(["2,3,4", "3", "1,2", "4,5,8"]), n_h=n_h, reps=reps,
                    prec="bf16x2", steps=_log(rng, 50, 1000))
    if use == "batch":                          # uneven sizes
        return dict(use=use, J=rng.choice(["sk", "sk+gauss"]), N=rng.randint(40, 100), N2=_log(rng, 150, 2000),
                    n_ctx=rng.randint(4, 32), dims=rng.choice(["2,3,4,8", "3,4", "1,6"]), n_h=_log(rng, 2, 16),
                    reps=rng.randint(2, 8), prec=rng.choice(["bf16x2", "fp8"]), steps=_log(rng, 16, 100))
    if use == "scan":
        return dict(use=use, J=rng.choice(["sk", "gauss", "sparse"]), N=_log(rng, 10, 128), D=rng.randint(1, 4),
                    n_h=n_h, reps=reps, prec="bf16x2", steps=_log(rng, 100, 2000))
    prec = rng.choice(["bf16x2", "bf16x2", "fp8", "fp32", "fp64"])
    if prec == "fp64":
        return dict(use=use, J=rng.choice(["sk", "gauss"]), N=_log(rng, 8, 48), D=rng.randint(1, 4), n_h=n_h,
                    reps=rng.randint(2, 16), prec=prec, steps=_log(rng, 16, 300))
    if prec == "fp32":
        return dict(use=use, J=rng.choice(["sk", "ladder", "gauss"]), N=2 * _log(rng, 5, 60), D=rng.randint(1, 4),
                    n_h=n_h, reps=reps, prec=prec, steps=_log(rng, 16, 300))
    if rng.random() < 0.5:
        return dict(use=use, J=rng.choice(["sk", "gauss"]), N=_log(rng, 8, 128), D=rng.randint(1, 8), n_h=n_h,
                    reps=reps, prec=prec, steps=_log(rng, 50, 1000))
    if rng.random() < 0.2:
        return dict(use=use, J="ladder", N=2 * _log(rng, 256, 1024), D=rng.choice([2, 3]), n_h=n_h,
                    reps=rng.randint(2, 64), prec=prec, steps=_log(rng, 16, 200))
    return dict(use=use, J=rng.choice(["sk", "gauss"]), N=_log(rng, 129, 1000), D=rng.randint(1, 4), n_h=n_h,
                reps=reps, prec=prec, steps=_log(rng, 16, 100))


# ---- inputs, from the seed alone ---------------------------------------------------------

def _couplings(kind, N, rng):
    """Couplings and feedback strength eps = 0.5 / (their largest eigenvalue, large N)."""
    if kind == "ladder":
        i = np.arange(N)
        J = np.zeros((N, N))
        J[i, (i + 1) % N] = J[(i + 1) % N, i] = -1.0
        J[i, (i + N // 2) % N] = -1.0
        return J, 0.5 / 3.0
    if kind == "gauss":
        J = np.triu(rng.standard_normal((N, N)) / math.sqrt(N), 1)
        return J + J.T, 0.25
    J = (rng.integers(0, 2, size=(N, N)) * 2 - 1).astype(np.float64)
    if kind == "sparse":
        J *= rng.random((N, N)) < 0.2
    J = np.triu(J, 1)
    return J + J.T, 0.25 / math.sqrt(N if kind == "sk" else max(1.0, 0.2 * N))


def _systems(case, seed):
    """The contexts of a case as plain arrays: couplings, weights, dimension, pumps, run keys."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 77])
    R = case["n_h"] * case["reps"]
    h = 0.5 * (1.0 + (np.linspace(0.0, 1.0, case["n_h"]) if case["n_h"] > 1 else np.zeros(1)))
    anneal = case["use"] != "xy"

    def system(J, eps, D, kind, seg=None, w=None):
        return dict(J=J, eps=eps, D=D, h=h, R=R, w=w, seg=seg, real=kind == "gauss", anneal=anneal,
                    seeds=rng.integers(0, 2 ** 63, size=R, dtype=np.int64))

    if case["use"] == "packed":
        sizes = [int(n) for n in np.linspace(case["N"], case["N2"], case["n_ctx"])]
        graphs = [_couplings("sparse", n, rng) for n in sizes]
        out = []
        for members in packing.plan(sizes):
            p = packing.build([g[0] for g in graphs], members)
            w = packing.spin_weights(p, [graphs[i][1] for i in members])
            out.append(system(p.J, 1.0, case["D"], "sparse", p.seg_begin, w))
        return out
    if case["use"] == "batch":
        kinds, dims = case["J"].split("+"), [int(d) for d in case["dims"].split(",")]
        out = []
        for i in range(case["n_ctx"]):
            kind, D = kinds[(i // len(dims)) % len(kinds)], dims[i % len(dims)]
            N = int(round(case["N"] + (case["N2"] - case["N"]) * i / max(1, case["n_ctx"] - 1)))
            J, eps = _couplings(kind, N, rng)
            out.append(system(J, eps, D, kind))
        return out
    J, eps = _couplings(case["J"], case["N"], rng)
    return [system(J, eps, case["D"], case["J"])]


def _network(seed):
    """Parameters, input mean and inverse deviation of the exit network."""
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 78])
    theta = rng.standard_normal(chym.N_MLP_PARAMS).astype(np.float32) * np.float32(0.15)
    mean = rng.standard_normal(chym.N_FEATURES).astype(np.float32) * np.float32(0.1)
    istd = (0.5 + rng.random(chym.N_FEATURES)).astype(np.float32)
    return theta, mean, istd


def prepare(case, seed):
    st = dict(case=case, ctx=[], prm=[], sched=[], h=[], seeds=[], X=[], E=[], S=[], sys=[])
    K = case["steps"]
    for s in _systems(case, seed):
        N, D, R = len(s["J"]), s["D"], s["R"]
        ctx = chym.Context(s["J"], D, chym.J_REAL if s["real"] else chym.J_PM1)
        if s["w"] is not None:
            ctx.set_coupling_weights(s["w"])
        prec = PRECS[case["prec"]]
        st["ctx"].append(ctx)
        st["prm"].append(chym.Params(dt=DT, sigma=SIGMA, init_std=INIT_STD, gamma=GAMMA, kappa=KAPPA, eps=s["eps"],
                                     prec=prec))
        st["sched"].append(chym.Schedule(1, K // 2, K) if s["anneal"] else chym.Schedule(0, 0, 1))
        if case["use"] == "scan":      # host arrays
            st["h"].append(s["h"])
            st["seeds"].append(s["seeds"].view(np.uint64))
        else:
            st["h"].append(torch.from_numpy(s["h"]).cuda())
            st["seeds"].append(torch.from_numpy(s["seeds"]).cuda())
            dt = torch.float64 if case["prec"] == "fp64" else torch.float32
            st["X"].append(torch.empty(R, N, D, dtype=dt, device="cuda"))
            st["E"].append(torch.empty(R, dtype=torch.float64, device="cuda"))
            st["S"].append(torch.empty(R, (N + 63) // 64, dtype=torch.int64, device="cuda"))
        st["sys"].append(dict(R=R, seg=s["seg"]))
    if case["use"] in ("batch", "packed"):
        st["batch"] = chym.Batch(st["ctx"])
    if case["use"] == "learned":
        R = st["sys"][0]["R"]
        net = chym.MLP(seed=1, max_batch=R)
        net.set_params(*_network(seed))
        st["net"] = net
        dev = lambda *sh, dtype=torch.float32: torch.empty(*sh, dtype=dtype, device="cuda")
        st["snap"] = torch.empty_like(st["X"][0])
        st["F"], st["L"] = dev(R, chym.N_FEATURES), dev(R)
        st["counts"], st["order"] = dev(5, dtype=torch.int64), dev(R, dtype=torch.int32)
        st["grad"], st["loss"] = dev(chym.N_MLP_PARAMS), dev(1)
        st["y"] = (torch.arange(R, device="cuda") % 5 == 0).float()
    torch.cuda.synchronize()
    return st


def run(st):
    case, steps = st["case"], st["case"]["steps"]
    stream = torch.cuda.current_stream().cuda_stream
    n_h = case["n_h"]
    ctx, prm, sched = st["ctx"], st["prm"], st["sched"]
    if case["use"] == "scan":
        c = ctx[0]
        c.run(prm[0], st["h"][0], st["seeds"][0], steps, sched[0], stream)
        E = c.energy(stream=stream)
        s = c.stats(float(E.min()), n_bins=64, stream=stream)
        return {"E": E, "hits": s["hits"], "hist": s["hist"], "P_max": s["P_max"], "W_range": s["W_range"],
                "W_scan": s["W_scan"], "dE_mean": s["dE_mean"], "best_E": s["best_E"]}

    def start(i, n):
        ctx[i].run_device(prm[i], st["h"][i].data_ptr(), n_h, st["seeds"][i].data_ptr(), st["sys"][i]["R"], n,
                          sched[i], stream)

    out = {}
    if case["use"] in ("batch", "packed"):
        for i in range(len(ctx)):
            start(i, 0)
        st["batch"].run(prm, sched, steps, stream)
        for i, c in enumerate(ctx):
            if case["use"] == "packed":
                out["E%d" % i] = c.energy_segments(st["sys"][i]["seg"], stream)
            else:
                c.energy_device(st["E"][i].data_ptr(), 0, stream)
                out["E%d" % i] = st["E"][i]
            c.copy_state_device(st["X"][i].data_ptr(), stream)
            out["X%d" % i] = st["X"][i]
        return out
    c, X, E, S = ctx[0], st["X"][0], st["E"][0], st["S"][0]
    if case["use"] == "learned":
        R = st["sys"][0]["R"]
        start(0, steps // 2)
        c.copy_state_device(st["snap"].data_ptr(), stream)
        c.run_device(prm[0], 0, n_h, 0, R, steps - steps // 2, sched[0], stream)
        c.energy_device(E.data_ptr(), 0, stream)
        c.features_device(st["snap"].data_ptr(), 0.1, st["F"].data_ptr(), stream)
        st["net"].forward_device(st["F"].data_ptr(), R, st["L"].data_ptr(), stream)
        c.exit_scan_device(E.data_ptr(), -1.0, st["L"].data_ptr(), 0.0, 10 * steps, steps,
                           st["counts"].data_ptr(), st["order"].data_ptr(), stream)
        st["net"].grad_device(st["F"].data_ptr(), st["y"].data_ptr(), R, st["grad"].data_ptr(),
                              st["loss"].data_ptr(), stream)
        return {"E": E, "features": st["F"], "logits": st["L"], "counts": st["counts"], "order": st["order"],
                "grad": st["grad"], "loss": st["loss"]}
    start(0, steps)
    if case["use"] == "xy":
        c.readout_xy_device(E.data_ptr(), S.data_ptr(), stream)
    else:
        c.energy_device(E.data_ptr(), S.data_ptr(), stream)
    c.copy_state_device(X.data_ptr(), stream)
    return {"E": E, "spins": S, "X": X}


def work(case):
    """Couplings, pumps and keys read once, states and energies written once; coupling product
    and update of every step.  (The noise's integer work is not counted.)"""
    by = fl = 0.0
    el = 8 if case["prec"] == "fp64" else 4
    R = case["n_h"] * case["reps"]
    if case["use"] == "packed":
        shapes = [(int(n), case["D"]) for n in np.linspace(case["N"], case["N2"], case["n_ctx"])]
        kinds = ["sparse"] * len(shapes)
    elif case["use"] == "batch":
        n, dims, ks = case["n_ctx"], [int(d) for d in case["dims"].split(",")], case["J"].split("+")
        shapes = [(int(round(case["N"] + (case["N2"] - case["N"]) * i / max(1, n - 1))), dims[i % len(dims)])
                  for i in range(n)]
        kinds = [ks[(i // len(dims)) % len(ks)] for i in range(n)]
    else:
        shapes, kinds = [(case["N"], case["D"])], [case["J"]]
    for (N, D), kind in zip(shapes, kinds):
        nnz = 3 * N if kind == "ladder" else N * N // 5 if kind == "sparse" else N * N
        by += (el if kind == "gauss" else 1) * nnz + 16 * R + (0 if case["use"] in ("scan", "learned") else el * R * N * D)
        fl += float(case["steps"]) * R * D * (2.0 * nnz + 12.0 * N) + 2.0 * nnz * R
        if case["use"] == "learned":
            by += R * 4 * (chym.N_FEATURES + 1)
            fl += R * (2.0 * nnz * (D + 1) + 6.0 * 2 * (24 * 64 + 64 * 64 + 64))
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits, in plain torch -------------------------------------------------

_M = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & _M) ^ c1 ^ k0, p1 & _M, ((p0 >> 32) & _M) ^ c3 ^ k1, p0 & _M
        k0, k1 = (k0 + 0x9E3779B9) & _M, (k1 + 0xBB67AE85) & _M
    return c0, c1, c2, c3


def _normals(keys, N, D, tag, k):
    """Normals [R, N, D] of the documented noise counter (tag 0: step k, tag 1: initial state)."""
    R = len(keys)
    k0, k1 = (keys & _M).view(R, 1), ((keys >> 32) & _M).view(R, 1)
    if D <= 2:
        spins = torch.arange(-(-N * D // 4), device=keys.device)
        blocks = torch.full_like(spins, tag << 8)
    else:
        nb = (D + 3) // 4
        spins = torch.arange(N, device=keys.device).repeat_interleave(nb)
        blocks = (tag << 8) | torch.arange(nb, device=keys.device).repeat(N)
    z = torch.zeros(R, len(spins), dtype=torch.int64, device=keys.device)
    w = _philox(z + spins, z + blocks, z + (k & _M), z + (k >> 32), k0, k1)
    u = [(v.double() + 0.5) * 2.0 ** -32 for v in w]
    out = torch.empty(R, len(spins), 4, dtype=torch.float64, device=keys.device)
    for j in (0, 2):
        r, t = torch.sqrt(-2.0 * torch.log(u[j])), 2.0 * math.pi * u[j + 1]
        out[..., j], out[..., j + 1] = r * torch.cos(t), r * torch.sin(t)
    if D <= 2:
        return out.reshape(R, -1)[:, :N * D].reshape(R, N, D)
    return out.reshape(R, N, -1)[..., :D]


def _integrate(s, K, steps, x=None, k_from=0):
    J = torch.from_numpy(s["J"]).cuda()
    keys = torch.from_numpy(s["seeds"]).cuda()
    N, D, R = len(s["J"]), s["D"], s["R"]
    gain = torch.from_numpy(np.repeat(s["h"], R // len(s["h"])) - 1.0).cuda().view(R, 1, 1)
    w = torch.ones(N, dtype=torch.float64, device="cuda") if s["w"] is None else torch.from_numpy(s["w"]).cuda()
    if x is None:
        x = INIT_STD * _normals(keys, N, D, 1, 0)
    ka = K // 2
    for k in range(k_from, k_from + steps):
        a = 1.0 if not s["anneal"] or k < ka else max(0.0, 1.0 - (k - ka) / (K - ka))
        y = (J @ x.permute(1, 0, 2).reshape(N, R * D)).reshape(N, R, D).permute(1, 0, 2) * (s["eps"] * w.view(1, N, 1))
        if a != 1.0 and D > 1:
            y = torch.cat([y[..., :1], a * y[..., 1:]], dim=2)
        n2 = (x * x).sum(dim=2, keepdim=True)
        x = x + DT * (x * (gain - KAPPA * x * x - GAMMA * n2) + y) + SIGMA * math.sqrt(DT) * _normals(keys, N, D, 0, k)
    return x


def _energy(J, x):
    s = torch.where(x >= 0, 1.0, -1.0).double()
    return -((s @ J) * s).sum(dim=1)


def _best_axis(J, x):
    """Lowest Ising energy over the axes that round planar spins, one axis per interval."""
    phi = torch.atan2(x[..., 1], x[..., 0]) + 0.5 * math.pi
    phi = torch.sort(phi - math.pi * torch.floor(phi / math.pi), dim=1).values
    nxt = torch.cat([phi[:, 1:], phi[:, :1] + math.pi], dim=1)
    mid = 0.5 * (phi + nxt)
    best = None
    for i in range(mid.shape[1]):
        e = _energy(J, x[..., 0] * torch.cos(mid[:, i:i + 1]) + x[..., 1] * torch.sin(mid[:, i:i + 1]))
        best = e if best is None else torch.minimum(best, e)
    return best


def _features(J, x, xs, hrun, D):
    R, N, _ = x.shape
    rms = torch.sqrt((x[..., 0] ** 2).mean(dim=1))
    u = torch.sort(x[..., 0].abs() / rms.view(R, 1), dim=1).values
    f = [u[:, int(math.floor(j * (N - 1) / 11.0 + 0.5))] for j in range(12)]
    e, es = _energy(J, x[..., 0]), _energy(J, xs[..., 0])
    frac = lambda v: (v[..., 1:] ** 2).sum(dim=(1, 2)) / (v ** 2).sum(dim=(1, 2))
    norm = torch.sqrt((x * x).sum(dim=2))
    sg = x / norm.unsqueeze(2)
    ehs = -(torch.einsum("pq,rqd->rpd", J, sg) * sg).sum(dim=(1, 2))
    flips = ((x[..., 0] >= 0) != (xs[..., 0] >= 0)).double().mean(dim=1)
    one = torch.ones_like(rms)
    f += [e / N, (e - es) / N, frac(x), frac(x) - frac(xs), flips, ehs / N, norm.mean(dim=1), hrun, one * D / 8.0,
          one * math.log(N) / math.log(2048.0), one * 0.1, rms]
    return torch.stack(f, dim=1)


def _net(seed, F, y):
    theta, mean, istd = (torch.from_numpy(v).cuda() for v in _network(seed))
    p = theta.bfloat16().double().requires_grad_(True)
    F = (F - mean.double()) * istd.double()
    W1, b1, W2, b2, W3, b3 = torch.split(p, [64 * 24, 64, 64 * 64, 64, 64, 1])
    gelu = torch.nn.functional.gelu
    z = gelu(gelu(F @ W1.view(64, 24).T + b1) @ W2.view(64, 64).T + b2) @ W3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y)
    loss.backward()
    return z.detach(), p.grad, loss.detach().view(1)


def exact(case, seed):
    K = case["steps"]
    systems = _systems(case, seed)
    cost = sum(K * s["R"] * s["D"] * len(s["J"]) * (200.0 + len(s["J"])) for s in systems)
    if cost > 8e12 or K * len(systems) > 12000:
        return None     # would take too long in 64 bits
    out = {}
    for i, s in enumerate(systems):
        J = torch.from_numpy(s["J"]).cuda()
        if case["use"] == "learned":
            xs = _integrate(s, K, K // 2)
            x = _integrate(s, K, K - K // 2, xs, K // 2)
            hrun = torch.from_numpy(np.repeat(s["h"], s["R"] // len(s["h"]))).cuda()
            F = _features(J, x, xs, hrun, s["D"])
            z, g, loss = _net(seed, F, (torch.arange(s["R"], device="cuda") % 5 == 0).double())
            return {"E": _energy(J, x[..., 0]), "features": F, "logits": z, "counts": None, "order": None, "grad": g,
                    "loss": loss}
        x = _integrate(s, K, K)
        if case["use"] == "batch":
            out["E%d" % i], out["X%d" % i] = _energy(J, x[..., 0]), x
        elif case["use"] == "packed":
            b = s["seg"]
            out["E%d" % i] = torch.stack([_energy(J[lo:hi, lo:hi], x[:, lo:hi, 0]) for lo, hi in zip(b[:-1], b[1:])],
                                         dim=1).cpu().numpy()
            out["X%d" % i] = x
        elif case["use"] == "xy":
            return {"E": _best_axis(J, x), "spins": None, "X": x}
        elif case["use"] == "scan":
            E = _energy(J, x[..., 0])
            return {"E": E.cpu().numpy(), "hits": None, "hist": None, "P_max": None, "W_range": None, "W_scan": None,
                    "dE_mean": float((E - E.min()).mean()), "best_E": float(E.min())}
        else:
            return {"E": _energy(J, x[..., 0]), "spins": None, "X": x}
    return out
