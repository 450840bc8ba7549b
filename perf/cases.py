"""Performance cases of the MGEnKF library.

Each case is one thing that a user's program has the library do, through the
Python binding of the C ABI, at sizes of the workloads in
``paper_2012_10091_gb300/workloads.py`` and of the tests:

* ``cycle``     a handle's whole analysis cycle (forecast, analysis, correction);
* ``forecast``  a handle's forecast between two analyses (members and fine run);
* ``truth``     the stateless forecast that truth runs use (one grid, FP64);
* ``analysis``  a handle's analysis and fine correction at one time;
* ``batch``     one cycle of many independent problems of uneven sizes;
* ``cnn_infer`` the residual of the learned correction;
* ``cnn_train`` one training step of it (loss, gradients, Adam);
* ``dual``      one cycle of the Dual EnKF (inlet parameter estimation).

A handle's pass loads the state, runs and reads the result, all in device
memory, so every pass of a state does the same work on the same values.  The
batch and the training step carry their state on from pass to pass, as their
loops do.  Mixed-precision states are FP32 on the device: their inputs are
FP32 values held in FP64 (the type of the interface) and their results are
returned as FP32.  ``exact`` restates each case in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2012_10091_gb300 import mgenkf as M

DEV = "cuda"
GAMMA, PRANDTL, MACH = 1.4, 0.72, 0.3
NS_MU, BURGERS_NU = 1e-3, 0.01
EPS_TAG, THETA_TAG = 0x45505300, 0x54485441

# Flops per point and model step (an FMA counts 2): NS-2D SSP-RK3 423 (per
# stage 114 for dt L and 11 for the primitives, 48 for the stage updates),
# Burgers 32 with the compensated FP32 state, 30 in FP64.
NS_FLOPS, BURGERS_FLOPS_MIXED, BURGERS_FLOPS_FP64, INLET_FLOPS = 423, 32, 30, 36


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest workload (256 / 64 points, 32 members, 16 sensors): a
        # whole FP64 cycle is a chain of tiny launches
        _single("cycle_burgers_small_fp64", "cycle", "burgers", "fp64", nc=64, ratio=4, ne=32, ny=16, steps=20),
        # the large 1-D workload: one observation interval of 4331 model steps
        _single("forecast_burgers_large_mixed", "forecast", "burgers", "mixed", nc=4096, ratio=4, ne=128, ny=512,
                steps=4331),
        # its truth run over the same interval, in FP64
        dict(name="truth_burgers_large_fp64", kind="truth", model="burgers", n=16384, nprob=1, steps=4331),
        # the plain FP64 filter at those sizes: every product, factor and solve in FP64
        _single("analysis_burgers_large_fp64", "analysis", "burgers", "fp64", nc=4096, ratio=4, ne=128, ny=512,
                steps=1),
        # the 2-D shear layer, 512^2 / 128^2 with 64 members: forecast and analysis
        _single("forecast_ns_mixed", "forecast", "ns", "mixed", nc=128, ratio=4, ne=64, ny=2048, steps=10),
        _single("analysis_ns_mixed", "analysis", "ns", "mixed", nc=128, ratio=4, ne=64, ny=2048, steps=10),
        # the plain FP64 filter's forecast and the FP64 truth run of the 2-D model
        _single("forecast_ns_fp64", "forecast", "ns", "fp64", nc=64, ratio=4, ne=32, ny=512, steps=10),
        dict(name="truth_ns_fp64", kind="truth", model="ns", n=512, nprob=1, steps=10),
        # a service that cycles many uneven problems: a quarter of the 96-problem batch
        dict(name="batch_ns_mixed", kind="batch", problems=24, layout=0, steps=10),
        # the learned correction at 256^2 -> 1024^2: inference and a training step of 8 samples
        dict(name="cnn_infer_256", kind="cnn_infer", nc=256, batch=1),
        dict(name="cnn_train_256x8", kind="cnn_train", nc=256, batch=8),
        # the paper's parameter estimation: 800 / 200 nodes, 100 members, 80 sensors, 30 steps
        dict(name="dual_800_200", kind="dual", nc=200, ratio=4, ne=100, ny=80, steps=30),
    ]


def _single(name, kind, model, precision, nc, ratio, ne, ny, steps, form="ensemble"):
    return dict(name=name, kind=kind, model=model, precision=precision, nc=nc, ratio=ratio, ne=ne, ny=ny,
                steps=steps, form=form)


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["cycle", "forecast", "forecast", "truth", "truth", "analysis", "analysis", "batch", "cnn_infer",
                       "cnn_train", "dual"])
    if kind in ("cycle", "forecast", "analysis"):
        model = rng.choice(["burgers", "ns"])
        precision = rng.choice(["fp64", "mixed"])
        ratio = rng.choice([2, 4, 8] if model == "burgers" else [2, 4])
        if model == "burgers":
            nc = _log(rng, 32, 4096 if precision == "mixed" or kind == "analysis" else 1024)
            nc = min(nc, 16384 // ratio)
            if nc * ratio > 4096:  # a split fine grid: whole pieces on every side
                nc -= nc % 64
            ny = _log(rng, 8, min(512, nc * ratio // 2))
            steps = _log(rng, 5, 40) if kind != "forecast" else _log(rng, 20, 1500)
        else:
            nc = 8 * _log(rng, 1, 16 if precision == "mixed" or kind == "analysis" else 8)
            ny = 2 * _log(rng, 8, min(1024, nc * nc // 4))
            steps = _log(rng, 1, 10)
        ne = _log(rng, 8, 128)
        if model == "ns" and precision == "fp64" and kind != "analysis":
            ne = min(ne, 32)
        form = "direct" if ny <= ne and rng.random() < 0.5 else "ensemble"
        c = _single("", kind, model, precision, nc, ratio, ne, ny, steps, form)
    elif kind == "truth":
        if rng.random() < 0.5:
            n = _log(rng, 128, 16384)
            if n > 4096:
                n -= n % 64
            c = dict(kind=kind, model="burgers", n=n, nprob=1, steps=_log(rng, 20, 4331))
        else:
            c = dict(kind=kind, model="ns", n=8 * _log(rng, 4, 64), nprob=1, steps=_log(rng, 1, 10))
    elif kind == "batch":
        c = dict(kind=kind, problems=_log(rng, 2, 24), layout=rng.randrange(1, 1000), steps=_log(rng, 2, 10))
        if c["problems"] == 24:
            c["problems"] = 23
    elif kind in ("cnn_infer", "cnn_train"):
        c = dict(kind=kind, nc=_log(rng, 8, 256), batch=rng.randint(1, 8))
    else:
        nc, ratio = _log(rng, 25, 250), rng.choice([1, 2, 4])
        c = dict(kind=kind, nc=nc, ratio=ratio, ne=_log(rng, 10, 128), ny=_log(rng, 8, min(80, nc * ratio // 4)),
                 steps=_log(rng, 5, 40))
    c.pop("name", None)
    return c


def _batch_sizes(case):
    """(nc, ne, ny) per problem: coarse sides, members and observation counts of the batched workload."""
    g = np.random.default_rng([case["layout"], case["problems"]])
    return [(int(g.choice((64, 96, 128, 192))), int(g.choice((16, 32, 64, 128))), 2 * int(g.integers(128, 1025)))
            for _ in range(case["problems"])]


def work(case):
    """Bytes: the states and observations a pass takes in and the results it
    returns, each once.  Flops: the model steps at the counts above, and the
    analysis' products (S and its right-hand sides, Cholesky, solves, X T)."""
    k = case["kind"]
    if k in ("cycle", "forecast", "analysis"):
        d = _dims(case)
        out = 8 if case["precision"] == "fp64" else 4
        b = (d["nxf"] + d["ne"] * d["nx"]) * (8 + out)
        f = 0.0
        if k != "analysis":
            f += _step_flops(case["model"], case["precision"]) * case["steps"] * (d["nxf"] + d["ne"] * d["nx"]) / d["V"]
        if k != "forecast":
            f += _analysis_flops(d["nx"], d["nxf"], d["ne"], case["ny"])
            b += 8 * case["ny"]
        return dict(bytes=b, flops=f)
    if k == "truth":
        v, p = (1, case["n"]) if case["model"] == "burgers" else (4, case["n"] ** 2)
        n = case["nprob"] * p
        return dict(bytes=16 * v * n, flops=_step_flops(case["model"], "fp64") * case["steps"] * n)
    if k == "batch":
        b = f = 0.0
        for nc, ne, ny in _batch_sizes(case):
            pts = ne * nc * nc + 16 * nc * nc
            b += 4 * pts * 8 + 8 * ny
            f += NS_FLOPS * case["steps"] * pts + _analysis_flops(4 * nc * nc, 64 * nc * nc, ne, ny)
        return dict(bytes=b, flops=f)
    if k in ("cnn_infer", "cnn_train"):
        pl = case["batch"] * case["nc"] ** 2
        fwd = 2.0 * 9 * (8 * 32 + 32 * 32 + 32 * 64) * pl
        if k == "cnn_infer":
            return dict(bytes=4.0 * pl * (8 + 64), flops=fwd)
        return dict(bytes=4.0 * pl * (8 + 64) + 4 * 6 * M.CNN_NPARAMS, flops=3 * fwd - 2.0 * 9 * 8 * 32 * pl)
    nf, ne = case["nc"] * case["ratio"], case["ne"]
    f = INLET_FLOPS * case["steps"] * (nf + 2.0 * ne * case["nc"]) + 2 * _analysis_flops(case["nc"], nf, ne, case["ny"])
    return dict(bytes=16.0 * (nf + ne * case["nc"] + 2 * ne) + 8 * case["ny"], flops=f)


def _step_flops(model, precision):
    if model == "ns":
        return NS_FLOPS
    return BURGERS_FLOPS_MIXED if precision == "mixed" else BURGERS_FLOPS_FP64


def _analysis_flops(nx, nxf, ne, ny):
    products = ny * (ne * (ne + 1) + 2.0 * ne * (ne + 1))
    return products + ne ** 3 / 3.0 + 2.0 * ne * ne * (ne + 1) + 2.0 * nx * ne * (ne + 1) + 12.0 * nxf


def _dims(case):
    V, dim = (1, 1) if case["model"] == "burgers" else (4, 2)
    nc, nf = case["nc"], case["nc"] * case["ratio"]
    return dict(V=V, dim=dim, nc=nc, nf=nf, r=case["ratio"], ne=case["ne"], ny=case["ny"], nx=V * nc ** dim,
                nxf=V * nf ** dim)


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _randn(shape, g, dtype=torch.float64):
    return torch.randn(shape, generator=g, device=DEV, dtype=dtype)


def _burgers_states(n, count, g, noise=0.05):
    """Sum of sines with a random amplitude per state, and point noise."""
    x = torch.arange(n, device=DEV, dtype=torch.float64) * (2 * math.pi / n)
    phase = torch.tensor([0.3, 1.1, 2.7, 4.0, 5.2], device=DEV, dtype=torch.float64)
    k = torch.arange(1, 6, device=DEV, dtype=torch.float64)
    prof = (torch.sin(k[:, None] * x + phase[:, None]) / k[:, None]).sum(0)
    amp = 0.8 + 0.1 * _randn((count, 1), g)
    return amp * prof + noise * _randn((count, n), g)


def _ns_states(n, count, g, delta):
    """Double shear layer of thickness delta at Mach 0.3 with 1e-3 velocity noise, 4 x n x n per state."""
    y = torch.arange(n, device=DEV, dtype=torch.float64) / n
    base = torch.tanh((y - 0.5) / delta) - torch.tanh(y / delta) - torch.tanh((y - 1.0) / delta)
    u = base[None, :, None] + 1e-3 * _randn((count, n, n), g)
    v = 1e-3 * _randn((count, n, n), g)
    rho = torch.ones_like(u)
    E = 1.0 / (GAMMA * MACH ** 2) / (GAMMA - 1.0) + 0.5 * (u * u + v * v)
    return torch.stack([rho, u, v, E], 1)


def _ns_delta(nc):
    return 0.02 * max(1.0, 128.0 / nc)


def _dt(model, nf):
    if model == "burgers":
        return min(1e-3, 0.5 * 0.628 * (2 * math.pi / nf) ** 2 / BURGERS_NU)
    h = 1.0 / nf
    return min(0.5 * math.sqrt(3.0) * h / (1.0 + 1.0 / MACH), 0.8 * 2.51 * h * h / (8.0 * NS_MU * GAMMA / PRANDTL))


def _problem(model, nc, ratio, ne, ny, mixed, seed):
    """Fine state, members, observed nodes and observations of one filter."""
    nf = nc * ratio
    sigma = 0.05 if model == "burgers" else 0.01
    rng = np.random.default_rng([seed, 5])
    if model == "burgers":
        fine, members = _burgers_states(nf, 1, _gen(seed, 1))[0], _burgers_states(nc, ne, _gen(seed, 2))
        truth = _burgers_states(nf, 1, _gen(seed, 3), 0.0)[0]
        idx = np.sort(rng.choice(nf, size=ny, replace=False)).astype(np.int32)
        var = np.zeros(ny, np.int32)
    else:
        d = _ns_delta(nc)
        fine, members = _ns_states(nf, 1, _gen(seed, 1), d).reshape(-1), _ns_states(nc, ne, _gen(seed, 2), d)
        truth = _ns_states(nf, 1, _gen(seed, 3), d).reshape(-1)
        nodes = np.sort(rng.choice(nf * nf, size=ny // 2, replace=False)).astype(np.int32)
        idx, var = np.repeat(nodes, 2).astype(np.int32), np.tile(np.array([1, 2], np.int32), ny // 2)
    members = members.reshape(ne, -1)
    if mixed:
        fine, members = fine.float().double(), members.float().double()
    npts = nf if model == "burgers" else nf * nf
    pick = torch.as_tensor(var.astype(np.int64) * npts + idx, device=DEV)
    yobs = truth[pick] + sigma * torch.as_tensor(rng.standard_normal(ny), device=DEV)
    return dict(fine=fine.contiguous(), members=members.contiguous(), idx=idx, var=var, yobs=yobs, sigma=sigma,
                dt=_dt(model, nf), nc=nc, nf=nf, ratio=ratio, ne=ne, ny=ny, model=model, seed=int(seed) % (1 << 31))


def _handle(p, mixed, form="ensemble"):
    ns = p["model"] == "ns"
    return M.MGEnKF(model=M.MGENKF_NS2D if ns else M.MGENKF_BURGERS1D, n_fine=p["nf"], ratio=p["ratio"],
                    n_members=p["ne"], obs_index=p["idx"], obs_var=p["var"], length=1.0 if ns else 2 * math.pi,
                    dt=p["dt"], nu=NS_MU if ns else BURGERS_NU, obs_sigma=p["sigma"], seed=p["seed"],
                    precision=M.MGENKF_MIXED if mixed else M.MGENKF_FP64,
                    gain_form=M.MGENKF_GAIN_DIRECT if form == "direct" else M.MGENKF_GAIN_ENSEMBLE, gamma=GAMMA,
                    prandtl=PRANDTL)


def _truth_state(case, seed):
    if case["model"] == "burgers":
        return _burgers_states(case["n"], case["nprob"], _gen(seed, 3), 0.01)
    return _ns_states(case["n"], case["nprob"], _gen(seed, 3), _ns_delta(case["n"] / 4))


def _cnn_data(case, seed):
    """Coarse fields of analyses (corrections of 1e-2, states around a mean) and fine corrections."""
    n, B = case["nc"], case["batch"]
    g = _gen(seed, 1)
    f = torch.float32
    dC = 1e-2 * _randn((B, 4, n, n), g, f)
    mean = torch.tensor([1.0, 0.0, 0.0, 20.0], device=DEV, dtype=f).view(1, 4, 1, 1)
    scale = torch.tensor([0.05, 0.9, 0.1, 0.5], device=DEV, dtype=f).view(1, 4, 1, 1)
    xs = mean + scale * _randn((B, 4, n, n), g, f)
    target = torch.repeat_interleave(torch.repeat_interleave(dC, 4, 2), 4, 3)
    target = target + 5e-3 * _randn((B, 4, 4 * n, 4 * n), g, f)
    params = {}
    for (name, shape), std in zip(M.CNN_SHAPES, (math.sqrt(2 / 72), 0.05, math.sqrt(2 / 288), 0.05, 0.03, 0.02)):
        params[name] = (std * _randn(shape, g, f)).cpu().numpy()
    stats = dict(mu_in=np.array([0, 0, 0, 0, 1, 0, 0, 20], np.float32),
                 s_in=np.array([1e-2] * 4 + [0.05, 0.9, 0.1, 0.5], np.float32),
                 s_out=np.array([1.2e-2, 1.1e-2, 1e-2, 1.3e-2], np.float32))
    return dC.contiguous(), xs.contiguous(), target.contiguous(), params, stats


def _dual_data(case, seed):
    nc, r, ne, ny = case["nc"], case["ratio"], case["ne"], case["ny"]
    nf = nc * r
    rng = np.random.default_rng([seed, 9])
    length, u0, omega, t0 = 0.0125 * nf, 1.0, 2 * math.pi, 10.0

    def wave(n, a, b):  # a developed travelling wave of inlet amplitude a and phase b
        x = np.arange(n) * (length / n)
        return u0 * (1 + a * np.exp(-x / 4.0) * np.sin(omega * (t0 - x / u0) + b))

    theta = np.stack([0.05 * rng.standard_normal(ne), 0.3 + 0.05 * rng.standard_normal(ne)], 1)
    members = np.stack([wave(nc, a, b) for a, b in theta])
    theta_fine = theta.mean(0)
    fine = wave(nf, *theta_fine)
    idx = np.sort(rng.choice(np.arange(1, max(nf // 4, ny + 1)), size=ny, replace=False)).astype(np.int32)
    yobs = wave(nf, 0.2, 0.0)[idx] + 0.05 * rng.standard_normal(ny)
    return dict(nc=nc, nf=nf, r=r, ne=ne, ny=ny, length=length, u0=u0, omega=omega, t0=t0, dt=2e-4, nu=1 / 200.0,
                sigma=0.05, q=1e-6, theta=theta, members=members, theta_fine=theta_fine, fine=fine, idx=idx, yobs=yobs,
                seed=int(seed) % (1 << 31))


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case)
    if k in ("cycle", "forecast", "analysis"):
        mixed = case["precision"] == "mixed"
        p = _problem(case["model"], case["nc"], case["ratio"], case["ne"], case["ny"], mixed, seed)
        s.update(p=p, h=_handle(p, mixed, case["form"]), fine=torch.empty_like(p["fine"]),
                 members=torch.empty_like(p["members"]))
    elif k == "truth":
        s["q0"] = _truth_state(case, seed)
    elif k == "batch":
        ps = [_problem("ns", nc, 4, ne, ny, True, seed * 131 + j)
              for j, (nc, ne, ny) in enumerate(_batch_sizes(case))]
        hs = [_handle(p, True) for p in ps]
        for h, p in zip(hs, ps):
            M.mgenkf_set_state(h.h, p["fine"], p["members"])
        s["yobs"] = torch.cat([p["yobs"] for p in ps])
        for key in ("fine", "members"):
            flat = torch.empty(sum(p[key].numel() for p in ps), dtype=torch.float64, device=DEV)
            s[key], s[key + "_parts"] = flat, flat.split([p[key].numel() for p in ps])
        s["batch"] = M.Batch(hs)
        s["innov"] = torch.empty(len(ps), dtype=torch.float64, device=DEV)
    elif k in ("cnn_infer", "cnn_train"):
        dC, xs, target, params, stats = _cnn_data(case, seed)
        cnn = M.CNN(case["nc"], case["batch"])
        cnn.set_params(params, stats)
        s.update(cnn=cnn, dC=dC, xs=xs, target=target)
        if k == "cnn_infer":
            s["res"] = torch.empty_like(target)
        else:
            s["loss"] = torch.zeros(1, dtype=torch.float32, device=DEV)
    else:
        d = _dual_data(case, seed)
        s["d"] = d
        s["h"] = M.DualMGEnKF(d["nf"], d["r"], d["ne"], d["idx"], d["length"], d["dt"], d["nu"], d["sigma"], d["q"],
                              d["seed"], d["u0"], d["omega"])
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k in ("cycle", "forecast", "analysis"):
        p, h = s["p"], s["h"]
        h.set_state(p["fine"], p["members"])
        if k == "cycle":
            h.cycle(case["steps"], p["yobs"])
        elif k == "forecast":
            h.forecast(case["steps"])
        else:
            h.analyse(p["yobs"])
            h.prolong_correct()
        M.mgenkf_get_state(h.h, s["fine"], s["members"])
        if case["precision"] == "mixed":
            return s["fine"].float(), s["members"].float()
        return s["fine"], s["members"]
    if k == "truth":
        q = s["q0"].clone()
        ns = case["model"] == "ns"
        nf = case["n"]
        M.mgk_forecast(M.MGENKF_NS2D if ns else M.MGENKF_BURGERS1D, M.MGENKF_FP64, q, case["nprob"], nf,
                       1.0 if ns else 2 * math.pi, _dt(case["model"], nf), NS_MU if ns else BURGERS_NU, GAMMA, PRANDTL,
                       nsteps=case["steps"])
        return q
    if k == "batch":
        s["batch"].cycle(case["steps"], s["yobs"], s["innov"])
        for h, f, m in zip(s["batch"].runs, s["fine_parts"], s["members_parts"]):
            M.mgenkf_get_state(h.h, f, m)
        return s["fine"].float(), s["members"].float(), s["innov"].float()
    if k == "cnn_infer":
        s["cnn"].forward(s["dC"], s["xs"], case["batch"], s["res"])
        return s["res"]
    if k == "cnn_train":
        cnn = s["cnn"]
        cnn.loss_grad(s["dC"], s["xs"], s["target"], case["batch"], s["loss"])
        cnn.adam_step(3e-4)
        params, grads = cnn.get_params()
        return dict(loss=s["loss"], params=params, grads=grads)
    d, h = s["d"], s["h"]
    h.set_state(d["fine"], d["members"], d["theta"], d["theta_fine"], d["t0"])
    h.cycle(case["steps"], d["yobs"])
    return h.get_state()


# ---------------------------------------------------------------------------
# the same results from plain FP64 torch
# ---------------------------------------------------------------------------
def _philox_normals(seed, tag, ctr0, count):
    """Philox4x64-10 (Salmon et al., SC'11) with key (seed, tag) and counter
    (ctr0, block, 0, 0), Box-Muller on the lane pairs (0, 1) and (2, 3)."""
    u64 = np.uint64
    nb = (count + 3) // 4

    def mul(a, b):  # 64 x 64 -> (high, low)
        m = u64(0xFFFFFFFF)
        s = u64(32)
        a0, a1, b0, b1 = a & m, a >> s, b & m, b >> s
        t = a1 * b0 + ((a0 * b0) >> s)
        w = (t & m) + a0 * b1
        return a1 * b1 + (t >> s) + (w >> s), a * b

    c = [np.full(nb, ctr0, u64), np.arange(nb, dtype=u64), np.zeros(nb, u64), np.zeros(nb, u64)]
    k0, k1 = int(seed), int(tag)
    m0, m1 = np.full(nb, 0xD2E7470EE14C6C93, u64), np.full(nb, 0xCA5A826395121157, u64)
    for _ in range(10):
        h0, l0 = mul(m0, c[0])
        h1, l1 = mul(m1, c[2])
        c = [h1 ^ c[1] ^ u64(k0), l1, h0 ^ c[3] ^ u64(k1), l0]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) % (1 << 64), (k1 + 0xBB67AE8584CAA73B) % (1 << 64)
    u = [((x >> u64(11)) + u64(1)).astype(np.float64) * 2.0 ** -53 for x in c]
    z = np.empty((nb, 4))
    for q in (0, 2):
        rad = np.sqrt(-2.0 * np.log(u[q]))
        z[:, q], z[:, q + 1] = rad * np.cos(2 * np.pi * u[q + 1]), rad * np.sin(2 * np.pi * u[q + 1])
    return z.reshape(-1)[:count]


def _rk3(u, dtl, steps):
    for _ in range(steps):
        u1 = u + dtl(u)
        u2 = 0.75 * u + 0.25 * (u1 + dtl(u1))
        u = (u + 2.0 * (u2 + dtl(u2))) / 3.0
    return u


def _burgers_exact(u, length, dt, steps):
    dx = length / u.shape[-1]
    a, b = dt / (4 * dx), dt * BURGERS_NU / dx ** 2

    def dtl(v):
        e, w = torch.roll(v, -1, -1), torch.roll(v, 1, -1)
        return a * ((w - e) * (w + e)) + b * ((e - v) + (w - v))

    return _rk3(u, dtl, steps)


def _ns_exact(q, dt, steps):
    """q: count x 4 x n x n (x last)."""
    h = 1.0 / q.shape[-1]
    kappa = NS_MU * GAMMA / ((GAMMA - 1.0) * PRANDTL)
    E_, W_ = (lambda a: torch.roll(a, -1, -1)), (lambda a: torch.roll(a, 1, -1))
    N_, S_ = (lambda a: torch.roll(a, -1, -2)), (lambda a: torch.roll(a, 1, -2))

    def dtl(q):
        rho, mx, my, E = q.unbind(1)
        u, v = mx / rho, my / rho
        p = (GAMMA - 1.0) * (E - 0.5 * rho * (u * u + v * v))
        T = p / rho
        F = (mx, mx * u + p, mx * v, (E + p) * u)
        G = (my, my * u, my * v + p, (E + p) * v)
        L = [-(E_(f) - W_(f) + N_(g) - S_(g)) / (2 * h) for f, g in zip(F, G)]
        tu, tv = (N_(u) - S_(u)) / (2 * h), (N_(v) - S_(v)) / (2 * h)  # x-faces (x + 1/2)
        ux, vx, uy, vy = (E_(u) - u) / h, (E_(v) - v) / h, 0.5 * (tu + E_(tu)), 0.5 * (tv + E_(tv))
        txx, txy = NS_MU * (4 / 3 * ux - 2 / 3 * vy), NS_MU * (uy + vx)
        fe = txx * 0.5 * (u + E_(u)) + txy * 0.5 * (v + E_(v)) + kappa * (E_(T) - T) / h
        for i, f in ((1, txx), (2, txy), (3, fe)):
            L[i] = L[i] + (f - W_(f)) / h
        tu, tv = (E_(u) - W_(u)) / (2 * h), (E_(v) - W_(v)) / (2 * h)  # y-faces (y + 1/2)
        uy, vy, ux, vx = (N_(u) - u) / h, (N_(v) - v) / h, 0.5 * (tu + N_(tu)), 0.5 * (tv + N_(tv))
        tyy, txy = NS_MU * (4 / 3 * vy - 2 / 3 * ux), NS_MU * (uy + vx)
        fe = txy * 0.5 * (u + N_(u)) + tyy * 0.5 * (v + N_(v)) + kappa * (N_(T) - T) / h
        for i, f in ((1, txy), (2, tyy), (3, fe)):
            L[i] = L[i] + (f - S_(f)) / h
        return dt * torch.stack(L, 1)

    return _rk3(q, dtl, steps)


def _lagrange(s):
    """Weights of the cubic through nodes -1, 0, 1, 2 at s."""
    return [-s * (s - 1) * (s - 2) / 6, (s + 1) * (s - 1) * (s - 2) / 2, -(s + 1) * s * (s - 2) / 2,
            (s + 1) * s * (s - 1) / 6]


def _prolong(c, r, axis):
    """4-point Lagrange interpolation by r along an axis of a periodic grid."""
    parts = []
    for m in range(r):
        w = _lagrange(m / r)
        parts.append(sum(w[t] * torch.roll(c, 1 - t, axis) for t in range(4)))
    out = torch.stack(parts, axis + 1 if axis >= 0 else c.dim() + axis + 1)
    shape = list(c.shape)
    shape[axis] *= r
    return out.reshape(shape)


def _observe(x, p):
    """H^C of coarse states x (count x nx): the Lagrange row at each observed fine node."""
    nc, r, nf = p["nc"], p["ratio"], p["nf"]
    idx, var = p["idx"].astype(np.int64), p["var"].astype(np.int64)
    w = np.array([_lagrange(m / r) for m in range(r)])
    off = np.arange(-1, 3)
    if p["model"] == "burgers":
        taps = (idx[:, None] // r + off) % nc
        wt = w[idx % r]
    else:
        fy, fx = idx // nf, idx % nf
        ty, tx = (fy[:, None] // r + off) % nc, (fx[:, None] // r + off) % nc
        taps = (var[:, None, None] * nc * nc + ty[:, :, None] * nc + tx[:, None, :]).reshape(len(idx), -1)
        wt = (w[fy % r][:, :, None] * w[fx % r][:, None, :]).reshape(len(idx), -1)
    taps, wt = torch.as_tensor(taps, device=x.device), torch.as_tensor(wt, device=x.device)
    return (x[:, taps] * wt).sum(-1)


def _analysis_exact(fine, members, p):
    """Stochastic EnKF of the members and the prolonged coarse correction of the fine run."""
    ne, ny, nc, r = p["ne"], p["ny"], p["nc"], p["ratio"]
    if p["model"] == "burgers":
        xs = fine[::r].clone()
    else:
        xs = fine.view(4, p["nf"], p["nf"])[:, ::r, ::r].reshape(-1)
    eps = p["sigma"] * torch.as_tensor(_philox_normals(p["seed"], EPS_TAG, 0, ne * ny), device=DEV).view(ne, ny)
    yf, ys = _observe(members, p), _observe(xs[None], p)[0]
    Y = (yf - yf.mean(0)) / math.sqrt(ne - 1)
    Z = torch.cat([p["yobs"] + eps - yf, (p["yobs"] - ys)[None]])
    s2 = p["sigma"] ** 2
    S = torch.eye(ne, dtype=torch.float64, device=DEV) + Y @ Y.T / s2
    T = torch.linalg.solve(S, Y @ Z.T / s2)
    X = (members - members.mean(0)) / math.sqrt(ne - 1)
    D = T.T @ X
    dC = D[ne]
    if p["model"] == "burgers":
        corr = _prolong(dC, r, -1)
    else:
        corr = _prolong(_prolong(dC.view(4, nc, nc), r, -1), r, -2).reshape(-1)
    d = p["yobs"] - ys
    return fine + corr, members + D[:ne], torch.sqrt((d * d).mean())


def _forecast_exact(p, steps):
    nc, nf = p["nc"], p["nf"]
    if p["model"] == "burgers":
        return (_burgers_exact(p["fine"], 2 * math.pi, p["dt"], steps),
                _burgers_exact(p["members"], 2 * math.pi, p["dt"], steps))
    return (_ns_exact(p["fine"].view(1, 4, nf, nf), p["dt"], steps).reshape(-1),
            _ns_exact(p["members"].view(-1, 4, nc, nc), p["dt"], steps).reshape(p["ne"], -1))


def _cnn_forward_exact(dC, xs, w, stats):
    def conv(a, W, b):
        return torch.nn.functional.conv2d(torch.nn.functional.pad(a, (1, 1, 1, 1), mode="circular"), W, b)

    mu, sc = (stats[k].view(1, 8, 1, 1) for k in ("mu_in", "s_in"))
    a = (torch.cat([dC, xs], 1) - mu) / sc
    a = torch.relu(conv(a, w["W1"], w["b1"]))
    a = torch.relu(conv(a, w["W2"], w["b2"]))
    return torch.nn.functional.pixel_shuffle(conv(a, w["W3"], w["b3"]), 4) * stats["s_out"].view(1, 4, 1, 1)


def _cnn_exact(case, seed):
    dC, xs, target, params, stats = _cnn_data(case, seed)
    f64 = lambda a: torch.as_tensor(a, device=DEV).double()  # noqa: E731
    w = {k: f64(v).requires_grad_(case["kind"] == "cnn_train") for k, v in params.items()}
    stats = {k: f64(v) for k, v in stats.items()}
    if case["kind"] == "cnn_infer":
        return _cnn_forward_exact(f64(dC), f64(xs), w, stats)
    names = [k for k, _ in M.CNN_SHAPES]
    grads = {k: torch.zeros_like(w[k]) for k in names}
    loss = 0.0
    for b in range(case["batch"]):  # sample by sample: the FP64 convolutions' workspaces stay small
        x, y = f64(dC[b:b + 1]), f64(target[b:b + 1])
        pred = _prolong(_prolong(x, 4, -1), 4, -2) + _cnn_forward_exact(x, f64(xs[b:b + 1]), w, stats)
        part = (((pred - y) / stats["s_out"].view(1, 4, 1, 1)) ** 2).mean() / case["batch"]
        for k, g in zip(names, torch.autograd.grad(part, [w[k] for k in names])):
            grads[k] += g
        loss += float(part)
    g = torch.cat([grads[k].reshape(-1) for k in names])
    p = torch.cat([w[k].detach().reshape(-1) for k in names])
    p = p - 3e-4 * g / (g.abs() + 1e-8)  # the first Adam step
    return dict(loss=torch.tensor([loss], dtype=torch.float64), params=p.cpu().numpy(), grads=g.cpu().numpy())


def _dual_exact(d):
    nc, nf, r, ne, ny = d["nc"], d["nf"], d["r"], d["ne"], d["ny"]

    def forecast(u, theta, steps):
        u, theta = np.atleast_2d(u).copy(), np.atleast_2d(theta)
        n, dt = u.shape[1], d["dt"]
        dx = d["length"] / n

        def rhs(v):
            f = 0.5 * v * v
            return (-(f[:, 2:] - f[:, :-2]) / (2 * dx)
                    + d["nu"] * (v[:, 2:] - 2 * v[:, 1:-1] + v[:, :-2]) / dx ** 2)

        def bc(inner, t):
            v = np.empty_like(u)
            v[:, 1:-1] = inner
            v[:, 0] = d["u0"] * (1 + theta[:, 0] * np.sin(d["omega"] * t + theta[:, 1]))
            v[:, -1] = 2 * v[:, -2] - v[:, -3]
            return v

        for s in range(steps):
            t = d["t0"] + s * dt
            u1 = bc(u[:, 1:-1] + dt * rhs(u), t + dt)
            u2 = bc(0.75 * u[:, 1:-1] + 0.25 * (u1[:, 1:-1] + dt * rhs(u1)), t + 0.5 * dt)
            u = bc(u[:, 1:-1] / 3 + 2 / 3 * (u2[:, 1:-1] + dt * rhs(u2)), t + dt)
        return u

    def rows(k):  # open grid: the cubic through 4 coarse nodes, one-sided at the ends
        j0 = np.minimum(np.maximum(k // r - 1, 0), nc - 4)
        s = k / r - j0
        w = np.stack([np.prod([(s - b) / (a - b) for b in range(4) if b != a], axis=0) for a in range(4)], 1)
        return j0[:, None] + np.arange(4), w

    def interp(x, tw):
        return (x[..., tw[0]] * tw[1]).sum(-1)

    def solve(xf, xs):
        yf = interp(xf, obs)
        Y = (yf - yf.mean(0)) / math.sqrt(ne - 1)
        Z = np.concatenate([d["yobs"] + eps - yf, (d["yobs"] - interp(xs, obs))[None]])
        s2 = d["sigma"] ** 2
        return np.linalg.solve(np.eye(ne) + Y @ Y.T / s2, Y @ Z.T / s2)

    def anomalies(a):
        return (a - a.mean(0)) / math.sqrt(ne - 1)

    obs, fine_rows = rows(d["idx"].astype(np.int64)), rows(np.arange(nf))
    eps = d["sigma"] * _philox_normals(d["seed"], EPS_TAG, 0, ne * ny).reshape(ne, ny)
    tau = math.sqrt(d["q"]) * _philox_normals(d["seed"], THETA_TAG, 0, 2 * ne).reshape(ne, 2)
    steps = d["steps"]
    fine = forecast(d["fine"], d["theta_fine"], steps)[0]
    theta_f = d["theta"] + tau
    xs = fine[::r][:nc]
    T = solve(forecast(d["members"], theta_f, steps), xs)
    theta = theta_f + (anomalies(theta_f).T @ T[:, :ne]).T
    xf = forecast(d["members"], theta, steps)
    T = solve(xf, xs)
    inc = anomalies(xf).T @ T
    return fine + interp(inc[:, ne], fine_rows), xf + inc[:, :ne].T, theta, theta.mean(0)


def exact(case, seed):
    k = case["kind"]
    if k in ("cycle", "forecast", "analysis"):
        p = _problem(case["model"], case["nc"], case["ratio"], case["ne"], case["ny"], case["precision"] == "mixed",
                     seed)
        fine, members = (p["fine"], p["members"]) if k == "analysis" else _forecast_exact(p, case["steps"])
        return (fine, members) if k == "forecast" else _analysis_exact(fine, members, p)[:2]
    if k == "truth":
        q, n = _truth_state(case, seed), case["n"]
        if case["model"] == "burgers":
            return _burgers_exact(q, 2 * math.pi, _dt("burgers", n), case["steps"])
        return _ns_exact(q, _dt("ns", n), case["steps"])
    if k == "batch":
        out = []
        for j, (nc, ne, ny) in enumerate(_batch_sizes(case)):
            p = _problem("ns", nc, 4, ne, ny, True, seed * 131 + j)
            f, m, innov = _analysis_exact(*_forecast_exact(p, case["steps"]), p)
            out.append((f, m.reshape(-1), innov.view(1)))
        return tuple(torch.cat([o[i] for o in out]) for i in range(3))
    if k in ("cnn_infer", "cnn_train"):
        return _cnn_exact(case, seed)
    return _dual_exact(dict(_dual_data(case, seed), steps=case["steps"]))
