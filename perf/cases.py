"""The work that users of this library have it do, as cases that a timing program can prepare and run.

Every case goes through the public entry points of ``paper_2403_03156_gb300.fsmp``: chains on
device-resident batches (``Context.run_device``), single events and streams of events from host
memory (``Context.submit`` / ``Context.poll``), the LucyDDM deconvolution (``Context.lucyddm``),
the deconvolution followed by chains from its state, and the entry point that allocates nothing
(``run_device_noalloc``). Inputs are simulated by ``workloads`` from the seed alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2403_03156_gb300 import fsmp, workloads

# kind -> (workload whose model and inputs it takes, precision, other context parameters)
KINDS = {
    # a bulk batch of uneven windows, 0.5 to 50 photo-electrons: the ordinary offline analysis
    "uneven": ("batched_uneven_100k", fsmp.FP32_REFRESH, dict(refresh_every=64)),
    # bulk low-occupancy data (dark-matter-like), half a warp per chain as the tuner picks for it
    "lowocc": ("lowocc_bulk_1m", fsmp.FP32_REFRESH, dict(refresh_every=64, pe_lanes=16)),
    # the MCP-PMT charge mixture
    "mcp": ("mcp_uneven_20k", fsmp.FP32_REFRESH, dict(refresh_every=64)),
    # long windows with 50 to 200 photo-electrons
    "pileup": ("highpileup_20k_1024", fsmp.FP32_REFRESH, dict(refresh_every=32)),
    # FP64 mode, the reference-quality run a user checks an analysis with
    "fp64": ("plain_fp64_256x128", fsmp.FP64, dict()),
    # events of 1 to 64 channels from host memory, as a readout hands them over
    "events": ("serving_20k_eps", fsmp.FP32_REFRESH, dict(refresh_every=64)),
    # the deconvolution alone
    "lucy": ("batched_uneven_100k", fsmp.FP32_REFRESH, dict(refresh_every=64)),
    # deconvolution, then chains from its state with PE-time histograms: the paper's whole path
    "lucy_chains": ("batched_uneven_100k", fsmp.FP32_REFRESH, dict(refresh_every=64)),
    # chains for a caller that cannot allocate device memory (static scratch, Sigma^-1 kernel)
    "noalloc": ("lowocc_bulk_1m", fsmp.FP32_REFRESH, dict(refresh_every=64)),
}
HIST_WIDTH = 1024  # grid points of a PE-time histogram (256 ns at 0.25 ns)


def listed():
    return [
        # one waveform, a short chain: a user's first call, where the launch and the chain's ends count
        dict(name="one_waveform", kind="lowocc", n=1, steps=200),
        # one event of a readout, submit to result: what its latency is made of
        dict(name="one_event", kind="events", n=1, steps=1500),
        # a burst of events through the serving loop
        dict(name="event_burst", kind="events", n=64, steps=1500),
        # bulk analysis of uneven windows, more chains than the GPU holds at once
        dict(name="uneven_20k", kind="uneven", n=20_000, steps=2000),
        # a run's worth that does not fill the GPU: odd count, short chains
        dict(name="uneven_777", kind="uneven", n=777, steps=1000),
        # bulk low-occupancy data
        dict(name="lowocc_100k", kind="lowocc", n=100_000, steps=1000),
        # MCP-PMT charges
        dict(name="mcp_5k", kind="mcp", n=5_000, steps=2000),
        # pile-up
        dict(name="pileup_1k", kind="pileup", n=1_000, steps=2000),
        # the FP64 configuration
        dict(name="fp64_256", kind="fp64", n=256, steps=1000),
        # the paper's 2000 Lucy iterations on a bulk batch
        dict(name="lucy_10k", kind="lucy", n=10_000, steps=2000),
        # the paper's whole path on a batch
        dict(name="lucy_chains_3k", kind="lucy_chains", n=3_001, steps=500),
        # chains without allocation
        dict(name="noalloc_2k", kind="noalloc", n=2_000, steps=300),
    ]


# ranges of drawn cases: waveforms (or events) and steps (or Lucy iterations)
RANGES = {
    "uneven": ((1, 20_000), (200, 2000)),
    "lowocc": ((1, 100_000), (200, 1000)),
    "mcp": ((16, 5_000), (200, 2000)),
    "pileup": ((8, 1_000), (200, 2000)),
    "fp64": ((8, 512), (200, 1000)),
    "events": ((1, 64), (300, 1500)),
    "lucy": ((1, 10_000), (50, 2000)),
    "lucy_chains": ((16, 4_000), (100, 500)),
    "noalloc": ((8, 4_000), (50, 300)),
}


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    size = [max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))
            for lo, hi in RANGES[kind]]
    return dict(kind=kind, n=size[0], steps=size[1])


def _params(kind):
    name, precision, more = KINDS[kind]
    return dict(workloads.CONFIGS[name]["params"], n_max=_n_max(kind), precision=precision, **more)


def _n_max(kind):
    cfg = workloads.CONFIGS[KINDS[kind][0]]
    return int(cfg.get("win_max", cfg["window"]))


@functools.lru_cache(maxsize=None)
def _context(kind):
    """One context per model, kept as a program keeps it. Contexts of device batches launch on the
    caller's stream only, so they carry one serving stream."""
    more = {} if kind == "events" else dict(n_streams=1)
    return fsmp.Context(_params(kind), **more)


def _burn(steps):
    return steps // 5


FLOATS = [n for n in fsmp.SUMMARY_DTYPE.names if fsmp.SUMMARY_DTYPE[n].kind == "f"]


def _device_outputs(out, W):
    """The summaries in a device buffer, field by field: 15 FP64 values, then 14 integers."""
    words = out.view(torch.float64).view(W, -1)
    got = {n: words[:, i] for i, n in enumerate(FLOATS)}
    got["counts"] = out.view(torch.int32).view(W, -1)[:, 2 * len(FLOATS):]
    return got


def _host_outputs(s):
    got = {n: s[n] for n in FLOATS}
    whole = s.view(np.int32).reshape(len(s), -1)[:, 2 * len(FLOATS):]
    got["counts"] = np.ascontiguousarray(whole)
    return got


def _batch(case, seed):
    """The waveforms of a device batch in decreasing expected cost, as the library's documents
    advise (the heaviest chains start first)."""
    kind = case["kind"]
    wl = workloads.make_workload(KINDS[kind][0], n_waveforms=case["n"], seed=seed)
    b = wl["batch"]
    cost = np.diff(b["offsets"]) * (1.0 + b["lambda0"])
    return workloads.subset(b, np.argsort(-cost, kind="stable"))


def _events(case, seed):
    """A readout's events: 1 to 64 channels each and lambda over its whole range, both spread
    evenly (event 0 has 32 channels and the middle lambda), so that the batch of another seed is
    other waveforms of the same size."""
    cfg = workloads.CONFIGS[KINDS["events"][0]]
    p, (_, lo, hi) = cfg["params"], cfg["lam"]
    rng = np.random.Generator(np.random.PCG64(seed))
    events, base = [], 0
    for i in range(case["n"]):
        nw = 1 + (37 * i + 31) % 64
        lam = lo * (hi / lo) ** ((0.618034 * i + 0.5) % 1.0)
        t0 = float(rng.uniform(p["t0_lo"], p["t0_hi"]))
        b, _ = workloads.simulate(p, np.full(nw, lam), np.full(nw, t0), rng, "uniform", cfg["win_min"], cfg["win_max"])
        b.update(seed=seed, index_base=base, n_steps=case["steps"], burn_in=_burn(case["steps"]))
        base += nw
        events.append(b)
    return events


def _fixed(samples, W, longest):
    """The samples at the front of a buffer with room for W of the longest windows."""
    buf = np.zeros(W * longest, np.float32)
    buf[:len(samples)] = samples
    return buf


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, kind=kind, seed=seed, steps=case["steps"], burn=_burn(case["steps"]))
    if kind == "events":
        return dict(state, ctx=_context(kind), events=_events(case, seed))
    b = _batch(case, seed)
    W = case["n"]
    dev = torch.device("cuda", 0)
    # windows are as long as their data asks: a buffer for the longest keeps one size
    t = dict(samples=torch.from_numpy(_fixed(b["samples"], W, _n_max(kind))).to(dev), offsets=torch.from_numpy(b["offsets"]).to(dev),
             lambda0=torch.from_numpy(b["lambda0"]).to(dev), t_origin_ns=torch.from_numpy(b["t_origin_ns"]).to(dev),
             wf_ids=torch.from_numpy(b["wf_ids"].astype(np.int64)).to(dev),
             out=torch.zeros(W * fsmp.SUMMARY_DTYPE.itemsize, dtype=torch.uint8, device=dev))
    if "T_lo" in b and not kind.startswith("lucy"):
        t["T_lo"], t["T_hi"] = torch.from_numpy(b["T_lo"]).to(dev), torch.from_numpy(b["T_hi"]).to(dev)
    if kind == "lucy_chains":
        t["pe_hist"] = torch.zeros((W, HIST_WIDTH), dtype=torch.int32, device=dev)
    state.update(t=t, longest=int(np.diff(b["offsets"]).max()), outputs=_device_outputs(t["out"], W))
    if kind == "noalloc":
        state["params"] = _params(kind)
    else:
        state["ctx"] = _context(kind)
    return state


def run(state):
    kind, steps, burn = state["kind"], state["steps"], state["burn"]
    if kind == "events":
        return _run_events(state["ctx"], state["events"])
    t, seed, longest = state["t"], state["seed"], state["longest"]
    if kind == "noalloc":
        fsmp.run_device_noalloc(state["params"], t, steps, burn, seed=seed, n_max_hint=longest)
        return state["outputs"]
    ctx = state["ctx"]
    if kind == "lucy":
        return ctx.lucyddm(t, n_iter=steps, with_q=True, n_max_hint=longest)
    if kind == "lucy_chains":
        start = ctx.lucyddm(t, n_iter=2000, n_max_hint=longest)
        t["pe_hist"].zero_()
        ctx.run_device(dict(t, **{k: start[k] for k in ("T_lo", "T_hi", "t0_init", "z_init", "n_init")}), steps,
                       burn, seed=seed, n_max_hint=longest)
        return dict(state["outputs"], start=start, pe_hist=t["pe_hist"])
    ctx.run_device(t, steps, burn, seed=seed, n_max_hint=longest)
    return state["outputs"]


def _run_events(ctx, events):
    for i, e in enumerate(events):
        if ctx.submit(e, request_id=i) != fsmp.OK:
            raise RuntimeError("an event was not admitted")
    got = {}
    while len(got) < len(events):
        for r in ctx.poll(len(events), 1000):
            if r["status"] != fsmp.OK:
                raise RuntimeError("an event failed")
            got[r["request_id"]] = r["summaries"]
    return _host_outputs(np.concatenate([got[i] for i in range(len(events))]))


# ---------------------------------------------------------------- work

def _mean_of(spec):
    if spec[0] == "loguniform":
        return (spec[2] - spec[1]) / math.log(spec[2] / spec[1])
    return float(spec[1]) if spec[0] == "fixed" else 0.5 * (spec[1] + spec[2])


def work(case):
    """Bytes: the waveforms and their parameters once, the outputs once. Operations of a chain
    step with p photo-electrons overlapping the proposed one (p = the mean count): its column
    against the residual (2 L_V), the overlap sums and the quadratic form over p x p entries
    (2 p^2), and on the half of the steps that accept, the row products (2 p^2), the update of
    C^-1 (4 entries' operations on p^2 / 2 entries) and the residual. A Lucy iteration: the two
    correlations by the response."""
    kind, steps = case["kind"], case["steps"]
    name = KINDS[kind][0]
    cfg = workloads.CONFIGS[name]
    p = workloads.CONFIGS[name]["params"]
    LV = workloads.pulse_support_samples(p)
    lam = _mean_of(cfg["lam"])
    W = case["n"] * (0.5 * sum(cfg["wf_per_event"]) if kind == "events" else 1)
    n = {"trimmed": 150.0, "uniform": 288.0}.get(cfg["window"]) or float(cfg["window"])
    nbytes = W * (4.0 * n + 4 + 8 * 3 + 8 + fsmp.SUMMARY_DTYPE.itemsize)
    step = 2 * LV + 2 * lam * lam + 0.5 * (2 * lam * lam + 2 * lam * lam + 4 * LV)
    lucy = 2.0 * LV * (2 * n + LV - 1)
    if kind == "lucy":
        cap = p["n_cap"]
        return dict(bytes=W * (4.0 * n + 12 + 4 * (n + LV - 1) + 4 * cap + 24), flops=W * steps * lucy)
    flops = W * steps * step
    if kind == "lucy_chains":
        flops += W * 2000 * lucy
        nbytes += W * (4.0 * HIST_WIDTH + 4 * p["n_cap"] + 24)  # the histograms, the start
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------- 64-bit values

def exact(case, seed):
    """FP64 chains step by step from the model's definition (log p(w | z) by Cholesky of every
    proposed state), and the deconvolution in FP64 where it is small. The other chains' decisions
    hang on their 32-bit rounding, step after step: they have no 64-bit value."""
    if case["kind"] == "fp64":
        return _exact_chains(case, seed)
    if case["kind"] == "lucy" and case["n"] * case["steps"] <= 20_000_000:
        return _exact_lucy(case, seed)
    return None


def _ser(p):
    """The single-electron response on the PE grid: the shifted ex-Gaussian, peak 1, cut after
    the last grid point above ser_eps and rounded up to whole samples."""
    s, tau, g, R = p["ser_sigma"], p["ser_tau"], p["grid_ns"], round(p["dt_sample_ns"] / p["grid_ns"])
    v = []
    for m in range(int(math.ceil((8 * s + 50 * tau) / g)) + 1):
        x = m * g - 4 * s
        v.append(math.exp((s * s - 2 * x * tau) / (2 * tau * tau)) * math.erfc((s * s - x * tau) / (math.sqrt(2) * s * tau)))
    v = np.array(v) / max(v)
    last = int(np.nonzero(np.abs(v) >= p["ser_eps"])[0][-1])
    Lt = -(-(last + 1) // R) * R
    return v[:Lt], R


def _phi(p, x):
    s, tau = p["phi_p1"], p["phi_p2"]
    c = math.erfc((s * s - x * tau) / (math.sqrt(2) * s * tau))
    return math.exp((s * s - 2 * x * tau) / (2 * tau * tau) + math.log(c)) / (2 * tau) if c > 0 else 0.0


def _philox(step, block, seed, ids):
    """Philox4x64-10 of counter (step, block, 0, 0) under the keys (seed, id), as uniforms [4, W]."""
    mask = (1 << 32) - 1

    def mul(m, x):  # 64 x 64 -> 128 bits: (high, low)
        a0, a1 = np.uint64(m & mask), np.uint64(m >> 32)
        b0, b1 = x & np.uint64(mask), x >> np.uint64(32)
        t = a0 * b0
        u = a1 * b0 + (t >> np.uint64(32))
        v = a0 * b1 + (u & np.uint64(mask))
        return a1 * b1 + (u >> np.uint64(32)) + (v >> np.uint64(32)), np.uint64(m) * x

    W = len(ids)
    c = [np.full(W, step, np.uint64), np.full(W, block, np.uint64), np.zeros(W, np.uint64), np.zeros(W, np.uint64)]
    k0, k1 = np.full(W, seed, np.uint64), ids.astype(np.uint64)
    for r in range(10):
        if r:
            k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
        h0, l0 = mul(0xD2E7470EE14C6C93, c[0])
        h1, l1 = mul(0xCA5A826395121157, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return [((x >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for x in c]


def _exact_chains(case, seed):
    p = _params(case["kind"])
    b = _batch(case, seed)
    W, steps, burn = case["n"], case["steps"], _burn(case["steps"])
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    f8 = dict(dtype=torch.float64, device=dev)
    V, R = _ser(p)
    Lt, g, cap, n = len(V), p["grid_ns"], p["n_cap"], _n_max(case["kind"])
    Vt = torch.tensor(np.append(V, 0.0), **f8)
    w = torch.from_numpy(b["samples"].astype(np.float64)).to(dev).view(W, n)
    mu, q, se2 = p["mu_q"], p["sigma_q"] ** 2, p["sigma_noise"] ** 2
    r = se2 / q
    k0_lo, k0_hi = math.ceil(p["t0_lo"] / g - 1e-9), math.floor(p["t0_hi"] / g + 1e-9)
    T = n * R  # the PE solution space is the whole window [0, T)
    d0 = -k0_hi - 1
    phi = np.array([_phi(p, d * g) for d in range(d0, T - k0_lo + 1)])
    lphi = torch.tensor(np.where(phi > 0, np.log(np.where(phi > 0, phi, 1.0)), -np.inf), **f8)
    cphi = torch.tensor(np.cumsum(phi), **f8)
    lam = torch.from_numpy(b["lambda0"]).to(dev)
    log_lam, logJ, J = torch.log(lam), math.log(p["jump_J"]), p["jump_J"]
    xs = torch.arange(n, device=dev) * R

    def columns(j):  # a_j over the window, [W, n]
        i = xs[None, :] - j[:, None]
        return Vt[torch.where((i >= 0) & (i < Lt), i, Lt)]

    eye = torch.eye(cap, **f8)
    rows = torch.arange(W, device=dev)

    def score(A):  # log p(w | z), log |Sigma|, sum of C^-1 A^T y
        y = w - mu * A.sum(1)
        C = A @ A.transpose(1, 2) + r * eye
        Lc = torch.linalg.cholesky(C)
        h = torch.bmm(A, y[:, :, None])
        v = torch.cholesky_solve(h, Lc)
        logdet = n * math.log(se2) + 2 * torch.log(torch.diagonal(Lc, dim1=1, dim2=2)).sum(1) - cap * math.log(r)
        quad = ((y * y).sum(1) - (h * v).sum((1, 2))) / se2
        return -0.5 * (n * math.log(2 * math.pi) + logdet + quad), logdet, v.sum((1, 2))

    z = torch.zeros((W, cap), dtype=torch.int64, device=dev)
    N = torch.zeros(W, dtype=torch.int64, device=dev)
    k0 = torch.full((W,), k0_lo + (k0_hi - k0_lo) // 2, dtype=torch.int64, device=dev)
    A = torch.zeros((W, cap, n), **f8)
    logL, logdet, sv = score(A)
    slots = torch.arange(cap, device=dev)[None, :]
    sums = {k: torch.zeros(W, **f8) for k in ("N", "N2", "K", "K2", "Q", "Q2", "w", "w2")}
    hist = torch.zeros((W, cap + 1), **f8)
    neg = torch.tensor(-math.inf, **f8)
    for step in range(steps):
        u = [torch.from_numpy(x).to(dev) for blk in (0, 1) for x in _philox(step, blk, seed, b["wf_ids"])]
        # the event time
        D = torch.round(torch.sqrt(-2 * torch.log(u[0])) * torch.cos(2 * math.pi * u[1]) / g).long()
        kp = k0 + D
        inside = (kp >= k0_lo) & (kp <= k0_hi)
        kc = torch.where(inside, kp, k0)
        live = slots < N[:, None]
        diff = torch.where(live, lphi[z - kc[:, None] - d0] - lphi[z - k0[:, None] - d0], 0.0).sum(1)
        la0 = torch.where(inside, diff, neg)
        k0 = torch.where(torch.log(u[2]) < la0, kp, k0)
        # the jump: 0 birth, 1 death, 2 update
        jump = torch.where(N == 0, 0, torch.where(u[3] < J, 0, torch.where(u[3] < 2 * J, 1, 2)))
        base = cphi[-1 - k0 - d0]
        tot = cphi[T - 1 - k0 - d0] - base
        jb = (torch.searchsorted(cphi, base + u[4] * tot, right=True) + d0 + k0).clamp(0, T - 1)
        kk = torch.minimum((u[4] * N.double()).long(), (N - 1).clamp(min=0))
        jm = z[rows, kk]
        Du = torch.round(torch.sqrt(-2 * torch.log(u[5])) * torch.cos(2 * math.pi * u[6]) / g).long()
        ju = jm + Du
        in_T = (ju >= 0) & (ju < T)
        juc = torch.where(in_T, ju, jm)
        lu_new, lu_old = lphi[juc - k0 - d0], lphi[jm - k0 - d0]
        birth, death, update = jump == 0, jump == 1, jump == 2
        noop = update & (Du == 0)
        valid = (birth & (N < cap)) | death | (update & ~noop & in_T & torch.isfinite(lu_new))
        slot = torch.where(birth, N.clamp(max=cap - 1), kk)
        jp = torch.where(birth, jb, juc)
        zn, An = z.clone(), A.clone()
        last = (N - 1).clamp(min=0)
        put = torch.where(death, z[rows, last], jp)
        zn[rows, slot] = put
        An[rows, slot] = torch.where(death[:, None], A[rows, last], columns(jp))
        dr = rows[death]
        zn[dr, last[death]] = 0
        An[dr, last[death]] = 0.0
        An[~valid], zn[~valid] = A[~valid], z[~valid]
        logL2, logdet2, sv2 = score(An)
        lPhi = torch.log(tot * g)
        prior = torch.where(birth, log_lam + lPhi - torch.log(N.double() + 1) + logJ * (N == 0).double(),
                            torch.where(death, -log_lam - lPhi + torch.log(N.clamp(min=1).double()) - logJ * (N == 1).double(),
                                        lu_new - lu_old))
        la = torch.where(valid, logL2 - logL + prior, neg)
        acc = valid & (torch.log(u[7]) < la)
        z, A = torch.where(acc[:, None], zn, z), torch.where(acc[:, None, None], An, A)
        logL, logdet, sv = torch.where(acc, logL2, logL), torch.where(acc, logdet2, logdet), torch.where(acc, sv2, sv)
        N = N + acc.long() * torch.where(birth, 1, torch.where(death, -1, 0))
        if step >= burn:
            Q = N.double() * mu + sv
            wt = g * torch.where(slots < N[:, None], z, 0).sum(1).double() / (N.double() + 1)
            for k, x in (("N", N.double()), ("K", k0.double() * g), ("Q", Q), ("w", wt)):
                sums[k] += x
                sums[k + "2"] += x * x
            hist[rows, N] += 1
    m = {k: v / (steps - burn) for k, v in sums.items()}
    zero = torch.zeros(W, **f8)
    return dict(mean_N=m["N"], var_N=m["N2"] - m["N"] ** 2, mean_t0=m["K"], var_t0=m["K2"] - m["K"] ** 2, mean_Q=m["Q"],
                var_Q=m["Q2"] - m["Q"] ** 2, logL=logL, logdet=logdet, drift_max=None, alg_bytes=None,
                lambda_hat=_lambda_hat(hist, lam), mean_wt=m["w"], var_wt=m["w2"] - m["w"] ** 2, mean_we=zero, var_we=zero)


def _lambda_hat(hist, lam0):
    """argmax over lambda >= 0 of -lambda + log sum_N h_N (lambda / lambda0)^N, row by row: a
    scan of (0, the largest N], then Newton steps from its best point."""
    ks = torch.arange(hist.shape[1], dtype=torch.float64, device=hist.device)
    lh = torch.log(hist)  # -inf where nothing was counted
    top = (ks * (hist > 0)).amax(1)
    grid = torch.arange(1, 2001, dtype=torch.float64, device=hist.device) / 2000

    def ll(lam):  # [W, G]
        return -lam + torch.logsumexp(lh[:, None, :] + ks * torch.log(lam / lam0[:, None])[:, :, None], 2)

    lam = torch.clamp(top, min=1.0)[:, None] * grid
    at = torch.stack([ll(lam[:, i:i + 250]).amax(1) for i in range(0, 2000, 250)], 1).amax(1)
    best = torch.cat([ll(lam[:, i:i + 250]) for i in range(0, 2000, 250)], 1).argmax(1)
    x = lam.gather(1, best[:, None])[:, 0]
    for _ in range(60):
        pw = torch.softmax(lh + ks * torch.log(x / lam0)[:, None], 1)
        E = (pw * ks).sum(1)
        var = (pw * ks * ks).sum(1) - E * E
        H = var - E
        nx = torch.where(H < 0, x - (-1 + E / x) * x * x / torch.where(H < 0, H, -1.0), E)
        x = torch.where(nx > 0, nx, x / 2)
    at = torch.maximum(at, ll(x[:, None])[:, 0])
    return torch.where((top == 0) | (lh[:, 0] >= at), torch.zeros_like(x), x)


def _exact_lucy(case, seed):
    p = _params(case["kind"])
    b = _batch(case, seed)
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    f8 = dict(dtype=torch.float64, device=dev)
    V, R = _ser(p)
    v = V[::R]
    S, LV = v.sum(), len(v)
    lens = np.diff(b["offsets"])
    n, W = int(lens.max()), case["n"]
    d = np.zeros((W, n))
    for i in range(W):
        d[i, :lens[i]] = np.maximum(b["samples"][b["offsets"][i]:b["offsets"][i + 1]].astype(np.float64), 0) / S
    d, ln = torch.tensor(d, **f8), torch.tensor(lens, device=dev)
    # K[tau + LV - 1, t] = v(t - tau)
    K = torch.zeros((n + LV - 1, n), **f8)
    for m in range(LV):
        t = torch.arange(n, device=dev)
        K[t - m + LV - 1, t] = float(v[m] / S)
    nq = ln + LV - 1
    q = torch.where(torch.arange(n + LV - 1, device=dev)[None, :] < nq[:, None], (d.sum(1) / nq)[:, None], 0.0)
    for _ in range(case["steps"]):
        wr = q @ K
        q = q * (torch.where(wr > 0, d / torch.where(wr > 0, wr, 1.0), 0.0) @ K.T)
    flat = torch.cat([q[i, :int(nq[i])] for i in range(W)])
    flat = torch.cat([flat, torch.zeros(W * (_n_max(case["kind"]) + LV - 1) - len(flat), **f8)])
    return dict(T_lo=None, T_hi=None, t0_init=None, z_init=None, n_init=None, status=None, q=flat)
