"""What a user of this library has it do, as cases that can be timed and compared.

Every case goes through the package's public entry points (``Hawkes``,
``Batch``, ``MLP`` and the samplers' ``HawkesTarget`` / ``SurrogateField``) on
the synthetic county-structured workloads of ``synth``.  The kinds:

  step      one MCMC step: a fresh location draw, then the FP32
            log-likelihood and gradient over every pair (synchronous call)
  bgtime    the same with eq. 2's time-only background and s_j = 1, on
            integer-day times with many ties (case counts reported by day)
  spatial   the same step with the exact spatial skip, which long runs at
            paper scale use
  f64       the FP64 reference path (the plain method)
  hmc       one exact evaluation of lockstep HMC chains: the location draw,
            staging, the one sweep launch and the reductions as a CUDA graph
  mh        one log-likelihood-only evaluation of the paper's univariate
            sampler: 30 chains, exact underflow skip
  regions   a batch of regional subsets of uneven size, captured as a graph
  train     Adam steps of the surrogate network
  predict   the surrogate's prediction inside a leapfrog step

The FP32 paths form their pair terms and partial sums in FP32, so their
numbers are returned in that type; the FP64 path's are returned in FP64.
"""
import functools
import math

import numpy as np
import torch

from paper_2407_11349_gb300 import hmc, synth
from paper_2407_11349_gb300.hawkes import (HAWKES_BG_TIME, HAWKES_F32, HAWKES_F64, HAWKES_MODEL1,
                                           HAWKES_SKIP_SPATIAL, HAWKES_SKIP_UNDERFLOW, MLP, Batch, Hawkes)

SEED_RESAMPLE = 2


def listed():
    return [
        # the smallest workload of the configurations: latency and launches
        {"name": "step_2k", "kind": "step", "data": "grid", "n": 2000},
        # a regional subset's size, odd, with daily ties: a few row tiles
        {"name": "step_17k_ties", "kind": "step", "data": "grid_ties", "n": 17103},
        # the mid-size workload: N = 100,000 over 1,200 days
        {"name": "step_100k", "kind": "step", "data": "grid", "n": 100_000},
        # the paper's scale, the headline benchmark's step
        {"name": "step_1m", "kind": "step", "data": "voronoi", "n": 1_000_000},
        # eq. 2 as printed, daily counts
        {"name": "bgtime_30k_ties", "kind": "bgtime", "data": "grid_ties", "n": 30_011},
        # the paper's scale with the exact spatial skip (HMC at N = 1M runs on it)
        {"name": "spatial_1m", "kind": "spatial", "data": "voronoi", "n": 1_000_000},
        # the plain method in FP64 on the smallest workload
        {"name": "f64_2k", "kind": "f64", "data": "grid", "n": 2000},
        # exact HMC, 4 chains of 50,000 clustered events
        {"name": "hmc_4x50k", "kind": "hmc", "n": 50_000, "chains": 4},
        # the paper's sampler at its chain count, 20,000 events
        {"name": "mh_30x20k", "kind": "mh", "n": 20_000, "chains": 30},
        # 16 regional subsets, 5k to 200k events, in one launch
        {"name": "regions_16", "kind": "regions", "n": 5000, "ratio": 40.0, "count": 16},
        # surrogate training at the samplers' batch size
        {"name": "train_b512", "kind": "train", "batch": 512, "steps": 20, "n": 4096},
        # a leapfrog step of 4 surrogate-driven chains
        {"name": "predict_4", "kind": "predict", "chains": 4, "n": 4096},
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "bgtime", "spatial", "spatial", "f64", "hmc", "mh", "regions", "train",
                       "predict"])
    if kind == "step":
        return {"kind": kind, "data": rng.choice(["grid", "grid_ties", "voronoi"]), "n": _between(rng, 300, 250_000)}
    if kind == "bgtime":
        return {"kind": kind, "data": rng.choice(["grid", "grid_ties"]), "n": _between(rng, 300, 120_000)}
    if kind == "spatial":
        return {"kind": kind, "data": rng.choice(["grid", "grid_ties", "voronoi"]), "n": _between(rng, 3000, 1_000_000)}
    if kind == "f64":
        return {"kind": kind, "data": rng.choice(["grid", "grid_ties"]), "n": _between(rng, 300, 12_000)}
    if kind == "hmc":
        c = rng.randint(1, 8)
        return {"kind": kind, "n": _between(rng, 1000, 100_000 // c + 1000), "chains": c}
    if kind == "mh":
        c = rng.randint(2, 30)
        return {"kind": kind, "n": _between(rng, 1000, 40_000), "chains": c}
    if kind == "regions":
        return {"kind": kind, "n": _between(rng, 500, 5000), "ratio": float(rng.randint(2, 40)),
                "count": rng.randint(2, 16)}
    if kind == "train":
        return {"kind": kind, "batch": 64 * rng.randint(1, 64), "steps": rng.randint(5, 40), "n": _between(rng, 200, 20_000)}
    return {"kind": "predict", "chains": _between(rng, 1, 4096), "n": _between(rng, 200, 20_000)}


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _voronoi():
    """The 3,143 irregular counties (the map is the same for every seed)."""
    return synth.voronoi_counties(3143, 4500.0, 2800.0, np.random.default_rng(2))


@functools.lru_cache(maxsize=4)
def _dataset(kind, n, seed):
    if kind == "voronoi":
        return synth.voronoi_dataset(n, seed=seed, counties=_voronoi())
    if n <= 10_000:  # the small workload: 100 days on a 20 x 20 grid of counties
        ds = synth.grid_dataset(n, 100.0, 20, 20, seed=seed)
    else:            # the mid-size one: 1,200 days on a 60 x 60 grid
        ds = synth.grid_dataset(n, 1200.0, 60, 60, seed=seed)
    return synth.integer_day_times(ds) if kind == "grid_ties" else ds


def _params(seed):
    return synth.chain_params(1, seed=seed)[0]


def _eta(case, seed):
    return np.log(synth.chain_params(case["chains"], seed=seed))


def _training_set(case, seed):
    """Log-parameters around a starting point and a smooth log-likelihood-like
    surface with its gradient (what warmup records, in shape and scale)."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    eta0 = np.log(np.asarray(synth.DEFAULT_PARAMS))
    scale = rng.uniform(0.01, 0.05, 6)
    z = rng.normal(size=(n, 6))
    A = rng.normal(size=(6, 6)) / 6.0
    H = np.eye(6) + A @ A.T
    cubic = rng.uniform(-0.1, 0.1, 6)
    ll = -5e4 - 0.5 * np.einsum("ni,ij,nj->n", z, H, z) + z ** 3 @ cubic
    grad = (-(z @ H) + 3.0 * z ** 2 * cubic) / scale
    return eta0 + z * scale, np.column_stack([ll, grad]), eta0, scale


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "bgtime", "spatial", "f64"):
        ds = _dataset(case["data"], case["n"], seed)
        hk = Hawkes(0).load(ds)
        flags = {"step": HAWKES_F32, "bgtime": HAWKES_F32 | HAWKES_BG_TIME | HAWKES_MODEL1,
                 "spatial": HAWKES_F32 | HAWKES_SKIP_SPATIAL, "f64": HAWKES_F64}[kind]
        p = _params(seed)
        if kind == "spatial":  # the order of the events belongs to loading them
            hk.loglik_grad(p, flags)
        return {"kind": kind, "hk": hk, "p": p, "flags": flags, "k": 0}
    if kind in ("hmc", "mh"):
        ds = synth.clustered_dataset(case["n"], T=1200.0, nx=40, ny=40, seed=seed)
        tgt = hmc.HawkesTarget(ds, case["chains"], seed=SEED_RESAMPLE,
                               flags=HAWKES_SKIP_UNDERFLOW if kind == "mh" else 0)
        eta = _eta(case, seed)
        if kind == "mh":
            tgt.eval_loglik(eta)  # makes the log-likelihood-only batches
        return {"kind": kind, "tgt": tgt, "eta": eta, "k": 0}
    if kind == "regions":
        base = _dataset("voronoi", 250_000, seed)
        sizes = synth.regional_sizes(case["count"], case["n"], case["ratio"])
        stream = torch.cuda.Stream()
        hks = [Hawkes(0, stream.cuda_stream).load(d) for d in synth.regional_subsets(base, sizes, seed=seed)]
        P = len(hks)
        batch = Batch(hks, [SEED_RESAMPLE] * P, list(range(P)), HAWKES_F32, stream.cuda_stream)
        dp = torch.from_numpy(synth.chain_params(P, seed=seed)).cuda()
        out = torch.zeros((P, 7), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        batch.capture(dp.data_ptr(), out.data_ptr())
        return {"kind": kind, "batch": batch, "dp": dp, "out": out, "stream": stream, "k": 0}
    X, Y, eta0, scale = _training_set(case, seed)
    net = MLP(0, seed=seed)
    net.set_data(X, Y)
    if kind == "train":
        net.train(50, batch=case["batch"], lr=1e-3, seed=seed)  # past Adam's first steps
        return {"kind": kind, "net": net, "batch": case["batch"], "steps": case["steps"], "seed": seed}
    rng = np.random.default_rng(seed + 1)
    return {"kind": kind, "field": hmc.SurrogateField(net, case["chains"]),
            "eta": eta0 + rng.normal(size=(case["chains"], 6)) * scale}


# ----------------------------------------------------------------------------
# One pass
# ----------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind in ("step", "bgtime", "spatial"):
        hk, k = state["hk"], state["k"]
        state["k"] = k + 1
        hk.resample(SEED_RESAMPLE, 0, k)
        ll, g = hk.loglik_grad(state["p"], state["flags"])
        return {"loglik": ll, "grad": g.astype(np.float32)}
    if kind == "f64":
        ll, g = state["hk"].loglik_grad(state["p"], state["flags"])
        return {"loglik": np.float64(ll), "grad": g}
    if kind == "hmc":
        state["k"] += 1
        ll, g = state["tgt"].resample_eval(state["k"], state["eta"])
        return {"loglik": ll.astype(np.float32), "grad": g.astype(np.float32)}
    if kind == "mh":
        state["k"] += 1
        ll, _ = state["tgt"].resample_eval_loglik(state["k"], state["eta"])
        return {"loglik": ll.astype(np.float32)}
    if kind == "regions":
        state["k"] += 1
        state["batch"].run(state["dp"].data_ptr(), state["k"], state["out"].data_ptr())
        state["batch"].wait()
        o = state["out"].cpu().numpy().astype(np.float32)
        return {"loglik": o[:, 0], "grad": o[:, 1:]}
    if kind == "train":
        loss = state["net"].train(state["steps"], batch=state["batch"], lr=1e-3, seed=state["seed"])
        return {"loss": loss, "params": state["net"].get_params()}
    ll, g = state["field"](state["eta"])
    return {"loglik": ll.astype(np.float32), "grad": g.astype(np.float32)}


# ----------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------
# Floating-point operations per unordered pair (a fused multiply-add is two,
# an exponential one): differences, r^2 and dt^2 (7), the background exponent
# and its exponential (2), its three moments at the row and at the column
# (10), the excitation exponent and its exponential (5), its moments (5).
FLOPS_PAIR = 29
FLOPS_PAIR_BGT = 24  # no r^2 in the background exponent and no r^2 moment
FLOPS_PAIR_LL = 18   # the two sums of the log-likelihood alone
EVENT_BYTES = 44     # t, x, y, s in FP64, tie range and county as 32-bit words
# Share of the unordered pairs with a term above 2^-126 at these parameters
# (counted on samples of the workloads' pairs): what the spatial skip needs.
NEAR = {"voronoi": 1.85e-3, "grid": 2.35e-3, "grid_ties": 2.35e-3}


def _pairs(n):
    return 0.5 * n * (n - 1)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "step" or kind == "f64":
        return {"bytes": EVENT_BYTES * n + 56, "flops": FLOPS_PAIR * _pairs(n)}
    if kind == "bgtime":
        return {"bytes": EVENT_BYTES * n + 56, "flops": FLOPS_PAIR_BGT * _pairs(n)}
    if kind == "spatial":
        near = NEAR[case["data"]] if n > 10_000 else 0.15  # 100 days on 1,000 x 1,000 km: a denser map
        return {"bytes": EVENT_BYTES * n + 56, "flops": FLOPS_PAIR * near * _pairs(n)}
    if kind == "hmc":
        return {"bytes": (EVENT_BYTES * n + 56) * case["chains"], "flops": FLOPS_PAIR * _pairs(n) * case["chains"]}
    if kind == "mh":
        # the underflow skip leaves the pairs within 93 days (background) or
        # about 437 days (excitation) of 1,200
        near = 0.6 * _pairs(n)
        return {"bytes": (EVENT_BYTES * n + 56) * case["chains"], "flops": FLOPS_PAIR_LL * near * case["chains"]}
    if kind == "regions":
        sizes = synth.regional_sizes(case["count"], case["n"], case["ratio"])
        return {"bytes": EVENT_BYTES * sum(sizes), "flops": FLOPS_PAIR * sum(_pairs(m) for m in sizes)}
    w = 7 * 256 + 256 * 256 + 256 * 7
    if kind == "train":  # forward, weight and activation gradients; weights, two moments and gradient
        return {"bytes": case["steps"] * (69639 * 4 * 6 + case["batch"] * 56), "flops": case["steps"] * 6.0 * w * case["batch"]}
    return {"bytes": 69639 * 4 + case["chains"] * 13 * 8, "flops": 2.0 * w * case["chains"]}


# ----------------------------------------------------------------------------
# The same in 64 bits, without the library
# ----------------------------------------------------------------------------

def _mulhi(a, b):
    """High 64 bits of the product of an array of uint64 and a constant."""
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    a0, a1, b0, b1 = a & m, a >> s, np.uint64(b & 0xFFFFFFFF), np.uint64(b >> 32)
    mid = a1 * b0 + ((a0 * b0) >> s)
    return a1 * b1 + (mid >> s) + (((mid & m) + a0 * b1) >> s)


def _philox4x64(i, iteration, key0, key1):
    """Philox4x64-10 (Salmon et al. 2011) with counter (i, iteration, 0, 0)."""
    M0, M1, W0, W1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157, 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B
    c = [i.astype(np.uint64), np.full(i.shape, iteration, np.uint64), np.zeros(i.shape, np.uint64),
         np.zeros(i.shape, np.uint64)]
    for r in range(10):
        k0 = np.uint64((key0 + r * W0) & 0xFFFFFFFFFFFFFFFF)
        k1 = np.uint64((key1 + r * W1) & 0xFFFFFFFFFFFFFFFF)
        h0, l0 = _mulhi(c[0], M0), c[0] * np.uint64(M0)
        h1, l1 = _mulhi(c[2], M1), c[2] * np.uint64(M1)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _locations(ds, stream, iteration):
    """The location draw: an area-weighted triangle of the county, then the
    square-root barycentric map."""
    tri, xy = ds.counties.tri_county, ds.counties.tri_xy
    area = 0.5 * np.abs((xy[:, 2] - xy[:, 0]) * (xy[:, 5] - xy[:, 1]) - (xy[:, 4] - xy[:, 0]) * (xy[:, 3] - xy[:, 1]))
    first = np.searchsorted(tri, np.arange(ds.counties.n))
    last = np.searchsorted(tri, np.arange(ds.counties.n), side="right") - 1
    with np.errstate(over="ignore"):
        w = _philox4x64(np.arange(ds.n), iteration, SEED_RESAMPLE, stream)
    u = [(v >> np.uint64(11)).astype(np.float64) / 9007199254740992.0 for v in w[:3]]
    pick = np.empty(ds.n, dtype=np.int64)
    order = np.argsort(ds.county, kind="stable")
    bounds = np.searchsorted(ds.county[order], np.arange(ds.counties.n + 1))
    for c in range(ds.counties.n):
        idx = order[bounds[c]:bounds[c + 1]]
        cum = np.cumsum(area[first[c]:last[c] + 1])
        pick[idx] = first[c] + np.minimum(np.searchsorted(cum, u[0][idx] * cum[-1], side="right"), cum.size - 1)
    v, r1 = xy[pick], np.sqrt(u[1])
    w0, w1, w2 = 1.0 - r1, r1 * (1.0 - u[2]), r1 * u[2]
    return w0 * v[:, 0] + w1 * v[:, 2] + w2 * v[:, 4], w0 * v[:, 1] + w1 * v[:, 3] + w2 * v[:, 5]


def _loglik64(t, x, y, s, p, bg_time=False):
    """eqs. 2-4 over all ordered pairs in FP64: ell and its six partials."""
    mu, tx, tt, th, om, h = (float(v) for v in p)
    t, x, y, s = (torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda") for a in (t, x, y, s))
    n = t.numel()
    cb = 1.0 / (math.sqrt(2 * math.pi) * tx * tx * tt) * (1.0 if bg_time else 1.0 / (2 * math.pi))
    ce = om / (2 * math.pi * h * h)
    tN = t[-1]
    is2 = 1.0 / (s * s)
    total = torch.zeros(7, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // n)
    for a in range(0, n, step):
        ti = t[a:a + step]
        d = ti[:, None] - t[None, :]
        r2 = (x[a:a + step, None] - x[None, :]).square_().add_((y[a:a + step, None] - y[None, :]).square_())
        B = d.square().mul_(-0.5 / (tt * tt))
        if not bg_time:
            B.sub_(r2 * (0.5 / (tx * tx)))
        B.exp_().mul_(d != 0).mul_(cb)
        SB, SBt = B.sum(1), (B * d).mul_(d).sum(1)
        SBr = torch.zeros_like(SB) if bg_time else (B * r2).sum(1)
        del B
        q = r2.mul_(is2[None, :])
        E = (q * (-0.5 / (h * h))).sub_(om * d)
        E.masked_fill_(d <= 0, -math.inf).exp_().mul_(is2[None, :]).mul_(ce)
        SE, SEt, SEq = E.sum(1), (E * d).sum(1), (E * q).sum(1)
        del E, q, d, r2
        lam = mu * SB + th * SE
        on = lam >= 1e-40
        il = torch.where(on, 1.0 / lam, torch.zeros_like(lam))
        ua, ub = (tN - ti) / tt, -ti / tt
        Pa, Pb = torch.special.ndtr(ua), torch.special.ndtr(ub)
        pa, pb = (torch.exp(-0.5 * v * v) / math.sqrt(2 * math.pi) for v in (ua, ub))
        ea = torch.exp(-om * (tN - ti))
        total += torch.stack([
            (torch.log(torch.clamp(lam, min=1e-40)) - mu * (Pa - Pb) - th * (1 - ea)).sum(),
            (SB * il - (Pa - Pb)).sum(),
            (mu * (SBr / tx ** 3 - 2 * SB / tx) * il).sum(),
            (mu * (SBt / tt ** 3 - SB / tt) * il - mu * (-pa * ua + pb * ub) / tt).sum(),
            (SE * il - (1 - ea)).sum(),
            (th * (SE / om - SEt) * il - th * (tN - ti) * ea).sum(),
            (th * (SEq / h ** 3 - 2 * SE / h) * il).sum()])
    o = total.cpu().numpy()
    return o[0], o[1:]


EXACT_PAIRS = 3e10  # ordered pairs that stay well within 20 s


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "bgtime", "spatial", "f64"):
        if float(case["n"]) ** 2 > EXACT_PAIRS:
            return None
        ds = _dataset(case["data"], case["n"], seed)
        x, y = (ds.x, ds.y) if kind == "f64" else _locations(ds, 0, 0)
        s = np.ones(ds.n) if kind == "bgtime" else ds.s
        ll, g = _loglik64(ds.t, x, y, s, _params(seed), bg_time=kind == "bgtime")
        return {"loglik": np.float64(ll), "grad": g}
    if kind in ("hmc", "mh"):
        if case["chains"] * float(case["n"]) ** 2 > EXACT_PAIRS:
            return None
        ds = synth.clustered_dataset(case["n"], T=1200.0, nx=40, ny=40, seed=seed)
        p = np.exp(_eta(case, seed))
        out = [_loglik64(ds.t, *_locations(ds, c, 1), ds.s, p[c]) for c in range(case["chains"])]
        ll = np.array([o[0] for o in out])
        return {"loglik": ll} if kind == "mh" else {"loglik": ll, "grad": np.stack([o[1] for o in out]) * p}
    if kind == "regions":
        sizes = synth.regional_sizes(case["count"], case["n"], case["ratio"])
        if sum(float(m) ** 2 for m in sizes) > EXACT_PAIRS:
            return None
        P = len(sizes)
        p = synth.chain_params(P, seed=seed)
        subs = synth.regional_subsets(_dataset("voronoi", 250_000, seed), sizes, seed=seed)
        out = [_loglik64(d.t, *_locations(d, k, 1), d.s, p[k]) for k, d in enumerate(subs)]
        return {"loglik": np.array([o[0] for o in out]), "grad": np.stack([o[1] for o in out])}
    # The network's weights are made by the library's own generator, so its
    # outputs have no value without it.
    return None
