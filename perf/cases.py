"""The work a user of this library has it do, as measurable cases.

Each case is one pass through the public entry points (the Python binding of
include/ppl.h) on inputs made from a seed:

  linefit     likelihood weighting on the line-fitting model with its records
              and log-weights, optionally followed by resampling with the
              record gather (the maximum taken from the summary)
  suffstat    the same with the factor from the data's sufficient statistics
  resample    systematic resampling with the gather of the particles' state
  population  the posterior summary of a given weighted population, then its
              resampling with the maximum taken from that summary
  logsumexp   the normalisation of given log-weights
  smc         the whole bootstrap filter (all T steps in one call)
  batched     many line-fitting data sets of uneven size in one launch
  learned     many data sets under proposals near their posteriors
  train       a training step of the proposal network

`exact` restates the method in 64-bit torch (its own Philox, Box-Muller, model,
normalisation, backpropagation), sharing no code with the library.

A posterior summary is a struct of FP64 fields holding numbers that the
library forms from FP32 log-weights and FP32 moments; a program that goes on
with them in torch takes them as one FP32 row per population, and so do these
cases.  The indices of the best traces are not among the outputs: which of two
traces that tie to the last bits of an FP32 log-weight comes first is a matter
of rounding.  Their log-weights (max_lw, deg_max_lw) are, and so are all
log-weights wherever the call writes them.
"""
import math

import numpy as np
import torch

import paper_2010_08454_gb300 as ppl

POINTS_MAX = 1 << 32      # traces x points of the largest line-fitting case
DEGS = (2, 3, 4, 5)       # the line-fitting model's degree prior
PRIOR_SIGMA, OBS_SIGMA = 10.0, 0.5
TRUE_CUBIC = (1.0, -2.0, 0.0, 0.5)  # y = 1 - 2x + 0.5x^3
FLOAT_FIELDS = {"evidence": (0, 2), "ess": (2, 3), "max_lw": (3, 4), "p_n": (7, 11),
                "mean_c": (11, 17), "deg_mean": (17, 41), "deg_var": (41, 65),
                "deg_max_lw": (65, 69)}  # 8-byte words of a summary


def listed():
    return [
        # the paper's line-fitting example at its own size: 32 points, 10^5
        # particles; latency and launches count
        {"name": "linefit_1e5x32", "kind": "linefit", "n": 100000, "L": 32, "resample": False},
        # the benchmark's step: 2^24 traces x 256 points, then resampling
        {"name": "linefit_2e24x256", "kind": "linefit", "n": 1 << 24, "L": 256, "resample": True},
        # a long data set: more points than one SM's shared memory stages
        {"name": "linefit_2e19x5000", "kind": "linefit", "n": 1 << 19, "L": 5000,
         "resample": False},
        # the benchmark's population by sufficient statistics
        {"name": "suffstat_2e24x256", "kind": "suffstat", "n": 1 << 24, "L": 256},
        # one resampling step of a small filter with a 6-float state (24 B)
        {"name": "resample_1e5x24B", "kind": "resample", "n": 100000, "m": 100000, "words": 6,
         "scale": 1.0},
        # a reweighted population of 32-byte records, summarised and resampled
        {"name": "population_2e24", "kind": "population", "n": 1 << 24, "scale": 1.0},
        # normalisation on its own, at the benchmark's size
        {"name": "logsumexp_2e24", "kind": "logsumexp", "n": 1 << 24, "scale": 20.0},
        # a small tracking filter: per-step latency counts
        {"name": "smc_1e4xT100", "kind": "smc", "n": 10000, "T": 100},
        # the benchmark's filter
        {"name": "smc_2e20xT200", "kind": "smc", "n": 1 << 20, "T": 200},
        # the benchmark's batch: 4096 data sets of 16 to 4096 points, 2^10 to
        # 2^16 particles each
        {"name": "batched_4096", "kind": "batched", "sets": 4096, "n_lo": 1 << 10,
         "n_hi": 1 << 16, "l_lo": 16, "l_hi": 4096},
        # the benchmark's 1024 held-out sets under their proposals
        {"name": "learned_1024x2e16", "kind": "learned", "sets": 1024, "n": 1 << 16},
        # one training step of the proposal network at the benchmark's batch (a
        # run is thousands of them; one, because the BF16 roundings of a step's
        # activations carry any difference in summation order on to the next)
        {"name": "train_b1024", "kind": "train", "batch": 1024, "steps": 1},
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["linefit", "linefit", "suffstat", "resample", "resample", "population",
                       "logsumexp", "smc", "batched", "learned", "train"])
    if kind == "linefit":
        L = log_int(1, 8192)
        return {"kind": kind, "n": log_int(1000, min(1 << 24, POINTS_MAX // (2 * L))), "L": L,
                "resample": rng.random() < 0.5}
    if kind == "suffstat":
        return {"kind": kind, "n": log_int(1000, 1 << 24), "L": log_int(8, 2048)}
    if kind == "resample":
        n = log_int(1000, 1 << 24)
        m = n if rng.random() < 0.7 else log_int(1000, 1 << 23)
        return {"kind": kind, "n": n, "m": m, "words": rng.choice([1, 3, 4, 6, 8, 12]),
                "scale": round(math.exp(rng.uniform(math.log(0.3), math.log(30.0))), 3)}
    if kind == "population":
        return {"kind": kind, "n": log_int(1000, 1 << 24),
                "scale": round(math.exp(rng.uniform(math.log(0.3), math.log(30.0))), 3)}
    if kind == "logsumexp":
        return {"kind": kind, "n": log_int(1000, 1 << 25),
                "scale": round(math.exp(rng.uniform(math.log(0.3), math.log(30.0))), 3)}
    if kind == "smc":
        return {"kind": kind, "n": log_int(1000, 1 << 20), "T": log_int(10, 200)}
    if kind == "batched":
        n_hi, l_hi = log_int(1 << 11, 1 << 16), log_int(32, 4096)
        return {"kind": kind, "sets": log_int(16, 2048), "n_lo": log_int(500, n_hi // 2),
                "n_hi": n_hi, "l_lo": log_int(1, l_hi // 2), "l_hi": l_hi}
    if kind == "learned":
        sets = log_int(16, 1024)
        return {"kind": kind, "sets": sets, "n": log_int(1000, min(1 << 18, (1 << 26) // sets))}
    return {"kind": kind, "batch": log_int(100, 4096), "steps": 1}


# ---- inputs ---------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _line_data(L, seed):
    r = np.random.default_rng([int(seed), L])
    x = r.uniform(-1.0, 1.0, L)
    y = sum(c * x ** k for k, c in enumerate(TRUE_CUBIC)) + OBS_SIGMA * r.standard_normal(L)
    return (torch.from_numpy(x.astype(np.float32)).cuda(),
            torch.from_numpy(y.astype(np.float32)).cuda())


def _batch_data(case, seed):
    """Uneven data sets: sizes log-uniform, true degree uniform, coefficients N(0, 1)."""
    r = np.random.default_rng([int(seed), case["sets"]])
    B = case["sets"]

    def log_uniform(lo, hi):
        v = np.floor(np.exp(r.uniform(np.log(lo), np.log(hi + 1), B)))
        return np.clip(v, lo, hi).astype(np.int64)

    L, N = log_uniform(case["l_lo"], case["l_hi"]), log_uniform(case["n_lo"], case["n_hi"])
    deg = r.integers(DEGS[0], DEGS[-1] + 1, B)
    coef = r.standard_normal((B, 6)) * (np.arange(6) <= deg[:, None])
    own = np.repeat(np.arange(B), L)
    x = r.uniform(-1.0, 1.0, len(own))
    y = OBS_SIGMA * r.standard_normal(len(own))
    for k in range(6):
        y += coef[own, k] * x ** k
    return (x.astype(np.float32), y.astype(np.float32), np.concatenate([[0], np.cumsum(L)]),
            np.concatenate([[0], np.cumsum(N)]))


def _held_out(sets, seed):
    """Data sets of 32 points drawn from the model's own prior, [sets, 32] FP32."""
    r = np.random.default_rng([int(seed), sets, 32])
    deg = r.integers(DEGS[0], DEGS[-1] + 1, sets)
    coef = PRIOR_SIGMA * r.standard_normal((sets, 6)) * (np.arange(6) <= deg[:, None])
    x = r.uniform(-1.0, 1.0, (sets, 32))
    y = OBS_SIGMA * r.standard_normal((sets, 32))
    for k in range(6):
        y += coef[:, k:k + 1] * x ** k
    return torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(y.astype(np.float32)).cuda()


def _near_posterior(x, y):
    """Proposal rows [sets, 48] FP32 as a trained network gives them: every
    degree's posterior mean and a standard deviation somewhat above the
    posterior's conditional one, degree logits near the posterior's."""
    x, y = x.double(), y.double()
    out = torch.zeros(x.shape[0], 48, dtype=torch.float64, device=x.device)
    base = 0
    for k, n in enumerate(DEGS):
        d = n + 1
        phi = torch.stack([x ** j for j in range(d)], 2)
        prec = phi.transpose(1, 2) @ phi / OBS_SIGMA ** 2 + torch.eye(d, device=x.device).double() / PRIOR_SIGMA ** 2
        b = (phi.transpose(1, 2) @ y.unsqueeze(2) / OBS_SIGMA ** 2).squeeze(2)
        mu = torch.linalg.solve(prec, b)
        sd = 1.5 / torch.diagonal(prec, dim1=1, dim2=2).sqrt()
        out[:, k] = 0.5 * (b * mu).sum(1) - 0.5 * torch.logdet(prec) - d * math.log(PRIOR_SIGMA)
        out[:, 4 + 2 * base:4 + 2 * (base + d):2] = mu / PRIOR_SIGMA
        out[:, 5 + 2 * base:5 + 2 * (base + d):2] = (sd / PRIOR_SIGMA).log().clamp(-8.5, 0.5)
        base += d
    out[:, :4] -= out[:, :4].max(1, keepdim=True).values
    out[:, :4].clamp_(min=-3.0)  # a network leaves every degree some mass
    return out.float().contiguous()


def _network(seed):
    r = np.random.default_rng([int(seed), 48])
    w = []
    for n_out, n_in in ((256, 64), (256, 256), (48, 256)):
        w.append(r.uniform(-1.0, 1.0, (n_out, n_in)) / math.sqrt(n_in))
        w.append(r.uniform(-0.05, 0.05, n_out))
    return torch.cat([torch.from_numpy(v.astype(np.float32)).reshape(-1) for v in w]).cuda()


def _records(n, seed):
    """Line-fitting records of a population: degree uniform, coefficients N(0, 1)."""
    g = _gen(seed)
    rec = torch.randn(n, 8, generator=g, device="cuda")
    deg = torch.randint(DEGS[0], DEGS[-1] + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    rec[:, :6] *= torch.arange(6, device="cuda") <= deg[:, None]
    rec[:, 6] = deg.view(torch.float32)
    rec[:, 7] = torch.arange(n, device="cuda", dtype=torch.int32).view(torch.float32)
    return rec


def _summary_views(res, rows):
    """Buffers and views of summaries: the FP32 rows and the two whole-number fields."""
    f32 = torch.empty(rows, 74, dtype=torch.float32, device="cuda")
    words = res.view(torch.float64).view(rows, 74)
    out = {k: f32[:, a:b] for k, (a, b) in FLOAT_FIELDS.items()}
    out["n_particles"] = res.view(torch.int64).view(rows, 74)[:, 5]
    out["map_deg_n_deg"] = res.view(torch.int32).view(rows, 148)[:, 12:14]
    return {"f32": f32, "words": words, "views": out}


def _taken(v):
    v["f32"].copy_(v["words"])
    return v["views"]


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "seed": int(seed), "case": case}
    if k in ("linefit", "suffstat"):
        n = case["n"]
        s["model"] = ppl.poly_model()
        s["x"], s["y"] = _line_data(case["L"], seed)
        s["ws"] = ppl.workspace(s["model"], n, case["L"])
        s["res"] = ppl.result_tensor()
        s["sum"] = _summary_views(s["res"], 1)
        s["lw"] = torch.empty(n, dtype=torch.float32, device="cuda")
        s["rec"] = ppl.poly_particles(n)
        if case.get("resample"):
            s["anc"] = torch.empty(n, dtype=torch.int32, device="cuda")
            s["out"] = torch.empty_like(s["rec"])
    elif k == "resample":
        g = _gen(seed)
        s["lw"] = case["scale"] * torch.randn(case["n"], generator=g, device="cuda")
        s["state"] = torch.randn(case["n"], case["words"], generator=g, device="cuda")
        s["out"] = torch.empty(case["m"], case["words"], device="cuda")
        s["anc"] = torch.empty(case["m"], dtype=torch.int32, device="cuda")
        s["ws"] = ppl.workspace(ppl.poly_model(), max(case["n"], case["m"]))
    elif k == "population":
        n = case["n"]
        s["model"] = ppl.poly_model()
        s["rec"] = _records(n, seed)
        s["lw"] = case["scale"] * torch.randn(n, generator=_gen(seed + 1), device="cuda")
        s["res"] = ppl.result_tensor()
        s["sum"] = _summary_views(s["res"], 1)
        s["out"] = torch.empty_like(s["rec"])
        s["anc"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["ws"] = ppl.workspace(s["model"], n)
    elif k == "logsumexp":
        s["lw"] = case["scale"] * torch.randn(case["n"], generator=_gen(seed), device="cuda")
        s["out"] = torch.empty(4, dtype=torch.float64, device="cuda")
        s["ws"] = ppl.workspace(ppl.poly_model(), case["n"])
    elif k == "smc":
        r = np.random.default_rng([int(seed), case["T"]])
        x, y = 0.0, np.zeros(case["T"], dtype=np.float32)
        for t in range(case["T"]):
            x = 0.9 * x + r.standard_normal()
            y[t] = x + 0.5 * r.standard_normal()
        s["model"] = ppl.lgssm_model()
        s["y"] = torch.from_numpy(y).cuda()
        s["ws"] = ppl.workspace(s["model"], case["n"], case["T"])
        s["out"] = {"x": torch.empty(case["n"], device="cuda"),
                    "lw": torch.empty(case["n"], device="cuda"),
                    "log_z": torch.empty(1, dtype=torch.float64, device="cuda"),
                    "resampled": torch.empty(case["T"], dtype=torch.int32, device="cuda"),
                    "ess": torch.empty(case["T"], dtype=torch.float64, device="cuda")}
    elif k in ("batched", "learned"):
        s["model"] = ppl.poly_model()
        if k == "batched":
            x, y, doff, poff = _batch_data(case, seed)
            s["x"], s["y"] = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
            ppt, bps = 4, 4
        else:
            s["x"], s["y"] = _held_out(case["sets"], seed)
            s["prop"] = _near_posterior(s["x"], s["y"])
            doff = np.arange(case["sets"] + 1, dtype=np.int64) * 32
            poff = np.arange(case["sets"] + 1, dtype=np.int64) * case["n"]
            ppt, bps = 8, 2
        s["doff"], s["poff"] = torch.from_numpy(doff).cuda(), torch.from_numpy(poff).cuda()
        s["ws"] = ppl.batched_workspace(doff, poff)
        s["plan"] = ppl.ppl_batched_prepare(s["model"], doff, poff, ppt, bps, s["ws"])
        s["res"] = ppl.batch_results_tensor(case["sets"])
        s["sum"] = _summary_views(s["res"], case["sets"])
    else:
        s["model"] = ppl.poly_model()
        s["init"] = _network(seed)
        s["params"] = torch.empty_like(s["init"])
        s["m"], s["v"] = torch.empty_like(s["init"]), torch.empty_like(s["init"])
        s["loss"] = torch.empty(case["steps"], dtype=torch.float64, device="cuda")
        s["ws"] = ppl.proposal_workspace(case["batch"])
    return s


def run(s):
    k, case, seed = s["kind"], s["case"], s["seed"]
    if k in ("linefit", "suffstat"):
        fn = ppl.ppl_infer_is_instance if k == "linefit" else ppl.ppl_infer_is_suffstat
        fn(s["model"], s["x"], s["y"], case["n"], seed, 0, out=s["res"], lw_out=s["lw"],
           particles_out=s["rec"], ws=s["ws"])
        out = {"summary": _taken(s["sum"]), "lw": s["lw"], "records": s["rec"].view(torch.int32)}
        if case.get("resample"):
            anc, new = ppl.ppl_resample_gather(case["n"], seed, s["lw"], s["rec"],
                                               max_lw_dev=ppl.result_max_lw(s["res"]),
                                               state_out=s["out"], ancestors=s["anc"], ws=s["ws"])
            out["ancestors"], out["resampled"] = anc, new.view(torch.int32)
        return out
    if k == "resample":
        anc, new = ppl.ppl_resample_gather(case["m"], seed, s["lw"], s["state"],
                                           state_out=s["out"], ancestors=s["anc"], ws=s["ws"])
        return {"ancestors": anc, "state": new}
    if k == "population":
        ppl.ppl_posterior_reduce(s["model"], s["rec"], s["lw"], out=s["res"], ws=s["ws"])
        out = {"summary": _taken(s["sum"])}
        anc, new = ppl.ppl_resample_gather(case["n"], seed, s["lw"], s["rec"],
                                           max_lw_dev=ppl.result_max_lw(s["res"]),
                                           state_out=s["out"], ancestors=s["anc"], ws=s["ws"])
        out["ancestors"], out["resampled"] = anc, new.view(torch.int32)
        return out
    if k == "logsumexp":
        return {"stats": ppl.ppl_logsumexp(s["lw"], out=s["out"], ws=s["ws"])}
    if k == "smc":
        o = ppl.ppl_smc_run(s["model"], s["y"], case["n"], seed, ws=s["ws"], out=s["out"])
        return {name: o[name] for name in ("x", "lw", "log_z", "resampled", "ess")}
    if k == "batched":
        ppl.ppl_infer_is_batched(s["model"], s["x"], s["y"], s["doff"], s["poff"], seed,
                                 s["plan"], s["res"], s["ws"])
        return {"summary": _taken(s["sum"])}
    if k == "learned":
        ppl.ppl_infer_is_learned(s["model"], s["x"], s["y"], s["doff"], s["poff"], seed,
                                 s["plan"], s["prop"], s["res"], s["ws"])
        return {"summary": _taken(s["sum"])}
    # the first step of a training run from its initial parameters
    s["params"].copy_(s["init"])
    s["m"].zero_()
    s["v"].zero_()
    ppl.ppl_proposal_train_init(s["params"], case["batch"], s["ws"])
    ppl.ppl_proposal_train_steps(s["model"], s["params"], s["m"], s["v"],
                                 case["batch"] * case["steps"], case["batch"], case["steps"],
                                 seed, 1e-3, s["loss"], s["ws"])
    return {"params": s["params"], "m": s["m"], "v": s["v"], "loss": s["loss"]}


def work(case):
    k = case["kind"]
    if k == "linefit":
        # data in, log-weight and record out; Horner and the square per point
        # at the mean coefficient count 4.5
        n, L = case["n"], case["L"]
        b = 8 * L + 36 * n
        if case["resample"]:  # log-weight and record in, ancestor and record out
            b += 72 * n
        return {"bytes": b, "flops": n * L * 10}
    if k == "suffstat":
        # per trace d (d + 1) / 2 multiply-adds and d squares, d = 3..6
        return {"bytes": 8 * case["L"] + 36 * case["n"], "flops": case["n"] * 34}
    if k == "resample":
        w = 4 * case["words"]
        return {"bytes": (4 + w) * (case["n"] + case["m"]), "flops": 16 * case["n"]}
    if k == "population":
        # record and log-weight in, ancestor and record out; weighted moments
        return {"bytes": 72 * case["n"], "flops": case["n"] * 45}
    if k == "logsumexp":
        return {"bytes": 4 * case["n"] + 32, "flops": 4 * case["n"]}
    if k == "smc":
        return {"bytes": 8 * case["n"] + 16 * case["T"], "flops": case["n"] * case["T"] * 60}
    if k == "batched":
        def mean(lo, hi):
            return (hi - lo) / math.log(hi / lo)
        L, N = mean(case["l_lo"], case["l_hi"] + 1), mean(case["n_lo"], case["n_hi"] + 1)
        return {"bytes": case["sets"] * (8 * L + 592), "flops": case["sets"] * N * L * 10}
    if k == "learned":
        return {"bytes": case["sets"] * (8 * 32 + 192 + 592),
                "flops": case["sets"] * case["n"] * (32 * 10 + 60)}
    weights = 64 * 256 + 256 * 256 + 256 * 48
    return {"bytes": 4 * 3 * 2 * weights, "flops": case["steps"] * case["batch"] * 6 * weights}


# ---- the same in 64 bits ----------------------------------------------------
def _philox(seed, particle, instance, purpose, block):
    """Philox4x32-10 words (Salmon et al., SC'11) as int64 tensors holding 32 bits."""
    mask = 0xFFFFFFFF
    c = [particle, instance, torch.zeros_like(particle),
         torch.zeros_like(particle) + ((purpose << 16) | 0) + block]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wrap modulo 2^64: their bits are right
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
    return c


def _normals(wa, wb):
    ua = ((wa >> 9).double() + 0.5) * 2.0 ** -23
    ub = ((wb >> 9).double() + 0.5) * 2.0 ** -23
    rho = torch.sqrt(-2.0 * torch.log(ua))
    return rho * torch.cos(2 * math.pi * ub), rho * torch.sin(2 * math.pi * ub)


def _trace_words(seed, particle, instance, purpose):
    a = _philox(seed, particle, instance, purpose, 0)
    b = _philox(seed, particle, instance, purpose, 1)
    z = [*_normals(a[0], a[1]), *_normals(a[2], a[3]), *_normals(b[0], b[1])]
    return torch.stack(z, -1), b[2]


def _prior_traces(seed, particle, instance, purpose=1):
    """(degree, coefficients) of the model's prior, FP64."""
    z, w = _trace_words(seed, particle, instance, purpose)
    deg = DEGS[0] + ((w * len(DEGS)) >> 32)
    c = PRIOR_SIGMA * z
    return deg, c * (torch.arange(6, device=c.device) <= deg[..., None])


def _factor(c, x, y):
    """-sum_l (y_l - f(x_l))^2 / (2 sigma^2) of traces c [n, 6], FP64."""
    phi = torch.stack([x ** k for k in range(6)])
    r = c @ phi
    r -= y
    return r.square_().sum(-1) * (-0.5 / OBS_SIGMA ** 2)


class _Weighted:
    """Weighted sums per degree, merged over chunks: [D, ...] with the running maximum."""

    def __init__(self, dev):
        self.m = torch.full((4,), -math.inf, dtype=torch.float64, device=dev)
        self.S = torch.zeros(4, 14, dtype=torch.float64, device=dev)
        self.ref = torch.zeros(4, 6, dtype=torch.float64, device=dev)
        self.n = 0

    def add(self, deg, c, lw):
        for k, n in enumerate(DEGS):
            at = deg == n
            v = torch.where(at, lw, torch.full_like(lw, -math.inf))
            m, i = v.max(0)
            if not bool(m > -math.inf):
                continue
            if not bool(self.m[k] > -math.inf):
                self.ref[k] = c[i]
            new = torch.maximum(m, self.m[k])
            w = torch.exp(v - new)
            d = c - self.ref[k]
            wd = w[:, None] * d
            s = torch.cat([w.sum()[None], (w * w).sum()[None], wd.sum(0), (wd * d).sum(0)])
            f = torch.exp(self.m[k] - new)
            self.S[k] *= f
            self.S[k, 1] *= f
            self.S[k] += s
            self.m[k] = new
        self.n += lw.numel()

    def row(self):
        """The 74 words of a summary (whole-number words 0)."""
        out = torch.zeros(74, dtype=torch.float64, device=self.m.device)
        M = self.m.max()
        e = torch.exp(self.m - M)
        s, s2 = (self.S[:, 0] * e).sum(), (self.S[:, 1] * e * e).sum()
        out[1] = M + torch.log(s)
        out[0] = out[1] - math.log(self.n)
        out[2], out[3] = s * s / s2, M
        p = self.S[:, 0] * e / s
        has = self.S[:, 0] > 0
        S0 = torch.where(has, self.S[:, 0], torch.ones_like(self.m))[:, None]
        sh = self.S[:, 2:8] / S0
        mean = (self.ref + sh) * has[:, None]
        var = (self.S[:, 8:14] / S0 - sh * sh).clamp(min=0) * has[:, None]
        out[7:11] = p
        out[11:17] = (p[:, None] * mean).sum(0)
        out[17:41], out[41:65] = mean.reshape(-1), var.reshape(-1)
        out[65:69] = self.m
        return out


def _exact_summary(rows):
    out = {k: rows[:, a:b] for k, (a, b) in FLOAT_FIELDS.items()}
    out["n_particles"] = None
    out["map_deg_n_deg"] = None
    return out


def _whole(n):
    return torch.arange(n, device="cuda", dtype=torch.int64)


def _exact_linefit(case, seed):
    x, y = (v.double() for v in _line_data(case["L"], seed))
    acc, lws = _Weighted("cuda"), []
    step = max(1 << 12, min(1 << 19, (1 << 27) // case["L"]))
    for i0 in range(0, case["n"], step):
        i = i0 + _whole(min(step, case["n"] - i0))
        deg, c = _prior_traces(seed, i, torch.zeros_like(i))
        lws.append(_factor(c, x, y))
        acc.add(deg, c, lws[-1])
    out = {"summary": _exact_summary(acc.row()[None]), "lw": torch.cat(lws), "records": None}
    if case.get("resample"):
        out["ancestors"] = out["resampled"] = None
    return out


def _exact_population(case, seed):
    rec = _records(case["n"], seed)
    lw = case["scale"] * torch.randn(case["n"], generator=_gen(seed + 1), device="cuda")
    acc = _Weighted("cuda")
    for i0 in range(0, case["n"], 1 << 20):
        r = rec[i0:i0 + (1 << 20)]
        acc.add(r[:, 6].contiguous().view(torch.int32), r[:, :6].double(), lw[i0:i0 + (1 << 20)].double())
    return {"summary": _exact_summary(acc.row()[None]), "ancestors": None, "resampled": None}


def _rows(parts):
    """Summary rows of many populations at once: the sums of _Weighted per (set, degree)."""
    m, S, ref, n = parts
    rows = []
    for b in range(m.shape[0]):
        a = _Weighted(m.device)
        a.m, a.S, a.ref, a.n = m[b], S[b], ref[b], n[b]
        rows.append(a.row())
    return torch.stack(rows)


def _exact_batched(case, seed):
    x, y, doff, poff = _batch_data(case, seed)
    x, y = torch.from_numpy(x).cuda().double(), torch.from_numpy(y).cuda().double()
    rows = []
    for b in range(case["sets"]):
        n, xb, yb = int(poff[b + 1] - poff[b]), x[doff[b]:doff[b + 1]], y[doff[b]:doff[b + 1]]
        i = _whole(n)
        deg, c = _prior_traces(seed, i, torch.full_like(i, b))
        lw = torch.cat([_factor(part, xb, yb) for part in c.split(max(1, (1 << 27) // len(xb)))])
        rows.append(_segment(deg, c, lw))
    return {"summary": _exact_summary(_rows(tuple(torch.stack(v) if torch.is_tensor(v[0]) else v
                                                  for v in zip(*rows))))}


def _segment(deg, c, lw):
    """(m, S, ref, n) of one population without a host read (four degrees at once)."""
    at = deg[None] == torch.tensor(DEGS, device=deg.device)[:, None]
    v = torch.where(at, lw[None], torch.full_like(lw, -math.inf)[None])
    m, i = v.max(1)
    ref = c[i]
    w = torch.exp(v - torch.where(m > -math.inf, m, torch.zeros_like(m))[:, None])
    A = torch.stack([torch.stack([w[k].sum(), w[k].square().sum()]) for k in range(4)])
    mom = []
    for k in range(4):
        d = c - ref[k]
        mom.append(torch.cat([w[k] @ d, w[k] @ (d * d)]))
    return m, torch.cat([A, torch.stack(mom)], 1), ref, lw.numel()


def _exact_learned(case, seed):
    if case["sets"] * case["n"] > 1 << 26:
        return None
    x, y = _held_out(case["sets"], seed)
    prop = _near_posterior(x, y).double()
    x, y = x.double(), y.double()
    base = [0, 3, 7, 12]
    rows = []
    for b in range(case["sets"]):
        i = _whole(case["n"])
        z, w6 = _trace_words(seed, i, torch.full_like(i, b), 1)
        q = torch.log_softmax(prop[b, :4], 0)
        # the degree choice is a comparison of FP32 cumulative masses
        o = prop[b, :4].float()
        e = torch.exp(o - o.max())
        cum = torch.cumsum(e / e.sum(), 0).double()
        u = ((w6 >> 9).double() + 0.5) * 2.0 ** -23
        k = (u[:, None] >= cum[:3]).sum(1)
        slot = torch.tensor(base, device=u.device)[k][:, None] + torch.arange(6, device=u.device)
        live = torch.arange(6, device=u.device) <= (k + 2)[:, None]
        slot = torch.where(live, slot, torch.zeros_like(slot))
        t = prop[b, 5 + 2 * slot].clamp(-9.0, 1.0)
        mu, sd = PRIOR_SIGMA * prop[b, 4 + 2 * slot], PRIOR_SIGMA * torch.exp(t)
        c = (mu + sd * z) * live
        # log N(c; 0, sigma^2) - log N(c; mu, s^2), live coefficients
        dens = -0.5 * (c / PRIOR_SIGMA) ** 2 + t + 0.5 * z * z
        lw = -math.log(4.0) - q[k] + (dens * live).sum(1) + _factor(c, x[b], y[b])
        rows.append(_segment(k + 2, c, lw))
    return {"summary": _exact_summary(_rows(tuple(torch.stack(v) if torch.is_tensor(v[0]) else v
                                                  for v in zip(*rows))))}


def _bf16(v):
    return v.float().bfloat16().double()


def _exact_train(case, seed):
    """Adam on the mean -log q in 64 bits, rounding where the method's
    definition holds BF16 (weights, features, activations and their gradients)."""
    B = case["batch"]
    sizes = ((256, 64), (256, 256), (48, 256))
    p = _network(seed).double()
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for s in range(case["steps"]):
        i = s * B + _whole(B)
        deg, c = _prior_traces(seed, i, torch.zeros_like(i), 5)
        w = _philox(seed, i[:, None].expand(B, 32).contiguous(), torch.zeros(B, 32, device="cuda", dtype=torch.int64), 5,
                    2 + _whole(32)[None])
        x = (2.0 * ((w[0] >> 9).double() + 0.5) * 2.0 ** -23 - 1.0).float().double()
        e = _normals(w[1], w[2])[0]
        y = OBS_SIGMA * e
        for k in range(6):
            y = y + c[:, k:k + 1] * x ** k
        x, at = torch.sort(x, dim=1, stable=True)
        y = torch.gather(y, 1, at).float() / 10.0
        feat = _bf16(torch.stack([x, y.double()], 2).reshape(B, 64))
        W, b, off = [], [], 0
        for n_out, n_in in sizes:
            W.append(_bf16(p[off:off + n_out * n_in].reshape(n_out, n_in)))
            off += n_out * n_in
            b.append(p[off:off + n_out])
            off += n_out
        h1 = _bf16(torch.relu(feat @ W[0].T + b[0]))
        h2 = _bf16(torch.relu(h1 @ W[1].T + b[1]))
        out = h2 @ W[2].T + b[2]
        k = deg - 2
        logq = torch.log_softmax(out[:, :4], 1)
        g = torch.zeros_like(out)
        g[:, :4] = torch.exp(logq) - torch.nn.functional.one_hot(k, 4)
        loss = -torch.gather(logq, 1, k[:, None])[:, 0]
        slot = torch.tensor([0, 3, 7, 12], device="cuda")[k][:, None] + torch.arange(6, device="cuda")
        live = torch.arange(6, device="cuda") <= deg[:, None]
        im = torch.where(live, 4 + 2 * slot, torch.full_like(slot, 4))
        om, os = torch.gather(out, 1, im), torch.gather(out, 1, im + 1)
        t = os.clamp(-9.0, 1.0)
        sd = PRIOR_SIGMA * torch.exp(t)
        z = (c - PRIOR_SIGMA * om) / sd
        loss = loss + ((0.5 * math.log(2 * math.pi) + math.log(PRIOR_SIGMA) + t + 0.5 * z * z) * live).sum(1)
        g.scatter_add_(1, im, torch.where(live, -z / sd * PRIOR_SIGMA, torch.zeros_like(z)))
        inside = live & (os > -9.0) & (os < 1.0)
        g.scatter_add_(1, im + 1, torch.where(inside, 1.0 - z * z, torch.zeros_like(z)))
        g /= B
        gb = _bf16(g)
        d2 = _bf16((gb @ W[2]) * (h2 > 0))
        d1 = _bf16((d2 @ W[1]) * (h1 > 0))
        grad = torch.cat([(d1.T @ feat).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0),
                          (gb.T @ h2).reshape(-1), g.sum(0)])
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        p = p - 1e-3 * (m / (1 - 0.9 ** (s + 1))) / (torch.sqrt(v / (1 - 0.999 ** (s + 1))) + 1e-8)
        losses.append(loss.sum())
    return {"params": p, "m": m, "v": v, "loss": torch.stack(losses)}


def exact(case, seed):
    k, seed = case["kind"], int(seed)
    if k in ("linefit", "suffstat"):
        return _exact_linefit(case, seed)
    if k == "population":
        return _exact_population(case, seed)
    if k == "logsumexp":
        lw = (case["scale"] * torch.randn(case["n"], generator=_gen(seed), device="cuda")).double()
        m, i = lw.max(0)
        e = torch.exp(lw - m)
        return {"stats": torch.stack([m + torch.log(e.sum()), e.sum() ** 2 / e.square().sum(), m,
                                      i.double()])}
    if k == "batched":
        return _exact_batched(case, seed)
    if k == "learned":
        return _exact_learned(case, seed)
    if k == "train":
        return _exact_train(case, seed)
    # ancestors are whole numbers of a fixed-point definition, and a filter's
    # particles follow from them: there is no other value in 64 bits
    return None
