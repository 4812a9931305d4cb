"""The work that a user of this library has it do, as timed cases.

Each kind of case below is one pass through the public entry points of
`paper_2308_16877_gb300.hpac`, at the sizes of the benchmark's configurations
(`bench.py`) and of the tests, from the smallest region call to the large
hydro mesh. `listed()` names the fixed cases, `draw()` gives further ones of
the same ranges, `exact()` the results in 64 bits without this library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_16877_gb300 import hpac
from paper_2308_16877_gb300 import workloads as W

GAMMA = 5.0 / 3.0
RATE = W.BS_RATE
# input scales (e, v, dv, q) of the hydro's iACT knob, as in the benchmark
HYDRO_SCALE = (1.0 / W.HYDRO_E0, 1.0, 10.0, 1.0 / ((GAMMA - 1.0) * W.HYDRO_E0))
# normalisation of the EOS surrogate for the ranges of eos_states()
EOS_SHIFT, EOS_SCALE = (1.0e5, 1.0, 0.0, 1.25e3), (1.0 / 5.8e4, 1.0 / 0.23, 1.0 / 0.0115, 1.0 / 1.6e3)


def listed():
    return [
        # the smallest calls: 65,536 options priced exactly, under TAF and
        # under perforation, as a user does to compare them
        dict(name="bs_compare_65536", kind="bs_compare", options=65536, hsize=4, psize=8, thresh=0.005,
             level=0, skip=4),
        # TAF over a large option book, scored by MAPE against exact prices
        dict(name="bs_taf_16m", kind="bs_taf", options=1 << 24, hsize=4, psize=8, thresh=0.005, level=0,
             metric=0),
        # iACT over an odd number of options (rows without 16-byte alignment),
        # with the decision mask, scored by RMSE
        dict(name="bs_iact_5m_odd", kind="bs_iact", options=5000011, tsize=8, tperwarp=32, thresh=0.05,
             level=1, metric=1),
        # the 64^3 hydro configuration, exact, whole run
        dict(name="hydro_exact_64", kind="hydro", n=64, steps=100, technique=0, tsize=0, tperwarp=0,
             thresh=0.0),
        # the large hydro mesh with iACT tables kept across steps on its EOS
        # (the first steps of the benchmark's headline run)
        dict(name="hydro_iact_256", kind="hydro", n=256, steps=20, technique=2, tsize=4, tperwarp=4,
             thresh=1e-3),
        # the design-space exploration: 256 configurations x 32 uneven regions
        dict(name="sweep_256x21m", kind="sweep", regions=32, lo=12, hi=22, odd=0, configs=256, block=128,
             per_sm=8, tile=4),
        # the learned surrogate serving 16M options
        dict(name="surrogate_infer_16m", kind="infer", options=1 << 24, hidden=64),
        # the surrogate's training: 64 batches of 8192 samples
        dict(name="surrogate_train_8192", kind="train", options=1 << 19, batch=8192, hidden=64),
        # gradients through the EOS surrogate, with respect to its inputs and
        # its weights, by autograd, at an odd size
        dict(name="surrogate_vjp_300007", kind="vjp", options=300007, hidden=128),
        # American options on the longest tree
        dict(name="binomial_1024", kind="binomial", members=4096, points=4, steps=1024, technique=0,
             thresh=0.0),
        # one K-Means iteration over 4M observations
        dict(name="kmeans_4m", kind="kmeans", options=1 << 22, clusters=16),
        # neighbour-box forces in double precision under block-level TAF
        dict(name="lavamd_taf_16", kind="lavamd", boxes=16, particles=100, technique=1, thresh=0.02, level=2),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm (so odd as often as even)."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["bs_compare", "bs_taf", "bs_iact", "hydro", "sweep", "infer", "train", "vjp",
                       "binomial", "kmeans", "lavamd"])
    if kind == "bs_compare":
        return dict(kind=kind, options=_log_int(rng, 4096, 1 << 20), hsize=rng.choice([1, 2, 3, 4, 5, 8, 16]),
                    psize=rng.choice([1, 4, 8, 16]), thresh=rng.choice([0.005, 0.05, 0.5]), level=rng.randrange(3),
                    skip=rng.randrange(2, 11))
    if kind == "bs_taf":
        return dict(kind=kind, options=_log_int(rng, 1 << 16, 1 << 24), hsize=rng.choice([1, 2, 3, 4, 5, 8, 16]),
                    psize=rng.choice([1, 4, 8, 16, 64]), thresh=rng.choice([0.005, 0.02, 0.1, 0.5]),
                    level=rng.randrange(3), metric=rng.randrange(2))
    if kind == "bs_iact":
        return dict(kind=kind, options=_log_int(rng, 1 << 16, 1 << 23), tsize=rng.choice([1, 2, 4, 5, 8, 16]),
                    tperwarp=rng.choice([1, 2, 4, 8, 16, 32]), thresh=rng.choice([0.02, 0.05, 0.2]),
                    level=rng.randrange(3), metric=rng.randrange(2))
    if kind == "hydro":
        n = _log_int(rng, 16, 160)
        tech = rng.choice([0, 0, 2])
        return dict(kind=kind, n=n, steps=rng.randrange(5, 40), technique=tech, tsize=rng.choice([4, 8]) if tech else 0,
                    tperwarp=rng.choice([1, 4, 32]) if tech else 0, thresh=1e-3 if tech else 0.0)
    if kind == "sweep":
        lo = rng.randrange(9, 13)
        return dict(kind=kind, regions=rng.randrange(3, 33), lo=lo, hi=lo + rng.randrange(2, 9), odd=rng.randrange(2),
                    configs=rng.choice([32, 64, 128, 256]), block=rng.choice([64, 128, 256]),
                    per_sm=rng.choice([4, 8, 12]), tile=rng.choice([1, 2, 4, 8]))
    if kind == "infer":
        return dict(kind=kind, options=_log_int(rng, 1 << 14, 1 << 24), hidden=rng.choice([64, 128]))
    if kind == "train":
        return dict(kind=kind, options=_log_int(rng, 1 << 16, 1 << 20), batch=_log_int(rng, 1024, 1 << 16),
                    hidden=rng.choice([64, 128]))
    if kind == "vjp":
        return dict(kind=kind, options=_log_int(rng, 1 << 12, 1 << 20), hidden=rng.choice([64, 128]))
    if kind == "binomial":
        tech = rng.choice([0, 0, 1])
        return dict(kind=kind, members=_log_int(rng, 500, 4096), points=4, steps=rng.choice([200, 255, 512, 777, 1024]),
                    technique=tech, thresh=rng.choice([0.02, 0.1]) if tech else 0.0)
    if kind == "kmeans":
        return dict(kind=kind, options=_log_int(rng, 1 << 14, 1 << 22), clusters=_log_int(rng, 2, 64))
    return dict(kind="lavamd", boxes=rng.randrange(2, 13), particles=rng.choice([33, 64, 100, 128, 200]),
                technique=rng.choice([0, 0, 1]), thresh=rng.choice([0.02, 0.04]), level=rng.randrange(3))


# --------------------------------------------------------------------------
# inputs: the distributions of workloads.py, drawn on the device
# --------------------------------------------------------------------------

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 64 + stream)
    return g


def _uniform(g, n, lo, hi, dtype=torch.float64):
    return (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo).to(dtype)


def options_in(n, seed):
    """(4, n) float32 options, sorted by strike in runs of 32."""
    g = _gen(seed, 1)
    x = torch.empty(4, n, dtype=torch.float32, device="cuda")
    for d, (lo, hi) in enumerate((W.BS_SPOT, W.BS_STRIKE, W.BS_EXPIRY, W.BS_VOL)):
        x[d] = _uniform(g, n, lo, hi, torch.float32)
    full = n // 32 * 32
    order = torch.argsort(x[1, :full].view(-1, 32), dim=1, stable=True)
    for d in range(4):
        x[d, :full] = torch.gather(x[d, :full].view(-1, 32), 1, order).reshape(-1)
    return x


def eos_states(n, seed):
    """(4, n) float64 states e, v, dv, q of the EOS region."""
    g = _gen(seed, 2)
    x = torch.empty(4, n, dtype=torch.float64, device="cuda")
    x[0] = _uniform(g, n, 0.0, 2.0e5)
    x[1] = _uniform(g, n, 0.6, 1.4)
    x[2] = _uniform(g, n, -0.02, 0.02)
    x[3] = torch.where(x[2] < 0, _uniform(g, n, 0.0, 5.0e3), torch.zeros((), dtype=torch.float64, device="cuda"))
    return x


def mesh(n, seed):
    """Jittered node coordinates (flat, x fastest) and element energies."""
    g = _gen(seed, 3)
    h = 1.0 / n
    ax = torch.arange(n + 1, dtype=torch.float64, device="cuda") * h
    inside = torch.ones(n + 1, dtype=torch.float64, device="cuda")
    inside[0] = inside[n] = 0.0
    out = []
    for axis in (2, 1, 0):
        shape = [1, 1, 1]
        shape[axis] = n + 1
        d = _uniform(g, (n + 1) ** 3, -W.HYDRO_JITTER * h, W.HYDRO_JITTER * h).view(n + 1, n + 1, n + 1)
        out.append((ax.view(shape) + d * inside.view(shape)).reshape(-1).contiguous())
    e = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    e[0] = W.HYDRO_E0
    return out[0], out[1], out[2], e


def sweep_regions(c):
    sizes = [s - 13 * (j % 5) * c["odd"] for j, s in enumerate(W.sweep_region_sizes(c["regions"], c["lo"], c["hi"]))]
    out, off = [], 0
    for s in sizes:
        out.append((s, off, max(1, s // 8)))
        off += s
    return out, off


def sweep_knobs(c):
    every = W.sweep_configs()
    step = len(every) // c["configs"]
    return every[step // 2::step]


def portfolio(c, seed):
    return W.binomial_portfolio(c["members"], c["points"], seed=int(seed) % (1 << 31))


def observations(c, seed):
    """(8, n) float32 from overlapping blobs, and K initial centroids."""
    g = _gen(seed, 5)
    n, K = c["options"], c["clusters"]
    centres = _uniform(g, K * 8, -10.0, 10.0).view(8, K)
    labels = torch.randint(K, (n,), generator=g, device="cuda")
    x = torch.empty(8, n, dtype=torch.float32, device="cuda")
    for d in range(8):
        x[d] = (centres[d][labels] + 2.0 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)).float()
    return x, x[:, :K].t().contiguous()


def network(kind, hidden, seed):
    """Descriptor and seeded weights (float32, the library's layout) of a surrogate."""
    if kind == "eos":
        d = hpac.eos_desc(hidden)
        for k in range(4):
            d.feat_shift[k], d.feat_scale[k] = EOS_SHIFT[k], EOS_SCALE[k]
        d.out_shift, d.out_scale = 1.0, 0.05
    else:
        d = hpac.blackscholes_desc(hidden)
    D, H = d.n_feat, hidden
    g = np.random.Generator(np.random.PCG64([int(seed), 17]))
    u = lambda n, fan: g.uniform(-1.0, 1.0, n) / math.sqrt(fan)
    p = np.concatenate([u(H * D, D), 0.1 * u(H, 1), u(H * H, H), 0.1 * u(H, 1), u(H, H), 0.1 * u(1, 1)])
    return d, p.astype(np.float32)


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def prepare(case, seed):
    c, s = case, {"case": case}
    kind = c["kind"]
    if kind in ("bs_compare", "bs_taf", "bs_iact"):
        n = c["options"]
        s["x"] = options_in(n, seed)
        s["R"] = hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, s["x"], param=RATE, logical_threads=max(1, n // 8))
        s["out"] = torch.zeros(n, dtype=torch.float32, device="cuda")
        if kind == "bs_compare":
            s["taf"], s["perfo"] = torch.zeros_like(s["out"]), torch.zeros_like(s["out"])
        else:
            x64 = s["x"].double().contiguous()
            s["ref"] = torch.zeros(n, dtype=torch.float64, device="cuda")
            with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=RATE) as R:
                R.run_exact(x64, s["ref"])
        if kind == "bs_iact":
            s["mask"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
            s["scale"] = [1.0 / hi for _, hi in (W.BS_SPOT, W.BS_STRIKE, W.BS_EXPIRY, W.BS_VOL)]
    elif kind == "hydro":
        n = c["n"]
        s["init"] = dict(zip(("x", "y", "z", "e"), mesh(n, seed)))
        s["H"] = hpac.Hydro(n, *s["init"].values(), W.hydro_dt(n), logical_threads=n ** 3)
        s["H"].eos.set_persistent(c["technique"] != 0)
        s["knobs"] = None
        if c["technique"] == 2:
            s["scale"] = (hpac.C.c_double * 4)(*HYDRO_SCALE)
            s["knobs"] = hpac.hpac_iact_knobs(c["tsize"], c["tperwarp"], c["thresh"], hpac.HPAC_LEVEL_THREAD, 0,
                                              hpac.C.cast(s["scale"], hpac.C.POINTER(hpac.C.c_double)))
    elif kind == "sweep":
        regions, total = sweep_regions(c)
        s["x"] = options_in(total, seed)
        x64 = s["x"].double().contiguous()
        s["ref"] = torch.zeros(total, dtype=torch.float64, device="cuda")
        with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, x64, param=RATE) as R:
            R.run_exact(x64, s["ref"])
        s["knobs"] = sweep_knobs(c)
        s["taf"] = [j for j, k in enumerate(s["knobs"]) if k["tech"] == "taf"]
        s["perfo"] = [j for j, k in enumerate(s["knobs"]) if k["tech"] == "perfo"]
        s["sweep"] = hpac.Sweep(s["knobs"], regions, s["x"], s["ref"], RATE, c["block"], c["per_sm"], c["tile"])
    elif kind in ("infer", "train"):
        n = c["options"]
        s["x"] = options_in(n, seed)
        d, p = network("bs", c["hidden"], seed)
        s["S"] = hpac.Surrogate(d, p)
        s["out"] = torch.zeros(n, dtype=torch.float32, device="cuda")
        if kind == "train":
            with hpac.Region(hpac.HPAC_REGION_BLACKSCHOLES, s["x"], param=RATE) as R:
                R.run_exact(s["x"], s["out"])
    elif kind == "vjp":
        n = c["options"]
        d, p = network("eos", c["hidden"], seed)
        s["S"] = hpac.Surrogate(d, p)
        s["x"] = eos_states(n, seed).requires_grad_()
        s["w"] = torch.from_numpy(p).cuda().requires_grad_()
        s["gout"] = _uniform(_gen(seed, 6), n, -1.0, 1.0)
    elif kind == "binomial":
        s["x"] = torch.from_numpy(portfolio(c, seed)).cuda()
        s["out"] = torch.zeros(s["x"].shape[1], dtype=torch.float32, device="cuda")
        s["R"] = hpac.Region(hpac.HPAC_REGION_BINOMIAL, s["x"], param=RATE, logical_threads=c["members"],
                             block_threads=128, arg=c["steps"])
    elif kind == "kmeans":
        s["x"], s["cent"] = observations(c, seed)
        n = c["options"]
        s["R"] = hpac.Region(hpac.HPAC_REGION_KMEANS, s["x"], logical_threads=max(1, n // 8), arg=c["clusters"])
        s["R"].set_aux(s["cent"])
        s["ids"], s["prev"] = (torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(2))
        s["work"] = hpac.kmeans_workspace(c["clusters"])
    else:
        P = c["boxes"] ** 3 * c["particles"]
        s["rq"] = _uniform(_gen(seed, 7), 4 * P, 0.1, 1.0).view(4, P)
        s["fv"] = torch.zeros_like(s["rq"])
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "bs_compare":
        R, x = s["R"], s["x"]
        R.run_exact(x, s["out"])
        R.run_taf(x, s["taf"], c["hsize"], c["psize"], c["thresh"], c["level"])
        R.run_perfo(x, s["perfo"], hpac.HPAC_PERFO_SMALL, c["skip"], herded=True)
        return {"exact": s["out"], "taf": s["taf"], "perfo": s["perfo"]}
    if kind == "bs_taf":
        s["R"].run_taf(s["x"], s["out"], c["hsize"], c["psize"], c["thresh"], c["level"])
        return {"out": s["out"], "quality": hpac.quality(s["ref"], s["out"], c["metric"])}
    if kind == "bs_iact":
        s["R"].run_iact(s["x"], s["out"], c["tsize"], c["tperwarp"], c["thresh"], c["level"], in_scale=s["scale"],
                        mask=s["mask"])
        return {"out": s["out"], "mask": s["mask"], "quality": hpac.quality(s["ref"], s["out"], c["metric"])}
    if kind == "hydro":
        H = s["H"]
        for k, v in s["init"].items():
            H[k].copy_(v)
        hpac.hpac_hydro_init(H.state, torch.cuda.current_stream().cuda_stream)
        if c["technique"]:
            H.eos.reset_state()
        H.run(c["steps"], c["technique"], s["knobs"])
        return {k: H[k] for k in ("x", "y", "z", "u", "v", "w", "e", "p", "q", "vrel")}
    if kind == "sweep":
        s["sweep"].run()
        r = s["sweep"].results()
        out = {k: np.ascontiguousarray(r[k]) for k in ("invocations", "approximated", "skipped", "mape_terms")}
        # the relative errors of worthless options (prices down to 1e-300) make
        # these sums span the whole range of a double: mantissa and exponent
        out["rel_mantissa"], out["rel_exponent"] = np.frexp(r["sum_abs_rel"])
        out["taf_sum_sq"] = np.ascontiguousarray(r["sum_sq"][s["taf"]])
        out["perfo_sum_sq"] = np.ascontiguousarray(r["sum_sq"][s["perfo"]])
        return out
    if kind == "infer":
        s["S"].infer(s["x"], s["out"], RATE)
        return s["out"]
    if kind == "train":
        loss = s["S"].train(s["x"], s["out"], RATE, batch=c["batch"], epochs=1, lr=3e-3)
        return {"params": s["S"].params(), "loss": loss}
    if kind == "vjp":
        out = s["S"].apply(s["x"], s["w"], GAMMA)
        gx, gw = torch.autograd.grad(out, (s["x"], s["w"]), s["gout"])
        return {"out": out.detach(), "gx": gx, "gw": gw}
    if kind == "binomial":
        if c["technique"] == 1:
            s["R"].run_taf(s["x"], s["out"], 1, 2, c["thresh"], hpac.HPAC_LEVEL_BLOCK)
        else:
            s["R"].run_exact(s["x"], s["out"])
        return s["out"]
    if kind == "kmeans":
        s["ids"], s["prev"] = s["prev"], s["ids"]
        s["R"].run_exact(s["x"], s["ids"])
        changed = hpac.kmeans_update(s["x"], s["ids"], s["cent"], s["work"], prev=s["prev"])
        return {"ids": s["ids"], "centroids": s["cent"], "changed": changed}
    return hpac.lavamd(s["rq"], c["boxes"], c["particles"], W.LAVAMD_A2, technique=c["technique"], level=c["level"],
                       hsize=4, psize=8, thresh=c["thresh"], fv=s["fv"])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    c = case
    kind = c["kind"]
    if kind == "bs_compare":
        n = c["options"]
        return {"bytes": 20 * n * 2 + 20 * n * (c["skip"] - 1) // c["skip"], "flops": 3 * 70 * n}
    if kind in ("bs_taf", "bs_iact"):
        n = c["options"]
        return {"bytes": (20 + 12 + (1 if kind == "bs_iact" else 0)) * n, "flops": 90 * n}
    if kind == "hydro":
        E, N = c["n"] ** 3, (c["n"] + 1) ** 3
        # per step: u, v, w, x, y, z read and written and 1/m read per node;
        # e, p, q, v read and written and V0 read per element
        return {"bytes": c["steps"] * (104 * N + 72 * E), "flops": c["steps"] * (54 * N + 240 * E)}
    if kind == "sweep":
        total, cfg = sweep_regions(c)[1], c["configs"]
        return {"bytes": 24 * total, "flops": total * (70 + 12 * cfg)}
    if kind in ("infer", "train"):
        n, H = c["options"], c["hidden"]
        f = 2 * (5 * H + H * H + H) + 20 * H
        return {"bytes": 20 * n, "flops": f * n if kind == "infer" else 4 * f * n}
    if kind == "vjp":
        n, H = c["options"], c["hidden"]
        return {"bytes": (32 + 8 + 8 + 32) * n, "flops": 4 * n * (2 * (4 * H + H * H + H) + 20 * H)}
    if kind == "binomial":
        n, N = c["members"] * c["points"], c["steps"]
        return {"bytes": 20 * n, "flops": n * (N * (N + 1) // 2) * 6}
    if kind == "kmeans":
        n = c["options"]
        return {"bytes": 40 * n, "flops": n * (24 * c["clusters"] + 8)}
    B, NP = c["boxes"], c["particles"]
    pairs = (3 * B - 2) ** 3 * NP * NP
    return {"bytes": 64 * B ** 3 * NP, "flops": pairs * 40 // (1 if c["technique"] == 0 else 2)}


# --------------------------------------------------------------------------
# the results in 64 bits
# --------------------------------------------------------------------------

def _bs64(x):
    S, K, T, sig = x.double()
    sst = sig * T.sqrt()
    d1 = ((S / K).log() + (RATE + 0.5 * sig * sig) * T) / sst
    cdf = lambda z: 0.5 * torch.special.erfc(-z * math.sqrt(0.5))
    return S * cdf(d1) - K * (-RATE * T).exp() * cdf(d1 - sst)


def _mlp64(f, p, D, H):
    """Network output of features f (n, D) with weights p (float64)."""
    cut = [H * D, H, H * H, H, H, 1]
    W1, b1, W2, b2, w3, b3 = torch.split(p, cut)
    gelu = lambda z: torch.nn.functional.gelu(z, approximate="tanh")
    h1 = gelu(f @ W1.view(H, D).t() + b1)
    h2 = gelu(h1 @ W2.view(H, H).t() + b2)
    return h2 @ w3 + b3


def _bs_features64(x, d):
    S, K, T, sig = x.double()
    f0 = (S / K).log()
    f1 = sig * T.sqrt()
    f3 = ((f0 + (RATE + 0.5 * sig * sig) * T) / f1).clamp(-10.0, 10.0)
    f = torch.stack([f0, f1, RATE * T, f3, sig], 1)
    return ((f - torch.tensor(list(d.feat_shift)[:5], dtype=torch.float64, device="cuda"))
            * torch.tensor(list(d.feat_scale)[:5], dtype=torch.float64, device="cuda"))


def _chunks(n, size=1 << 20):
    return [slice(i, min(n, i + size)) for i in range(0, n, size)]


def _hydro64(c, seed):
    """The exact hydro run: forces as the gradient of sum (p + q) V."""
    n, dt = c["n"], W.hydro_dt(c["n"])
    x, y, z, e = mesh(n, seed)
    pos = torch.stack([x, y, z]).view(3, n + 1, n + 1, n + 1)

    def volume(r):
        P = [r[:, d:n + d, b:n + b, a:n + a] for d in (0, 1) for b in (0, 1) for a in (0, 1)]
        s1, s2 = (P[2] - P[1]) + (P[6] - P[3]), (P[4] - P[2]) + (P[5] - P[6])
        trip = lambda a, b, d: (a * torch.linalg.cross(b, d, dim=0)).sum(0)
        return (trip(s1, P[7] - P[2], P[3] - P[0]) + trip(s2, P[7] - P[4], P[6] - P[0])
                - trip(s1 + s2, P[7] - P[1], P[5] - P[0])) / 12.0

    V0 = volume(pos)
    mass = torch.zeros(n + 1, n + 1, n + 1, dtype=torch.float64, device="cuda")
    for d in (0, 1):
        for b in (0, 1):
            for a in (0, 1):
                mass[d:n + d, b:n + b, a:n + a] += 0.125 * V0
    e = e.view(n, n, n)
    p, q, vrel, vel = (GAMMA - 1.0) * e, torch.zeros_like(e), torch.ones_like(e), torch.zeros_like(pos)
    for _ in range(c["steps"]):
        r = pos.detach().requires_grad_()
        force, = torch.autograd.grad(((p + q) * volume(r)).sum(), r)
        vel = vel + dt * force / mass
        vel[0, :, :, 0], vel[1, :, 0, :], vel[2, 0, :, :] = 0.0, 0.0, 0.0
        pos = pos + dt * vel
        V = volume(pos)
        v1 = torch.where(V == V0, torch.ones_like(V), V / V0)
        dv = v1 - vrel
        du = V.clamp(min=0.0) ** (1.0 / 3.0) * dv / (v1 * dt)
        cs = (GAMMA * p.clamp(min=0.0) * v1).sqrt()
        q = torch.where(dv < 0, (4.0 * du * du + 0.5 * cs * du.abs()) / v1, torch.zeros_like(e))
        v0 = v1 - dv
        num = e * v0 - 0.5 * dv * ((GAMMA - 1.0) * e + 2.0 * q * v0)
        p = torch.where(num < 0, torch.zeros_like(e), (GAMMA - 1.0) * num / (v0 * (v1 + 0.5 * (GAMMA - 1.0) * dv)))
        e, vrel = p * v1 / (GAMMA - 1.0), v1
    out = dict(x=pos[0], y=pos[1], z=pos[2], u=vel[0], v=vel[1], w=vel[2], e=e, p=p, q=q, vrel=vrel)
    return {k: v.reshape(-1) for k, v in out.items()}


def _dropped(k, n, T):
    """Dropped invocations of one region under a perforation configuration (torch bool)."""
    i = torch.arange(n, device="cuda")
    key = i // T if k.get("herded", 1) else i
    m = k["m"]
    if k["kind"] == hpac.HPAC_PERFO_SMALL:
        return key % m == m - 1
    if k["kind"] == hpac.HPAC_PERFO_LARGE:
        return key % m != 0
    cut = n * m // 100
    if k["kind"] == hpac.HPAC_PERFO_INI:
        return i < cut
    if k["kind"] == hpac.HPAC_PERFO_FINI:
        return i >= n - cut
    wrap = lambda v: v - (1 << 64) if v >= 1 << 63 else v   # 64-bit constants as signed
    z = (key ^ wrap(int(k.get("seed", 0)))) + wrap(0x9E3779B97F4A7C15)
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * wrap(0x94D049BB133111EB)
    z = z ^ ((z >> 31) & ((1 << 33) - 1))
    return ((z >> 40) & ((1 << 24) - 1)) < int(math.floor(k["rate"] * 16777216.0))


def _sweep64(c, seed):
    """Perforation's squared errors: a dropped invocation leaves 0, so its
    squared error is the price's square; kept ones have none in 64 bits."""
    regions, total = sweep_regions(c)
    ref = _bs64(options_in(total, seed))
    knobs = [k for k in sweep_knobs(c) if k["tech"] == "perfo"]
    sq = np.zeros((len(knobs), len(regions)))
    for r, (n, off, T) in enumerate(regions):
        a2 = ref[off:off + n] ** 2
        for j, k in enumerate(knobs):
            sq[j, r] = float(torch.dot(_dropped(k, n, T).double(), a2))
    return {"invocations": None, "approximated": None, "skipped": None, "mape_terms": None, "rel_mantissa": None,
            "rel_exponent": None, "taf_sum_sq": None, "perfo_sum_sq": sq}


def _binomial64(c, seed):
    x = torch.from_numpy(portfolio(c, seed)).cuda().double()
    N, out = c["steps"], []
    for sl in _chunks(x.shape[1], 4096):
        S0, X, T, sig = (v[:, None] for v in x[:, sl])
        dt = T / N
        v = sig * dt.sqrt()
        u, a = v.exp(), (RATE * dt).exp()
        pu = (a - 1.0 / u) / (u - 1.0 / u)
        S = S0 * (v * (2.0 * torch.arange(N + 1, device="cuda", dtype=torch.float64) - N)).exp()
        V = (S - X).clamp(min=0.0)
        for n in range(N - 1, -1, -1):
            S = S[:, :n + 1] * u
            V = torch.maximum((pu / a) * V[:, 1:n + 2] + ((1.0 - pu) / a) * V[:, :n + 1], S - X)
        out.append(V[:, 0])
    return torch.cat(out)


def _kmeans64(c, seed):
    x, cent = observations(c, seed)
    n, K = c["options"], c["clusters"]
    ids = torch.empty(n, dtype=torch.int64, device="cuda")
    for sl in _chunks(n, 1 << 19):
        xs = x[:, sl].double()
        ids[sl] = torch.stack([((xs - cent[k].double()[:, None]) ** 2).sum(0) for k in range(K)]).argmin(0)
    count = torch.bincount(ids, minlength=K).double()
    mean = torch.stack([torch.zeros(K, dtype=torch.float64, device="cuda").index_add_(0, ids, x[d].double())
                        for d in range(8)], 1) / count.clamp(min=1.0)[:, None]
    mean = torch.where(count[:, None] > 0, mean, cent.double())
    return {"ids": ids.double(), "centroids": mean, "changed": None}


def _lavamd64(c, seed):
    B, NP = c["boxes"], c["particles"]
    rq = _uniform(_gen(seed, 7), 4 * B ** 3 * NP, 0.1, 1.0).view(4, B, B, B, NP)
    fv = torch.zeros_like(rq)
    own = lambda d: slice(max(0, -d), B - max(0, d))
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                h = (slice(None), own(dz), own(dy), own(dx))
                o = (slice(None), own(-dz), own(-dy), own(-dx))
                a, b = rq[h], rq[o]
                for m in range(NP):
                    d = a[:3] - b[:3, ..., m:m + 1]
                    t = b[3, ..., m:m + 1] * (-W.LAVAMD_A2 * (d * d).sum(0)).exp()
                    fv[h][0] += t
                    fv[h][1:] += 2.0 * t * d
    return fv.view(4, -1)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "bs_compare":
        n, T = c["options"], max(1, c["options"] // 8)
        y = _bs64(options_in(n, seed))
        kept = (torch.arange(n, device="cuda") // T) % c["skip"] != c["skip"] - 1
        return {"exact": y, "taf": None, "perfo": torch.where(kept, y, torch.zeros_like(y))}
    if kind == "hydro" and c["technique"] == 0:
        return _hydro64(c, seed)
    if kind == "sweep":
        return _sweep64(c, seed)
    if kind == "infer":
        x = options_in(c["options"], seed)
        d, p = network("bs", c["hidden"], seed)
        p = torch.from_numpy(p).cuda().double()
        y = [_mlp64(_bs_features64(x[:, sl], d), p, 5, c["hidden"]) for sl in _chunks(c["options"])]
        return x[0].double() * (d.out_shift + d.out_scale * torch.cat(y))
    if kind == "train":
        x = options_in(c["options"], seed)
        d, p = network("bs", c["hidden"], seed)
        f, mult, H, n = _bs_features64(x, d), x[0].double(), c["hidden"], c["options"]
        t = (_bs64(x) / mult - d.out_shift) / d.out_scale
        p = torch.from_numpy(p).cuda().double().requires_grad_()
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        batches = -(-n // c["batch"])
        for k, sl in enumerate(_chunks(n, c["batch"])):
            g, = torch.autograd.grad(((_mlp64(f[sl], p, 5, H) - t[sl]) ** 2).mean(), p)
            with torch.no_grad():
                lr = 0.5 * 3e-3 * (1.0 + math.cos(math.pi * k / batches))
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                p -= lr * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        with torch.no_grad():
            loss = sum(float(((_mlp64(f[sl], p, 5, H) - t[sl]) ** 2).sum()) for sl in _chunks(n)) / n
        return {"params": p.detach(), "loss": loss}
    if kind == "vjp":
        H, n = c["hidden"], c["options"]
        d, w = network("eos", H, seed)
        x = eos_states(n, seed).requires_grad_()
        w = torch.from_numpy(w).cuda().double().requires_grad_()
        e, v1, dv, q = x
        f = ((x.t() - torch.tensor(EOS_SHIFT, dtype=torch.float64, device="cuda"))
             * torch.tensor(EOS_SCALE, dtype=torch.float64, device="cuda"))
        u = e - dv * q
        mult = torch.where(u > 0, (GAMMA - 1.0) * u / v1, torch.zeros_like(u))
        out = (mult * (d.out_shift + d.out_scale * _mlp64(f, w, 4, H))).clamp(min=0.0)
        gx, gw = torch.autograd.grad(out, (x, w), _uniform(_gen(seed, 6), n, -1.0, 1.0))
        return {"out": out.detach(), "gx": gx, "gw": gw}
    if kind == "binomial" and c["technique"] == 0:
        return _binomial64(c, seed)
    if kind == "kmeans":
        return _kmeans64(c, seed)
    if kind == "lavamd" and c["technique"] == 0 and c["boxes"] <= 12:
        return _lavamd64(c, seed)
    return None
