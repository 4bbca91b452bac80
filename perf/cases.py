"""The work a user of this library has it do, one case per dict.

Chains of Swendsen-Wang sweeps (one lattice, a batch of lattices, a served
group of short jobs, the few-cluster update, the simple-cubic lattice) and
cluster labeling (percolation masks, grey-level images), each through the
public calls a program makes.  ``prepare`` gives what such a program holds
before the call, ``run`` is one pass, ``exact`` computes the same results
from the definitions in include/swccl.h with plain torch in 64-bit integers.
"""
import math
import random
import statistics
import weakref

import torch

import paper_1105_5804_gb300 as sw

M32 = 0xFFFFFFFF
WARM = 20           # sweeps from the hot start before a chain is measured


def listed():
    return [
        # A small chain run for its averages: L = 64, many sweeps per call, then the observables.  Launches count.
        {"name": "chain_ising_64", "kind": "chain", "L": 64, "q": 2, "ratio": 1.0, "n": 100},
        # The benchmark lattice: critical Ising, L = 16384, a few sweeps, then the observables and the spins.
        {"name": "chain_ising_16384", "kind": "chain", "L": 16384, "q": 2, "ratio": 1.0, "n": 4},
        # The paper's Table I size with q = 4 states at its critical point.
        {"name": "chain_potts4_8192", "kind": "chain", "L": 8192, "q": 4, "ratio": 1.0, "n": 4},
        # One step of a pipeline that hands in new spins: three states, a side no tile divides.
        {"name": "io_potts3_1000", "kind": "io", "L": 1000, "q": 3, "ratio": 1.0, "n": 10},
        # The few-cluster update, 16 x 16 seed blocks, p_flip = 1/2.
        {"name": "few_ising_4096", "kind": "few", "L": 4096, "q": 2, "ratio": 1.0, "n": 8, "ell": 16},
        # Independent replicas of uneven size and temperature advanced together, then every chain read.
        {"name": "batch_64_chains", "kind": "batch", "chains": 64, "L_min": 64, "L_max": 2048, "n": 50, "mix": 2024},
        # A group of short jobs as a server runs it: a batch made in a workspace, 10 sweeps, observables, destroyed.
        {"name": "serve_sw_group", "kind": "serve", "chains": 6, "L_min": 128, "L_max": 640, "n": 10, "mix": 7},
        # Simple-cubic critical Ising chain.
        {"name": "cubic_ising_256", "kind": "cubic", "X": 256, "Y": 256, "Z": 256, "q": 2, "n": 4},
        # The labeling workload: critical bond percolation, periodic 4096 x 4096.
        {"name": "label_perc_4096", "kind": "label", "H": 4096, "W": 4096, "periodic": True, "call": "label"},
        # One small grid by the call that allocates nothing.  Latency counts.
        {"name": "label_small_200x300", "kind": "label", "H": 200, "W": 300, "periodic": True, "call": "noalloc"},
        # Segmentation of one large image of odd sides: pixels to bonds to labels, open boundaries.
        {"name": "segment_5003x7001", "kind": "segment", "images": 1, "side_min": 5003, "side_max": 7001, "mix": 0},
        # A served group of segmentation requests of any size.
        {"name": "segment_group_8", "kind": "segment", "images": 8, "side_min": 256, "side_max": 1536, "mix": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "io", "few", "batch", "serve", "cubic", "label", "label", "segment",
                       "segment"])
    if kind in ("chain", "io", "few"):
        L = 4 * max(1, _log(rng, 16, 1024))
        c = {"kind": kind, "L": L, "q": rng.choice([2, 2, 3, 4]), "ratio": rng.choice([1.0, 1.0, 0.6, 1.4]),
             "n": max(1, min(100, (1 << 26) // (L * L)))}
        if kind == "few":
            c["ell"] = rng.choice([d for d in (1, 2, 4, 8, 16, 32) if L % d == 0])
        return c
    if kind in ("batch", "serve"):
        hi = 4 * _log(rng, 64, 256)
        return {"kind": kind, "chains": rng.randint(4, 48) if kind == "batch" else rng.randint(1, 12), "L_min": 64,
                "L_max": hi, "n": rng.randint(5, 30) if kind == "batch" else 10, "mix": rng.randint(1, 10 ** 6)}
    if kind == "cubic":
        return {"kind": kind, "X": _log(rng, 16, 256), "Y": _log(rng, 16, 256), "Z": _log(rng, 16, 256),
                "q": rng.choice([2, 3]), "n": 4}
    if kind == "label":
        H, W = _log(rng, 16, 4096), _log(rng, 16, 4096)
        return {"kind": kind, "H": H, "W": W, "periodic": rng.random() < 0.5,
                "call": rng.choice(["label", "ws", "noalloc"] if H * W <= 4 << 20 else ["label", "ws"])}
    lo = rng.randint(64, 1024)
    return {"kind": kind, "images": rng.randint(1, 8), "side_min": lo, "side_max": lo + rng.randint(1, 1024),
            "mix": rng.randint(1, 10 ** 6)}


# --------------------------------------------------------------------------- sizes and couplings of a case
def _beta(q, ratio=1.0):
    """ratio times the critical inverse temperature (Ising convention for q = 2)."""
    return ratio * math.log(1.0 + math.sqrt(q)) * (0.5 if q == 2 else 1.0)


def _chains(c):
    """Sizes and inverse temperatures of a batch: L log-uniform in steps of 32 (a batch) or 4 (served jobs), beta
    spread over [0.9, 1.1] of the critical one."""
    rng = random.Random(c["mix"])
    step = 32 if c["kind"] == "batch" else 4
    L = [min(c["L_max"], step * max(1, round(_log(rng, c["L_min"], c["L_max"]) / step))) // 4 * 4
         for _ in range(c["chains"])]
    beta = [_beta(2, 0.9 + 0.2 * r / max(1, len(L) - 1)) for r in range(len(L))]
    return L, beta


def _images(c):
    if not c["mix"]:
        return [(c["side_min"], c["side_max"])]
    rng = random.Random(c["mix"])
    return [(rng.randint(c["side_min"], c["side_max"]), rng.randint(c["side_min"], c["side_max"]))
            for _ in range(c["images"])]


def _grey_image(H, W, seed):
    """Gaussian-blurred white noise (sigma = 3, reflecting edges) in 8 equally likely grey levels."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn(H, W, generator=g, device="cuda")
    r = 12
    tap = [math.exp(-0.5 * (k / 3.0) ** 2) for k in range(-r, r + 1)]
    for dim in (0, 1):
        n = z.shape[dim]
        out = torch.zeros_like(z)
        for k in range(-r, r + 1):
            i = torch.arange(k, n + k, device="cuda") % (2 * n)
            out += (tap[k + r] / sum(tap)) * z.index_select(dim, torch.where(i < n, i, 2 * n - 1 - i))
        z = out
    z /= math.sqrt(sum((a / sum(tap)) ** 2 for a in tap) ** 2)      # the blurred field's standard deviation
    cuts = torch.tensor([statistics.NormalDist().inv_cdf(k / 8) for k in range(1, 8)], device="cuda")
    return torch.bucketize(z, cuts).to(torch.uint8).reshape(-1).contiguous()


class _Handle:
    """A library handle that is destroyed with the state that holds it."""

    def __init__(self, h, destroy):
        self.h = h
        weakref.finalize(self, destroy, h)


# --------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    c, k = dict(case), case["kind"]
    s = {"case": c, "seed": seed}
    if k in ("chain", "io", "few"):
        L, q = c["L"], c["q"]
        h = sw.sw_create_ex(L, q, _beta(q, c["ratio"]), 1.0, sw.SW_CONV_AUTO, seed, True)
        s["chain"] = _Handle(h, sw.sw_destroy)
        if k == "few":
            sw.sw_set_update(h, sw.SW_UPDATE_FEW, c["ell"], sw.sw_prob_threshold(0.5))
        sw.sw_sweep(h, WARM)
        sw.sw_observables(h)
        s["spins"] = torch.empty(L * L, dtype=torch.int8, device="cuda")
        if k == "io":
            s["inp"] = sw.sw_get_spins(h, torch.empty_like(s["spins"]))
            s["obs"] = torch.empty(c["n"], 1 + q, dtype=torch.int64, device="cuda")
    elif k == "batch":
        L, beta = _chains(c)
        b = sw.sw_batch_create(L, [2] * len(L), beta, [seed * 1000 + r for r in range(len(L))], sw.SW_CONV_ISING, True)
        s["batch"] = _Handle(b, sw.sw_batch_destroy)
        sw.sw_batch_sweep(b, WARM)
        rows = torch.empty(WARM, 3, dtype=torch.int64, device="cuda")
        for r in range(len(L)):
            sw.sw_batch_observables_async(b, r, 2, rows)
        sw.sw_batch_sync(b)
        s["L"] = L
        s["obs"] = torch.empty(len(L), c["n"], 3, dtype=torch.int64, device="cuda")
        s["spins"] = torch.empty(sum(x * x for x in L), dtype=torch.int8, device="cuda")
        s["views"] = s["spins"].split([x * x for x in L])
    elif k == "serve":
        s["L"], s["beta"] = _chains(c)
        s["ws"] = torch.empty(sw.sw_batch_device_bytes(s["L"], [2] * len(s["L"])), dtype=torch.uint8, device="cuda")
        s["obs"] = torch.empty(len(s["L"]), c["n"], 3, dtype=torch.int64).pin_memory()
        s["stream"] = torch.cuda.Stream()
        s["spins"] = torch.empty(sum(x * x for x in s["L"]), dtype=torch.int8, device="cuda")
        s["views"] = s["spins"].split([x * x for x in s["L"]])
    elif k == "cubic":
        h = sw.sw3_create(c["X"], c["Y"], c["Z"], c["q"], _cubic_T(c["q"]), seed, True)
        s["chain"] = _Handle(h, sw.sw3_destroy)
        sw.sw3_sweep(h, WARM)
        sw.sw3_observables(h)
        s["spins"] = torch.empty(c["X"] * c["Y"] * c["Z"], dtype=torch.int8, device="cuda")
    elif k == "label":
        N = c["H"] * c["W"]
        s["mask"] = torch.empty(sw.mask_bytes(N), dtype=torch.uint8, device="cuda")
        sw.ccl_perc_mask(seed, s["mask"], c["H"], c["W"])
        s["labels"] = torch.empty(N, dtype=torch.int32, device="cuda")
        if c["call"] == "ws":
            s["ws"] = torch.empty(sw.ccl_workspace_bytes(c["H"], c["W"]), dtype=torch.uint8, device="cuda")
    else:
        hw = _images(c)
        s["H"], s["W"] = [x[0] for x in hw], [x[1] for x in hw]
        s["px"] = [_grey_image(H, W, seed * 100 + j) for j, (H, W) in enumerate(hw)]
        s["mask"] = [torch.empty(sw.mask_bytes(H * W), dtype=torch.uint8, device="cuda") for H, W in hw]
        s["labels"] = [torch.empty(H * W, dtype=torch.int32, device="cuda") for H, W in hw]
        size = sw.ccl_workspace_bytes(*hw[0]) if len(hw) == 1 else sw.ccl_batch_workspace_bytes(s["H"], s["W"])
        s["ws"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    return s


def _cubic_T(q):
    """Activation threshold near the simple-cubic critical point (Ising K_c = 0.2217 in the +-1 convention)."""
    return sw.sw_threshold_for(q, 0.2216546 if q == 2 else 0.5505, 1.0, sw.SW_CONV_AUTO)


def run(s):
    c, k = s["case"], s["case"]["kind"]
    if k in ("chain", "few"):
        h = s["chain"].h
        sw.sw_sweep(h, c["n"])
        obs = sw.sw_observables(h, c["n"])
        return {"obs": obs, "spins": sw.sw_get_spins(h, s["spins"])}
    if k == "io":
        h = s["chain"].h
        sw.sw_sweep_io(h, c["n"], s["inp"], s["obs"], s["spins"])
        sw.sw_sync(h)
        return {"obs": s["obs"], "spins": s["spins"]}
    if k == "batch":
        b = s["batch"].h
        sw.sw_batch_sweep(b, c["n"])
        for r in range(len(s["L"])):
            sw.sw_batch_observables_async(b, r, 2, s["obs"][r])
        for r, L in enumerate(s["L"]):
            sw.sw_batch_get_spins(b, r, L, s["views"][r])
        return {"obs": s["obs"], "spins": s["spins"]}
    if k == "serve":
        with torch.cuda.stream(s["stream"]):
            b = sw.sw_batch_create_ws(s["L"], [2] * len(s["L"]), s["beta"],
                                      [s["seed"] * 1000 + r for r in range(len(s["L"]))], s["ws"], sw.SW_CONV_ISING,
                                      True, s["stream"])
            sw.sw_batch_set_graph(b, False)
            sw.sw_batch_sweep(b, c["n"])
            for r in range(len(s["L"])):
                sw.sw_batch_observables_async(b, r, 2, s["obs"][r])
            for r, L in enumerate(s["L"]):
                sw.sw_batch_get_spins(b, r, L, s["views"][r])
            sw.sw_batch_destroy(b)
        return {"obs": s["obs"], "spins": s["spins"]}
    if k == "cubic":
        h = s["chain"].h
        sw.sw3_sweep(h, c["n"])
        obs = sw.sw3_observables(h, c["n"])
        return {"obs": obs, "spins": sw.sw3_get_spins(h, s["spins"])}
    if k == "label":
        if c["call"] == "ws":
            return sw.ccl_label_ws(s["mask"], s["labels"], c["H"], c["W"], c["periodic"], s["ws"])
        call = sw.ccl_label if c["call"] == "label" else sw.ccl_label_noalloc
        return call(s["mask"], s["labels"], c["H"], c["W"], c["periodic"])
    for px, m, H, W in zip(s["px"], s["mask"], s["H"], s["W"]):
        sw.ccl_bonds_from_pixels(px, m, H, W, False)
    if len(s["px"]) == 1:
        sw.ccl_label_ws(s["mask"][0], s["labels"][0], s["H"][0], s["W"][0], False, s["ws"])
    else:
        sw.ccl_label_batch(s["mask"], s["labels"], s["H"], s["W"], [False] * len(s["H"]), s["ws"])
    return {"labels": s["labels"], "mask": s["mask"]}


# --------------------------------------------------------------------------- what a pass cannot do without
PHILOX_OPS = 60     # 32-bit integer operations of one draw: 10 rounds of two wide products and four XORs


def work(case):
    """bytes: a sweep reads and writes every spin; labeling reads 2 bits (from pixels: 1 byte, and writes the 2 bits)
    and writes 4 bytes per site.  flops: integer operations of the bond draws (two sites per draw, one in 3D), one
    comparison and one AND per bond; labeling: one operation per bond."""
    k = case["kind"]
    if k == "label":
        N = case["H"] * case["W"]
        return {"bytes": 4.25 * N, "flops": 2.0 * N}
    if k == "segment":
        N = sum(H * W for H, W in _images(case))
        return {"bytes": 5.25 * N, "flops": 4.0 * N}
    if k == "cubic":
        N = case["X"] * case["Y"] * case["Z"]
        return {"bytes": 2.0 * N * case["n"], "flops": (PHILOX_OPS + 6.0) * N * case["n"]}
    N = sum(x * x for x in _chains(case)[0]) if k in ("batch", "serve") else case["L"] ** 2
    return {"bytes": 2.0 * N * case["n"], "flops": (PHILOX_OPS / 2 + 4.0) * N * case["n"]}


# --------------------------------------------------------------------------- the same from the definitions
def _philox(c0, sweep, tag, seed):
    """Philox4x32-10 words of counters c0 (int64 tensor), as four int64 tensors."""
    x = [c0 & M32, torch.full_like(c0, sweep & M32), torch.full_like(c0, sweep >> 32), torch.full_like(c0, tag)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        pa, pb = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((pb >> 32) & M32) ^ x[1] ^ k0, pb & M32, ((pa >> 32) & M32) ^ x[3] ^ k1, pa & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x


def _roots(n, a, b):
    """Smallest index of each component of the graph with edges a[i] - b[i]."""
    par = torch.arange(n, device=a.device)
    while a.numel():
        pa, pb = par[a], par[b]
        live = pa != pb
        a, b, pa, pb = a[live], b[live], pa[live], pb[live]
        par.scatter_reduce_(0, torch.maximum(pa, pb), torch.minimum(pa, pb), "amin")
        while True:
            up = par[par]
            if torch.equal(up, par):
                break
            par = up
    return par


def _sweep(s, sides, q, T, seed, k, few=None):
    """Sweep k of a chain: s is an int64 tensor of the lattice's shape (sides, slowest axis first)."""
    n, flat = s.numel(), s.reshape(-1)
    i = torch.arange(n, device=s.device).reshape(sides)
    if len(sides) == 2:
        w = _philox(torch.arange((n + 1) // 2, device=s.device), k, 0, seed)
        words = [torch.stack((w[d], w[d + 2]), 1).reshape(-1)[:n] for d in range(2)]
    else:
        words = _philox(i.reshape(-1), k, 5, seed)
    a, b = [], []
    for d in range(len(sides)):
        j = i.roll(-1, len(sides) - 1 - d).reshape(-1)
        on = ((flat[j] == flat) & (words[d] < T)).nonzero().reshape(-1)
        a.append(on)
        b.append(j[on])
    root = _roots(n, torch.cat(a), torch.cat(b))
    w = _philox(i.reshape(-1), k, 1, seed)
    if few is None:
        return ((w[0] * q) >> 32)[root].reshape(sides)
    ell, P = few
    L, B = sides[0], sides[0] // ell
    blk = torch.arange(ell * ell, device=s.device)
    v = _philox(blk, k, 4, seed)
    seeds = (blk // ell * B + ((v[1] * B) >> 32)) * L + blk % ell * B + ((v[0] * B) >> 32)
    moves = torch.zeros(n, dtype=torch.bool, device=s.device)
    moves[root[seeds]] = True
    moves &= w[1] < P
    step = torch.where(moves, 1 + ((w[0] * (q - 1)) >> 32), 0)
    return ((flat + step[root]) % q).reshape(sides)


def _counts(s, q):
    eq = sum(int((s == s.roll(-1, d)).sum()) for d in range(s.dim()))
    return [eq] + [int((s == x).sum()) for x in range(q)]


def _chain(sides, q, T, seed, warm, n, few=None):
    """Spins after warm + n sweeps from the hot start, and the observables of the last n (a pipeline step's first pass
    hands in the spins after the warm-up, which changes nothing)."""
    N = math.prod(sides)
    i = torch.arange(N, device="cuda")
    s = ((_philox(i, 0, 2, seed)[0] * q) >> 32).reshape(sides)
    obs = []
    for k in range(warm + n):
        s = _sweep(s, sides, q, T, seed, k, few)
        if k >= warm:
            obs.append(_counts(s, q))
    return {"obs": torch.tensor(obs, dtype=torch.int64), "spins": s.reshape(-1)}


def _threshold(K):
    return min(1 << 32, math.floor(-math.expm1(-K) * 4294967296.0))


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("chain", "io", "few"):
        L, q = c["L"], c["q"]
        if L * L * (WARM + c["n"]) > 2 ** 31:
            return None                                      # about half a minute
        K = _beta(q, c["ratio"]) * (2.0 if q == 2 else 1.0)
        return _chain((L, L), q, _threshold(K), seed, WARM, c["n"], (c["ell"], 1 << 31) if k == "few" else None)
    if k in ("batch", "serve"):
        L, beta = _chains(c)
        warm = WARM if k == "batch" else 0
        if len(L) * (warm + c["n"]) > 600:
            return None
        out = [_chain((x, x), 2, _threshold(2.0 * b), seed * 1000 + r, warm, c["n"])
               for r, (x, b) in enumerate(zip(L, beta))]
        return {"obs": torch.stack([o["obs"] for o in out]), "spins": torch.cat([o["spins"] for o in out])}
    if k == "cubic":
        if c["X"] * c["Y"] * c["Z"] * (WARM + c["n"]) > 2 ** 31:
            return None
        K = 2.0 * 0.2216546 if c["q"] == 2 else 0.5505
        return _chain((c["Z"], c["Y"], c["X"]), c["q"], _threshold(K), seed, WARM, c["n"])
    if k == "label":
        H, W = c["H"], c["W"]
        i = torch.arange(H * W, device="cuda")
        w = _philox(torch.arange((H * W + 1) // 2, device="cuda"), 0, 3, seed)
        on = [torch.stack((w[d], w[d + 2]), 1).reshape(-1)[:H * W].reshape(H, W) < 1 << 31 for d in range(2)]
        return _labels(on, H, W, c["periodic"])
    out = {"labels": [], "mask": []}
    for j, (H, W) in enumerate(_images(c)):
        px = _grey_image(H, W, seed * 100 + j).reshape(H, W)
        on = [px == px.roll(-1, 1), px == px.roll(-1, 0)]
        on[0][:, -1] = on[1][-1, :] = False
        bits = (on[0].to(torch.int64) + 2 * on[1].to(torch.int64)).reshape(-1)
        bits = torch.nn.functional.pad(bits, (0, -bits.numel() % 4)).reshape(-1, 4)
        out["mask"].append((bits * torch.tensor([1, 4, 16, 64], device="cuda")).sum(1))
        out["labels"].append(_labels(on, H, W, False))
    return out


def _labels(on, H, W, periodic):
    if not periodic:
        on[0][:, -1] = on[1][-1, :] = False
    i = torch.arange(H * W, device="cuda").reshape(H, W)
    a = [i[on[d]] for d in range(2)]
    b = [i.roll(-1, 1 - d)[on[d]] for d in range(2)]
    return _roots(H * W, torch.cat(a), torch.cat(b))
