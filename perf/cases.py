"""The calls that users of grng spend their time in, as measurable cases.

A case is one call (or one launch, or one burst) through the package's public
entry points, on an engine that keeps its place in its sequence from pass to
pass as a user's does.  The sizes are the library's own workloads: the RNG
burner's batches (one FP32 uniform fill of 10^3 .. 10^8 numbers), the fill
sweep up to 10^9 outputs over both engines and the distribution / dtype
pairs, 16384 substreams, the table of 4096 batched requests, the transform of
caller-supplied words and FastCaloSim-shaped bursts through the server.

listed() names the representative ones, draw() gives others of the same
ranges, prepare() / run() are a user's program, work() is what a pass cannot
do without, and exact() evaluates the same outputs in 64 bits with plain torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_01329_gb300 as grng

ENGINES = {"philox": grng.PHILOX4X32X10, "mrg": grng.MRG32K3A}

# name -> (kind, dtype, p0, p1)
DISTS = {
    "bits": (grng.BITS, grng.U32, 0.0, 0.0),
    "uniform_f32": (grng.UNIFORM, grng.F32, 0.0, 1.0),
    "uniform_f32_range": (grng.UNIFORM, grng.F32, 2.0, 5.0),
    "uniform_f64": (grng.UNIFORM, grng.F64, 0.0, 1.0),
    "uniform_f64_pm1": (grng.UNIFORM, grng.F64, -1.0, 1.0),
    "uniform_f64_range": (grng.UNIFORM, grng.F64, 2.0, 5.0),
    "gaussian_f32": (grng.GAUSSIAN, grng.F32, 0.0, 1.0),
    "gaussian_f64": (grng.GAUSSIAN, grng.F64, 0.0, 1.0),
    "gaussian_f64_affine": (grng.GAUSSIAN, grng.F64, -3.0, 0.25),
    "lognormal_f32": (grng.LOGNORMAL, grng.F32, 0.0, 1.0),
    "lognormal_f64": (grng.LOGNORMAL, grng.F64, 0.0, 0.5),
    "gaussian_icdf_f32": (grng.GAUSSIAN_ICDF, grng.F32, 0.0, 1.0),
    "gaussian_icdf_f64": (grng.GAUSSIAN_ICDF, grng.F64, 0.0, 1.0),
    "lognormal_icdf_f32": (grng.LOGNORMAL_ICDF, grng.F32, 0.0, 1.0),
}

# the distributions of the batched request table
BATCH_DISTS = ["bits", "uniform_f32", "gaussian_f32", "lognormal_f32", "uniform_f64_pm1"]

TORCH_TYPE = {grng.U32: torch.int32, grng.F32: torch.float32, grng.F64: torch.float64}

MRG_STRIDE_LOG2, PHILOX_STRIDE_LOG2 = 76, 40


def listed():
    return [
        # the burner's small batches: one call whose cost is its latency
        {"name": "philox uniform f32 1e3", "call": "fill", "engine": "philox", "dist": "uniform_f32", "n": 10**3},
        # the burner's largest batch, the paper's headline fill
        {"name": "philox uniform f32 1e8", "call": "fill", "engine": "philox", "dist": "uniform_f32", "n": 10**8},
        # Monte Carlo in double precision
        {"name": "philox uniform f64 1e8", "call": "fill", "engine": "philox", "dist": "uniform_f64", "n": 10**8},
        # noise arrays of an odd length, one call after another: the word
        # phase moves from call to call
        {"name": "philox gaussian f32 3e7+1", "call": "fill", "engine": "philox", "dist": "gaussian_f32",
         "n": 3 * 10**7 + 1},
        # the sweep's double precision normals
        {"name": "philox gaussian f64 1e8", "call": "fill", "engine": "philox", "dist": "gaussian_f64", "n": 10**8},
        # an ordinary fill on the sequential engine
        {"name": "mrg uniform f32 1e6", "call": "fill", "engine": "mrg", "dist": "uniform_f32", "n": 10**6},
        # the sweep's largest size: raw words for a consumer of its own
        {"name": "mrg bits 1e9", "call": "fill", "engine": "mrg", "dist": "bits", "n": 10**9},
        # one substream per parallel worker, both engines at their customary spacing
        {"name": "mrg substreams f64 16384", "call": "substreams", "engine": "mrg", "dist": "gaussian_f64",
         "streams": 16384, "n": 16384},
        {"name": "philox substreams 16384", "call": "substreams", "engine": "philox", "dist": "uniform_f32",
         "streams": 16384, "n": 16384},
        # 4096 generators with mixed distributions and sizes, one launch
        {"name": "batch 4096", "call": "batch", "count": 4096, "lo": 64, "hi": 1 << 20},
        # words from elsewhere, transformed
        {"name": "transform gaussian f32 1e8", "call": "transform", "dist": "gaussian_f32", "n": 10**8},
        # a burst of calorimeter events through the server: 3 uniforms and 1
        # gaussian a hit, waited for event by event
        {"name": "serve 48 events", "call": "serve", "events": 48, "hits": 8000},
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n | 1 if rng.random() < 0.4 else n

    call = rng.choice(["fill"] * 6 + ["substreams", "batch", "transform", "serve"])
    if call == "fill":
        return {"call": "fill", "engine": rng.choice(["philox", "mrg"]), "dist": rng.choice(sorted(DISTS)),
                "n": size(10**3, 2 * 10**8)}
    if call == "substreams":
        n = size(64, 65536)
        return {"call": "substreams", "engine": rng.choice(["philox", "mrg"]), "dist": rng.choice(sorted(DISTS)),
                "streams": size(16, max(16, min(16384, 10**8 // n))), "n": n}
    if call == "batch":
        return {"call": "batch", "count": size(8, 4096), "lo": 64, "hi": size(1 << 14, 1 << 20)}
    if call == "transform":
        return {"call": "transform", "dist": rng.choice(sorted(DISTS)), "n": size(10**3, 2 * 10**8)}
    return {"call": "serve", "events": rng.randint(4, 60), "hits": size(500, 20000)}


def distribution(name):
    kind, dtype, p0, p1 = DISTS[name]
    return grng.Distribution(kind, dtype, p0, p1)


def words_of(name, n):
    """Words of the engine's sequence that n outputs consume."""
    kind, dtype = DISTS[name][:2]
    if kind in (grng.GAUSSIAN, grng.LOGNORMAL):
        n = (n + 1) // 2 * 2
    return n * (2 if dtype == grng.F64 else 1)


def batch_table(case):
    """(distribution, size, element offset in its dtype's pool) per request."""
    r = np.random.Generator(np.random.PCG64(case["count"]))
    sizes = np.rint(np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"])))
    which = r.integers(0, len(BATCH_DISTS), size=case["count"])
    used = {grng.U32: 0, grng.F32: 0, grng.F64: 0}
    table = []
    for n, k in zip(sizes.astype(np.int64).tolist(), which.tolist()):
        dtype = DISTS[BATCH_DISTS[k]][1]
        table.append((BATCH_DISTS[k], n, used[dtype]))
        used[dtype] += (n + 63) // 64 * 64  # each output at a 256-byte boundary, as allocators place them
    return table, used


def event_hits(case):
    """Hits per event: lognormal around the case's mean."""
    r = np.random.Generator(np.random.PCG64(case["events"]))
    hits = np.rint(np.exp(r.normal(math.log(case["hits"]) - 0.32, 0.8, size=case["events"])))
    return np.clip(hits, 100, 200000).astype(np.int64).tolist()


def engine_seed(seed):
    return 2021 + 7919 * (int(seed) % (1 << 40))


def prepare(case, seed):
    call, s0 = case["call"], engine_seed(seed)
    if call == "fill":
        d = distribution(case["dist"])
        return {"call": call, "dist": d, "engine": grng.Engine(ENGINES[case["engine"]], s0),
                "out": torch.empty(case["n"], dtype=TORCH_TYPE[d.dtype], device="cuda")}
    if call == "substreams":
        d = distribution(case["dist"])
        log2 = MRG_STRIDE_LOG2 if case["engine"] == "mrg" else PHILOX_STRIDE_LOG2
        return {"call": call, "dist": d, "engine": grng.Engine(ENGINES[case["engine"]], s0), "n": case["n"],
                "streams": case["streams"], "stride": 1 << log2,
                "out": torch.empty(case["n"] * case["streams"], dtype=TORCH_TYPE[d.dtype], device="cuda")}
    if call == "batch":
        table, used = batch_table(case)
        pools = {t: torch.zeros(max(u, 64), dtype=TORCH_TYPE[t], device="cuda") for t, u in used.items()}
        reqs = []
        for i, (name, n, at) in enumerate(table):
            d = distribution(name)
            reqs.append((grng.Engine(grng.PHILOX4X32X10, s0 + i), d, pools[d.dtype][at:at + n]))
        batch = grng.Batch(reqs)
        return {"call": call, "batch": batch, "out": [pools[grng.U32], pools[grng.F32], pools[grng.F64]]}
    if call == "transform":
        d = distribution(case["dist"])
        return {"call": call, "dist": d, "words": given_words(case, seed),
                "out": torch.empty(case["n"], dtype=TORCH_TYPE[d.dtype], device="cuda")}
    reqs = [grng.serve_request(s0 + i, [(distribution("uniform_f32"), 3 * h), (distribution("gaussian_f32"), h)])
            for i, h in enumerate(event_hits(case))]
    return {"call": call, "server": grng.Server(256 << 20), "requests": reqs, "tickets": []}


def given_words(case, seed):
    g = torch.Generator(device="cuda").manual_seed(engine_seed(seed))
    return torch.randint(-(1 << 31), 1 << 31, (words_of(case["dist"], case["n"]),), dtype=torch.int32, device="cuda",
                         generator=g)


def run(state):
    call = state["call"]
    if call == "fill":
        return grng.generate(state["dist"], state["engine"], state["out"])
    if call == "substreams":
        return grng.generate_substreams(state["dist"], state["engine"], state["out"], state["n"], state["streams"],
                                        state["stride"])
    if call == "batch":
        state["batch"].launch()
        return state["out"]
    if call == "transform":
        return grng.transform_words(state["dist"], state["words"], state["out"])
    server = state["server"]
    for t in state["tickets"]:  # the consumer is done with the last burst
        server.release(t)
    state["tickets"] = [server.submit(q) for q in state["requests"]]
    return [server.output(t).view(torch.float32) for t in state["tickets"]]


# integer and floating point operations an output cannot do without: the
# engine's per word (Philox: 10 rounds of 2 products and 4 exclusive ors per 4
# words; MRG32k3a: 4 products, 2 sums, 2 reductions, the combination), then the
# transform's per output
ENGINE_OPS = {"philox": 15, "mrg": 12, "given": 0}


def transform_ops(name):
    kind, dtype = DISTS[name][:2]
    if kind == grng.BITS:
        return 0
    if kind == grng.UNIFORM:
        return 4
    return (25 if dtype == grng.F32 else 60) + (10 if kind in (grng.LOGNORMAL, grng.LOGNORMAL_ICDF) else 0)


def work(case):
    call = case["call"]
    engine = "given" if call == "transform" else case.get("engine", "philox")
    if call == "batch":
        parts = [(name, n) for name, n, _ in batch_table(case)[0]]
    elif call == "serve":
        h = sum(event_hits(case))
        parts = [("uniform_f32", 3 * h), ("gaussian_f32", h)]
    else:
        parts = [(case["dist"], case["n"] * case.get("streams", 1))]
    nbytes = flops = 0
    for name, n in parts:
        w = words_of(name, n)
        nbytes += n * (8 if DISTS[name][1] == grng.F64 else 4) + (4 * w if call == "transform" else 0)
        flops += w * ENGINE_OPS[engine] + n * transform_ops(name)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------ 64-bit values
M32 = 0xFFFFFFFF
MRG_M = (4294967087, 4294944443)


def mul_hi_lo(m, c):
    """High and low words of m * c, m a constant and c int64 tensors below 2^32."""
    a = (c & 0xFFFF) * m
    b = (c >> 16) * m + (a >> 16)
    return b >> 16, ((b & 0xFFFF) << 16) | (a & 0xFFFF)


def philox_blocks(key, counter):
    """[blocks, 4] words of the counter blocks `counter` (below 2^63), key an int or a tensor."""
    c = [counter & M32, counter >> 32, torch.zeros_like(counter), torch.zeros_like(counter)]
    k0, k1 = key & M32, key >> 32
    for _ in range(10):
        h0, l0 = mul_hi_lo(0xD2511F53, c[0])
        h1, l1 = mul_hi_lo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return torch.stack(c, 1)


def philox_words(seed, first, count):
    """Words [first, first + count) of a stream, `first` a multiple of 4."""
    b = torch.arange((count + 3) // 4, dtype=torch.int64, device="cuda") + first // 4
    return philox_blocks(seed, b).view(-1)[:count]


def mul_mod(a, b, m):
    return (((a * (b >> 16)) % m << 16) + a * (b & 0xFFFF)) % m


def mat_pow(a, e, m):
    r = [[int(i == j) for j in range(3)] for i in range(3)]
    mul = lambda x, y: [[sum(x[i][k] * y[k][j] for k in range(3)) % m for j in range(3)] for i in range(3)]  # noqa: E731
    while e:
        if e & 1:
            r = mul(r, a)
        a, e = mul(a, a), e >> 1
    return r


def mrg_words(seed, starts_log2, streams, count):
    """[streams, count] words of the substreams 2^starts_log2 words apart."""
    per = max(1, min(count, 65536 * 4 // streams))  # lanes of a stream
    steps = -(-count // per)
    mats = ([[0, 1, 0], [0, 0, 1], [MRG_M[0] - 810728, 1403580, 0]],
            [[0, 1, 0], [0, 0, 1], [MRG_M[1] - 1370589, 0, 527612]])
    states = []
    for a, m, x in ((mats[0], MRG_M[0], [1, 1, seed % MRG_M[0]]), (mats[1], MRG_M[1], [1, 1, 1])):
        state = [torch.tensor([v], dtype=torch.int64, device="cuda") for v in x]
        # lane states by doubling: [0, 2^k) jumped by 2^k units gives [2^k, 2^(k+1))
        for total, unit in ((per, steps), (streams, 1 << starts_log2)):
            wide, k = state, 0
            base = state[0].numel()
            while wide[0].numel() < total * base:
                j = mat_pow(a, unit << k, m)
                more = [(mul_mod(wide[0], torch.tensor(r[0], device="cuda"), m) +
                         mul_mod(wide[1], torch.tensor(r[1], device="cuda"), m) +
                         mul_mod(wide[2], torch.tensor(r[2], device="cuda"), m)) % m for r in j]
                wide = [torch.cat([p, q]) for p, q in zip(wide, more)]
                k += 1
            state = [v[:total * base] for v in wide]
        states.append(state)
    (x0, x1, x2), (y0, y1, y2) = states
    words = torch.empty(steps, streams * per, dtype=torch.int64, device="cuda")
    for i in range(steps):
        xn = (1403580 * x1 + 810728 * (MRG_M[0] - x0)) % MRG_M[0]
        yn = (527612 * y2 + 1370589 * (MRG_M[1] - y0)) % MRG_M[1]
        x0, x1, x2, y0, y1, y2 = x1, x2, xn, y1, y2, yn
        torch.remainder(xn - yn, MRG_M[0], out=words[i])
    return words.view(steps, streams, per).permute(1, 2, 0).reshape(streams, steps * per)[:, :count]


def values(name, w, n):
    """The n outputs per row of the words w [rows, words], in 64 bits."""
    kind, dtype, p0, p1 = DISTS[name]
    if kind == grng.BITS:
        return None
    pair = kind in (grng.GAUSSIAN, grng.LOGNORMAL)
    icdf = kind in (grng.GAUSSIAN_ICDF, grng.LOGNORMAL_ICDF)
    if dtype == grng.F64:
        w = w.reshape(w.shape[0], -1, 2)
        k = ((w[..., 0] << 20) | (w[..., 1] >> 12)) if icdf else ((w[..., 0] << 21) | (w[..., 1] >> 11))
        bits = 52 if icdf else 53
    else:
        k, bits = (w >> 9, 23) if icdf else (w >> 8, 24)
    if icdf:
        # u = (k + 1/2) 2^-bits through the nearer tail, where it is exact
        upper = k >= 1 << (bits - 1)
        tail = torch.where(upper, (1 << bits) - 1 - k, k)
        z = torch.special.ndtri((2 * tail + 1).double() * 2.0 ** -(bits + 1))
        x = torch.where(upper, -z, z)
    elif pair:
        k = k.reshape(k.shape[0], -1, 2)
        rho = torch.sqrt(-2.0 * torch.log((k[..., 0] + 1).double() * 2.0**-bits))
        # the angle by its octant's exact fraction of a turn
        turn = k[..., 1]
        quarter, rest = turn >> (bits - 2), turn & ((1 << (bits - 2)) - 1)
        ang = rest.double() * (2.0 ** -(bits - 1) * math.pi)
        c, s = torch.cos(ang), torch.sin(ang)
        cq = torch.where(quarter % 2 == 0, c, s) * torch.where((quarter == 1) | (quarter == 2), -1.0, 1.0)
        sq = torch.where(quarter % 2 == 0, s, c) * torch.where(quarter >= 2, -1.0, 1.0)
        x = torch.stack([rho * cq, rho * sq], -1).reshape(k.shape[0], -1)
    else:
        x = p0 + (p1 - p0) * (k.double() * 2.0**-bits)
    x = x[:, :n]
    if kind != grng.UNIFORM:
        x = p0 + p1 * x
    return torch.exp(x) if kind in (grng.LOGNORMAL, grng.LOGNORMAL_ICDF) else x


PART = 1 << 24  # words at a time, so that the intermediate tensors stay small


def philox_values(name, seed, first, n):
    out = []
    total = words_of(name, n)
    for at in range(0, total, PART):
        w = philox_words(seed, first + at, min(PART, total - at))
        left = n - at * n // total if at else n
        out.append(values(name, w[None], left)[0])
    return torch.cat(out)[:n]


def exact(case, seed):
    call, s0 = case["call"], engine_seed(seed)
    if call in ("fill", "substreams", "transform") and case["dist"] == "bits":
        return None
    if call == "transform":
        w = given_words(case, seed)
        return torch.cat([values(case["dist"], (p.to(torch.int64) & M32)[None], case["n"])[0]
                          for p in w.split(PART)])[:case["n"]]
    if call == "fill" and case["engine"] == "philox":
        return philox_values(case["dist"], s0, 0, case["n"])
    if call == "fill":
        w = mrg_words(s0, 0, 1, words_of(case["dist"], case["n"])).reshape(-1)
        return torch.cat([values(case["dist"], p[None], case["n"])[0] for p in w.split(PART)])[:case["n"]]
    if call == "substreams":
        name, n, streams = case["dist"], case["n"], case["streams"]
        words = words_of(name, n)
        rows, out = max(1, PART // words), []
        if case["engine"] == "mrg":
            for part in mrg_words(s0, MRG_STRIDE_LOG2, streams, words).split(rows):
                out.append(values(name, part, n))
        else:
            blocks = torch.arange((words + 3) // 4, dtype=torch.int64, device="cuda")
            for at in range(0, streams, rows):
                k = torch.arange(at, min(at + rows, streams), dtype=torch.int64, device="cuda")
                b = (k[:, None] << (PHILOX_STRIDE_LOG2 - 2)) + blocks[None]
                w = philox_blocks(s0, b.reshape(-1)).view(len(k), -1)[:, :words]
                out.append(values(name, w, n))
        return torch.cat(out).reshape(-1)
    if call == "batch":
        table, used = batch_table(case)
        pools = {t: torch.zeros(max(u, 64), dtype=torch.float64, device="cuda") for t, u in used.items()}
        for i, (name, n, at) in enumerate(table):
            if name != "bits":
                pools[DISTS[name][1]][at:at + n] = philox_values(name, s0 + i, 0, n)
        return [None, pools[grng.F32], pools[grng.F64]]
    return [torch.cat([philox_values("uniform_f32", s0 + i, 0, 3 * h),
                       values("gaussian_f32", philox_words(s0 + i, 0, 4 * h + 4)[3 * h:4 * h + h % 2][None], h)[0]])
            for i, h in enumerate(event_hits(case))]
