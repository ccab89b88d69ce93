"""Batched persistent launch (grng_batch_*) vs single calls and the oracle.

A batch must give every request exactly what the same grng_generate calls in
table order would give (requests of one engine follow each other in its
sequence), continue every sequence on the next launch (device-resident
offsets), replay identically from a CUDA graph, and leave the engines at the
right offsets after commit.  The full table: 4096 Philox engines, log-uniform
sizes in [64, 2^20], five distributions.
"""

import numpy as np
import pytest

import oracle
from paper_2109_01329_gb300 import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TDT = {0: torch.int32, 1: torch.float32, 2: torch.float64}


@pytest.fixture(scope="module")
def g():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2109_01329_gb300 as grng

    return grng


def _close(kind, dtype, got, ref):
    if kind in (0, 1):
        a = got.view(np.uint32 if got.dtype.itemsize == 4 else np.uint64)
        b = ref.view(np.uint32 if ref.dtype.itemsize == 4 else np.uint64)
        return np.array_equal(a, b)
    tol = 2e-6 if dtype == 1 else 1e-14
    return bool(np.all(np.abs(got.astype(np.float64) - ref) <= tol * np.maximum(1.0, np.abs(ref))))


def _host(t):
    a = t.cpu().numpy()
    return a.view(np.uint32) if a.dtype == np.int32 else a


VARS = [(0, 0, 0.0, 0.0), (1, 1, 0.0, 1.0), (1, 1, -2.5, 7.0), (1, 2, 0.0, 1.0),
        (1, 2, -1.0, 1.0), (1, 2, 2.0, 5.0), (2, 1, 0.5, 2.0), (3, 1, 0.0, 1.0),
        (2, 2, 0.0, 1.0), (3, 2, 0.25, 0.5), (4, 1, 0.0, 1.0), (5, 2, 0.0, 0.5)]


def _mixed_requests(g, seed=3, count=60):
    """Requests over all variants, odd sizes, misaligned pointers, shared engines."""
    rng = np.random.Generator(np.random.PCG64(seed))
    shared = [g.Engine(0, 1000 + k, int(rng.integers(0, 1 << 40))) for k in range(4)]
    reqs, meta = [], []
    for i in range(count):
        kind, dtype, p0, p1 = VARS[i % len(VARS)]
        n = int(rng.choice([0, 1, 2, 3, 5, 7, 64, 999, 4096, 70001]))
        pofs = int(rng.integers(0, 4)) if dtype != 2 else int(rng.integers(0, 2))
        buf = torch.empty(n + pofs + 1, dtype=TDT[dtype], device="cuda")
        out = buf[pofs:pofs + n]
        if i % 5 == 0:
            eng = shared[i % 4]
        else:
            eng = g.Engine(0, 7 * i + 1, int(rng.integers(0, 1 << 20)))
        reqs.append((eng, g.Distribution(kind, dtype, p0, p1), out, n))
        meta.append((kind, dtype, p0, p1, n))
    return reqs, meta, shared


def _expected_starts(g, reqs, meta):
    """Start offset of each request: its engine's offset plus earlier requests' words."""
    pos, starts = {}, []
    for (eng, dist, out, n), (kind, dtype, p0, p1, _) in zip(reqs, meta):
        key = id(eng)
        if key not in pos:
            pos[key] = eng.offset
        starts.append(pos[key])
        pos[key] += oracle.words_for(kind, dtype, n)
    return starts, pos


def _clone_requests(g, reqs):
    """The same requests on fresh engines with the same sharing and offsets."""
    fresh = {}
    out = []
    for (e, d, o, n) in reqs:
        if id(e) not in fresh:
            fresh[id(e)] = g.Engine(0, e.state[1], e.offset)
        out.append((fresh[id(e)], d, torch.empty_like(o), n))
    return out


def test_batch_equals_oracle_and_continues(g):
    reqs, meta, shared = _mixed_requests(g)
    starts, ends = _expected_starts(g, reqs, meta)
    seeds = [r[0].state[1] for r in reqs]
    b = g.Batch(reqs, ipt=2)
    b.launch()
    torch.cuda.synchronize()
    for i, ((eng, dist, out, n), (kind, dtype, p0, p1, _)) in enumerate(zip(reqs, meta)):
        ref = oracle.generate(0, seeds[i], starts[i], kind, dtype, p0, p1, n)
        assert _close(kind, dtype, _host(out), ref), f"request {i} {meta[i]} launch 1"
    # engines are untouched until commit
    assert all(r[0].offset == s for r, s in zip(reqs, starts) if id(r[0]) not in
               {id(e) for e in shared})
    # second launch: every engine advanced by all of its requests' words
    adv = {k: ends[k] - min(s for r, s in zip(reqs, starts) if id(r[0]) == k) for k in ends}
    b.launch()
    torch.cuda.synchronize()
    for i, ((eng, dist, out, n), (kind, dtype, p0, p1, _)) in enumerate(zip(reqs, meta)):
        ref = oracle.generate(0, seeds[i], starts[i] + adv[id(eng)], kind, dtype, p0, p1, n)
        assert _close(kind, dtype, _host(out), ref), f"request {i} {meta[i]} launch 2"
    b.commit()
    for (eng, _, _, _) in reqs:
        first = min(s for r, s in zip(reqs, starts) if r[0] is eng)
        assert eng.offset == first + 2 * adv[id(eng)]


def test_batch_graph_replay_equals_launches(g):
    reqs_a, meta, _ = _mixed_requests(g, seed=9, count=30)
    reqs_b = _clone_requests(g, reqs_a)
    ba = g.Batch(reqs_a, ipt=4)
    bb = g.Batch(reqs_b, ipt=4)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        ba.launch(stream=s)  # warm-up outside capture
        s.synchronize()
        with torch.cuda.graph(graph, stream=s):
            ba.launch(stream=s)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    # ba ran 1 eager launch + 3 replays = 4 launches (capturing does not execute)
    for _ in range(4):
        bb.launch()
    torch.cuda.synchronize()
    for (ea, da, oa, na), (eb, db, ob, nb) in zip(reqs_a, reqs_b):
        assert torch.equal(oa.view(torch.uint8), ob.view(torch.uint8))


def test_autotune_keeps_outputs(g):
    reqs, meta, _ = _mixed_requests(g, seed=4, count=20)
    b = g.Batch(reqs, ipt=1)
    b.launch()
    torch.cuda.synchronize()
    before = [r[2].clone() for r in reqs]
    # rewind: a fresh identical batch tuned then launched once
    reqs2 = _clone_requests(g, reqs)
    b2 = g.Batch(reqs2, ipt=1)
    ipt, ctas, ms = b2.autotune()
    assert ipt in (1, 2, 4, 8, 16, 32) and 1 <= ctas <= 32 and ms > 0
    b2.launch()
    torch.cuda.synchronize()
    for x, r in zip(before, reqs2):
        assert torch.equal(x.view(torch.uint8), r[2].view(torch.uint8))


@pytest.mark.parametrize("phased", [False, True], ids=["offset0", "word_phases"])
def test_4096_request_batch_equals_per_request(g, phased):
    """The 4096-request table, bit for bit against one grng_generate per
    request; with phased engines every request starts at a word offset of
    random phase mod 4 (the state of engines that have run before), so the
    groups straddle Philox blocks."""
    table = W.batched_requests(4096)
    rng0 = np.random.Generator(np.random.PCG64(77))
    offs = rng0.integers(0, 1 << 40, len(table)) if phased else np.zeros(len(table), np.int64)
    outs, reqs, singles = [], [], []
    for q, off in zip(table, offs):
        name, kind, dtype, p0, p1 = q["dist"]
        n = q["n"]
        d = g.Distribution(kind, dtype, p0, p1)
        out = torch.empty(n, dtype=TDT[dtype], device="cuda")
        reqs.append((g.Engine(0, q["seed"], int(off)), d, out, n))
        ref = torch.empty(n, dtype=TDT[dtype], device="cuda")
        g.generate(d, g.Engine(0, q["seed"], int(off)), ref)
        singles.append(ref)
    b = g.Batch(reqs, ipt=4)
    b.autotune()
    b.launch()
    torch.cuda.synchronize()
    bad = [i for i, (r, s) in enumerate(zip(reqs, singles))
           if not torch.equal(r[2].view(torch.uint8), s.view(torch.uint8))]
    assert not bad, f"{len(bad)} requests differ, first {bad[:5]}"
    # spot-check against the oracle
    rng = np.random.Generator(np.random.PCG64(1))
    for i in rng.integers(0, len(table), 24):
        q = table[int(i)]
        name, kind, dtype, p0, p1 = q["dist"]
        m = min(q["n"], 4096)
        ref = oracle.generate(0, q["seed"], int(offs[int(i)]), kind, dtype, p0, p1, m)
        assert _close(kind, dtype, _host(reqs[int(i)][2][:m]), ref)


def test_every_tuner_geometry_gives_the_same_outputs(g):
    """The output is a function of the word index only, so every launch
    geometry the autotuner tries (ipt x CTAs per SM) must give the outputs of
    the same grng_generate calls; each launch continues every sequence."""
    reqs, meta, _ = _mixed_requests(g, seed=9, count=40)
    refs = _clone_requests(g, reqs)
    b = g.Batch(reqs, ipt=8)  # workspace sized for ipt = 1: every ipt fits
    for ipt in (1, 2, 4, 8, 16, 32):
        for ctas in (1, 2, 4, 6, 8, 12, 16):
            b.set_config(ipt, ctas)
            b.launch()
            torch.cuda.synchronize()
            for (e, d, o, n), (er, dr, orf, nr) in zip(reqs, refs):
                g.generate(dr, er, orf, n=nr)
            torch.cuda.synchronize()
            for k, ((e, d, o, n), (er, dr, orf, nr)) in enumerate(zip(reqs, refs)):
                assert torch.equal(o[:n].view(torch.uint8), orf[:nr].view(torch.uint8)), \
                    (ipt, ctas, k)
    b.commit()
    for (e, d, o, n), (er, dr, orf, nr) in zip(reqs, refs):
        assert e.offset == er.offset


def test_set_config_refuses_a_map_that_does_not_fit(g):
    # 2^22 FP32 outputs are 2^20 groups: 4096 tiles at ipt 1, 512 at ipt 8
    d = g.Distribution.uniform(0.0, 1.0)
    reqs = [(g.Engine(0, 5, 0), d, torch.empty(1 << 22, dtype=torch.float32, device="cuda"),
             1 << 22)]
    b = g.Batch(reqs, ipt=8, tunable=False)
    b.set_config(16, 4)  # larger tiles: a smaller map, fits
    with pytest.raises(g.GrngError):
        b.set_config(1, 4)


@pytest.mark.parametrize("heavy", [False, True])
def test_launches_continue_across_carries_and_tile_runs(g, heavy):
    """Requests long enough for runs of several tiles, starting before, across and
    after a carry out of the low 32 bits of the block counter, at every word
    phase and from misaligned outputs: each of three launches equals the
    per-request calls bit for bit, and commit moves the engines by all three.
    Without the FP64 fixed-point transforms the lighter kernel takes them."""
    dists = [(0, 0), (1, 1), (1, 2), (2, 1), (3, 1), (4, 1)] + ([(2, 2), (3, 2), (4, 2)] if heavy else [])
    reqs, refs = [], []
    for i, (kind, dtype) in enumerate(dists * 4):
        n = (3, 1001, 8191 * 4 + 1, 300_003)[i // len(dists)]
        off = ((1 << 34) - 2 * n + i, (1 << 66) - n // 2 - i, i, 5 + i)[i % 4]
        d = g.Distribution(kind, dtype, 0.0, 1.0 if kind else 0.0)
        buf = torch.zeros(n + 4, dtype=TDT[dtype], device="cuda")
        reqs.append((g.Engine(0, 100 + i, off), d, buf[i % 3:i % 3 + n]))
        refs.append((g.Engine(0, 100 + i, off), d, torch.zeros(n, dtype=TDT[dtype], device="cuda"), buf, i % 3))
    b = g.Batch(reqs)
    for _ in range(3):
        b.launch()
        for (_, d, out), (e, _, ref, buf, lead) in zip(reqs, refs):
            g.generate(d, e, ref)
        torch.cuda.synchronize()
        for i, ((_, d, out), (_, _, ref, buf, lead)) in enumerate(zip(reqs, refs)):
            assert torch.equal(out.contiguous().view(torch.uint8), ref.view(torch.uint8)), (i, d)
            assert not buf[:lead].any() and not buf[lead + ref.numel():].any(), (i, d)
    b.commit()
    for (e, _, _), (r, _, _, _, _) in zip(reqs, refs):
        assert e.offset == r.offset


@pytest.mark.parametrize("kind, dtype", [(0, 0), (1, 1), (1, 2), (2, 1), (3, 1), (4, 1)])
def test_every_phase_at_the_edges_of_tiles_and_chunks(g, kind, dtype):
    """Sizes around a group, a warp's one and two chunks of 31 groups and a tile of
    256 groups, at every word phase and output alignment: equal to the
    per-request call bit for bit, nothing written outside."""
    epg = 2 if dtype == 2 else 4  # elements per group
    sizes = [m * epg + d for m in (0, 1, 2, 30, 31, 61, 62, 63, 256, 257, 258, 512, 1000) for d in (-1, 0, 1, 2)]
    d = g.Distribution(kind, dtype, 0.0, 1.0 if kind else 0.0)
    reqs, refs = [], []
    for i, n in enumerate(n for n in sizes if n > 0):
        for phase in range(4):
            lead = (i + phase) % 3 if i % 2 else 0
            buf = torch.zeros(n + 8, dtype=TDT[dtype], device="cuda")
            reqs.append((g.Engine(0, i, phase), d, buf[lead:lead + n]))
            refs.append((g.Engine(0, i, phase), torch.zeros(n, dtype=TDT[dtype], device="cuda"), buf, lead))
    for ipt in (1, 8):
        b = g.Batch(reqs, ipt=ipt)
        b.launch()
        for e, ref, _, _ in refs:
            g.generate(d, e.copy(), ref)
        torch.cuda.synchronize()
        for (e, ref, buf, lead) in refs:
            n = ref.numel()
            assert torch.equal(buf[lead:lead + n].clone().view(torch.uint8), ref.view(torch.uint8)), (n, e.offset, lead)
            assert not buf[:lead].any() and not buf[lead + n:].any(), (n, e.offset, lead)


def test_launches_after_overlapping_ones_continue_past_all(g):
    """Launches of one batch left to overlap on two streams, with unequal grids
    between: those after them still give the per-request calls' outputs at the
    launches' number of advances, and commit moves the engines by all of them."""
    dists = [(0, 0), (1, 1), (2, 1), (1, 2)]
    reqs, refs = [], []
    for i, (kind, dtype) in enumerate(dists * 6):
        n = (1003, 70_001, 1 << 18)[i % 3]
        d = g.Distribution(kind, dtype, 0.0, 1.0 if kind else 0.0)
        reqs.append((g.Engine(0, i, 5 * i), d, torch.empty(n, dtype=TDT[dtype], device="cuda")))
        refs.append(g.Engine(0, i, 5 * i))
    b = g.Batch(reqs)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    total = 0
    for ctas in (32, 1, 4):
        b.set_config(8, ctas)
        torch.cuda.synchronize()
        for _ in range(20):
            for s in streams:
                b.launch(stream=s)
                total += 1
        torch.cuda.synchronize()
        b.launch()
        total += 1
        torch.cuda.synchronize()
        for i, ((_, d, out), start) in enumerate(zip(reqs, refs)):
            e = start.copy()
            e.skip_ahead((total - 1) * g.words_for(d, out.numel()))
            want = torch.empty_like(out)
            g.generate(d, e, want)
            assert torch.equal(out.view(torch.uint8), want.view(torch.uint8)), (ctas, i)
    b.commit()
    for (e, d, out), start in zip(reqs, refs):
        assert e.offset == start.offset + total * g.words_for(d, out.numel())


@pytest.mark.parametrize("run", [2, 8])
@pytest.mark.parametrize("heavy", [False, True])
def test_merged_tiles_with_carries_splits_and_ragged_ends(g, heavy, run):
    """Batches of enough tiles that a CTA takes two or eight at a time, those of one
    request as one: requests that end inside a run, start misaligned, at every word
    phase, with a Box-Muller pair split by the output's start, and before and
    across a carry out of the low block counter word equal the per-request calls bit
    for bit."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    dists = [(0, 0), (1, 1), (2, 1), (3, 1)] + ([(2, 2), (3, 2), (4, 2)] if heavy else [(1, 2), (4, 1)])
    # tiles of 256 groups: this many of them over the requests below
    per = (16 * sms * run + 16 * sms // 2) // (2 * len(dists)) + 3
    reqs, refs, tiles = [], [], 0
    for i, (kind, dtype) in enumerate(dists * 2):
        epg = 2 if dtype == 2 else 4
        n = (per * 256 + 37 * i) * epg + i % 3
        words = oracle.words_for(kind, dtype, n)
        off = ((1 << 34) - words // 3 + i, i, (1 << 34) - 2 * words - i)[i % 3] & ~(1 if dtype == 2 and i % 2 else 0)
        lead = i % 4 if dtype != 2 else i % 2
        d = g.Distribution(kind, dtype, 0.0, 1.0 if kind else 0.0)
        buf = torch.zeros(n + 8, dtype=TDT[dtype], device="cuda")
        reqs.append((g.Engine(0, 100 + i, off), d, buf[lead:lead + n]))
        refs.append((g.Engine(0, 100 + i, off), buf, lead))
        tiles += -(-(lead + n) // (256 * epg))
    assert min(8, tiles // (16 * sms)) == run
    b = g.Batch(reqs)
    b.set_config(1, 32)
    for _ in range(2):
        b.launch()
        for (_, d, out), (e, buf, lead) in zip(reqs, refs):
            want = torch.empty_like(out)
            g.generate(d, e, want)
            torch.cuda.synchronize()
            assert torch.equal(out.clone().view(torch.uint8), want.view(torch.uint8)), (d, lead, out.numel())
            assert not buf[:lead].any() and not buf[lead + out.numel():].any(), (d, lead)
