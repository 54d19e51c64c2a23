"""Parity of the CUDA path (through the C ABI) with the CPU oracle.

Integer results -- sites, mismatch counts, amplicons, pass flags, sequences
-- must be identical; the fp32 Tm must be within 0.01 deg C of the oracle's
fp64 value (NaN where the oracle has NaN).  Inputs are seeded synthetic
workloads; nothing here is produced by the CUDA path and then trusted.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2509_13300_gb300 import ah, build, synth

pytestmark = pytest.mark.gpu
TM_TOL = 0.01  # deg C


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = ah.Context(0)
    yield c
    c.close()


def gpu_run(ctx, w, table=None):
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in w.pairs]
        if table is not None:
            for p in pids:
                ctx.ah_set_nn_table(p, table)
        sites = ctx.scan(sid, pids)
        tm, ps = ctx.tm(sid, pids, sites)
        amps = ctx.pair(sid, pids, sites)
        amps_tm = ctx.pair(sid, pids, sites, ps)
        seqs, offs = ctx.fetch(sid, amps)
    finally:
        ctx.ah_unload_genomes(sid)
    return dict(sites=sites, tm=tm, pass_=ps, amps=amps, amps_tm=amps_tm, seqs=seqs, offs=offs)


def oracle_run(w, table=None):
    sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, w.pairs)
    tm, ps = oracle.tm(w.seq, w.contig_off, sites, w.pairs, table)
    amps = oracle.pair(sites, w.pairs)
    amps_tm = oracle.pair(sites, w.pairs, ps)
    seqs, offs = oracle.fetch(w.seq, w.contig_off, amps)
    return dict(sites=sites, tm=tm, pass_=ps, amps=amps, amps_tm=amps_tm, seqs=seqs, offs=offs)


def assert_parity(g, o, min_sites=1):
    assert len(g["sites"]) == len(o["sites"]), (len(g["sites"]), len(o["sites"]))
    assert len(o["sites"]) >= min_sites
    assert g["sites"].tobytes() == o["sites"].tobytes()
    tg, to = g["tm"].astype(np.float64), o["tm"]
    nan_g, nan_o = np.isnan(tg), np.isnan(to)
    assert np.array_equal(nan_g, nan_o)
    if (~nan_o).any():
        err = np.abs(tg[~nan_o] - to[~nan_o]).max()
        assert err <= TM_TOL, err
    assert np.array_equal(g["pass_"], o["pass_"])
    assert g["amps"].tobytes() == o["amps"].tobytes()
    assert g["amps_tm"].tobytes() == o["amps_tm"].tobytes()
    assert np.array_equal(g["offs"], o["offs"])
    assert g["seqs"] == o["seqs"]


def test_tiny_workload(ctx):
    """Plain method, tiny: 200 kbp, 3 contigs, 10 planted amplicons, k = 2."""
    w = synth.tiny(0)
    o = oracle_run(w)
    assert_parity(gpu_run(ctx, w), o, min_sites=10)
    # the same with the paper's default 50 deg C threshold (Sec. 3.2)
    w.pairs = [dict(w.pairs[0], tm_min=50.0)]
    o2 = oracle_run(w)
    assert 0 < o2["pass_"].sum() < len(o2["pass_"]) or len(o2["pass_"]) == 0
    assert_parity(gpu_run(ctx, w), o2)


@pytest.mark.parametrize("seed,k,clamp", [(1, 0, 0), (2, 1, 0), (3, 2, 1), (4, 3, 0), (5, 4, 2), (6, 5, 0),
                                          (7, 7, 0), (8, 9, 3), (9, 10, 0)])
def test_random_small_with_edge_letters(ctx, seed, k, clamp):
    """Short primers so hits are frequent; lower case, IUPAC letters and gaps in
    the genome; several contigs including tiny ones; k from 0 to 10."""
    max_len = 900 if k < 4 else 200 if k < 7 else 80
    w = synth.random_small(seed, n_bases=60_000 // (1 + k // 3) + 777 * seed, n_contigs=7, L_f=7 + k + seed % 3,
                           L_r=6 + k + seed % 2, k=k, codes_f="RNY"[: 1 + seed % 3], codes_r="SBD"[: 1 + seed % 3],
                           lower_frac=0.05, iupac_frac=0.003, min_len=30, max_len=max_len)
    w.pairs = [dict(w.pairs[0], clamp=clamp, tm_min=float(seed * 3))]
    assert_parity(gpu_run(ctx, w), oracle_run(w))


@pytest.mark.parametrize("clamp", [0, 3])
def test_longest_primers_with_planted_sites(ctx, clamp):
    """Primers of the longest supported length (32, the width of a window word)
    and 31, planted on both strands with 0..6 substitutions at k = 4, some
    across contig ends and next to no-base runs: the whole path equals the
    oracle."""
    rng = np.random.default_rng(77 + clamp)
    fwd = synth.random_primer(rng, 32, "RYNSW")
    rev = synth.random_primer(rng, 31, "KMY")
    n = 400_000
    g = synth.random_bases(rng, n, 0.5)
    for s0 in rng.integers(0, n - 100, 60):
        g[s0:s0 + int(rng.integers(1, 40))] = ord("N")
    for j in range(80):
        a = int(rng.integers(0, n - 2600))
        f = synth._draw_oligo(rng, fwd, int(rng.integers(0, 7)))
        r = synth._revcomp(synth._draw_oligo(rng, rev, int(rng.integers(0, 7))))
        gap = int(rng.integers(100, 2400))
        left, right = (f, r) if j % 2 == 0 else (r, f)  # FR and RF
        g[a:a + len(left)] = np.frombuffer(left.encode(), np.uint8)
        g[a + 32 + gap:a + 32 + gap + len(right)] = np.frombuffer(right.encode(), np.uint8)
    cuts = np.sort(rng.choice(np.arange(1, n), 6, replace=False)).astype(np.uint64)
    off = np.concatenate([[0], cuts, [n]]).astype(np.uint64)
    w = synth.Workload("longest", g, off, np.zeros(len(off) - 1, np.uint32),
                       [synth.pcr_params(fwd, rev, k=4, min_len=100, max_len=3000, clamp=clamp)],
                       np.zeros(0, dtype=synth.PLANT_DTYPE))
    o = oracle_run(w)
    assert len(o["sites"]) >= 40 and len(o["amps"]) >= 10
    assert_parity(gpu_run(ctx, w), o)


def test_thread_per_site_tm_at_high_degeneracy(ctx):
    """Primers of 8,192 and 4,096 oligos (six N and an R; six N), enough chance
    sites (above 32,768) for the thread-per-site Tm: every site's maximum over
    all oligos within 0.01 C of the oracle's enumeration of every oligo, the
    pass flags exact at a threshold near the median, and the whole path equal."""
    rng = np.random.default_rng(5)
    fwd, rev = "ANCNGNTNANCR", "CNNGNNTANNGC"
    n = 3_200_000
    g = synth.random_bases(rng, n, 0.5)
    off = np.array([0, 400_000, 1_300_000, 2_500_000, n], np.uint64)
    w = synth.Workload("degenerate", g, off, np.zeros(4, np.uint32),
                       [synth.pcr_params(fwd, rev, k=1, min_len=30, max_len=60, tm_min=31.0)],
                       np.zeros(0, dtype=synth.PLANT_DTYPE))
    o = oracle_run(w)
    assert len(o["sites"]) > 32768 and 0.2 < o["pass_"].mean() < 0.8
    assert_parity(gpu_run(ctx, w), o)


def test_k_at_least_length_reports_every_window(ctx):
    w = synth.random_small(21, n_bases=5000, n_contigs=3, L_f=6, L_r=5, k=6, min_len=5, max_len=40)
    assert_parity(gpu_run(ctx, w), oracle_run(w), min_sites=19000)


def test_several_pairs_in_one_pass(ctx):
    rng = np.random.default_rng(5)
    w = synth.random_small(33, n_bases=120_000, n_contigs=5, L_f=12, L_r=10, k=2, min_len=40, max_len=2000)
    pairs = [w.pairs[0]]
    for j in range(4):
        f = synth.random_primer(rng, 10 + j, "RY")
        r = synth.random_primer(rng, 11 + j, "N")
        pairs.append(synth.pcr_params(f, r, k=j % 4, min_len=20 + j, max_len=1500, tm_min=20.0))
    w.pairs = pairs
    assert_parity(gpu_run(ctx, w), oracle_run(w))


def test_many_sites_take_the_thread_per_site_tm_path(ctx):
    """Over 32,768 sites, so ah_tm runs the one-thread-per-site kernel; its
    maximum is within 0.01 C of the oracle's, and with the threshold put
    exactly on an oracle site value (such sites are deferred to the exact
    decision) every pass flag is still the fp64 one."""
    w = synth.random_small(41, n_bases=300_000, n_contigs=4, L_f=11, L_r=10, k=4, codes_f="RYN", codes_r="SWK",
                           min_len=30, max_len=300)
    o = oracle_run(w)
    assert len(o["sites"]) >= 40_000
    ok = ~np.isnan(o["tm"])
    med = float(np.median(o["tm"][ok]))
    at_site = float(o["tm"][ok][np.argmin(np.abs(o["tm"][ok] - med))])
    for thr in (med + 0.003, at_site):
        w.pairs = [dict(w.pairs[0], tm_min=thr)]
        o = oracle_run(w)
        assert 0 < o["pass_"].sum() < len(o["pass_"])
        assert_parity(gpu_run(ctx, w), o)
    # ah_run, twice: the first run overflows the one-synchronisation sizes and
    # finishes step by step; the second (the last count was large) queues only
    # the scan in ah_run_begin and finishes in ah_run_end
    p = w.pairs[0]
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
        runs = [ctx.run(sid, [pid], tm_filter=True) for _ in range(2)]
    finally:
        ctx.ah_unload_genomes(sid)
    o_amps = oracle.pair(o["sites"], w.pairs, o["pass_"])
    o_seqs, o_offs = oracle.fetch(w.seq, w.contig_off, o_amps)
    for r in runs:
        assert r["sites"].tobytes() == o["sites"].tobytes()
        assert np.array_equal(r["pass_"], o["pass_"])
        ok = ~np.isnan(o["tm"])
        assert np.abs(r["tm"][ok].astype(np.float64) - o["tm"][ok]).max() <= TM_TOL
        assert r["amps"].tobytes() == o_amps.tobytes() and r["seqs"] == o_seqs


def test_scan_wait_limit_reports_timeout_and_the_context_stays_usable(ctx):
    """Failure detection without a fault: each warp's first slice waits on a
    barrier that no copy will complete (20 us limit); the scan gives up, waits
    for its warps' real copies still in flight and ah_scan returns
    AH_ERR_TIMEOUT; the next scan on the same context is exact."""
    w = synth.random_small(51, n_bases=3_000_000, n_contigs=3, L_f=16, L_r=15, k=2, min_len=30, max_len=900)
    p = w.pairs[0]
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
        ctx.debug_scan_stall(True)
        try:
            with pytest.raises(ah.AHError) as e:
                ctx.scan(sid, [pid])
            assert e.value.status == ah.AH_ERR_TIMEOUT
        finally:
            ctx.debug_scan_stall(False)
        sites = ctx.scan(sid, [pid])
    finally:
        ctx.ah_unload_genomes(sid)
    assert sites.tobytes() == oracle.scan(w.seq, w.contig_off, w.contig_genome, w.pairs).tobytes()


@pytest.mark.parametrize("fwd,rev,k", [
    ("ACGTTGCAAC", "GGTACCATTG", 1),            # network over a part of the positions
    ("NNNNNN", "NNNACNNN", 0),                  # nothing, or two positions, to count
    ("RYSWKMRYSW", "BDHVRYBDH", 2),             # no single-base position: no complements
    ("ACGNBDHRYSWKAC", "TGCANNNNNNACGT", 2),  # complements beside single bases, N left out
    ("ACGTACGTACGTACGTACGTACGTACGTACGT", "TTGACWSKMRYBDHANACGTACGGTACGATCA", 9),
])
@pytest.mark.parametrize("n_bases", [31, 32 * 1024 - 1, 32 * 1024 + 1, 5 * 32 * 1024, 300_007])
def test_scan_filter_at_tile_edges(ctx, fwd, rev, k, n_bases):
    """The scan's network counts only some positions and lets other starts through to the exact
    count: sites equal the oracle's on sets around a tile's size, with runs of non-bases."""
    rng = np.random.default_rng(n_bases + k)
    seq = synth.random_bases(rng, n_bases, 0.5).copy()
    for s0 in rng.integers(0, n_bases, 1 + n_bases // 2000):
        seq[s0:s0 + int(rng.integers(1, 90))] = ord("N")
    for i, L in ((0, len(fwd)), (1, len(rev))):  # planted sites, also at the very end
        for at in [n_bases - L] + list(rng.integers(0, max(1, n_bases - L), 5)):
            if 0 <= at <= n_bases - L:
                oligo = synth._draw_oligo(rng, (fwd, rev)[i], int(rng.integers(0, k + 1)))
                seq[at:at + L] = np.frombuffer((oligo if i == 0 else synth._revcomp(oligo)).encode(), np.uint8)
    cuts = np.unique(rng.integers(1, n_bases, 4))
    off = np.concatenate([[0], cuts, [n_bases]]).astype(np.uint64)
    gen = np.zeros(len(off) - 1, np.uint32)
    pairs = [synth.pcr_params(fwd, rev, k=k, min_len=20, max_len=400)]
    want = oracle.scan(seq, off, gen, pairs)
    sid = ctx.load(seq, off, gen)
    try:
        got = ctx.scan(sid, [ctx.ah_set_primers(fwd, rev, pairs[0])])
    finally:
        ctx.ah_unload_genomes(sid)
    assert got.tobytes() == want.tobytes(), (len(got), len(want))


def test_full_collection_workload_against_the_oracle(ctx):
    """The whole 100-genome collection workload (0.41 Gbp, 1,777 contigs, the
    960-oligo pair, k = 3, Tm threshold 50 C) through ah_run, against the oracle
    on every genome: sites, pass flags, Tm-filtered amplicons and sequences."""
    import os
    import bench
    w = bench.workload(1, 100)
    p = w.pairs[0]
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
        g = ctx.run(sid, [pid], tm_filter=True)
    finally:
        ctx.ah_unload_genomes(sid)
    cores = os.cpu_count() or 1
    s = oracle.scan(w.seq, w.contig_off, w.contig_genome, w.pairs, n_threads=cores)
    tm, ps = oracle.tm(w.seq, w.contig_off, s, w.pairs, n_threads=cores)
    a = oracle.pair(s, w.pairs, ps)
    q, qo = oracle.fetch(w.seq, w.contig_off, a)
    assert len(s) > 5000 and len(a) > 100
    assert g["sites"].tobytes() == s.tobytes()
    ok = ~np.isnan(tm)
    assert np.array_equal(np.isnan(g["tm"]), ~ok)
    assert np.abs(g["tm"][ok].astype(np.float64) - tm[ok]).max() <= TM_TOL
    assert np.array_equal(g["pass_"], ps)
    assert g["amps"].tobytes() == a.tobytes()
    assert g["seqs"] == q and np.array_equal(g["offs"].astype(np.uint64), qo.astype(np.uint64))


@pytest.mark.parametrize("device_input", [False, True])
def test_2bit_load_gives_the_letters(ctx, device_input):
    """ah_load_genomes_2bit over 70 Mbp (two host staging chunks, a tiny
    contig, a contig ending inside a tile, N runs, IUPAC letters, gaps and
    lower case): fetching every contig whole gives the input upper-cased with
    every non-ACGT letter as N, exactly as the ASCII load does."""
    import torch
    rng = np.random.default_rng(23)
    n = 70_000_003
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n)].copy()
    lower = rng.random(n) < 0.01
    seq[lower] += 32
    for s0 in rng.integers(0, n - 200, 3000):  # runs of other letters
        seq[s0:s0 + int(rng.integers(1, 120))] = np.frombuffer(b"NRY-", np.uint8)[int(rng.integers(0, 4))]
    off = np.array([0, 5, 40_000_000, 40_032_781, 69_999_000, n], dtype=np.uint64)
    gen = np.array([0, 0, 1, 1, 2], dtype=np.uint32)
    codes, gaps = ah.encode_2bit(seq)
    src = torch.from_numpy(codes).cuda() if device_input else codes
    amps = np.zeros(len(off) - 1, dtype=ah.AMPLICON_DTYPE)
    amps["genome"] = gen
    amps["contig"] = np.arange(len(off) - 1)
    amps["end"] = np.diff(off.astype(np.int64))
    up = np.where((seq >= 97) & (seq <= 122), seq - 32, seq).astype(np.uint8)
    want = np.where(np.isin(up, np.frombuffer(b"ACGT", np.uint8)), up, ord("N")).astype(np.uint8).tobytes()
    for load in ("2bit", "ascii"):
        if load == "2bit":
            sid = ctx.ah_load_genomes_2bit(src, n, gaps, off, gen)
        else:
            sid = ctx.load(seq, off, gen)
        try:
            got, offs = ctx.fetch(sid, amps)
        finally:
            ctx.ah_unload_genomes(sid)
        assert got == want, load
        assert np.array_equal(offs.astype(np.int64), off.astype(np.int64))


def test_2bit_load_scan_parity(ctx):
    """The whole path on a set loaded from 2-bit codes equals the oracle on the
    letters (short primers, lower case, IUPAC letters and gaps, tiny contigs)."""
    w = synth.random_small(61, n_bases=90_000, n_contigs=7, L_f=9, L_r=8, k=2, codes_f="RN", codes_r="SB",
                           lower_frac=0.05, iupac_frac=0.01, min_len=30, max_len=600)
    codes, gaps = ah.encode_2bit(w.seq)
    sid = ctx.ah_load_genomes_2bit(codes, len(w.seq), gaps, w.contig_off, w.contig_genome)
    try:
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in w.pairs]
        sites = ctx.scan(sid, pids)
        tm, ps = ctx.tm(sid, pids, sites)
        amps = ctx.pair(sid, pids, sites)
        amps_tm = ctx.pair(sid, pids, sites, ps)
        seqs, offs = ctx.fetch(sid, amps)
    finally:
        ctx.ah_unload_genomes(sid)
    g = dict(sites=sites, tm=tm, pass_=ps, amps=amps, amps_tm=amps_tm, seqs=seqs, offs=offs)
    assert_parity(g, oracle_run(w), min_sites=50)


def test_2bit_loads_in_flight_on_two_streams(ctx):
    """Two 2-bit loads queued back to back on two streams, without waiting
    (the batched form's pattern): each set keeps its own no-base runs, so both
    give their letters."""
    import torch
    rng = np.random.default_rng(31)
    seqs, srcs, gapss, offs = [], [], [], []
    for j, n in enumerate((9_000_017, 7_500_001)):
        seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n)].copy()
        for s0 in rng.integers(0, n - 200, 4000 + 3000 * j):
            seq[s0:s0 + int(rng.integers(1, 60))] = ord("N")
        codes, gaps = ah.encode_2bit(seq)
        seqs.append(seq)
        srcs.append(torch.from_numpy(codes).cuda())
        gapss.append(gaps)
        offs.append(np.array([0, n // 3, n], dtype=np.uint64))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    sids = [ctx.ah_load_genomes_2bit(srcs[j], len(seqs[j]), gapss[j], offs[j], np.zeros(2, np.uint32), streams[j])
            for j in range(2)]
    try:
        for j in range(2):
            amps = np.zeros(2, dtype=ah.AMPLICON_DTYPE)
            amps["contig"] = [0, 1]
            amps["end"] = np.diff(offs[j].astype(np.int64))
            got, _ = ctx.fetch(sids[j], amps)
            want = np.where(seqs[j] == ord("N"), ord("N"), seqs[j]).astype(np.uint8).tobytes()
            assert got == want, j
    finally:
        for sid in sids:
            ctx.ah_unload_genomes(sid)


def test_host_loads_queued_without_waiting(ctx):
    """AH_LOAD_HOST_ASYNC: host loads (2-bit and ASCII, pinned buffers, several
    sets queued back to back on two streams while a run is pending) return
    before their copies finish; every set still gives its letters, and a run on
    each equals the oracle's."""
    import torch
    rng = np.random.default_rng(47)
    w = synth.random_small(62, n_bases=300_000, n_contigs=5, L_f=9, L_r=8, k=2, codes_f="RN", codes_r="SB",
                           min_len=30, max_len=600)
    p = w.pairs[0]
    pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
    o = oracle_run(w)
    seqs, srcs = [], []
    for j, n in enumerate((5_000_011, 3_200_003, 4_100_000)):
        seq = np.frombuffer(b"ACGTacgt", np.uint8)[rng.integers(0, 8, n)].copy()
        for s0 in rng.integers(0, n - 200, 2000):
            seq[s0:s0 + int(rng.integers(1, 60))] = ord("N")
        seqs.append(seq)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    # a run in flight on the small set while the big host loads are queued
    sid0 = ctx.load(w.seq, w.contig_off, w.contig_genome)
    sids, keep = [], []
    try:
        for j, seq in enumerate(seqs):
            off = np.array([0, len(seq) // 2, len(seq)], np.uint64)
            if j % 2 == 0:
                codes, gaps = ah.encode_2bit(seq)
                host = torch.from_numpy(codes).pin_memory()
                sids.append(ctx.ah_load_genomes_2bit(host, len(seq), gaps, off, np.zeros(2, np.uint32),
                                                     streams[j % 2], host_async=True))
            else:
                host = torch.from_numpy(seq).pin_memory()
                sids.append(ctx.ah_load_genomes(host, len(seq), off, np.zeros(2, np.uint32), streams[j % 2],
                                                host_async=True))
            keep.append(host)  # unchanged until the set is ready
        r = ctx.run(sid0, [pid], tm_filter=True)
        assert r["sites"].tobytes() == o["sites"].tobytes() and r["amps"].tobytes() == o["amps_tm"].tobytes()
        for j, seq in enumerate(seqs):
            amps = np.zeros(2, dtype=ah.AMPLICON_DTYPE)
            amps["contig"] = [0, 1]
            amps["end"] = [len(seq) // 2, len(seq) - len(seq) // 2]
            got, _ = ctx.fetch(sids[j], amps)
            up = np.where(seq == ord("N"), ord("N"), seq & 0xDF).astype(np.uint8).tobytes()
            assert got == up, j
    finally:
        for sid in sids:
            ctx.ah_unload_genomes(sid)
        ctx.ah_unload_genomes(sid0)
    with pytest.raises(ah.AHError) as e:
        ctx._check(ctx._lib.ah_load_genomes_2bit_ex(ctx.h, ah._ptr(np.zeros(4, np.uint8)), 16, None, 0,
                                                    ah._ptr(np.array([0, 16], np.uint64)), 1,
                                                    ah._ptr(np.zeros(1, np.uint32)), 1, ah.ctypes.byref(
                                                        ah.ctypes.c_uint32()), None))
    assert e.value.status == ah.AH_ERR_ARG  # the reversed flag has no 2-bit form


def test_2bit_load_rejects_bad_gaps(ctx):
    codes = np.zeros(25, np.uint8)
    off, gen = np.array([0, 100], np.uint64), np.zeros(1, np.uint32)
    for bad in ([[10, 0]], [[10, 5], [12, 3]], [[90, 20]], [[50, 5], [10, 5]]):
        with pytest.raises(ah.AHError) as e:
            ctx.ah_load_genomes_2bit(codes, 100, np.array(bad, np.uint64), off, gen)
        assert e.value.status == ah.AH_ERR_ARG


def test_collection_spanning_many_tiles(ctx):
    """Genome-collection generator at reduced size: ~5 Mbp, 6 genomes, many
    contigs, N runs, planted operons with 0-4 substitutions, the 960-oligo pair."""
    w = synth.collection(seed=1, n_genomes=6, len_lo=4e5, len_hi=1.5e6, max_subs=4)
    o = oracle_run(w)
    assert len(o["amps"]) >= 3
    assert_parity(gpu_run(ctx, w), o)


def test_paper_primer_pairs(ctx):
    """The four benchmark pairs printed in the paper (Sec. 2.3) on one collection."""
    pairs = [synth.pcr_params(f, r, k=2, min_len=100, max_len=3000, tm_min=50.0)
             for f, r in synth.PAPER_PAIRS.values()]
    w = synth.collection(seed=4, n_genomes=3, len_lo=3e5, len_hi=8e5, pairs=pairs, plant_max=4, max_subs=2)
    assert_parity(gpu_run(ctx, w), oracle_run(w))


@pytest.mark.parametrize("salt", [0, 1, 5])
def test_salt_methods_and_ions(ctx, salt):
    w = synth.tiny(0)
    w.pairs = [dict(w.pairs[0], saltcorr=salt, K_mM=10.0, Tris_mM=20.0, Mg_mM=1.5, dNTPs_mM=0.2,
                    dnac1_nM=400.0, dnac2_nM=100.0, tm_min=45.0)]
    assert_parity(gpu_run(ctx, w), oracle_run(w))


@pytest.mark.parametrize("salt", [2, 3, 4, 6, 7, -1])
def test_salt_methods_not_offered_are_rejected(ctx, salt):
    """Only the salt methods the oracle pins to published values (0, 1, 5) are offered."""
    p = dict(synth.tiny(0).pairs[0], saltcorr=salt)
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers(p["fwd"], p["rev"], p)
    assert e.value.status == ah.AH_ERR_ARG


def test_custom_nn_table_with_mismatch_terms(ctx):
    """A table with non-zero mismatch stacks and mismatch-specific terminal
    terms, passed to both sides; includes entries that make some duplex
    entropies positive, which forces the enumeration path on the GPU."""
    rng = np.random.default_rng(12)
    t = oracle.default_table()
    ta = ah.NNTable()
    H = np.array(t.stack_dH)
    S = np.array(t.stack_dS)
    zero = (H == 0)
    H[zero] = np.round(rng.uniform(-3, 4, zero.sum()), 1)
    S[zero] = np.round(rng.uniform(-12, 12, zero.sum()), 1)
    TH = np.round(rng.uniform(-1, 3, 16), 1)
    TS = np.round(rng.uniform(-4, 6, 16), 1)
    for tt in (t, ta):
        tt.stack_dH[:] = list(H)
        tt.stack_dS[:] = list(S)
        tt.term_dH[:] = list(TH)
        tt.term_dS[:] = list(TS)
    w = synth.tiny(0)
    w.pairs = [dict(w.pairs[0], tm_min=30.0)]
    g = gpu_run(ctx, w, table=ta)
    o = oracle_run(w, table=t)
    assert_parity(g, o)


def test_threshold_decisions_at_the_boundary(ctx):
    """tm_min set at (and a hair either side of) oracle Tm values: the pass
    flags must still equal the fp64 decisions."""
    w = synth.tiny(0)
    o = oracle_run(w)
    vals = o["tm"][~np.isnan(o["tm"])]
    assert len(vals) > 3
    for v in (vals[0], vals[len(vals) // 2] + 1e-9, vals[-1] - 1e-9):
        w.pairs = [dict(w.pairs[0], tm_min=float(v))]
        assert_parity(gpu_run(ctx, w), oracle_run(w))


def test_threshold_band_decisions(ctx):
    """tm_min placed inside the 0.01 deg C band around site Tm values, at
    offsets from 1e-12 to 9e-3: the pass flags equal the fp64 decisions (the
    fp64 sign test decides most, exhaustive enumeration the closest), and the
    reported Tm stays within 0.01 of the oracle and on the side of its flag."""
    w = synth.tiny(0)
    o_sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, w.pairs)
    o_tm, _ = oracle.tm(w.seq, w.contig_off, o_sites, w.pairs)
    vals = np.unique(o_tm[~np.isnan(o_tm)])
    vals = vals[np.linspace(0, len(vals) - 1, min(5, len(vals))).astype(int)]
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        p0 = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])
        sites = ctx.scan(sid, [p0])
        assert sites.tobytes() == o_sites.tobytes()
        for v in vals:
            for d in (0.0, 1e-12, -1e-12, 1e-9, -1e-9, 1e-6, -1e-6, 1e-4, -1e-4, 3e-3, -3e-3, 9e-3, -9e-3):
                p = dict(w.pairs[0], tm_min=float(v) + d)
                pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
                tm, ps = ctx.tm(sid, [pid], sites)
                e_tm, e_ps = oracle.tm(w.seq, w.contig_off, o_sites, [p])
                assert np.array_equal(ps, e_ps), (v, d)
                ok = ~np.isnan(e_tm)
                assert np.abs(tm[ok].astype(np.float64) - e_tm[ok]).max() <= TM_TOL
                tmin = np.float32(p["tm_min"])
                assert np.all((tm[ok] >= tmin) == (ps[ok] == 1)), (v, d)
    finally:
        ctx.ah_unload_genomes(sid)


def test_device_resident_buffers(ctx):
    """Inputs and outputs in device memory (torch CUDA tensors) give the same
    records as host buffers."""
    import torch
    w = synth.tiny(0)
    o = oracle_run(w)
    seq_d = torch.from_numpy(w.seq).cuda()
    sid = ctx.ah_load_genomes(seq_d, len(w.seq), w.contig_off, w.contig_genome)
    pid = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])
    n = len(o["sites"])
    sites_d = torch.zeros(n * 16, dtype=torch.uint8, device="cuda")
    assert ctx.ah_scan(sid, [pid], sites_d, n) == n
    assert sites_d.cpu().numpy().tobytes() == o["sites"].tobytes()
    tm_d = torch.zeros(n, dtype=torch.float32, device="cuda")
    ps_d = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ctx.ah_tm(sid, [pid], sites_d, n, tm_d, ps_d)
    assert np.nanmax(np.abs(tm_d.cpu().numpy() - o["tm"])) <= TM_TOL
    m = len(o["amps"])
    amps_d = torch.zeros(m * 28, dtype=torch.uint8, device="cuda")
    assert ctx.ah_pair(sid, [pid], sites_d, None, n, amps_d, m) == m
    assert amps_d.cpu().numpy().tobytes() == o["amps"].tobytes()
    total = int(o["offs"][-1])
    seq_out = torch.zeros(total, dtype=torch.uint8, device="cuda")
    offs_d = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ctx.ah_fetch(sid, amps_d, m, seq_out, total, offs_d)
    assert seq_out.cpu().numpy().tobytes() == o["seqs"]
    assert np.array_equal(offs_d.cpu().numpy().astype(np.uint64), o["offs"])
    ctx.ah_unload_genomes(sid)


def test_errors_are_reported_not_raised_on_device(ctx):
    w = synth.tiny(0)
    p = dict(w.pairs[0])
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers("ACGX", p["rev"], p)
    assert e.value.status == ah.AH_ERR_PRIMER
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers("ACGT", p["rev"], p)  # shorter than 5
    assert e.value.status == ah.AH_ERR_PRIMER
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers("NNNNNNNNNNNN", p["rev"], p)  # degeneracy 4^12 > 10000
    assert e.value.status == ah.AH_ERR_PRIMER
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers(p["fwd"], p["rev"], dict(p, k=11))
    assert e.value.status == ah.AH_ERR_PRIMER
    with pytest.raises(ah.AHError) as e:
        ctx.ah_set_primers(p["fwd"], p["rev"], dict(p, min_len=10, max_len=5))
    assert e.value.status == ah.AH_ERR_ARG
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
    with pytest.raises(ah.AHError) as e:  # size query: cap = 0 reports the count with AH_ERR_OVERFLOW
        ctx.ah_scan(sid, [pid], None, 0)
    assert e.value.status == ah.AH_ERR_OVERFLOW
    n = e.value.needed
    assert n > 2
    small = np.zeros(n - 1, dtype=ah.SITE_DTYPE)
    with pytest.raises(ah.AHError) as e:
        ctx.ah_scan(sid, [pid], small, n - 1)
    assert e.value.status == ah.AH_ERR_OVERFLOW and e.value.needed == n
    assert not small.view(np.uint8).any()
    with pytest.raises(ah.AHError) as e:
        ctx.ah_scan(sid + 100, [pid], None, 0)
    assert e.value.status == ah.AH_ERR_ARG
    # a site record outside its contig is rejected before any kernel uses it
    bad = np.zeros(1, dtype=ah.SITE_DTYPE)
    bad["contig"] = 2
    bad["pos"] = 10 ** 9
    with pytest.raises(ah.AHError) as e:
        ctx.tm(sid, [pid], bad)
    assert e.value.status == ah.AH_ERR_ARG
    ctx.ah_unload_genomes(sid)
    # the context is still usable afterwards
    assert_parity(gpu_run(ctx, w), oracle_run(w))


def test_memory_budget_is_enforced():
    build.build()
    w = synth.tiny(0)
    with ah.Context(0, mem_budget_bytes=1 << 16) as c:
        with pytest.raises(ah.AHError) as e:
            c.load(w.seq, w.contig_off, w.contig_genome)
        assert e.value.status == ah.AH_ERR_BUDGET
        assert c.device_bytes() < (1 << 16)


def test_empty_and_degenerate_sets(ctx):
    p = synth.tiny(0).pairs[0]
    pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
    # no bases at all, one empty contig
    sid = ctx.ah_load_genomes(np.zeros(1, np.uint8), 0, np.array([0, 0], np.uint64), np.array([0], np.uint32))
    assert ctx.ah_scan(sid, [pid], None, 0) == 0  # zero sites fit in capacity 0
    ctx.ah_unload_genomes(sid)
    # contigs shorter than the primers, empty contigs in between, all-N contig
    seq = np.frombuffer(b"ACGTACG" + b"N" * 50 + b"ACGT", np.uint8).copy()
    off = np.array([0, 7, 7, 57, 61], np.uint64)
    sid = ctx.ah_load_genomes(seq, len(seq), off, np.array([0, 0, 1, 1], np.uint32))
    assert ctx.ah_scan(sid, [pid], None, 0) == 0
    ctx.ah_unload_genomes(sid)


def test_pack_classifies_every_byte_value(ctx):
    """All 256 byte values, at every offset within a 4-byte word and across
    tile boundaries: exactly A/C/G/T in either case are bases, all else N."""
    rng = np.random.default_rng(3)
    vals = np.tile(np.arange(256, dtype=np.uint8), 600)
    seq = np.concatenate([vals, rng.permutation(vals), np.frombuffer(b"ACGTacgtN" * 5000, np.uint8)])
    off = np.array([0, 70_001, len(seq)], np.uint64)  # a contig boundary inside a word
    sid = ctx.ah_load_genomes(seq, len(seq), off, np.array([0, 1], np.uint32))
    amps = np.zeros(2, dtype=ah.AMPLICON_DTYPE)
    amps["contig"] = [0, 1]
    amps["end"] = [70_001, len(seq) - 70_001]
    got, goff = ctx.fetch(sid, amps)
    want, woff = oracle.fetch(seq, off, amps)
    ctx.ah_unload_genomes(sid)
    assert np.array_equal(goff, woff) and got == want


def test_pack_single_non_bases_in_base_tiles(ctx):
    """Tiles of bases (either case) with single non-base bytes scattered through
    them, at word, row and tile edges: the packer's fast all-bases test must
    send every such column to the exact per-byte test."""
    rng = np.random.default_rng(11)
    n = 7 * 32768 + 1234
    seq = rng.choice(np.frombuffer(b"ACGTacgt", np.uint8), n)
    others = np.array([v for v in range(256) if v not in b"ACGTacgt"], np.uint8)
    edges = [0, 3, 4, 1023, 1024, 31 * 1024, 32767, 32768, 32768 + 31 * 1024 + 1023, 3 * 32768 + 5 * 1024 + 511]
    pos = np.unique(np.concatenate([edges, rng.integers(0, n, 60)]))
    seq[pos] = rng.choice(others, len(pos))
    off = np.array([0, n], np.uint64)
    sid = ctx.ah_load_genomes(seq, n, off, np.array([0], np.uint32))
    amps = np.zeros(1, dtype=ah.AMPLICON_DTYPE)
    amps["end"] = [n]
    got, goff = ctx.fetch(sid, amps)
    want, woff = oracle.fetch(seq, off, amps)
    ctx.ah_unload_genomes(sid)
    assert np.array_equal(goff, woff) and got == want


@pytest.mark.parametrize("tm_filter", [True, False])
def test_run_equals_separate_calls_and_oracle(ctx, tm_filter):
    """ah_run (the fused path) gives the records of ah_scan/ah_tm/ah_pair/ah_fetch
    and of the oracle; too-small outputs are reported, not written."""
    w = synth.collection(seed=2, n_genomes=4, len_lo=3e5, len_hi=9e5)
    w.pairs = [dict(w.pairs[0], tm_min=50.0)]
    o = oracle_run(w)
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    pid = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])
    r = ctx.run(sid, [pid], tm_filter=tm_filter)
    amps = o["amps_tm"] if tm_filter else o["amps"]
    seqs, offs = oracle.fetch(w.seq, w.contig_off, amps)
    assert r["sites"].tobytes() == o["sites"].tobytes()
    assert np.array_equal(r["pass_"], o["pass_"])
    ok = ~np.isnan(o["tm"])
    assert np.array_equal(np.isnan(r["tm"]), ~ok) and np.abs(r["tm"][ok] - o["tm"][ok]).max() <= TM_TOL
    assert r["amps"].tobytes() == amps.tobytes() and len(amps) > 0
    assert r["seqs"] == seqs and np.array_equal(r["offs"], offs)
    # capacity one short on the amplicons: counts reported, sites still written
    n, m = len(r["sites"]), len(r["amps"])
    sites = np.zeros(n, dtype=ah.SITE_DTYPE)
    small = np.zeros(m, dtype=ah.AMPLICON_DTYPE)
    out = ah.RunOut(sites.ctypes.data, n, 0, None, None, small.ctypes.data, m - 1, 0, None, 0, 0, None,
                    1 if tm_filter else 0, 0)
    with pytest.raises(ah.AHError) as e:
        ctx.ah_run(sid, [pid], out)
    assert e.value.status == ah.AH_ERR_OVERFLOW
    assert out.n_sites == n and out.n_amplicons == m and out.n_seq == len(seqs)
    assert sites.tobytes() == o["sites"].tobytes() and not small.view(np.uint8).any()
    ctx.ah_unload_genomes(sid)


def test_many_sites_take_the_device_wide_paths(ctx):
    """More than 16384 sites (device-wide sort instead of the one-block sort)
    and more than 65536 values in the pairing prefix sum (device-wide scan)."""
    w = synth.random_small(41, n_bases=20_000, n_contigs=8, L_f=6, L_r=5, k=6, min_len=12, max_len=12)
    o = oracle_run(w)
    assert len(o["sites"]) > 65536
    assert_parity(gpu_run(ctx, w), o)


def _run_into_device(ctx, sid, pid, caps, tm_filter=True):
    """ah_run into device buffers (torch) with the given capacities (sites,
    amplicons, sequence bytes); returns (status, out struct, host copies)."""
    import torch
    ns, na, nq = caps
    u8 = dict(dtype=torch.uint8, device="cuda")
    b = dict(sites=torch.zeros(max(ns, 1) * 16, **u8), tm=torch.zeros(max(ns, 1), dtype=torch.float32, device="cuda"),
             ps=torch.zeros(max(ns, 1), **u8), amps=torch.zeros(max(na, 1) * 28, **u8),
             seq=torch.zeros(max(nq, 1), **u8), offs=torch.zeros(max(na, 1) + 1, dtype=torch.int64, device="cuda"))
    out = ah.RunOut(b["sites"].data_ptr(), ns, 0, b["tm"].data_ptr(), b["ps"].data_ptr(), b["amps"].data_ptr(), na, 0,
                    b["seq"].data_ptr(), nq, 0, b["offs"].data_ptr(), 1 if tm_filter else 0, 0)
    status = ah.AH_OK
    try:
        ctx.ah_run(sid, [pid], out)
    except ah.AHError as e:
        status = e.status
    torch.cuda.synchronize()
    return status, out, {k: v.cpu().numpy() for k, v in b.items()}


def test_run_into_device_buffers_and_every_fallback(ctx):
    """ah_run with device outputs: generous and exact capacities take the
    one-synchronisation path; a capacity one short on any output is reported
    with the true counts (the step-by-step path), and the next call with room
    is exact again."""
    w = synth.collection(seed=3, n_genomes=3, len_lo=3e5, len_hi=9e5)
    w.pairs = [dict(w.pairs[0], tm_min=50.0)]
    o = oracle_run(w)
    n, m = len(o["sites"]), len(o["amps_tm"])
    seqs, offs = oracle.fetch(w.seq, w.contig_off, o["amps_tm"])
    q = len(seqs)
    assert n > 0 and m > 0
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    pid = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])

    def check_all(b):
        assert b["sites"][:16 * n].tobytes() == o["sites"].tobytes()
        assert np.array_equal(b["ps"][:n], o["pass_"])
        assert b["amps"][:28 * m].tobytes() == o["amps_tm"].tobytes()
        assert b["seq"][:q].tobytes() == seqs
        assert np.array_equal(b["offs"][:m + 1].astype(np.uint64), offs)

    for caps in [(n + 100, m + 100, q + 100), (n, m, q), (20000, 60000, 1 << 22)]:
        st, out, b = _run_into_device(ctx, sid, pid, caps)
        assert st == ah.AH_OK and (out.n_sites, out.n_amplicons, out.n_seq) == (n, m, q)
        check_all(b)
    for short in range(3):
        caps = [n, m, q]
        caps[short] -= 1
        st, out, b = _run_into_device(ctx, sid, pid, tuple(caps))
        assert st == ah.AH_ERR_OVERFLOW and (out.n_sites, out.n_amplicons, out.n_seq) == (n, m, q)
        if short != 0:
            assert b["sites"][:16 * n].tobytes() == o["sites"].tobytes()
    st, out, b = _run_into_device(ctx, sid, pid, (n, m, q))
    assert st == ah.AH_OK
    check_all(b)
    ctx.ah_unload_genomes(sid)


@pytest.mark.parametrize("case", ["sites_above_16384", "amplicons_above_16384", "amplicons_above_65535"])
def test_run_past_the_one_synchronisation_sizes(ctx, case):
    """Counts above what the one-synchronisation launches are sized for
    (sites, amplicons, sequence bytes) finish on the step-by-step path with
    the oracle's records, on the first call and on repeated calls; a small
    workload afterwards is exact again."""
    if case == "sites_above_16384":
        w = synth.random_small(41, n_bases=20_000, n_contigs=8, L_f=6, L_r=5, k=6, min_len=12, max_len=12)
    elif case == "amplicons_above_16384":
        w = synth.random_small(7, n_bases=120_000, n_contigs=1, L_f=5, L_r=5, k=1, codes_f="R", codes_r="Y",
                               min_len=12, max_len=100)
    else:
        w = synth.random_small(9, n_bases=100_000, n_contigs=1, L_f=5, L_r=5, k=1, codes_f="R", codes_r="Y",
                               min_len=10, max_len=250)
    o = oracle_run(w)
    seqs, offs = oracle.fetch(w.seq, w.contig_off, o["amps_tm"])
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    pid = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])
    for _ in range(2):
        r = ctx.run(sid, [pid], tm_filter=True)
        assert r["sites"].tobytes() == o["sites"].tobytes()
        assert np.array_equal(r["pass_"], o["pass_"])
        assert r["amps"].tobytes() == o["amps_tm"].tobytes()
        assert r["seqs"] == seqs and np.array_equal(r["offs"], offs)
    ctx.ah_unload_genomes(sid)
    t = synth.tiny(0)
    ot = oracle_run(t)
    sid = ctx.load(t.seq, t.contig_off, t.contig_genome)
    pid = ctx.ah_set_primers(t.pairs[0]["fwd"], t.pairs[0]["rev"], t.pairs[0])
    r = ctx.run(sid, [pid], tm_filter=False)
    assert r["sites"].tobytes() == ot["sites"].tobytes() and r["amps"].tobytes() == ot["amps"].tobytes()
    ctx.ah_unload_genomes(sid)


@pytest.mark.parametrize("source", ["device", "host"])
def test_run_begin_end_pipeline(ctx, source):
    """ah_run_begin / ah_run_end give ah_run's records; while a run is pending
    other calls are refused; three sets run as a pipeline (the next set packs on
    a second stream after the current scan, or, from host memory, is copied
    and packed while the run computes) each match the oracle."""
    import torch
    ws = [synth.collection(seed=s, n_genomes=2, len_lo=3e5, len_hi=6e5) for s in (4, 5, 6)]
    pair = dict(ws[0].pairs[0], tm_min=50.0)  # one pair for every set (the generator draws one per seed)
    for w in ws:
        w.pairs = [pair]
    p = ws[0].pairs[0]
    pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
    want = []
    for w in ws:
        o = oracle_run(w)
        seqs, offs = oracle.fetch(w.seq, w.contig_off, o["amps_tm"])
        want.append((o, seqs, offs))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    scan_done = torch.cuda.Event()
    dev = [torch.from_numpy(w.seq).cuda() for w in ws] if source == "device" else [w.seq for w in ws]
    torch.cuda.synchronize()
    cap = 20000
    u8 = dict(dtype=torch.uint8, device="cuda")
    b = dict(sites=torch.zeros(cap * 16, **u8), tm=torch.zeros(cap, dtype=torch.float32, device="cuda"),
             ps=torch.zeros(cap, **u8), amps=torch.zeros(cap * 28, **u8), seq=torch.zeros(1 << 22, **u8),
             offs=torch.zeros(cap + 1, dtype=torch.int64, device="cuda"))
    out = ah.RunOut(b["sites"].data_ptr(), cap, 0, b["tm"].data_ptr(), b["ps"].data_ptr(), b["amps"].data_ptr(), cap,
                    0, b["seq"].data_ptr(), 1 << 22, 0, b["offs"].data_ptr(), 1, 0)
    prev = ctx.ah_load_genomes(dev[0], len(ws[0].seq), ws[0].contig_off, ws[0].contig_genome, streams[0])
    total_amps = 0
    for i, w in enumerate(ws):
        ctx.ah_run_begin(prev, [pid], out, streams[i % 2], scan_done)
        with pytest.raises(ah.AHError) as e:  # refused while the run is pending
            ctx.ah_scan(prev, [pid], None, 0)
        assert e.value.status == ah.AH_ERR_ARG
        nxt = None
        if i + 1 < len(ws):
            if source == "device":
                streams[(i + 1) % 2].wait_event(scan_done)
            nxt = ctx.ah_load_genomes(dev[i + 1], len(ws[i + 1].seq), ws[i + 1].contig_off,
                                      ws[i + 1].contig_genome, streams[(i + 1) % 2])
        ctx.ah_run_end(out)
        torch.cuda.synchronize()
        o, seqs, offs = want[i]
        n, m, q = out.n_sites, out.n_amplicons, out.n_seq
        assert b["sites"][:16 * n].cpu().numpy().tobytes() == o["sites"].tobytes()
        assert np.array_equal(b["ps"][:n].cpu().numpy(), o["pass_"])
        assert b["amps"][:28 * m].cpu().numpy().tobytes() == o["amps_tm"].tobytes()
        total_amps += m
        assert b["seq"][:q].cpu().numpy().tobytes() == seqs
        assert np.array_equal(b["offs"][:m + 1].cpu().numpy().astype(np.uint64), offs)
        ctx.ah_unload_genomes(prev)
        prev = nxt
    assert total_amps > 0  # the first set carries planted amplicons of this pair
    with pytest.raises(ah.AHError):  # nothing pending
        ctx.ah_run_end(out)


@pytest.mark.parametrize("on_device", [False, True])
def test_decoy_sets_on_reversed_contigs(ctx, on_device):
    """A reversed (decoy) load gives, through every call and ah_run, the oracle's
    records on the contig-wise reversed collection; the off-target rate is the
    ratio of decoy to real amplicons."""
    import torch
    w = synth.collection(seed=2, n_genomes=4, len_lo=3e5, len_hi=9e5)
    w.pairs = [dict(w.pairs[0], tm_min=40.0)]
    rev = oracle.reverse_contigs(w.seq, w.contig_off)
    wr = synth.Workload(**{**w.__dict__, "seq": rev})
    o = oracle_run(wr)
    seq_in = torch.from_numpy(w.seq).cuda() if on_device else w.seq
    sid = ctx.ah_load_genomes(seq_in, len(w.seq), w.contig_off, w.contig_genome, reversed=True)
    try:
        pid = ctx.ah_set_primers(w.pairs[0]["fwd"], w.pairs[0]["rev"], w.pairs[0])
        sites = ctx.scan(sid, [pid])
        assert sites.tobytes() == o["sites"].tobytes() and len(sites) > 0
        tm, ps = ctx.tm(sid, [pid], sites)
        assert np.array_equal(ps, o["pass_"])
        ok = ~np.isnan(o["tm"])
        assert np.abs(tm[ok] - o["tm"][ok]).max() <= TM_TOL
        amps = ctx.pair(sid, [pid], sites)
        assert amps.tobytes() == o["amps"].tobytes()
        seqs, offs = ctx.fetch(sid, amps)
        assert seqs == o["seqs"] and np.array_equal(offs, o["offs"])
        r = ctx.run(sid, [pid], tm_filter=True)
        assert r["amps"].tobytes() == o["amps_tm"].tobytes()
    finally:
        ctx.ah_unload_genomes(sid)
    real = oracle.pair(oracle.scan(w.seq, w.contig_off, w.contig_genome, w.pairs), w.pairs)
    assert len(real) > 0
    rate = len(o["amps"]) / len(real)  # the off-target estimate this load supports
    assert 0.0 <= rate


def test_tm_threshold_sweep(ctx):
    """ah_tm_sweep: per threshold, the amplicons whose two sites pass, those that
    are FF/RR, and the genomes amplified, equal to the oracle's fp64 decisions --
    on a grid and at thresholds placed on (and within 1e-7 of) site Tm values."""
    w = synth.collection(seed=2, n_genomes=6, len_lo=3e5, len_hi=9e5)
    pair = w.pairs[0]
    sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, [pair])
    amps = oracle.pair(sites, [pair])
    tm64, _ = oracle.tm(w.seq, w.contig_off, sites, [pair])
    fin = np.unique(tm64[~np.isnan(tm64)])
    picks = fin[np.linspace(0, len(fin) - 1, 6).astype(int)]
    thr = list(np.arange(20.0, 72.0, 2.0)) + [float(v) for v in picks]
    thr += [float(picks[2]) + 1e-7, float(picks[3]) - 1e-7, float(picks[4]) + 1e-12]
    assert len(thr) <= 64
    want = []
    for T in thr:
        ok = tm64 >= T  # NaN compares false: fails every threshold
        live = ok[amps["left"]] & ok[amps["right"]]
        want.append((int(live.sum()), int((live & (amps["orient"] >= 2)).sum()),
                     len(set(amps["genome"][live].tolist()))))
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid = ctx.ah_set_primers(pair["fwd"], pair["rev"], pair)
        g_sites = ctx.scan(sid, [pid])
        assert g_sites.tobytes() == sites.tobytes()
        g_amps = ctx.pair(sid, [pid], g_sites)
        assert g_amps.tobytes() == amps.tobytes() and len(amps) > 0
        rows, n_genomes = ctx.ah_tm_sweep(sid, [pid], g_sites, g_amps, thr)
    finally:
        ctx.ah_unload_genomes(sid)
    assert n_genomes == len(set(w.contig_genome.tolist()))
    got = [tuple(int(x) for x in r) for r in rows]
    assert got == want
    assert want[0][0] > want[-10][0]  # the counts do move with the threshold


@pytest.mark.parametrize("case", ["collection", "repeats"])
def test_amplicon_variants_and_amplitypes(ctx, case):
    """ah_amplitypes: variant ids and per-genome amplitypes equal the plain
    definition on the fetched sequences (exact sequence identity)."""
    if case == "collection":
        w = synth.collection(seed=8, n_genomes=12, len_lo=2e5, len_hi=6e5)
    else:  # short primers on repeated genomes: many equal sequences and shared patterns
        base = synth.random_small(3, n_bases=30_000, n_contigs=2, L_f=6, L_r=6, k=1, min_len=20, max_len=300)
        reps = 5
        seq = np.concatenate([base.seq] * reps)
        n0 = len(base.seq)
        off = np.concatenate([base.contig_off[:-1] + r * n0 for r in range(reps)] + [[reps * n0]]).astype(np.uint64)
        gen = np.repeat(np.arange(reps, dtype=np.uint32), len(base.contig_off) - 1)
        seq[n0 + 100:n0 + 110] = ord("N")  # genome 1 differs a little
        w = synth.Workload(**{**base.__dict__, "seq": seq, "contig_off": off, "contig_genome": gen})
    pair = w.pairs[0]
    sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, [pair])
    amps = oracle.pair(sites, [pair])
    assert len(amps) > 3
    want_v, want_rows, want_nv, want_nt = oracle.amplitypes(w.seq, w.contig_off, amps)
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        variant, rows, nv, nt = ctx.amplitypes(sid, amps)
    finally:
        ctx.ah_unload_genomes(sid)
    assert np.array_equal(variant, want_v)
    assert [tuple(int(x) for x in r) for r in rows] == want_rows
    assert (nv, nt) == (want_nv, want_nt)
    if case == "repeats":
        assert nt < len(want_rows)  # some genomes share an amplitype


def test_device_generator_matches_cpu_twin(ctx):
    """ah_generate_bases writes, on the device, the same bytes as the CPU twin,
    for the whole collection and for ranges at other offsets."""
    import torch
    from paper_2509_13300_gb300 import countergen
    c = countergen.collection(seed=7, n_genomes=6, len_lo=2e5, len_hi=8e5)
    want = c.bases()
    out = torch.zeros(c.n_bases, dtype=torch.uint8, device="cuda")
    ctx.generate_bases(c, 0, c.n_bases, out)
    assert out.cpu().numpy().tobytes() == want.tobytes()
    for a, n in ((4, 1), (8, 4099), (40000, 123457), (c.n_bases - 1001 - (c.n_bases - 1001) % 4, 1001)):
        part = torch.zeros(n, dtype=torch.uint8, device="cuda")
        ctx.generate_bases(c, a, n, part)
        assert part.cpu().numpy().tobytes() == want[a:a + n].tobytes()
    with pytest.raises(ah.AHError):  # base0 not a multiple of 4
        ctx.generate_bases(c, 3, 10, out)
    # the same from the collection's tables on the device (stream-ordered calls)
    tables = ctx.device_tables(c)
    out.zero_()
    ctx.generate_bases(c, 0, c.n_bases, out, tables=tables)
    torch.cuda.synchronize()
    assert out.cpu().numpy().tobytes() == want.tobytes()
    for a, n in ((8, 4099), (40000, 123457)):
        part = torch.zeros(n, dtype=torch.uint8, device="cuda")
        ctx.generate_bases(c, a, n, part, tables=tables)
        torch.cuda.synchronize()
        assert part.cpu().numpy().tobytes() == want[a:a + n].tobytes()


def test_large_workload_shape_on_device_generated_genomes(ctx):
    """The large workload's shape (counter-generated genomes, k = 4, window
    100-3000, pairs of 960, 64 and 256 oligos scanned in one pass) on a small
    seed-7 collection generated on the device: sites, Tm and amplicons equal the
    oracle's on the CPU twin's bytes."""
    import torch
    from paper_2509_13300_gb300 import countergen
    rng = np.random.default_rng(7)
    p960 = synth.pcr_params("AGRRTTYGATYHTDGYTYAG", "YCNTTCCYTYDYRGTACT", k=4, min_len=100, max_len=3000,
                            tm_min=45.0)
    # oligo totals as the sum of the two primers' degeneracies: 32 + 32 and 128 + 128
    p64 = synth.pcr_params(synth.random_primer(rng, 19, "RYSWK"), synth.random_primer(rng, 21, "WKMRY"), k=4,
                           min_len=100, max_len=3000, tm_min=45.0)
    p256 = synth.pcr_params(synth.random_primer(rng, 22, "RYSWKMR"), synth.random_primer(rng, 24, "KMRYSWK"), k=4,
                            min_len=100, max_len=3000, tm_min=45.0)
    pairs = [p960, p64, p256]
    c = countergen.collection(seed=7, n_genomes=8, len_lo=2e5, len_hi=1e6, pairs=pairs)
    w = c.workload()
    o_sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, pairs)
    o_tm, o_ps = oracle.tm(w.seq, w.contig_off, o_sites, pairs)
    o_amps = oracle.pair(o_sites, pairs, o_ps)
    assert len(o_amps) > 0
    dev = torch.zeros(c.n_bases, dtype=torch.uint8, device="cuda")
    ctx.generate_bases(c, 0, c.n_bases, dev)
    sid = ctx.ah_load_genomes(dev, c.n_bases, c.contig_off, c.contig_genome)
    try:
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs]
        r = ctx.run(sid, pids, tm_filter=True)
    finally:
        ctx.ah_unload_genomes(sid)
    assert r["sites"].tobytes() == o_sites.tobytes()
    assert np.array_equal(r["pass_"], o_ps)
    ok = ~np.isnan(o_tm)
    assert np.abs(r["tm"][ok] - o_tm[ok]).max() <= TM_TOL
    assert r["amps"].tobytes() == o_amps.tobytes()


def _served_oracle(w, pair, genomes, k, tm_filter):
    """A request's result by the plain definition: the pair scanned at the
    request's k over the pool, sites of the named genomes kept, Tm and
    amplicon calling on those sites alone."""
    p = dict(pair, k=k)
    sites = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p])
    sites = sites[np.isin(sites["genome"], np.asarray(genomes, dtype=np.uint32))]
    passed = None
    if tm_filter and len(sites):
        _, passed = oracle.tm(w.seq, w.contig_off, sites, [p])
    amps = oracle.pair(sites, [p], passed)
    seqs, offs = oracle.fetch(w.seq, w.contig_off, amps)
    return sites, amps, seqs, offs


def test_served_requests_alone_and_in_the_mix(ctx):
    """ah_serve_*: every request's result is the same whether it runs alone
    (one request per batch), in large mixed batches, or in batches cut short
    by the memory budget, and equals the plain definition on the pool."""
    pairs = [synth.pcr_params(*synth.PAPER_PAIRS["Titan"], k=3, min_len=100, max_len=3000, tm_min=45.0),
             synth.pcr_params(*synth.PAPER_PAIRS["V3V4"], k=2, min_len=100, max_len=3000, tm_min=50.0)]
    w = synth.collection(seed=12, n_genomes=10, len_lo=1.5e5, len_hi=5e5, pairs=pairs, max_subs=3)
    n_g = int(w.contig_genome.max()) + 1
    rng = np.random.default_rng(5)
    reqs = []
    for i in range(24):
        g = rng.choice(n_g, size=int(rng.integers(1, n_g + 1)), replace=False)
        reqs.append((g.astype(np.uint32), int(rng.integers(len(pairs))), int(rng.integers(0, 4)),
                     bool(rng.integers(2))))
    reqs.append((np.zeros(0, np.uint32), 0, 2, True))                      # no genomes
    reqs.append((np.array([n_g + 5, 1, 1], np.uint32), 1, 1, False))       # unknown id and a duplicate
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs]
    try:
        def serve(max_batch, mem_budget, one_at_a_time):
            out = []
            with ah.Server(ctx, sid, mem_budget=mem_budget, max_batch=max_batch) as srv:
                if one_at_a_time:
                    for g, j, k, f in reqs:
                        out.append(srv.wait(srv.submit(g, pids[j], k, f)))
                else:
                    tickets = [srv.submit(g, pids[j], k, f) for g, j, k, f in reqs]
                    out = [srv.wait(t) for t in tickets]
            return out

        alone = serve(1, 1 << 30, True)
        mixed = serve(64, 1 << 30, False)
        budget = serve(64, 200_000, False)
        # the context is usable again after the servers stopped
        assert len(ctx.scan(sid, [pids[0]])) > 0
    finally:
        ctx.ah_unload_genomes(sid)
    assert max(x[4]["batch_size"] for x in mixed) > 8
    assert max(x[4]["batch_size"] for x in budget) < max(x[4]["batch_size"] for x in mixed)
    assert all(x[4]["batch_size"] == 1 for x in alone)
    total_amps = 0
    for n, ((g, j, k, f), a, m, b) in enumerate(zip(reqs, alone, mixed, budget)):
        for x in (m, b):
            assert x[0].tobytes() == a[0].tobytes(), n
            assert x[1].tobytes() == a[1].tobytes(), n
            assert x[2] == a[2] and np.array_equal(x[3], a[3]), n
        info = a[4]
        assert info["status"] == 0 and info["submit_ms"] <= info["start_ms"] <= info["done_ms"]
        want_s, want_a, want_q, want_o = _served_oracle(w, pairs[j], [x for x in g if x < n_g], k, f)
        assert a[0].tobytes() == want_s.tobytes(), n
        assert a[1].tobytes() == want_a.tobytes(), n
        assert a[2] == want_q and np.array_equal(a[3], want_o), n
        total_amps += len(want_a)
    assert total_amps > 10


def test_profile_hmm_build_and_scores(ctx):
    """ah_hmm_build / ah_hmm_score / ah_hmm_forward: the profile trained on the
    exact-match amplicons of an operon family (training set taken end to end: a
    k = 0 run and its fetched sequences) equals the oracle's (fp32 of its fp64
    scores), and the fp32 Viterbi and Forward scores of every k = 2 amplicon and
    of random regions are within the fp32 accumulation bound of the oracle's
    fp64 scores."""
    import torch
    w = synth.operon_family(seed=21, n_genomes=16)
    p = w.pairs[0]
    p0 = dict(p, k=0)
    s0 = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p0])
    a0 = oracle.pair(s0, [p0])
    q0, o0 = oracle.fetch(w.seq, w.contig_off, a0)
    train = [q0[int(o0[i]):int(o0[i + 1])].decode() for i in range(len(a0))]
    assert len(train) >= 8
    ref, T, E = oracle.hmm_build(train)
    s2 = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p])
    a2 = oracle.pair(s2, [p])
    rng = np.random.default_rng(3)  # unrelated regions in either orientation
    extra = np.zeros(40, dtype=oracle.AMPLICON_DTYPE)
    lens = np.diff(w.contig_off.astype(np.int64))
    for r in extra:
        c = int(rng.integers(len(lens)))
        L = int(rng.integers(200, 900))
        s = int(rng.integers(0, lens[c] - L))
        r["genome"], r["contig"], r["start"], r["end"], r["orient"] = w.contig_genome[c], c, s, s + L, rng.integers(2)
    amps = np.concatenate([a2, extra])
    q2, o2 = oracle.fetch(w.seq, w.contig_off, amps)
    seqs = [q2[int(o2[i]):int(o2[i + 1])].decode() for i in range(len(amps))]
    want = np.array([oracle.hmm_viterbi(T, E, x) for x in seqs])
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid0 = ctx.ah_set_primers(p0["fwd"], p0["rev"], p0)
        r0 = ctx.run(sid, [pid0], tm_filter=False)
        gtrain = [r0["seqs"][int(r0["offs"][i]):int(r0["offs"][i + 1])].decode() for i in range(len(r0["amps"]))]
        assert gtrain == train
        hid = ctx.hmm_build(gtrain)
        m, gref, gt, ge = ctx.hmm_tables(hid)
        assert (m, gref) == (T.shape[0] - 1, ref)
        assert np.array_equal(np.isinf(gt), np.isinf(T))
        fin = ~np.isinf(T)
        assert np.abs(gt[fin] - T[fin]).max() <= 1e-5
        assert np.abs(ge - E).max() <= 1e-5
        got = ctx.hmm_score(sid, hid, amps)
        got_f = ctx.hmm_forward(sid, hid, amps)
        # device records and scores give the same
        dev_amps = torch.from_numpy(amps.view(np.uint8).copy()).cuda()
        dev_out = torch.zeros(len(amps), dtype=torch.float32, device="cuda")
        ctx.hmm_score(sid, hid, dev_amps, n=len(amps), out=dev_out)
        assert np.array_equal(dev_out.cpu().numpy(), got)
        with pytest.raises(ah.AHError):
            ctx.hmm_score(sid, hid + 99, amps)
        bad = amps[:1].copy()
        bad["end"] = lens[bad["contig"][0]] + 5
        with pytest.raises(ah.AHError):
            ctx.hmm_score(sid, hid, bad)
        ctx.hmm_free(hid)
    finally:
        ctx.ah_unload_genomes(sid)
    # fp32 accumulation along one path of N = n + m moves: the rounding of each
    # addition is at most 2^-24 of the partial sum, and N roundings of either
    # sign add up like a random walk (sqrt(N)); a partial sum is at most the
    # final score plus the remaining terms, about N times the mean table entry.
    # Ten standard deviations of that walk (observed errors are ~1/30 of it).
    pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
    N = np.array([len(x) for x in seqs]) + m
    tol = 10.0 * np.sqrt(N) * 2.0 ** -24 * (np.abs(want) + N * pmean) + 1e-4
    err = np.abs(got.astype(np.float64) - want)
    assert (err <= tol).all(), (err.max(), tol.min())
    assert want[:len(a2)].min() > want[len(a2):].max()  # family members above unrelated regions
    # Forward: the same walk, plus per log-sum step an absolute error of a few
    # 2^-23 from log2(1 + 2^d) (exp2f / log2f within 2 ulp)
    want_f = np.array([oracle.hmm_forward(T, E, x) for x in seqs])
    tol_f = 10.0 * np.sqrt(N) * (2.0 ** -24 * (np.abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4
    err_f = np.abs(got_f.astype(np.float64) - want_f)
    assert (err_f <= tol_f).all(), (err_f.max(), tol_f.min())
    assert (want_f >= want - 1e-9).all() and (got_f >= got - 1e-3).all()  # the sum is at least the best path


@pytest.mark.parametrize("kernel", ["wave", "rows"])
def test_profile_hmm_kernels_on_profiles_of_several_lengths(ctx, kernel, monkeypatch):
    """Both scoring kernels (the warp wavefront and the block-per-group kernel,
    forced by AH_HMM_KERNEL for both scores) against the oracle's fp64 Viterbi
    and Forward scores, on profiles of m + 1 = 40, 129, 255 and 640 columns
    (the wavefront's stripes hold 128: a lone partial stripe, a last stripe of
    one column, a nearly full one, five full ones) and on amplicons of 0, 1 and
    2 letters up to 1,700."""
    monkeypatch.setenv("AH_HMM_KERNEL", kernel)
    w = synth.operon_family(seed=21, n_genomes=16)
    p = w.pairs[0]
    p0 = dict(p, k=0)
    s0 = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p0])
    a0 = oracle.pair(s0, [p0])
    q0, o0 = oracle.fetch(w.seq, w.contig_off, a0)
    train = [q0[int(o0[i]):int(o0[i + 1])].decode() for i in range(len(a0))]
    assert min(len(x) for x in train) >= 254
    s2 = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p])
    amps = oracle.pair(s2, [p])[:24]
    rng = np.random.default_rng(8)
    lens = np.diff(w.contig_off.astype(np.int64))
    extra = np.zeros(24, dtype=oracle.AMPLICON_DTYPE)
    for q, r in enumerate(extra):
        c = int(rng.integers(len(lens)))
        L = [0, 1, 2][q] if q < 3 else int(rng.integers(3, 1700))
        s = int(rng.integers(0, lens[c] - L))
        r["genome"], r["contig"], r["start"], r["end"], r["orient"] = w.contig_genome[c], c, s, s + L, q % 2
    amps = np.concatenate([amps, extra])
    qa, oa = oracle.fetch(w.seq, w.contig_off, amps)
    seqs = [qa[int(oa[i]):int(oa[i + 1])].decode() for i in range(len(amps))]
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        for cut in (39, 128, 254, None):
            tr = [x[:cut] for x in train] if cut else train
            _, T, E = oracle.hmm_build(tr)
            m = T.shape[0] - 1
            assert m == (cut or m)
            hid = ctx.hmm_build(tr)
            got = ctx.hmm_score(sid, hid, amps).astype(np.float64)
            got_f = ctx.hmm_forward(sid, hid, amps).astype(np.float64)
            ctx.hmm_free(hid)
            want = np.array([oracle.hmm_viterbi(T, E, x) for x in seqs])
            want_f = np.array([oracle.hmm_forward(T, E, x) for x in seqs])
            fin = ~np.isinf(T)
            # the fp32 accumulation bound of the test above (a random walk of
            # roundings along one path of N = n + m moves, ten standard deviations)
            pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
            N = np.array([len(x) for x in seqs]) + m
            tol = 10.0 * np.sqrt(N) * 2.0 ** -24 * (np.abs(want) + N * pmean) + 1e-4
            tol_f = 10.0 * np.sqrt(N) * (2.0 ** -24 * (np.abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4
            assert np.isfinite(got).all() and np.isfinite(got_f).all(), (cut, kernel)
            err, err_f = np.abs(got - want), np.abs(got_f - want_f)
            assert (err <= tol).all(), (cut, kernel, err.max(), int(err.argmax()))
            assert (err_f <= tol_f).all(), (cut, kernel, err_f.max(), int(err_f.argmax()))
    finally:
        ctx.ah_unload_genomes(sid)


@pytest.mark.parametrize("m,n", [(1, 3), (127, 9), (128, 1), (255, 700), (256, 5), (257, 13), (511, 40), (1100, 3)])
def test_profile_hmm_wavefront_stripes_and_tasks(ctx, m, n):
    """The wavefront at its stripes' edges (a narrow profile of at most 128 columns, stripes of
    256: full, one column over), with fewer and more amplicons than blocks, from empty to longer
    than the profile, and under a memory budget that leaves it few blocks' buffers: Viterbi and
    Forward against the oracle in fp64."""
    rng = np.random.default_rng(m * 1000 + n)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    ref = acgt[rng.integers(0, 4, m)].tobytes().decode()
    train = [ref, ref] + [synth._mutate(rng, ref, 0.03, 0.02) or "A" for _ in range(6)]
    seqs = [synth._mutate(rng, ref, 0.05, 0.03) for _ in range(n)]
    seqs[0] = ""
    if n > 2:
        seqs[1] = acgt[rng.integers(0, 4, 2 * m + 70)].tobytes().decode()  # unrelated and longer
        seqs[2] = ref[m // 2:] + "N" + ref[:m // 3]
    body = "".join(seqs) + "A"
    seq = np.frombuffer(body.encode(), np.uint8).copy()
    off = np.array([0, len(seq)], np.uint64)
    amps = np.zeros(n, dtype=ah.AMPLICON_DTYPE)
    ends = np.cumsum([len(x) for x in seqs])
    amps["end"], amps["start"] = ends, ends - [len(x) for x in seqs]
    ref_i, T, E = oracle.hmm_build(train)
    some = np.unique(np.concatenate([np.arange(min(n, 6)), rng.integers(0, n, 6)]))
    want = np.array([oracle.hmm_viterbi(T, E, seqs[i]) for i in some])
    want_f = np.array([oracle.hmm_forward(T, E, seqs[i]) for i in some])
    got = {}
    with ah.Context(0, 12 << 20) as small:  # boundary buffers get at most 1/16 of it
        for name, c in (("full", ctx), ("budget", small)):
            sid = c.load(seq, off, np.zeros(1, np.uint32))
            hid = c.hmm_build(train)
            got[name] = c.hmm_score(sid, hid, amps), c.hmm_forward(sid, hid, amps)
            c.hmm_free(hid)
            c.ah_unload_genomes(sid)
    # the bound of the parity test above: ten standard deviations of a walk of fp32 roundings
    fin = ~np.isinf(T)
    pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
    N = np.array([len(seqs[i]) for i in some]) + len(T) - 1
    for v, f in got.values():
        tol = 10.0 * np.sqrt(N) * 2.0 ** -24 * (np.abs(want) + N * pmean) + 1e-4
        assert (np.abs(v[some].astype(np.float64) - want) <= tol).all()
        tol_f = 10.0 * np.sqrt(N) * (2.0 ** -24 * (np.abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4
        assert (np.abs(f[some].astype(np.float64) - want_f) <= tol_f).all()
    every = 1e-4 + 1e-5 * np.abs(got["full"][0])
    assert (np.abs(got["full"][0] - got["budget"][0]) <= every).all()  # also the amplicons the oracle did not score


@pytest.mark.parametrize("lens", [[1, 1, 31, 32, 33], [639, 640, 641, 640, 639], [1279, 1281, 1920, 1280, 5]])
def test_amplitype_hash_groups_and_tables(ctx, lens):
    """Variants and amplitypes of records of the hash's group sizes (32 letters a row, 640 a group),
    in both orientations, across tile ends, with N, with copies in several genomes and with
    sequences that differ in one letter or only in length, against the plain definition; a bad
    record is refused."""
    rng = np.random.default_rng(sum(lens))
    base = synth.random_bases(rng, max(lens), 0.5).copy()
    genomes, recs, pos = [], [], 0
    for g in range(7):
        parts, at = [], 0
        for c in range(60):
            body = base[:lens[int(rng.integers(len(lens)))]].copy()
            if rng.random() < 0.3:
                body[int(rng.integers(len(body)))] = rng.choice(list(b"ACGTN"))
            rc = bool(rng.integers(2))
            stored = np.frombuffer(synth._revcomp(body.tobytes().decode().replace("N", "A")).encode(), np.uint8) if rc else body
            gap = synth.random_bases(rng, int(rng.integers(0, 40)), 0.5)
            parts += [gap, stored]
            recs.append((g, g, at + len(gap), at + len(gap) + len(body), 0, 0, 1 if rc else int(rng.choice([0, 2, 3])), 0, 0, 0))
            at += len(gap) + len(body)
        genomes.append(np.concatenate(parts))
    seq = np.concatenate(genomes)
    off = np.concatenate([[0], np.cumsum([len(x) for x in genomes])]).astype(np.uint64)
    amps = np.array(recs, dtype=ah.AMPLICON_DTYPE)
    want_v, want_rows, want_nv, want_nt = oracle.amplitypes(seq, off, amps)
    sid = ctx.load(seq, off, np.arange(len(genomes), dtype=np.uint32))
    try:
        variant, rows, nv, nt = ctx.amplitypes(sid, amps)
        assert np.array_equal(variant, want_v) and (nv, nt) == (want_nv, want_nt)
        assert np.array_equal(np.asarray(rows), np.asarray(want_rows))
        for f, v in (("genome", 6), ("orient", 4), ("contig", 99)):
            bad = amps.copy()
            bad[f][3] = v
            with pytest.raises(ah.AHError):
                ctx.amplitypes(sid, bad)
        again = ctx.amplitypes(sid, amps)
        assert np.array_equal(again[0], want_v)
    finally:
        ctx.ah_unload_genomes(sid)


@pytest.mark.parametrize("offset", [0, 1, 3, 4, 7, 8, 13, 15])
@pytest.mark.parametrize("reversed_", [False, True])
def test_packing_at_any_address_and_mirrored(ctx, offset, reversed_):
    """Device input at every kind of misalignment, forward and with its contigs reversed: the
    letters of every contig (sets ending inside, at and just past a tile; contigs from one letter
    to several tiles; letters of either case, N and other bytes) come back as the oracle gives them."""
    import torch
    rng = np.random.default_rng(offset)
    T = 32 * 1024
    for n in (5, T - 1, T, T + 33, 4 * T + 17):
        seq = synth.random_bases(rng, n, 0.5).copy()
        at = rng.integers(0, n, 1 + n // 500)
        seq[at] = rng.integers(0, 256, len(at), dtype=np.uint8)
        low = rng.random(n) < 0.2
        seq[low & (seq >= 65) & (seq <= 90)] += 32
        cuts = np.unique(rng.integers(1, n, 6)) if n > 10 else np.array([2])
        off = np.concatenate([[0], cuts, cuts[-1:], [n]]).astype(np.uint64)  # one empty contig
        gen = np.zeros(len(off) - 1, np.uint32)
        buf = torch.zeros(n + 64, dtype=torch.uint8, device="cuda")
        buf[:] = ord("C")  # neighbours of the input are bases
        buf[offset:offset + n] = torch.from_numpy(seq).cuda()
        torch.cuda.synchronize()
        amps = np.zeros(len(off) - 1, dtype=ah.AMPLICON_DTYPE)
        amps["contig"] = np.arange(len(amps))
        amps["end"] = np.diff(off.astype(np.int64))
        want, _ = oracle.fetch(oracle.reverse_contigs(seq, off) if reversed_ else seq, off, amps)
        sid = ctx.ah_load_genomes(buf[offset:], n, off, gen, reversed=reversed_)
        try:
            got, _ = ctx.fetch(sid, amps)
        finally:
            ctx.ah_unload_genomes(sid)
        assert got == want, n


@pytest.mark.parametrize("per_tile", [0, 1, 15, 16, 17, 900])
def test_2bit_packing_with_few_and_many_no_base_runs(ctx, per_tile):
    """2-bit loads whose tiles meet few no-base runs (masks per column) and many (marked position by
    position), runs across tile ends, over whole tiles and at the set's end: the letters come back."""
    import torch
    rng = np.random.default_rng(per_tile)
    T = 32 * 1024
    for n in (70, T - 3, 4 * T + 40):
        seq = synth.random_bases(rng, n, 0.5).copy()
        for t in range(0, n, T):
            for s0 in rng.integers(t, min(n, t + T), per_tile):
                seq[s0:s0 + int(rng.integers(1, 12))] = ord("N")
        if n > 2 * T:
            seq[T - 5:T + 40] = ord("N")      # across a tile end and its extension row
            seq[2 * T - 1:3 * T + 1] = ord("N")  # a whole tile
            seq[n - 9:] = ord("N")
        codes, gaps = ah.encode_2bit(seq)
        off = np.array([0, n], np.uint64)
        amps = np.zeros(1, dtype=ah.AMPLICON_DTYPE)
        amps["end"] = n
        for c in (codes, torch.from_numpy(codes).cuda()):
            torch.cuda.synchronize()
            sid = ctx.ah_load_genomes_2bit(c, n, gaps, off, np.zeros(1, np.uint32))
            try:
                got, _ = ctx.fetch(sid, amps)
            finally:
                ctx.ah_unload_genomes(sid)
            assert got == seq.tobytes(), n


@pytest.mark.parametrize("lengths,codes,n_sites", [([(32, 29)], ("RN", "BDHV"), 32768), ([(30, 31)], ("", "NNY"), 33001),
                                                   ([(12 + j, 27 - j) for j in range(16)], ("YW", "VK"), 60001)])
def test_thread_per_site_tm_over_window_offsets_and_primer_mixes(ctx, lengths, codes, n_sites):
    """Caller's sites at every offset of a window in its 16-byte groups and rows, across tile ends, on windows with
    other letters, for primers up to 32 long and sets of one to four bases, up to 16 pairs mixed at random: the
    maxima within 0.01 C of the oracle's (the bound of the entry point), NaN and pass flags the same."""
    rng = np.random.default_rng(n_sites)
    n = 5 * 32768 + 77
    seq = synth.random_bases(rng, n, 0.5).copy()
    seq[rng.integers(0, n, 60)] = ord("N")
    off = np.array([0, 40_001, 40_100, n], np.uint64)
    pairs = [synth.pcr_params(synth.random_primer(rng, lf, codes[0]), synth.random_primer(rng, lr, codes[1]), k=3,
                              min_len=30, max_len=900, tm_min=20.0) for lf, lr in lengths]
    sites = np.zeros(n_sites, dtype=ah.SITE_DTYPE)
    sites["contig"] = rng.choice(3, n_sites, p=[0.3, 0.1, 0.6])
    sites["pair"] = rng.integers(0, len(pairs), n_sites)
    sites["primer"] = rng.integers(0, 2, n_sites)
    sites["strand"] = rng.integers(0, 2, n_sites)
    size = np.diff(off.astype(np.int64))[sites["contig"]]
    sites["pos"] = rng.random(n_sites) * (size - 32 + 1)
    sid = ctx.load(seq, off, np.zeros(3, np.uint32))
    try:
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs]
        want, _ = oracle.tm(seq, off, sites, pairs)
        med = float(np.nanmedian(want))
        pairs = [dict(p, tm_min=med) for p in pairs]
        want, passed = oracle.tm(seq, off, sites, pairs)
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs]
        tm, ps = ctx.tm(sid, pids, sites)
    finally:
        ctx.ah_unload_genomes(sid)
    nan = np.isnan(want)
    assert 0 < nan.sum() < n_sites // 4 and 0.2 < passed.mean() < 0.8
    assert np.array_equal(np.isnan(tm), nan)
    assert np.abs(tm[~nan].astype(np.float64) - want[~nan]).max() <= TM_TOL
    assert np.array_equal(ps, passed)


@pytest.mark.parametrize("n_sites", [1, 31, 513, 8192, 8193, 16384])
@pytest.mark.parametrize("spread", [False, True])
def test_rank_sort_ranges(ctx, n_sites, spread):
    """Small runs sort their sites in 1,024 ranges of the key space: counts at the edges of what a thread holds in
    registers and of the path, hits spread over the set or in a few adjacent ranges, in canonical order."""
    rng = np.random.default_rng(n_sites)
    fwd, rev = "ACGTTGCAAGCT", "GGATCCATTCAG"
    n = 30_000_000 if spread else 16384 * 24 + 4096
    seq = np.full(n, ord("T"), np.uint8)
    at = np.sort(rng.choice(n // 24 - 2, n_sites, replace=False)) * 24 + 3
    words = [np.frombuffer(w.encode(), np.uint8) for w in (fwd, oracle_reverse_complement(fwd), rev,
                                                           oracle_reverse_complement(rev))]
    for p, w in zip(at, rng.integers(0, 4, n_sites)):
        seq[p:p + 12] = words[w]
    off = np.unique(np.r_[0, rng.integers(1, n, 5) // 24 * 24, n]).astype(np.uint64)
    gen = np.arange(len(off) - 1, dtype=np.uint32)
    pair = synth.pcr_params(fwd, rev, k=0, min_len=30, max_len=200)
    want = oracle.scan(seq, off, gen, [pair])
    sid = ctx.load(seq, off, gen)
    try:
        pid = ctx.ah_set_primers(fwd, rev, pair)
        got = ctx.scan(sid, [pid])
        run = ctx.run(sid, [pid])
    finally:
        ctx.ah_unload_genomes(sid)
    assert len(want) == n_sites
    assert got.tobytes() == want.tobytes() and run["sites"].tobytes() == want.tobytes()


def oracle_reverse_complement(s):
    return s[::-1].translate(str.maketrans("ACGT", "TGCA"))


@pytest.mark.parametrize("n_contigs,contig", [(1, 900), (40, 3000), (3, 1_200_000)])
@pytest.mark.parametrize("tm_filter", [False, True])
def test_run_pairs_in_one_launch_at_block_edges(ctx, n_contigs, contig, tm_filter):
    """A run's amplicons and sequence offsets come from one launch that scans counts over its blocks: no site, sites
    in one block and over many, with and without the Tm filter, first with outputs that are too small."""
    w = synth.random_small(contig, n_bases=n_contigs * contig, n_contigs=n_contigs, L_f=9, L_r=8, k=1, min_len=20,
                           max_len=400)
    p = dict(w.pairs[0], tm_min=-10.0)
    want = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p])
    _, passed = oracle.tm(w.seq, w.contig_off, want, [p])
    amps = oracle.pair(want, [p], passed if tm_filter else None)
    seqs, offs = oracle.fetch(w.seq, w.contig_off, amps)
    sid = ctx.load(w.seq, w.contig_off, w.contig_genome)
    try:
        pid = ctx.ah_set_primers(p["fwd"], p["rev"], p)
        for _ in range(2):
            r = ctx.run(sid, [pid], tm_filter=tm_filter)
            assert r["sites"].tobytes() == want.tobytes() and r["amps"].tobytes() == amps.tobytes()
            assert r["seqs"] == seqs and np.array_equal(r["offs"], offs)
    finally:
        ctx.ah_unload_genomes(sid)
    assert len(want) <= 16384 and (contig != 1_200_000 or len(want) > 4096)


@pytest.mark.parametrize("parts", [1, 2, 15, 16, 17, 40])
def test_mirrored_tiles_of_few_and_many_contigs(ctx, parts):
    """Contig ends at every place in a word and next to tile ends, about `parts` per tile (tiles of few parts are
    gathered part by part, others word by word), with runs of contigs of one to seven bases: the letters come back."""
    import torch
    rng = np.random.default_rng(parts)
    T = 32 * 1024
    for n in (37, T - 2, 3 * T + 33):
        cuts = [rng.integers(t, min(n, t + T), parts) for t in range(0, n, T)]
        near = [t + d for t in range(T, n, T) for d in (-1, 0, 1, 31, 32, 33)] if parts > 1 else []
        tiny = np.cumsum(rng.integers(1, 8, 9)) + int(rng.integers(0, max(1, n - 80)))
        off = np.unique(np.concatenate([[0, n], *cuts, near, tiny if parts in (2, 40) else []]))
        off = off[(off >= 0) & (off <= n)].astype(np.uint64)
        gen = np.arange(len(off) - 1, dtype=np.uint32)
        seq = synth.random_bases(rng, n, 0.5).copy()
        seq[rng.integers(0, n, 3)] = ord("N")
        amps = np.zeros(len(off) - 1, dtype=ah.AMPLICON_DTYPE)
        amps["contig"] = np.arange(len(amps))
        amps["end"] = np.diff(off.astype(np.int64))
        want, _ = oracle.fetch(oracle.reverse_contigs(seq, off), off, amps)
        buf = torch.from_numpy(np.concatenate([np.zeros(5, np.uint8), seq])).cuda()
        torch.cuda.synchronize()
        sid = ctx.ah_load_genomes(buf[5:], n, off, gen, reversed=True)
        try:
            got, _ = ctx.fetch(sid, amps)
        finally:
            ctx.ah_unload_genomes(sid)
        assert got == want, n


@pytest.mark.parametrize("pipelined", [False, True])
def test_run_on_a_device_without_room_for_the_pairing_cluster(pipelined):
    """A device slice without room for a cluster of 16 CTAs takes the step-by-step form: every output of a run, and
    of queued ones with the next load beside them, as where the cluster fits; the whole GPU has room for it."""
    w = synth.tiny(3)
    p = dict(w.pairs[0], tm_min=45.0)
    want = oracle.scan(w.seq, w.contig_off, w.contig_genome, [p])
    tm, passed = oracle.tm(w.seq, w.contig_off, want, [p])
    amps = oracle.pair(want, [p], passed)
    seqs, offs = oracle.fetch(w.seq, w.contig_off, amps)
    assert len(amps)
    with ah.Context(0) as c:
        pid = c.ah_set_primers(p["fwd"], p["rev"], p)
        sid = c.load(w.seq, w.contig_off, w.contig_genome)
        for on, launches in ((True, 1), (False, 4), (True, 1)):  # cluster; count, scan, total, write
            c.debug_pair_cluster(on)
            if pipelined:
                buf = dict(sites=np.zeros(len(want), ah.SITE_DTYPE), tm=np.zeros(len(want), np.float32),
                           pass_=np.zeros(len(want), np.uint8), amps=np.zeros(len(amps), ah.AMPLICON_DTYPE),
                           seq=np.zeros(len(seqs), np.uint8), offs=np.zeros(len(amps) + 1, np.uint64))
                o = ah.RunOut(buf["sites"].ctypes.data, len(want), 0, buf["tm"].ctypes.data, buf["pass_"].ctypes.data,
                              buf["amps"].ctypes.data, len(amps), 0, buf["seq"].ctypes.data, len(seqs), 0,
                              buf["offs"].ctypes.data, 1, 0)
                c.ah_run_begin(sid, [pid], o)
                other = c.load(w.seq, w.contig_off, w.contig_genome)
                c.ah_run_end(o)
                c.ah_unload_genomes(other)
                assert (o.n_sites, o.n_amplicons, o.n_seq) == (len(want), len(amps), len(seqs))
                r = dict(buf, seqs=buf["seq"].tobytes())
            else:
                caps = (len(want), len(amps), len(seqs))
                c.ah_set_profiling(1)
                r = c.run(sid, [pid], caps=caps)
                assert c.ah_get_profile("pair")[1] == launches
                c.ah_set_profiling(0)
            assert r["sites"].tobytes() == want.tobytes() and np.array_equal(r["pass_"], passed)
            assert r["amps"].tobytes() == amps.tobytes() and r["seqs"] == seqs and np.array_equal(r["offs"], offs)


def test_hmm_scores_leave_a_memory_budget_as_it_was():
    """The wavefront's buffers are the call's own: after it, a set loads that fills what the budget leaves beside
    everything the other kernel's call keeps."""
    import torch
    budget, m, n = 48 << 20, 300, 200
    rng = np.random.default_rng(12)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    ref = acgt[rng.integers(0, 4, m)].tobytes().decode()
    seq = acgt[rng.integers(0, 4, n * m)]
    amps = np.zeros(n, dtype=ah.AMPLICON_DTYPE)
    amps["start"] = np.arange(n) * m
    amps["end"] = amps["start"] + m
    device = torch.from_numpy(seq).cuda()
    torch.cuda.synchronize()
    off, gen = np.array([0, len(seq)], np.uint64), np.zeros(1, np.uint32)
    used = {}
    for kernel in ("rows", "wave"):
        with pytest.MonkeyPatch.context() as mp, ah.Context(0, budget) as c:
            mp.setenv("AH_HMM_KERNEL", kernel)
            sid = c.ah_load_genomes(device, len(seq), off, gen)
            hid = c.hmm_build([ref, ref, ref[:-1]])
            scores = c.hmm_score(sid, hid, amps)
            assert np.isfinite(scores).all()
            used[kernel] = c.device_bytes()
            if kernel == "rows":
                continue
            tile = 4 * (1024 + 32) * 4
            tiles = (budget - used["rows"] - 4096) // (tile + 8)
            big = torch.full((tiles * 32768,), ord("A"), dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            sid2 = c.ah_load_genomes(big, len(big), np.array([0, len(big)], np.uint64), gen)
            c.ah_unload_genomes(sid2)
            assert c.hmm_score(sid, hid, amps).tobytes() == scores.tobytes()
    assert used["wave"] > used["rows"] + (1 << 20)  # it did have buffers


@pytest.mark.parametrize("m,n,line", [(300, 3, 28), (1100, 700, 75), (3000, 3, 228), (3000, 700, 75)])
def test_viterbi_of_amplicons_shorter_than_the_profile(m, n, line, monkeypatch):
    """Viterbi scores go by rows up to a line in letters (of the longest of few amplicons, of the mean of many) and by
    the wavefront, which takes boundary buffers, above it; Forward always by the wavefront.  Scores at both sides of
    the line against the oracle in fp64."""
    rng = np.random.default_rng(m + n)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    ref = acgt[rng.integers(0, 4, m)].tobytes().decode()
    train = [ref, ref, ref[:-2]]
    seq = acgt[rng.integers(0, 4, 100_000)]
    seq[:m] = np.frombuffer(ref.encode(), np.uint8)
    _, T, E = oracle.hmm_build(train)
    fin = ~np.isinf(T)
    pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
    for L, wave in ((1, False), (line, False), (line + 1, True)):
        amps = np.zeros(n, dtype=ah.AMPLICON_DTYPE)
        amps["start"] = np.r_[7, rng.integers(0, len(seq) - L, n - 1)]
        amps["end"] = amps["start"] + L
        with ah.Context(0) as c:
            sid = c.load(seq, np.array([0, len(seq)], np.uint64), np.zeros(1, np.uint32))
            hid = c.hmm_build(train)
            monkeypatch.setenv("AH_HMM_KERNEL", "rows")
            c.hmm_score(sid, hid, amps)
            monkeypatch.delenv("AH_HMM_KERNEL")
            before = c.device_bytes()
            got = c.hmm_score(sid, hid, amps).astype(np.float64)
            assert (c.device_bytes() > before) == wave, L
            before = c.device_bytes()
            got_f = c.hmm_forward(sid, hid, amps).astype(np.float64)
            assert wave or c.device_bytes() > before, L
        some = [0, 1, n - 1]
        seqs = [seq[amps["start"][i]:amps["end"][i]].tobytes().decode() for i in some]
        want = np.array([oracle.hmm_viterbi(T, E, x) for x in seqs])
        want_f = np.array([oracle.hmm_forward(T, E, x) for x in seqs])
        # the bound of the parity test above: ten standard deviations of a walk of fp32 roundings
        N = L + m
        assert (np.abs(got[some] - want) <= 10.0 * np.sqrt(N) * 2.0 ** -24 * (np.abs(want) + N * pmean) + 1e-4).all()
        assert (np.abs(got_f[some] - want_f) <=
                10.0 * np.sqrt(N) * (2.0 ** -24 * (np.abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4).all()


@pytest.mark.parametrize("n_sites", [1025, 3000, 8200, 16384])
@pytest.mark.parametrize("where", ["first", "last", "two", "dozen", "mixed"])
def test_rank_sort_of_sites_crowded_into_few_ranges(ctx, n_sites, where):
    """Sites of a small run that lie in few of the 1,024 ranges of the key space: all in the first, all in the last
    ones, in two places, in a dozen, and half in one place with the rest spread; a second pair has no site."""
    rng = np.random.default_rng(n_sites)
    fwd, rev = "ACGTTGCAAGCT", "GGATCCATTCAG"
    n, room = 1 << 28, n_sites * 14 + 64
    spans = {"first": [(0, 1.0)], "last": [(n - room, 1.0)], "two": [(1000, 0.5), (n // 3, 0.5)],
             "dozen": [(n // 13 * j, 1 / 12) for j in range(12)], "mixed": [(n // 2, 0.5)]}[where]
    at = [s0 + 13 * np.arange(int(round(n_sites * part))) for s0, part in spans]
    if where == "mixed":
        at.append(rng.choice(n // 64 - 2, n_sites // 2, replace=False) * 64)
    at = np.unique(np.concatenate(at))[:n_sites]
    words = np.stack([np.frombuffer(w.encode(), np.uint8) for w in
                      (fwd, oracle_reverse_complement(fwd), rev, oracle_reverse_complement(rev))])
    seq = np.full(n, ord("N"), np.uint8)
    which = rng.integers(0, 4, len(at))
    for p, w in zip(at, which):
        seq[p:p + 12] = words[w]
    whole = (seq[at[:, None] + np.arange(12)] == words[which]).all(axis=1)  # (a plant may lie over another)
    off, gen = np.array([0, n // 5, n], np.uint64), np.array([0, 0], np.uint32)
    pairs = [synth.pcr_params(f, r, k=0, min_len=30, max_len=200) for f, r in ((fwd, rev), ("TTTTTTTTTTTTT", "TTTTTTTTTTTTTT"))]
    sid = ctx.load(seq, off, gen)
    try:
        pids = [ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs]
        run = ctx.run(sid, pids, tm_filter=False, caps=(n_sites + 64, 8 * n_sites, 1 << 22))
        alone = ctx.scan(sid, pids)
    finally:
        ctx.ah_unload_genomes(sid)
    got = run["sites"]
    contig = (at >= n // 5).astype(np.uint32)
    end = np.where(contig, n, n // 5)
    keep = (at + 12 <= end) & whole
    order = np.array([(0, 0), (0, 1), (1, 0), (1, 1)])[which]  # a copy at p: primer and strand
    assert keep.sum() > 1000 and len(got) == keep.sum()
    assert np.array_equal(got["pos"], (at - np.where(contig, n // 5, 0))[keep]) and np.array_equal(got["contig"], contig[keep])
    assert np.array_equal(got["primer"], order[keep, 0]) and np.array_equal(got["strand"], order[keep, 1])
    assert not got["mm"].any() and not got["pair"].any() and not got["genome"].any()
    assert alone.tobytes() == got.tobytes()


@pytest.mark.parametrize("spots,left,right", [(1, 1, 1), (1, 31, 33), (16, 16, 16), (25, 25, 25), (63, 30, 34),
                                              (512, 4, 4), (2048, 4, 4), (40, 90, 90)])
def test_run_of_hot_spots_that_lead_many_amplicons(ctx, spots, left, right):
    """Neighbouring sites that pair with one another, from one amplicon to more than the one-launch form holds: groups
    of 32 sites lie over all CTAs of the pairing's cluster, up to its last site; amplicons, sequences and offsets as
    the oracle gives them."""
    rng = np.random.default_rng(spots)
    fwd, rev = "ACGTTGCAAGCT", "GGATCCATTCAG"
    step = 14 * (left + right) + 2200
    n = spots * step + 500
    seq = np.full(n, ord("T"), np.uint8)
    words = [np.frombuffer(w.encode(), np.uint8) for w in (fwd, oracle_reverse_complement(rev))]
    for j in range(spots):
        for i in range(left + right):
            at = j * step + 14 * i + (int(rng.integers(100, 300)) if i >= left else 0)
            at = min(at, (j + 1) * step - 2000)
            seq[at:at + 12] = words[i >= left]
    off = np.array([0, n // step // 2 * step, n], np.uint64)
    gen = np.zeros(2, np.uint32)
    pair = synth.pcr_params(fwd, rev, k=0, min_len=30, max_len=14 * (left + right) + 400)
    want = oracle.scan(seq, off, gen, [pair])
    amps = oracle.pair(want, [pair])
    seqs, offs = oracle.fetch(seq, off, amps)
    assert len(want) and len(amps)
    sid = ctx.load(seq, off, gen)
    try:
        pid = ctx.ah_set_primers(fwd, rev, pair)
        for caps in ((len(want), len(amps), len(seqs)), (0, 0, 0)):
            r = ctx.run(sid, [pid], tm_filter=False, caps=caps)
            assert r["sites"].tobytes() == want.tobytes() and r["amps"].tobytes() == amps.tobytes()
            assert r["seqs"] == seqs and np.array_equal(r["offs"], offs)
    finally:
        ctx.ah_unload_genomes(sid)


def test_launch_counts_of_the_tm_stage_and_of_a_small_run():
    """The profile counts the kernels that a call launches: a small run is five (scan, site sort, Tm, pairing,
    sequences); the Tm stage one below the thread-per-site line, two from there on, and two under a table whose
    entropies may reach the concentration term (where many sites may need every oligo)."""
    w = synth.tiny(5)
    p = dict(w.pairs[0], tm_min=40.0)
    tables = {v: ah.NNTable() for v in (1.0, 10.0)}  # L - 1 stacks of 1 stay below it, of 10 do not
    for v, t in tables.items():
        t.stack_dS[:] = [v] * 256
    with ah.Context(0) as c:
        sid = c.load(w.seq, w.contig_off, w.contig_genome)
        pid = c.ah_set_primers(p["fwd"], p["rev"], p)
        c.ah_set_profiling(1)
        c.run(sid, [pid], caps=(64, 64, 1 << 16))
        assert c.ah_get_profile(None)[1] == 5
        for n, entropy, want in ((1, None, 1), (24575, None, 1), (24576, None, 2), (7, 1.0, 1), (7, 10.0, 2)):
            if entropy:
                c.ah_set_nn_table(pid, tables[entropy])
            sites = np.zeros(n, dtype=ah.SITE_DTYPE)
            sites["pos"] = np.arange(n) % 1000
            c.ah_set_profiling(1)
            c.tm(sid, [pid], sites)
            assert c.ah_get_profile("tm")[1] == want, n
        c.ah_set_profiling(0)


@pytest.mark.parametrize("m", [600, 1100, 1400, 1700, 2300, 2500, 2800, 3000])
def test_hmm_wavefront_uses_its_boundary_buffers_again(ctx, m):
    """Blocks with many tasks (a memory budget leaves one or two blocks for 24 amplicons of 3, 5, 6, 7, 9, 10, 11 and
    12 stripes), so that a buffer's turn comes round while a last stripe, which hands nothing on, lies between: the
    same scores as with a block per amplicon, and the oracle's."""
    rng = np.random.default_rng(m)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    ref = acgt[rng.integers(0, 4, m)].tobytes().decode()
    train = [ref, ref, ref[:-3], ref[5:]]
    seqs = [synth._mutate(rng, ref[:int(m * rng.uniform(0.2, 1.0))], 0.05, 0.02) for _ in range(22)]
    seqs += ["", ref + ref[:m // 4]]
    seq = np.frombuffer(("".join(seqs) + "A").encode(), np.uint8).copy()
    off = np.array([0, len(seq)], np.uint64)
    amps = np.zeros(len(seqs), dtype=ah.AMPLICON_DTYPE)
    ends = np.cumsum([len(x) for x in seqs])
    amps["end"], amps["start"] = ends, ends - [len(x) for x in seqs]
    got = []
    with ah.Context(0, 8 << 20) as small:
        for c in (ctx, small):
            sid = c.load(seq, off, np.zeros(1, np.uint32))
            hid = c.hmm_build(train)
            got.append((c.hmm_score(sid, hid, amps), c.hmm_forward(sid, hid, amps)))
            c.hmm_free(hid)
            c.ah_unload_genomes(sid)
    assert got[0][0].tobytes() == got[1][0].tobytes() and got[0][1].tobytes() == got[1][1].tobytes()
    _, T, E = oracle.hmm_build(train)
    fin = ~np.isinf(T)
    pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
    for i in (0, 22, 23):
        N = len(seqs[i]) + m
        # the bound of the parity test above: ten standard deviations of a walk of fp32 roundings
        want, want_f = oracle.hmm_viterbi(T, E, seqs[i]), oracle.hmm_forward(T, E, seqs[i])
        assert abs(float(got[0][0][i]) - want) <= 10.0 * np.sqrt(N) * 2.0 ** -24 * (abs(want) + N * pmean) + 1e-4
        assert abs(float(got[0][1][i]) - want_f) <= \
            10.0 * np.sqrt(N) * (2.0 ** -24 * (abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4


@pytest.mark.parametrize("kind", ["copies", "one deletion", "deletions by turns", "one insertion", "insertions by turns"])
@pytest.mark.parametrize("m,n_train", [(40, 40_000), (60, 20_000), (300, 4000), (500, 100), (500, 3000), (700, 700)])
def test_forward_on_odds_after_large_training_sets(ctx, m, n_train, kind):
    """The range of the scaled odds: profiles whose rare moves and letters have probabilities down to 1 / (training
    sequences + 4) and whose common ones include long deletions, single deletions in every other column, long and
    scattered insertions; amplicons that agree, end early, start late, are turned about, lie apart by a few letters
    or agree with nothing.  Forward (and Viterbi) against the oracle in fp64."""
    rng = np.random.default_rng(m)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    ref = acgt[rng.integers(0, 4, m)].tobytes().decode()

    def random(n):
        return acgt[rng.integers(0, 4, n)].tobytes().decode()

    a, b = m // 5, m // 2  # the columns of the variants
    ins = random(40)
    variants = {"copies": [ref], "one deletion": [ref[:a] + ref[b:]],
                "deletions by turns": [ref[:a] + ref[a:b:2] + ref[b:], ref[:a] + ref[a + 1:b:2] + ref[b:]],
                "one insertion": [ref[:a] + ins + ref[a:]],
                "insertions by turns": [ref[:a] + "".join(x + "A" for x in ref[a:b]) + ref[b:]]}[kind]
    train = [ref] * (n_train // 2 + 1)
    train += [variants[i % len(variants)] for i in range(n_train - len(train))]
    seqs = [ref, "", ref[:1], ref[:m // 3], ref[m // 3:], ref[m // 2:] + ref[:m // 2], random(m), random(2 * m),
            ref[:a] + random(30) + ref[a:], ref[:a] + ref[a + 6:], ref[:b] + random(3) + ref[b:], ref + random(50),
            random(50) + ref, ref[:a] + random(b - a) + ref[b:], "A" * m, ref[:b] + "A" * 200 + ref[b:],
            ref[::-1], ref + ref, ref[:a] + ref[a:b] * 2 + ref[b:], *variants]
    seqs += [synth._mutate(rng, v, 0.1, 0.1) for v in variants for _ in range(4)]
    seq = np.frombuffer(("".join(seqs) + "A").encode(), np.uint8).copy()
    amps = np.zeros(len(seqs), dtype=ah.AMPLICON_DTYPE)
    ends = np.cumsum([len(x) for x in seqs])
    amps["end"], amps["start"] = ends, ends - [len(x) for x in seqs]
    sid = ctx.load(seq, np.array([0, len(seq)], np.uint64), np.zeros(1, np.uint32))
    try:
        hid = ctx.hmm_build(train)
        _, ref_i, T, E = ctx.hmm_tables(hid)
        assert train[ref_i] == ref
        got, got_f = ctx.hmm_score(sid, hid, amps).astype(np.float64), ctx.hmm_forward(sid, hid, amps).astype(np.float64)
        ctx.hmm_free(hid)
    finally:
        ctx.ah_unload_genomes(sid)
    T, E = T.astype(np.float64), E.astype(np.float64)  # (the tables' own roundings are the other tests')
    want = np.array([oracle.hmm_viterbi(T, E, x) for x in seqs])
    want_f = np.array([oracle.hmm_forward(T, E, x) for x in seqs])
    fin = ~np.isinf(T)
    pmean = float(np.concatenate([np.abs(T[fin]), np.abs(E[1:]).ravel()]).mean())
    N = np.array([len(x) for x in seqs]) + m
    # the bound of the parity test above: ten standard deviations of a walk of fp32 roundings
    assert (np.abs(got - want) <= 10.0 * np.sqrt(N) * 2.0 ** -24 * (np.abs(want) + N * pmean) + 1e-4).all()
    tol_f = 10.0 * np.sqrt(N) * (2.0 ** -24 * (np.abs(want_f) + N * pmean) + 4 * 2.0 ** -23) + 1e-4
    assert (np.abs(got_f - want_f) <= tol_f).all(), (np.abs(got_f - want_f) / tol_f).max()


@pytest.mark.parametrize("tiles,per_claim", [(7295, 1), (7297, 2), (10_950, 3), (29_191, 8)])
def test_scan_tiles_claimed_several_at_a_time(tiles, per_claim, monkeypatch):
    """Large sets hand out their tiles in claims of up to eight (n_tiles / (24 CTAs) of them; one CTA per SM here, so
    that smaller sets do too), the last claim past the set's end: a site in every tile, at its edges and inside, is
    found once, and again in a second scan."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms != 152:
        pytest.skip("the sizes are for 152 SMs")
    assert min(8, max(1, tiles // (sms * 24))) == per_claim
    monkeypatch.setenv("AH_SCAN_TUNING", "4,0,0,4,2,1")
    fwd, rev = "ACGTTGCAAGCT", "GGATCCATTCAG"
    T = 32 * 1024
    n = tiles * T - 17
    rng = np.random.default_rng(tiles)
    at = np.arange(tiles) * T + rng.choice([0, 1, 31, 1023, 1024, T // 2, T - 40, T - 13, T - 11, T - 1], tiles)
    at[-1] = n - 12
    word = np.frombuffer(fwd.encode(), np.uint8)
    seq = torch.full((n,), ord("T"), dtype=torch.uint8, device="cuda")
    seq[torch.from_numpy(at[:, None] + np.arange(12)).cuda()] = torch.from_numpy(np.tile(word, (tiles, 1))).cuda()
    whole = np.r_[np.diff(at) >= 12, True] & np.r_[True, np.diff(at) >= 12]  # (a plant may lie over the next one)
    torch.cuda.synchronize()
    with ah.Context(0) as c:
        sid = c.ah_load_genomes(seq, n, np.array([0, n], np.uint64), np.zeros(1, np.uint32))
        pid = c.ah_set_primers(fwd, rev, synth.pcr_params(fwd, rev, k=0, min_len=30, max_len=200))
        for _ in range(2):
            got = c.scan(sid, [pid])
            assert np.array_equal(np.sort(got["pos"]), got["pos"]) and len(np.unique(got["pos"])) == len(got)
            assert np.isin(at[whole], got["pos"]).all() and np.isin(got["pos"], at).all()
            assert not got["primer"].any() and not got["strand"].any() and not got["mm"].any()
