"""What a user of this framework has it do, as cases to measure.

A case is one pass of a user's program over inputs it already holds: one or
several genome collections are loaded (packed) and run through the path of in
silico PCR -- primer matching, melting temperatures, pairing, sequences -- or
one of its stages is called on records the program kept, or amplicons are
analysed and scored.  Everything goes through the ctypes binding of the C ABI
(paper_2509_13300_gb300.ah), with device buffers where a program keeps its
results on the GPU and numpy arrays where the entry point returns them.

Genome collections are made on the GPU from the seed: genome lengths
log-uniform around the mean, geometric contig counts, a GC content per genome,
0.1 % of the bases in runs of N, and planted amplicons whose primer sites
carry 0..k substitutions, some of them copies of a common family.  Primers,
mismatch limits and windows belong to the case: a program keeps its primers
from one collection to the next.

exact() states the floating results in 64 bits with torch alone: a brute-force
scan and the maximum melting temperature over every oligo of the primer, and
the profile HMM's build, Viterbi and Forward recurrences.
"""
import math

import numpy as np
import torch

from paper_2509_13300_gb300 import ah, synth

# primer pairs of the published list, and synthetic ones of 16 to 960 oligos
PAIRS = {
    "V3V4": synth.PAPER_PAIRS["V3V4"],
    "V1V9": synth.PAPER_PAIRS["V1V9"],
    "Titan": synth.PAPER_PAIRS["Titan"],
    "mecA": synth.PAPER_PAIRS["mecA"],
    "p16": ("ACGGRTYCATGAACKTC", "TTGSACGMTAGCCWTAGC"),
    "p64": ("GCRTAYCCASTGAWCTKAG", "CAWGTTKACMGGRTTYACAGC"),
    "p256": ("ATRGCYATSGACWTTKGACMCR", "TGKCAMRTTACYGGSATWCAKTGC"),
    "p960": ("CTRAYGGKCMTSAWTHGADC", "GANCTYRAGKTWCSTTBAACGA"),
}
WINDOW = (100, 3000)


def _case(kind, **kw):
    return dict(kind=kind, **kw)


def listed():
    return [
        # a plasmid-sized genome kept loaded: one primer pair tried on it (the smallest call)
        _case("run", name="tiny_resident", load="resident", bases=200_000, genomes=1, pairs="p64:2", plants=10),
        # one bacterial genome of a collection buffer, at whatever address it starts: load, run, unload
        _case("run", name="genome_at_odd_address", load="device", bases=4_600_001, genomes=1, pairs="V1V9:2", plants=7,
              offset=3),
        # the genome collection with the 960-oligo pair: load, run, unload
        _case("run", name="collection_960oligos", load="device", bases=407_000_003, genomes=100, pairs="p960:3",
              plants=8),
        # the decoy collection (contigs reversed): the off-target rate of a primer pair
        _case("run", name="decoy_reversed", load="reversed", bases=100_000_007, genomes=25, pairs="Titan:3", plants=8),
        # a chunk of a large collection, three pairs at k = 4: load, run, unload
        _case("run", name="large_3pairs_k4", load="device", bases=4_000_000_001, genomes=1100,
              pairs="Titan:4,p64:4,p256:4", plants=8),
        # a batch streamed from pinned host memory as 2-bit codes, four pairs of k = 2, 3, 4, 2
        _case("run", name="batch_2bit_host", load="host2bit", bases=1_500_000_013, genomes=500,
              pairs="p16:2,p64:3,p256:4,p960:2", plants=8),
        # a resident pool searched for one published pair at a small k
        _case("run", name="pool_V3V4_k1", load="resident", bases=2_000_000_000, genomes=500, pairs="V3V4:1", plants=8),
        # a burst of requests to the server over a resident pool: genome subsets of Zipf-like sizes, two
        # pairs, k = 0, 1, 2, 3; every result is read back
        _case("served", name="served_burst", bases=1_000_000_000, genomes=250, pairs="V1V9:3,p64:3", plants=8,
              requests=24),
        # the stages called one by one on a kept site list of two pairs: melting temperatures, amplicons, sequences
        _case("stages", name="tm_pair_fetch", bases=1_200_000_000, genomes=300, pairs="Titan:4,p256:4", plants=100),
        # threshold sweep and amplitypes over the called amplicons of a collection
        _case("analysis", name="sweep_and_amplitypes", bases=150_000_000, genomes=600, pairs="Titan:3", plants=60,
              thresholds=31),
        # profile HMM: Viterbi scores of full-length amplicons, Forward scores of shorter ones
        _case("hmm", name="hmm_viterbi", amplicons=4000, template=1421, forward=False),
        _case("hmm", name="hmm_forward", amplicons=5000, template=420, forward=True),
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def pair_list(n, kmax):
        names = rng.sample(sorted(PAIRS), n)
        return ",".join("%s:%d" % (p, rng.randint(0 if p == "mecA" else 1, kmax)) for p in names)

    kind = rng.choice(["run"] * 6 + ["served", "stages", "stages", "analysis", "hmm", "hmm"])
    if kind == "run":
        load = rng.choice(["resident", "device", "device", "reversed", "host2bit", "host"])
        top = {"resident": 4e9, "device": 4e9, "reversed": 4e8, "host2bit": 1.5e9, "host": 4e8}[load]
        n = span(150_000, top)
        return _case("run", load=load, bases=n, genomes=max(1, min(1500, n // span(1_000_000, 8_000_000))),
                     pairs=pair_list(rng.choice([1, 1, 2, 3]), 4), plants=rng.randint(1, 15),
                     offset=rng.choice([0, 0, rng.randint(1, 15)]) if load == "device" else 0)
    if kind == "served":
        n = span(20_000_000, 1_000_000_000)
        return _case("served", bases=n, genomes=max(4, n // 4_000_000), pairs=pair_list(rng.choice([1, 2]), 3),
                     plants=8, requests=rng.randint(1, 24))
    if kind == "stages":
        n = span(3_000_000, 1_200_000_000)
        return _case("stages", bases=n, genomes=max(1, n // 4_000_000), pairs=pair_list(rng.choice([1, 2]), 4),
                     plants=rng.randint(5, 100))
    if kind == "analysis":
        n = span(2_000_000, 150_000_000)
        return _case("analysis", bases=n, genomes=max(1, n // 250_000), pairs="%s:%d" % (
            rng.choice(["Titan", "V1V9"]), rng.randint(2, 3)), plants=rng.randint(5, 60), thresholds=rng.randint(3, 64))
    fwd = rng.random() < 0.5
    template = span(100, 1500) if fwd else span(100, 2200)
    most = int((1.1e9 if fwd else 8.5e9) / (template + 40) ** 2)
    return _case("hmm", amplicons=max(1, min(8000, span(max(1, most // 40), max(2, most)))), template=template,
                 forward=fwd)


# ------------------------------------------------------------------ inputs
_SETS = synth._IUPAC_BASES
_LETTERS = np.frombuffer(b"ACGT", dtype=np.uint8)
_COMP = np.zeros(256, dtype=np.uint8)
_COMP[list(b"ACGTN")] = list(b"TGCAN")


def _pairs(case):
    out = []
    for item in case["pairs"].split(","):
        name, k = item.split(":")
        f, r = PAIRS[name]
        out.append(synth.pcr_params(f, r, k=int(k), min_len=WINDOW[0], max_len=WINDOW[1], tm_min=48.0))
    return out


def _oligos(rng, primer, subs):
    """len(subs) oligos of `primer` as ASCII rows, row i with subs[i] substitutions outside the sets."""
    n, L = len(subs), len(primer)
    out = np.empty((n, L), dtype=np.uint8)
    for j, ch in enumerate(primer):
        out[:, j] = np.frombuffer(_SETS[ch].encode(), dtype=np.uint8)[rng.integers(len(_SETS[ch]), size=n)]
    free = [j for j, ch in enumerate(primer) if ch != "N"]
    order = rng.random((n, len(free))).argsort(axis=1)
    for j, pos in enumerate(free):
        others = np.frombuffer("".join(b for b in "ACGT" if b not in _SETS[primer[pos]]).encode(), dtype=np.uint8)
        hit = (order < np.minimum(subs, len(free))[:, None])[:, j]
        out[hit, pos] = others[rng.integers(len(others), size=int(hit.sum()))]
    return out


def _layout(case, rng):
    """Genome and contig tables: (contig_off, contig_genome, genome offsets)."""
    G, n = case["genomes"], case["bases"]
    w = np.exp(rng.uniform(math.log(2.0), math.log(7.0), G))
    goff = np.concatenate([[0], np.round(np.cumsum(w) / w.sum() * n)]).astype(np.int64)
    nc = np.minimum(200, rng.geometric(0.05, G))
    starts, owner = [], []
    for g in range(G):
        a, b = int(goff[g]), int(goff[g + 1])
        cuts = np.unique(rng.integers(a + 1, max(a + 2, b), nc[g] - 1)) if nc[g] > 1 else np.zeros(0, np.int64)
        starts.append(np.concatenate([[a], cuts[cuts < b]]))
        owner.append(np.full(len(starts[-1]), g))
    off = np.append(np.concatenate(starts), n).astype(np.uint64)
    return off, np.concatenate(owner).astype(np.uint32), goff


def _collection(case, seed, family=False):
    """ASCII bases on the GPU, contig_off, contig_genome, pairs."""
    rng = np.random.default_rng([seed, 1])
    gen = torch.Generator(device="cuda").manual_seed(seed * 2654435761 % (1 << 62))
    pairs = _pairs(case)
    off, owner, goff = _layout(case, rng)
    n, G = case["bases"], case["genomes"]
    lead = case.get("offset", 0)
    buf = torch.empty(n + lead + 64, dtype=torch.uint8, device="cuda")
    seq = buf[lead:lead + n]
    lut = torch.tensor(list(b"GCAT"), dtype=torch.uint8, device="cuda")
    gc = rng.uniform(0.3, 0.7, G)
    for g in range(G):  # G, C below gc, A, T above it
        for a in range(int(goff[g]), int(goff[g + 1]), 1 << 27):
            b = min(int(goff[g + 1]), a + (1 << 27))
            u = torch.randint(0, 256, (b - a,), dtype=torch.uint8, device="cuda", generator=gen)
            t = [int(256 * gc[g] / 2), int(256 * gc[g]), int(128 * (1 + gc[g]))]
            seq[a:b] = lut[((u >= t[0]).to(torch.uint8) + (u >= t[1]) + (u >= t[2])).int()]
    runs = max(1, int(n * 0.001 / 50.5))  # 0.1 % of the bases in runs of N
    rs = torch.from_numpy(rng.integers(0, max(1, n - 100), runs)).cuda()
    rl = torch.from_numpy(rng.integers(1, 101, runs)).cuda()
    first = torch.repeat_interleave(rs - (rl.cumsum(0) - rl), rl)
    at = (first + torch.arange(first.numel(), device="cuda")).clamp_(max=n - 1)
    seq[at] = ord("N")
    # planted amplicons, whole: primer site, body, reverse-complemented site; every other one a
    # copy of one of four family bodies with a few substitutions (family: nearly all)
    P = G * case["plants"]
    body = 600 if family else 460
    fam = _LETTERS[rng.integers(4, size=(4, body))]
    own = np.repeat(np.arange(G), case["plants"])
    which = rng.integers(len(pairs), size=P)
    for i, p in enumerate(pairs):
        sel = np.nonzero(which == i)[0]
        m = len(sel)
        lf, lr = len(p["fwd"]), len(p["rev"])
        rows = np.empty((m, lf + body + lr), dtype=np.uint8)
        rows[:, :lf] = _oligos(rng, p["fwd"], rng.integers(0, p["k"] + 1, m))
        rows[:, lf:lf + body] = np.where((rng.random(m) < (0.9 if family else 0.5))[:, None],
                                         fam[rng.integers(4, size=m)], _LETTERS[rng.integers(4, size=(m, body))])
        hit = rng.random((m, body)) < 0.0005
        rows[:, lf:lf + body][hit] = _LETTERS[rng.integers(4, size=int(hit.sum()))]
        rows[:, lf + body:] = _COMP[_oligos(rng, p["rev"], rng.integers(0, p["k"] + 1, m))[:, ::-1]]
        flip = rng.random(m) < 0.5
        rows[flip] = _COMP[rows[flip][:, ::-1]]
        width = rows.shape[1]
        room = goff[own[sel] + 1] - goff[own[sel]] - width
        slot = np.minimum(room // (width + 8), 1 << 20).clip(1)  # slots, so that few plants overlap
        s = goff[own[sel]] + (rng.integers(0, slot) * (width + 8)).clip(0, room.clip(0))
        idx = torch.from_numpy(s[:, None] + np.arange(width)).cuda().clamp_(max=n - 1)
        val = torch.from_numpy(rows).cuda()
        for q in range(0, m, 4096):  # later plants win over earlier ones they overlap, in a fixed order
            flat, first_of = np.unique(idx[q:q + 4096].cpu().numpy().ravel()[::-1], return_index=True)
            v = val[q:q + 4096].cpu().numpy().ravel()[::-1][first_of]
            seq[torch.from_numpy(flat).cuda()] = torch.from_numpy(np.ascontiguousarray(v)).cuda()
    return seq, off, owner, pairs


def _expected_sites(pairs, n):
    """Sites of uniform random bases: the capacity a program sets aside (with a margin)."""
    total = 0.0
    for p in pairs:
        for primer in (p["fwd"], p["rev"]):
            d = np.zeros(len(primer) + 1)
            d[0] = 1.0
            for ch in primer:
                q = 1 - len(_SETS[ch]) / 4
                d = d * (1 - q) + np.concatenate([[0], d[:-1]]) * q
            total += 2 * d[:p["k"] + 1].sum()
    return total * n


def _encode_2bit(seq):
    """2-bit codes (GPU uint8) and no-base runs of ASCII bases on the GPU."""
    n = seq.numel()
    lut = torch.zeros(256, dtype=torch.uint8, device="cuda")
    for i, ch in enumerate(b"ACGT"):
        lut[ch] = i
    codes = torch.zeros((n + 3) // 4, dtype=torch.uint8, device="cuda")
    at = []
    for a in range(0, n, 1 << 27):
        s = seq[a:a + (1 << 27)]
        c = lut[s.int()]
        at.append(torch.nonzero(s == ord("N")).flatten() + a)
        if c.numel() % 4:
            c = torch.cat([c, torch.zeros(4 - c.numel() % 4, dtype=torch.uint8, device="cuda")])
        q = c.view(-1, 4)
        codes[a // 4:a // 4 + q.shape[0]] = q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)
    at = torch.cat(at).cpu().numpy().astype(np.uint64)
    if not len(at):
        return codes, np.zeros((0, 2), np.uint64)
    cut = np.nonzero(np.diff(at) != 1)[0]
    s = at[np.concatenate([[0], cut + 1])]
    e = at[np.append(cut, len(at) - 1)] + np.uint64(1)
    return codes, np.stack([s, e - s], axis=1)


def _u8(n):
    return torch.zeros(max(int(n), 1), dtype=torch.uint8, device="cuda")


class _Out:
    """Device output buffers of a run (zeroed once; a pass returns them whole, with the counts)."""

    def __init__(self, sites, amps, seq):
        self.caps = (int(sites), int(amps), int(seq))
        self.sites, self.tm = _u8(16 * sites), torch.zeros(int(sites), dtype=torch.float32, device="cuda")
        self.pass_, self.amps, self.seq = _u8(sites), _u8(28 * amps), _u8(seq)
        self.offs = torch.zeros(int(amps) + 1, dtype=torch.int64, device="cuda")

    def run_out(self):
        s, a, q = self.caps
        return ah.RunOut(self.sites.data_ptr(), s, 0, self.tm.data_ptr(), self.pass_.data_ptr(), self.amps.data_ptr(),
                         a, 0, self.seq.data_ptr(), q, 0, self.offs.data_ptr(), 1, 0)


def _records(buf, size):
    return buf.view(torch.int32).view(-1, size // 4)


def _room(case, pairs):
    """Site capacity a program sets aside (GC-rich and GC-poor genomes hold several times the mean)."""
    return int(8 * _expected_sites(pairs, case["bases"])) + 4 * case["genomes"] * case["plants"] + 16384


def prepare(case, seed):
    """Contexts, inputs on the GPU (or in pinned host memory), primers, and output buffers."""
    if case["kind"] == "hmm":
        return _prepare_hmm(case, seed)
    seq, off, owner, pairs = _collection(case, seed, family=case["kind"] == "analysis")
    ctx = ah.Context(0)
    n = case["bases"]
    st = dict(kind=case["kind"], ctx=ctx, n=n, off=off, owner=owner,
              pids=[ctx.ah_set_primers(p["fwd"], p["rev"], p) for p in pairs])
    torch.cuda.synchronize()
    room = _room(case, pairs)
    if case["kind"] == "run":
        st.update(load=case["load"], seq=seq, out=_Out(room, 60_000, 64 << 20))
        torch.cuda.synchronize()
        if case["load"] == "resident":
            st["sid"] = ctx.ah_load_genomes(seq, n, off, owner)
            ctx.ah_scan(st["sid"], st["pids"], st["out"].sites, room)  # the pool is ready (the load is stream-ordered)
            del st["seq"]
        elif case["load"] == "host2bit":
            codes, st["gaps"] = _encode_2bit(seq)
            st["seq"] = codes.cpu().pin_memory()
        elif case["load"] == "host":
            st["seq"] = seq.cpu().pin_memory()
        return st
    st["sid"] = ctx.ah_load_genomes(seq, n, off, owner)
    sites = _u8(16 * room)
    cap = 1 << 18
    amps = _u8(28 * cap)
    torch.cuda.synchronize()
    ns = ctx.ah_scan(st["sid"], st["pids"], sites, room)  # the set is ready (the load is stream-ordered)
    if case["kind"] == "served":  # pairs and k's belong to the case, the genomes asked for to the seed
        rng = np.random.default_rng([seed, 4])
        sizes = np.exp(rng.random(case["requests"]) * math.log(case["genomes"])).astype(int).clip(1)
        st["requests"] = [(rng.choice(case["genomes"], s, replace=False), st["pids"][i % len(pairs)],
                           (i // len(pairs)) % (pairs[i % len(pairs)]["k"] + 1)) for i, s in enumerate(sizes)]
        st["server"] = ah.Server(ctx, st["sid"])
        most = case["requests"] * room
        st["out"] = (np.zeros(most, ah.SITE_DTYPE), np.zeros(case["requests"] * 4096 * case["plants"], ah.AMPLICON_DTYPE),
                     np.zeros(case["requests"] << 22, np.uint8))
        return st
    # the collection stays loaded, its site list is kept on the device
    st.update(ns=ns, sites=sites, tm=torch.zeros(room, dtype=torch.float32, device="cuda"), pass_=_u8(room))
    if case["kind"] == "stages":
        st.update(amps=amps, cap=cap, seq=_u8(1 << 28), offs=torch.zeros(cap + 1, dtype=torch.int64, device="cuda"))
        return st
    na = ctx.ah_pair(st["sid"], st["pids"], st["sites"], None, ns, amps, cap)
    st.update(sites=sites[:16 * ns], amps=amps[:28 * na], cap=cap, thresholds=np.linspace(35.0, 65.0, case["thresholds"]))
    st["amps_host"] = st["amps"].cpu().numpy().view(ah.AMPLICON_DTYPE)
    st["out"] = np.zeros((2, cap), dtype=np.int32)
    return st


def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind == "hmm":
        if st["forward"]:
            ctx.hmm_forward(st["sid"], st["hmm"], st["amps"], st["n"], st["out"])
        else:
            ctx.hmm_score(st["sid"], st["hmm"], st["amps"], st["n"], st["out"])
        return {"score": st["out"]}
    if kind == "run":
        load = st["load"]
        if load == "resident":
            sid = st["sid"]
        elif load == "host2bit":
            sid = ctx.ah_load_genomes_2bit(st["seq"], st["n"], st["gaps"], st["off"], st["owner"], host_async=True)
        else:
            sid = ctx.ah_load_genomes(st["seq"], st["n"], st["off"], st["owner"], reversed=load == "reversed",
                                      host_async=load == "host")
        out = st["out"]
        o = ctx.ah_run(sid, st["pids"], out.run_out())
        if load != "resident":
            ctx.ah_unload_genomes(sid)
        return {"sites": _records(out.sites, 16), "tm": out.tm, "pass": out.pass_, "amps": _records(out.amps, 28),
                "offs": out.offs, "seq": out.seq, "counts": np.array([o.n_sites, o.n_amplicons, o.n_seq])}
    if kind == "served":
        tickets = [st["server"].submit(g, pid, k) for g, pid, k in st["requests"]]
        got = [st["server"].wait(t) for t in tickets]
        at = [0, 0, 0]
        for sites, amps, seq, _, _ in got:  # read back one after another
            for j, x in enumerate((sites, amps, np.frombuffer(seq, np.uint8))):
                st["out"][j][at[j]:at[j] + len(x)] = x
                at[j] += len(x)
        return {"sites": st["out"][0].view(np.int32), "amps": st["out"][1].view(np.int32), "seq": st["out"][2],
                "counts": np.array([[len(g[0]), len(g[1]), len(g[2])] for g in got])}
    if kind == "stages":
        ctx.ah_tm(st["sid"], st["pids"], st["sites"], st["ns"], st["tm"], st["pass_"])
        na = ctx.ah_pair(st["sid"], st["pids"], st["sites"], st["pass_"], st["ns"], st["amps"], st["cap"])
        ctx.ah_fetch(st["sid"], st["amps"], na, st["seq"], st["seq"].numel(), st["offs"])
        return {"tm": st["tm"], "pass": st["pass_"], "amps": _records(st["amps"], 28), "offs": st["offs"],
                "seq": st["seq"], "counts": np.array([st["ns"], na])}
    rows, n_genomes = ctx.ah_tm_sweep(st["sid"], st["pids"], st["sites"], st["amps"], st["thresholds"])
    variant, per_genome, n_variants, n_types = ctx.amplitypes(st["sid"], st["amps_host"])
    out = st["out"]
    out[0, :len(variant)] = variant
    out[1, :per_genome.size] = per_genome.ravel()
    return {"rows": rows.astype(np.int64), "genomes": n_genomes, "variant": out[0], "per_genome": out[1],
            "counts": np.array([len(variant), len(per_genome), n_variants, n_types])}


def work(case):
    if case["kind"] == "hmm":
        cols = case["template"] + 40
        cells = case["amplicons"] * cols * cols  # 10 adds, 6 maxima or sums per cell of the recurrence
        return {"bytes": case["amplicons"] * (cols // 2 + 32) + 52 * cols, "flops": 16 * cells}
    pairs = _pairs(case)
    n = case["bases"]
    sites = _expected_sites(pairs, n)
    plants = case["genomes"] * case["plants"]
    if case["kind"] == "run":
        read = {"host2bit": n // 4, "resident": n // 2}.get(case["load"], n)
        # per start, strand and primer position: one set test and one addition
        flops = 2 * n * sum(2 * (len(p["fwd"]) + len(p["rev"])) for p in pairs)
        return {"bytes": int(read + 21 * sites + plants * 540), "flops": flops}
    window = 12  # bytes of a packed window of at most 32 bases with its flags
    if case["kind"] == "served":
        g = case["genomes"]  # the mean of exp(U log g) genomes a request
        asked = case["requests"] * n * ((g - 1) / math.log(g) if g > 1 else 1) / g
        return {"bytes": int(asked / 2 + 16 * sites * asked / n + plants * 540 * asked / n),
                "flops": 2 * asked * 2 * (len(pairs[0]["fwd"]) + len(pairs[0]["rev"]))}
    if case["kind"] == "stages":
        return {"bytes": int((33 + window + 5) * sites + plants * (28 + 8 + 1.25 * 500)), "flops": int(sites * 640)}
    return {"bytes": int((16 + window) * sites + plants * (28 + 300 + 8)), "flops": int(sites * 2 * 16 * 20)}


# ------------------------------------------------------------------ the HMM's inputs
def _family(case, seed):
    """Training sequences and amplicons: copies of one template between two primer sites, with 2 %
    substitutions and 0.5 % single-letter insertions and deletions each.  Lists of uint8 codes 0..3."""
    rng = np.random.default_rng([seed, 2])
    m = case["template"] + 40
    template = rng.integers(0, 4, m)

    def copy():
        keep = rng.random(m) >= 0.005
        ins = rng.random(m) < 0.005
        sub = rng.random(m) < 0.02
        keep[:20] = keep[-20:] = True
        ins[:20] = ins[-20:] = sub[:20] = sub[-20:] = False
        t = np.where(sub, (template + rng.integers(1, 4, m)) % 4, template)
        out = np.repeat(t, keep.astype(np.int64) + ins)
        first = np.cumsum(keep.astype(np.int64) + ins) - (keep.astype(np.int64) + ins)
        out[first[ins]] = rng.integers(0, 4, int(ins.sum()))  # the inserted letter, before its column's
        return out.astype(np.uint8)

    train = [template.astype(np.uint8)] * 2 + [copy() for _ in range(14)]
    return train, [copy() for _ in range(case["amplicons"])]


def _prepare_hmm(case, seed):
    train, amps = _family(case, seed)
    rng = np.random.default_rng([seed, 3])
    ctx = ah.Context(0)
    n = len(amps)
    flip = rng.random(n) < 0.5
    margin = 37  # bases between amplicons (four contigs)
    lens = np.array([len(a) for a in amps])
    start = np.concatenate([[0], np.cumsum(lens + margin)])
    seq = rng.integers(0, 4, int(start[-1]) + margin).astype(np.uint8)
    for i, a in enumerate(amps):
        seq[start[i]:start[i] + lens[i]] = 3 - a[::-1] if flip[i] else a
    per = -(-n // 4)
    first = start[np.minimum(np.arange(5) * per, n)]
    first[4] = len(seq)
    contig = np.arange(n) // per
    rec = np.zeros(n, dtype=ah.AMPLICON_DTYPE)
    rec["genome"] = rec["contig"] = contig
    rec["start"] = start[:-1] - first[contig]
    rec["end"] = rec["start"] + lens
    rec["orient"] = flip
    ascii_ = torch.from_numpy(_LETTERS[seq]).cuda()
    torch.cuda.synchronize()
    sid = ctx.ah_load_genomes(ascii_, len(seq), first.astype(np.uint64), np.arange(4, dtype=np.uint32))
    hid = ctx.hmm_build([bytes(_LETTERS[t]) for t in train])
    return dict(kind="hmm", ctx=ctx, sid=sid, hmm=hid, forward=case["forward"], n=n, ascii=ascii_,
                amps=torch.from_numpy(rec.view(np.uint8).copy()).cuda(),
                out=torch.empty(n, dtype=torch.float32, device="cuda"))


# ------------------------------------------------------------------ 64-bit results
# unified Watson-Crick stacks of SantaLucia (1998): dH (kcal/mol), dS (cal/(K mol)) by top dinucleotide
_DH = np.array([[-7.9, -8.4, -7.8, -7.2], [-8.5, -8.0, -10.6, -7.8], [-8.2, -9.8, -8.0, -8.4], [-7.2, -8.2, -8.5, -7.9]])
_DS = np.array([[-22.2, -22.4, -21.0, -20.4], [-22.7, -19.9, -27.2, -21.0], [-22.2, -24.4, -19.9, -22.4],
                [-21.3, -22.2, -22.7, -22.2]])


def _bits(primer):
    return [sum(1 << "ACGT".index(b) for b in _SETS[ch]) for ch in primer]


def _exact_tm_group(primer, windows, minus, p):
    """Maximum Tm over the primer's oligos for windows (n, L) of codes 0..3 (4: no base -> NaN)."""
    L = len(primer)
    sets = [["ACGT".index(b) for b in _SETS[ch]] for ch in primer]
    grid = torch.cartesian_prod(*[torch.tensor(s) for s in sets]) if L > 1 else torch.tensor(sets[0])[:, None]
    grid = grid.view(-1, L).cuda()
    t = torch.where(minus[:, None], windows.flip(1), 3 - windows).long()  # template base opposite each position
    bad = (windows > 3).any(1)
    t.clamp_(0, 3)
    oh = torch.nn.functional.one_hot(grid[:, :-1] * 4 + grid[:, 1:], 16).double().view(len(grid), -1)
    tab = torch.zeros(2, 16, 16, dtype=torch.float64, device="cuda")  # [H or S][template pair][oligo pair]
    for x in range(4):
        for y in range(4):
            for k, d in enumerate((_DH, _DS)):
                tab[k, (3 - x) * 4 + 3 - y, x * 4 + y] = d[x, y]
    gc = torch.tensor([0, 1, 1, 0], dtype=torch.float64, device="cuda")
    ends = gc[grid[:, 0]] + gc[grid[:, -1]]
    endH, endS = 2 * 2.3 + ends * (0.1 - 2.3), 2 * 4.1 + ends * (-2.8 - 4.1)
    c = 1.987 * math.log((p["dnac1_nM"] - p["dnac2_nM"] / 2) * 1e-9) + 0.368 * (L - 1) * math.log(p["Na_mM"] / 1000)
    out = torch.empty(len(windows), dtype=torch.float64, device="cuda")
    for a in range(0, len(windows), 1 << 16):
        q = t[a:a + (1 << 16)]
        idx = q[:, :-1] * 4 + q[:, 1:]
        H = tab[0][idx].view(len(q), -1) @ oh.T + endH
        S = tab[1][idx].view(len(q), -1) @ oh.T + endS
        out[a:a + (1 << 16)] = (1000 * H / (S + c)).amax(1) - 273.15
    out[bad] = math.nan
    return out


def _exact_site_tm(case, seed):
    seq, off, _, pairs = _collection(case, seed)
    n = case["bases"]
    offs = torch.from_numpy(off.astype(np.int64)).cuda()
    lut = torch.full((256,), 4, dtype=torch.uint8, device="cuda")
    for i, ch in enumerate(b"ACGT"):
        lut[ch] = i
    code = torch.empty(n, dtype=torch.uint8, device="cuda")
    for a in range(0, n, 1 << 27):
        code[a:a + (1 << 27)] = lut[seq[a:a + (1 << 27)].int()]
    del seq
    if case.get("load") == "reversed":
        flip = torch.empty_like(code)
        for a, b in zip(off[:-1].tolist(), off[1:].tolist()):
            flip[a:b] = code[a:b].flip(0)
        code = flip
    one = torch.tensor([1, 2, 4, 8, 0], dtype=torch.uint8, device="cuda")
    tms = []
    for p in pairs:
        keys, vals = [], []
        for primer_i, primer in enumerate((p["fwd"], p["rev"])):
            L = len(primer)
            fwd = _bits(primer)
            rc = [int("{:04b}".format(b)[::-1], 2) for b in fwd[::-1]]
            found, minus = [], []
            for strand, masks in enumerate((fwd, rc)):
                for a in range(0, max(0, n - L + 1), 1 << 27):
                    m = min(1 << 27, n - L + 1 - a)
                    bit = one[code[a:a + m + L - 1].int()]
                    acc = torch.zeros(m, dtype=torch.uint8, device="cuda")
                    for i, mk in enumerate(masks):
                        if mk != 15:
                            acc += (bit[i:i + m] & mk) == 0
                        else:
                            acc += bit[i:i + m] == 0
                    at = torch.nonzero(acc <= p["k"]).flatten() + a
                    end = offs[torch.searchsorted(offs, at, right=True)]
                    at = at[at + L <= end]
                    found.append(at)
                    minus.append(torch.full_like(at, strand))
            at, strand = torch.cat(found), torch.cat(minus)
            w = code[at[:, None] + torch.arange(L, device="cuda")] if len(at) else code[:0].view(0, L)
            vals.append(_exact_tm_group(primer, w.long(), strand == 1, p))
            keys.append(at * 4 + primer_i * 2 + strand)
        tms.append(torch.cat(vals)[torch.cat(keys).argsort()])
    tms.append(torch.zeros(_room(case, pairs) - sum(len(t) for t in tms), dtype=torch.float64, device="cuda"))
    return torch.cat(tms)


def _exact_profile(train):
    """Move and emission scores (bits) of the profile of the training sequences, the first as reference."""
    ref = train[0].astype(np.int64)
    m = len(ref)
    ct, ce = np.zeros((m + 1, 3, 3)), np.zeros((m + 1, 4))
    for s in train:
        n = len(s)
        d = np.zeros((n + 1, m + 1), dtype=np.int64)
        d[0] = np.arange(m + 1)
        cols = np.arange(m + 1)
        for i in range(1, n + 1):
            best = np.empty(m + 1, dtype=np.int64)
            best[0] = i
            best[1:] = np.minimum(d[i - 1, :-1] + (ref != s[i - 1]), d[i - 1, 1:] + 1)
            d[i] = np.minimum.accumulate(best - cols) + cols  # a gap step costs 1 per column
        i, j, moves = n, m, []
        while i or j:
            if i and j and d[i, j] == d[i - 1, j - 1] + (ref[j - 1] != s[i - 1]):
                moves.append(0)
                i, j = i - 1, j - 1
            elif i and d[i, j] == d[i - 1, j] + 1:
                moves.append(1)
                i -= 1
            else:
                moves.append(2)
                j -= 1
        frm = col = pos = 0
        for to in reversed(moves):
            ct[col, frm, to] += 1
            if to != 1:
                col += 1
            if to == 0:
                ce[col, s[pos]] += 1
            if to != 2:
                pos += 1
            frm = to
        ct[m, frm, 0] += 1
    ct += 1
    ct[m, :, 2] = 0
    with np.errstate(divide="ignore"):
        t = np.log2(ct / ct.sum(2, keepdims=True))
    t[0, 2] = -np.inf
    e = np.log2((ce + 1) / (ce.sum(1, keepdims=True) + 4) * 4)
    e[0] = 0
    return t, e


def _exact_hmm(case, seed):
    train, amps = _family(case, seed)
    t, e = (torch.from_numpy(x).cuda() for x in _exact_profile(train))
    m, n = len(t) - 1, len(amps)
    lens = torch.tensor([len(a) for a in amps], device="cuda")
    rows = int(lens.max())
    letters = np.zeros((rows, n), dtype=np.int64)
    for i, a in enumerate(amps):
        letters[:len(a), i] = a
    letters = torch.from_numpy(letters).cuda()
    ln2 = math.log(2.0)
    neg = torch.full((n, 1), -math.inf, dtype=torch.float64, device="cuda")
    if case["forward"]:
        def add(*v):
            return torch.logsumexp(torch.stack(v) * ln2, 0) / ln2

        def along(v):
            return torch.logcumsumexp(v * ln2, 1) / ln2
    else:
        def add(*v):
            return torch.stack(v).amax(0)

        def along(v):
            return torch.cummax(v, 1).values
    tdd = torch.cat([torch.zeros(2, dtype=torch.float64, device="cuda"), t[1:m, 2, 2]]).cumsum(0)  # D_1 .. D_j

    def deletes(M, I):
        b = add(M[:, :-1] + t[:-1, 0, 2], I[:, :-1] + t[:-1, 1, 2])
        return torch.cat([neg, along(b - tdd[1:]) + tdd[1:]], 1)

    M = torch.full((n, m + 1), -math.inf, dtype=torch.float64, device="cuda")
    M[:, 0] = 0
    I = torch.full_like(M, -math.inf)
    D = deletes(M, I)
    score = torch.empty(n, dtype=torch.float64, device="cuda")
    for i in range(rows + 1):
        done = lens == i
        if bool(done.any()):
            score[done] = add(M[done, m] + t[m, 0, 0], I[done, m] + t[m, 1, 0], D[done, m] + t[m, 2, 0])
        if i == rows:
            break
        x = letters[i]
        nM = add(M[:, :-1] + t[:-1, 0, 0], I[:, :-1] + t[:-1, 1, 0], D[:, :-1] + t[:-1, 2, 0]) + e[1:, x].T
        I = add(M + t[:, 0, 1], I + t[:, 1, 1], D + t[:, 2, 1])
        M = torch.cat([neg, nM], 1)
        D = deletes(M, I)
    return score


def exact(case, seed):
    if case["kind"] == "hmm":
        return {"score": _exact_hmm(case, seed)}
    if case["kind"] == "run":
        return {"sites": None, "tm": _exact_site_tm(case, seed), "pass": None, "amps": None, "offs": None, "seq": None,
                "counts": None}
    if case["kind"] == "stages":
        return {"tm": _exact_site_tm(case, seed), "pass": None, "amps": None, "offs": None, "seq": None, "counts": None}
    return None
