"""The work whose speed this library is judged by: complete junction-detection builds.

Every case is one build of a genome set through the public entry points of
``paper_1602_05856_gb300.twopaco`` -- host strings through a ``Context``, a device-resident
``DeviceBuild`` launched kernel by kernel or replayed as a captured graph, or a streamed build
from page-locked host memory -- over the sizes, k-mer lengths, filter sizes, round counts and
options that the repository's configurations, tests and bench use.

Two recipes draw the genomes on the GPU, from the seed alone:

* ``star``: an ancestor with a repeat family and independent descendants of it (SNPs, short
  indels, a large deletion, inversions) -- the bacterial collections;
* ``tree``: ``genomes_gpu.mammal_set``, leaves of a random tree over an ancestor that is 45%
  repeats -- the mammal-scale sets.
"""
import numpy as np
import torch

from paper_1602_05856_gb300 import genomes_gpu
from paper_1602_05856_gb300 import twopaco as T

_BASES = dict(recipe="star", genomes=7, length=5_555_000, contigs=1, snp=0.01, indel=0.001, k=25,
              filter_log2=28, hashes=4, rounds=1, both_strands=True, split_at_n=False,
              partial=False, edges=False, api="graph")


def _case(name=None, **fields):
    c = dict(_BASES, **fields)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest served request: two windows of 0.1 Mbp, host strings in, host arrays out
        _case("served_small", genomes=2, length=100_000, filter_log2=21, api="host"),
        # a middling served request (0.1-50 Mbp windows, log-uniform: a few Mbp each), k = 31
        _case("served_k31", genomes=5, length=2_236_000, k=31, filter_log2=27, api="host"),
        # the plain single build: four 1 Mbp genomes, a 2^24-bit filter with three hashes
        _case("plain_single", genomes=4, length=1_000_000, snp=0.005, indel=0.0005, filter_log2=24,
              hashes=3),
        # the bacterial-scale set at k = 25: the everyday build, its filter inside L2
        _case("bacterial_k25"),
        # the same at k = 31 with the compacted graph's edges, launched call by call
        _case("bacterial_k31_edges", k=31, edges=True, api="launches"),
        # the paper's other k-mer length, k = 100 (four-word k-mers)
        _case("bacterial_k100", k=100),
        # draft assemblies: many contigs per genome, runs of N that end a string
        _case("drafts_split_n", length=3_000_001, genomes=12, contigs=57, split_at_n=True),
        # the batched 62-genome set in one build, a filter at the edge of L2
        _case("batched_k25", genomes=62, length=5_455_000, filter_log2=30),
        # the same genomes with two-word k-mers
        _case("batched_k63", genomes=62, length=5_455_000, k=63, filter_log2=30),
        # a slice of the mammal-scale set in four rounds, its filter beyond L2
        _case("tree_rounds4", recipe="tree", genomes=8, length=25_000_000, filter_log2=31, rounds=4),
        # a quarter of the mammal-scale set: 6 Gbp, four rounds, the headline's bits per base
        _case("tree_large", recipe="tree", genomes=8, length=750_000_000, filter_log2=34, rounds=4),
        # streamed from page-locked host memory, k = 31, a 1 GiB filter
        _case("tree_streamed_k31", recipe="tree", genomes=8, length=100_000_000, k=31, filter_log2=33,
              rounds=4, api="streamed"),
    ]


def _log_uniform(rng, lo, hi):
    return int(lo * (hi / lo) ** rng.random())


def draw(rng):
    """A served request, a bacterial collection or a mammal-scale set."""
    kind = rng.choice(("served", "star", "star", "star", "tree", "tree"))
    hashes = rng.choice((3, 4, 4, 5, 6))
    if kind == "served":
        genomes = rng.randint(2, 20)
        length = _log_uniform(rng, 100_000, 4_000_000) | 1
        return _case(genomes=genomes, length=length, k=rng.choice((25, 31)), hashes=hashes,
                     filter_log2=(8 * genomes * length - 1).bit_length(), api="host")
    if kind == "star":
        genomes = _log_uniform(rng, 2, 62)
        length = _log_uniform(rng, 300_000, 5_500_000) | 1
        split = rng.random() < 0.25
        return _case(genomes=genomes, length=length, hashes=hashes, snp=rng.choice((0.005, 0.01)),
                     contigs=rng.choice((1, 1, _log_uniform(rng, 2, 300))),
                     k=rng.choice((15, 21, 25, 25, 27, 31, 45, 63, 64, 100, 127)),
                     filter_log2=(rng.randint(4, 10) * genomes * length - 1).bit_length(),
                     both_strands=rng.random() < 0.9, split_at_n=split,
                     partial=rng.random() < 0.15, edges=rng.random() < 0.2,
                     api=rng.choice(("graph", "launches")))
    rounds = rng.choice((2, 3, 4, 4, 8, 16))
    length = _log_uniform(rng, 4_000_000, 500_000_000 * 4 // max(rounds, 4)) | 1
    return _case(recipe="tree", genomes=8, length=length, rounds=rounds, hashes=hashes,
                 k=rng.choice((21, 25, 25, 27, 31, 63)),
                 filter_log2=(rng.randint(6, 14) * 8 * length // rounds).bit_length(),
                 api=rng.choice(("graph", "graph", "streamed")) if length < 100_000_000 else "graph")


def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda")


def _codes(g, n, lo=0, hi=4):
    return torch.randint(lo, hi, (n,), dtype=torch.uint8, generator=g, device="cuda")


def _descendant(g, rng, anc, snp, indel):
    """The ancestor with a large deletion, SNPs, 1-10 bp indels and inversions (2-bit codes)."""
    cut = int(rng.integers(0, anc.numel() // 6 + 1))
    at = int(rng.integers(0, anc.numel() - cut + 1))
    s = torch.cat((anc[:at], anc[at + cut:]))
    n = s.numel()
    s = torch.where(_rand(g, n) < snp, (s + _codes(g, n, 1, 4)) % 4, s)
    event = _rand(g, n)
    count = torch.ones(n, dtype=torch.int64, device="cuda")
    size = _codes(g, n, 1, 11).long()
    count += torch.where(event < indel / 2, size, 0)  # insertions after a base
    gone = torch.zeros(n + 11, dtype=torch.int32, device="cuda")  # deletions: +1 at the start, -1 past the end
    d = torch.nonzero((event >= indel / 2) & (event < indel)).squeeze(1)
    gone.index_add_(0, d, torch.ones_like(d, dtype=torch.int32))
    gone.index_add_(0, d + size[d], -torch.ones_like(d, dtype=torch.int32))
    count[torch.cumsum(gone, 0)[:n] > 0] = 0
    at = torch.repeat_interleave(count)
    first = torch.ones(at.numel(), dtype=torch.bool, device="cuda")
    first[1:] = at[1:] != at[:-1]
    s = torch.where(first, s[at], _codes(g, at.numel()))
    for _ in range(s.numel() // 250_000):
        ln = int(rng.integers(1_000, 50_001))
        a = int(rng.integers(0, s.numel() - ln))
        s[a:a + ln] = 3 - torch.flip(s[a:a + ln], [0])
    return s


def _star(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    anc = _codes(g, case["length"])
    family = _codes(g, 1_500)
    for a in rng.integers(0, max(1, anc.numel() - 1_500), size=max(1, anc.numel() // 185_000)):
        anc[a:a + 1_500] = torch.where(_rand(g, 1_500) < 0.02, _codes(g, 1_500), family)
    ascii_of = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
    out = []
    for _ in range(case["genomes"]):
        s = ascii_of[_descendant(g, rng, anc, case["snp"], case["indel"]).long()]
        if case["split_at_n"]:  # assembly gaps: about 50 per Mbp, log-uniform lengths up to 5 kbp
            for a in rng.integers(0, s.numel(), size=max(1, s.numel() // 20_000)):
                s[a:a + int(np.exp(rng.uniform(0, np.log(5_000))))] = ord("n" if rng.random() < 0.1 else "N")
        cuts = np.sort(rng.integers(0, s.numel() + 1, size=case["contigs"] - 1))
        bounds = [0, *cuts.tolist(), s.numel()]
        out += [s[a:b] for a, b in zip(bounds[:-1], bounds[1:])]
    return out


def _genomes(case, seed):
    """(all bases in one CUDA tensor, string offsets)."""
    if case["recipe"] == "star":
        return genomes_gpu.concat_device(_star(case, seed))
    return genomes_gpu.concat_device(genomes_gpu.mammal_set(case["length"], case["genomes"], seed))


def _capacity(case):
    """Room for output positions, by the recipe alone: every position of a bacterial collection;
    of a mammal-scale set 27% are junctions."""
    return int(case["genomes"] * case["length"] * (1.02 if case["recipe"] == "star" else 0.31))


def _reserve(case, m):
    """(table slots, candidate-list units) as a program sizes a resident build's: half a table
    slot per base for a bacterial collection, as a served request does, and the measured shares
    of a mammal-scale set (a few percent of a round's positions are distinct candidates)."""
    if case["recipe"] == "tree":
        per_round = m // case["rounds"]
        return 1 << max(20, int(per_round * 0.15).bit_length()), per_round // 2
    return 1 << max(16, (m // 2 - 1).bit_length()), 0


def prepare(case, seed):
    bases, off = _genomes(case, seed)
    m = int(off[-1])
    bits = 1 << case["filter_log2"]
    opts = dict(hashes=case["hashes"], both_strands=case["both_strands"],
                split_at_n=case["split_at_n"], partial=case["partial"])
    if case["api"] == "host":
        b = bases.cpu().numpy()
        seqs = [b[int(off[t]):int(off[t + 1])] for t in range(len(off) - 1)]
        return {"case": case, "context": T.Context(), "seqs": seqs, "bits": bits,
                "options": T.Options(**opts), "counts": np.zeros(len(seqs), np.int64),
                "positions": np.zeros(_capacity(case), np.int64)}
    slots, records = _reserve(case, m)
    streamed = case["api"] == "streamed"
    host = bases.cpu().pin_memory() if streamed else None
    build = T.DeviceBuild(bases, off, case["k"], bits, case["rounds"],
                          T.Options(table_slots=slots, candidate_records=records, **opts),
                          capacity=_capacity(case), resident=not streamed)
    build.out_positions.zero_()
    state = {"case": case, "build": build}
    if streamed:
        state["host"] = host
        state["staging"] = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    if case["edges"]:  # at most one 56-byte edge per junction
        state["edge_offsets"] = torch.zeros(len(off), dtype=torch.int64, device="cuda")
        state["edges"] = torch.zeros((_capacity(case), 7), dtype=torch.int64, device="cuda")
    if case["api"] == "graph":
        build.capture()
    return state


def run(state):
    case = state["case"]
    if case["api"] == "host":  # the junctions into the program's own arrays, string by string
        found, _ = state["context"].build(state["seqs"], case["k"], state["bits"], case["rounds"],
                                          state["options"], copy=False)
        at = 0
        for t, pos in enumerate(found):
            state["positions"][at:at + pos.size] = pos.view(np.int64)
            state["counts"][t] = pos.size
            at += pos.size
        return {"counts": state["counts"], "positions": state["positions"]}
    b = state["build"]
    if case["api"] == "streamed":
        b.run_streamed(state["host"], state["staging"])
    else:
        b.run()
    out = {"offsets": b.out_offsets, "positions": b.out_positions}
    if case["edges"]:
        e = state["edges"]
        T.twopaco_edges_device(b.ws_ptr, b.offsets.data_ptr(), b.n_seqs, b.out_offsets.data_ptr(),
                               b.out_positions.data_ptr(), state["edge_offsets"].data_ptr(),
                               e.data_ptr(), e.shape[0], torch.cuda.current_stream().cuda_stream)
        out.update(edge_offsets=state["edge_offsets"], edges=e)
    return out


def work(case):
    """The input bytes read once and the outputs written once. The share of positions that are
    junctions is the recipe's: next to any of the other genomes' differences, or 26% on a tree."""
    m = case["genomes"] * case["length"]
    if case["recipe"] == "star":
        m *= 11 / 12  # the mean large deletion
        share = 1 - (1 - case["snp"] - case["indel"]) ** case["genomes"]
    else:
        share = 0.26
    return {"bytes": m * (1 + share * (8 + (56 if case["edges"] else 0))), "flops": 0}


def exact(case, seed):
    """The junction positions by their definition, with sorted k-mers: small sets of one-word
    k-mers on both strands."""
    if case["k"] > 31 or case["genomes"] * case["length"] > 2_000_000 or case["split_at_n"] or \
            case["partial"] or case["edges"] or not case["both_strands"]:
        return None
    bases, off = _genomes(case, seed)
    code = np.zeros(256, np.uint64)
    code[list(b"ACGT")] = range(4)
    x, k = code[bases.cpu().numpy()], case["k"]
    m, off = x.size, off.astype(np.int64)
    n = max(0, m - k + 1)
    f, r = np.zeros(n, np.uint64), np.zeros(n, np.uint64)
    for j in range(k):
        f = (f << np.uint64(2)) | x[j:j + n]
        r |= (np.uint64(3) - x[j:j + n]) << np.uint64(2 * j)
    string = np.searchsorted(off, np.arange(n), "right") - 1
    pos = np.flatnonzero(np.arange(n) + k <= off[string + 1])
    begins, ends = pos == off[string[pos]], pos + k == off[string[pos] + 1]
    before, after = x[np.maximum(pos - 1, 0)], x[np.minimum(pos + k, m - 1)]
    _, which = np.unique(np.minimum(f, r)[pos], return_inverse=True)
    mask = np.zeros(which.max(initial=-1) + 1, np.uint64)
    one = np.uint64(1)
    for here, pred, succ in ((f[pos] <= r[pos], before, after),
                             (r[pos] <= f[pos], np.uint64(3) - after, np.uint64(3) - before)):
        inner = here & ~begins & ~ends
        np.bitwise_or.at(mask, which[inner], (one << pred[inner]) | (np.uint64(16) << succ[inner]))
    np.bitwise_or.at(mask, which[begins | ends], np.uint64(256))
    several = np.array([bin(v & 15).count("1") > 1 or bin(v >> 4 & 15).count("1") > 1 or v >> 8
                        for v in range(512)], bool)
    found = pos[several[mask.astype(np.int64)][which]]
    at = np.searchsorted(found, off)
    positions = np.zeros(_capacity(case), np.int64)
    positions[:found.size] = found - off[string[found]]
    if case["api"] == "host":
        return {"counts": np.diff(at), "positions": positions}
    return {"offsets": at.astype(np.int64), "positions": positions}
