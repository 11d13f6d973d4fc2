"""The work that a user of this framework has it do, as cases that can be timed.

Every case goes through the public entry points of
``paper_0804_3643_gb300.binding`` as the README's examples and the serving
loop call them.  Inputs are the synthetic banks of
``paper_0804_3643_gb300.synth`` (its length, composition, homolog and
low-complexity model), in the sizes of that module's workloads and of the
benchmark.  All outputs are integer records (bytes), residue codes, offsets
or counts, so two correct versions give equal ones; no output is a floating
or rounded number, and there is no ``exact``.  Records go into buffers that
the caller keeps, sized once for the case and zero behind the records.

Kinds of case:

compare     two protein banks compared from their codes: both indexed, then
            searched (stages 0-3.1), optionally with the S0 filter
query       a few proteins against a resident, indexed bank: the query bank is
            indexed and searched, as the serving loop does for a batch
plan        a planned search of a fixed query bank against a resident bank,
            replayed as a CUDA graph
load        a large bank indexed, and a first query against it
ungapped    stages 1-2 alone on two indexed banks, the hits sorted
extend      stage 3.1 alone on a list of hits (``fixed``: the entry point that
            allocates nothing, into the caller's buffer)
align       stage 3.2 and the trace-back fields of a search's records
translated  a nucleotide bank translated in six frames, indexed and searched
            against proteins (``both``: against a second translated bank)
"""
import math

import numpy as np
import torch

from paper_0804_3643_gb300 import binding as B
from paper_0804_3643_gb300 import synth

RESIDUES = 331.0        # mean residues of a synthetic protein
PAIR_RATE = 1.97e-4     # pairs of equal key per pair of residues
HIT_RATE = 1.76e-3      # stage-2 hits per pair at S1 = 38 (ordinary banks)
LOW_HIT_RATE = 2.2e-2   # the same for banks with low-complexity runs


def listed():
    return [
        # the whole comparison at the size of the headline benchmark
        {"name": "compare 10000x100000", "kind": "compare", "n1": 10000, "n2": 100000, "planted": 0.05},
        # a small comparison, where launches, copies and waits count
        {"name": "compare 200x2000", "kind": "compare", "n1": 200, "n2": 2000, "planted": 0.10},
        # banks with low-complexity runs: few keys hold most pairs, and one pair in some forty is a hit
        {"name": "compare low complexity", "kind": "compare", "n1": 10000, "n2": 10000, "planted": 0.0, "lowc": 0.20},
        # the lossy filter of Section 4.2, at sizes that are no round numbers
        {"name": "compare filtered", "kind": "compare", "n1": 3001, "n2": 29989, "planted": 0.05, "s0": 53},
        # a serving batch of the mean request size against the resident bank
        {"name": "query 250 resident", "kind": "query", "n1": 250, "n2": 1000000},
        # the smallest request: latency
        {"name": "query 2 resident", "kind": "query", "n1": 2, "n2": 1000000},
        # a fixed query set replayed as a CUDA graph
        {"name": "plan 20 replayed", "kind": "plan", "n1": 20, "n2": 200000},
        # a service's start: the bank indexed, and its first query
        {"name": "load 500000", "kind": "load", "n1": 1, "n2": 500000},
        # the ungapped hits themselves, sorted
        {"name": "ungapped 1000x20000", "kind": "ungapped", "n1": 1000, "n2": 20000, "planted": 0.05},
        # stage 3.1 for a caller that allocates nothing
        {"name": "extend 60001 fixed", "kind": "extend", "hits": 60001, "fixed": True},
        # full gapped alignments of the headline comparison's records
        {"name": "align 10000x100000", "kind": "align", "n1": 10000, "n2": 100000, "planted": 0.05},
        # proteins against a translated nucleotide bank
        {"name": "translated 2000x20M", "kind": "translated", "n1": 2000, "nt": 20000000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compare", "compare", "low", "filtered", "query", "plan", "load", "ungapped", "extend", "align",
                       "translated"])
    c = {"kind": kind}
    if kind in ("compare", "filtered", "align"):
        c.update(n1=_log(rng, 200, 10000), n2=_log(rng, 2000, 100000), planted=rng.choice([0.0, 0.05, 0.1]))
    elif kind == "low":
        c.update(kind="compare", n1=_log(rng, 1000, 10000), n2=_log(rng, 1000, 10000), planted=0.0,
                 lowc=rng.choice([0.05, 0.1, 0.2]))
    elif kind == "query":
        c.update(n1=_log(rng, 1, 500), n2=_log(rng, 100000, 1000000))
        if rng.random() < 0.3:
            c["align"] = True  # the service's other answer: alignments
    elif kind == "plan":
        c.update(n1=_log(rng, 1, 250), n2=_log(rng, 20000, 500000))
    elif kind == "load":
        c.update(n1=_log(rng, 1, 4), n2=_log(rng, 50000, 800000))
    elif kind == "ungapped":
        c.update(n1=_log(rng, 200, 3000), n2=_log(rng, 2000, 50000), planted=0.05)
    elif kind == "extend":
        c.update(hits=_log(rng, 100, 4000000))
        c["fixed"] = c["hits"] <= 65536 and rng.random() < 0.5
    else:
        c.update(n1=_log(rng, 100, 4000), nt=_log(rng, 300000, 30000000))
        if rng.random() < 0.3:
            c.update(n1=max(10, c["n1"] // 4), both=True)
    if c["kind"] == "filtered":
        c.update(kind="compare", s0=rng.choice([45, 53, 60]))
    if c["kind"] != "load" and rng.random() < 0.25:
        # BLAST's other gap costs for BLOSUM62, and a threshold beside the calibrated one
        c.update(gap_open=rng.choice([9, 10, 12]), gap_extend=rng.choice([1, 2]), s1=rng.choice([36, 40, 44]))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _params(case):
    own = {k: case[k] for k in ("gap_open", "gap_extend", "s1") if k in case}
    return B.plast_default_params(**own) if own else None


def _codes(bank):
    d = B.DeviceBank.from_host(bank.codes, bank.seq_off)
    return d.codes, d.seq_off


def _zeros(n, nbytes):
    return torch.zeros(n * nbytes, dtype=torch.uint8, device="cuda")


def _residues(case):
    """Expected residues of the two banks that are searched."""
    if case["kind"] == "translated":
        return (2.0 * 1024 if case.get("both") else RESIDUES) * case["n1"], 2.0 * case["nt"]
    return RESIDUES * case["n1"], RESIDUES * case["n2"]


def _room(case, hits=False):
    """Records (or stage-2 hits) that the caller's buffer holds: two to three times what such banks give."""
    r1, r2 = _residues(case)
    pairs = PAIR_RATE * r1 * r2
    if case.get("lowc"):
        return int(4e-2 * pairs) + 500000
    return int((5e-3 if hits else 7e-4) * pairs) + int(300 * case.get("planted", 0.0) * case.get("n2", 0)) + 100000


def _pair(case, seed):
    """(bank 1, bank 2) on the host, bank 2 carrying homologs of bank 1."""
    rng = np.random.default_rng(seed)
    lowc = case.get("lowc", 0.0)
    b1 = synth.protein_bank(rng, case["n1"], lowcomplex_frac=lowc)
    b2 = synth.protein_bank(rng, case["n2"], homolog_source=b1, planted_frac=case["planted"], lowcomplex_frac=lowc)
    return b1, b2


def _large_bank(rng, n):
    """(codes, offsets) of n background proteins, the residues drawn on the device."""
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(synth.protein_lengths(rng, n), out=off[1:])
    g = torch.Generator(device="cuda")
    g.manual_seed(int(rng.integers(1 << 62)))
    cdf = torch.from_numpy(np.cumsum(synth.RR_FREQ)).to("cuda", torch.float32)
    codes = torch.empty(int(off[-1]), dtype=torch.int8, device="cuda")
    step = 1 << 26
    for s in range(0, codes.numel(), step):
        u = torch.rand(min(step, codes.numel() - s), generator=g, device="cuda")
        codes[s:s + u.numel()] = torch.searchsorted(cdf, u, right=True).clamp_(max=19).to(torch.int8)
    return codes, torch.from_numpy(off).cuda()


def _indexed(bank):
    return B.plast_index_bank(*_codes(bank))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "params": _params(case)}
    if kind in ("compare", "query", "load", "translated"):
        st["out"] = _zeros(_room(case), B.GAPPED_BYTES)
    if kind == "compare":
        b1, b2 = _pair(case, seed)
        st.update(q=_codes(b1), t=_codes(b2))
    elif kind in ("query", "plan", "load"):
        rng = np.random.default_rng(seed)
        st["q"] = _codes(synth.random_protein_bank(rng, case["n1"]))
        large = _large_bank(rng, case["n2"])
        if kind == "load":
            st["t"] = large
        else:
            st["bank"] = B.plast_index_bank(*large)
        if kind == "plan":
            st["plan"] = B.Plan(B.plast_index_bank(*st["q"]), st["bank"], max_hits=_room(case, hits=True),
                                max_records=_room(case), params=st["params"])
            st["plan"].records.zero_()
            st["stream"] = torch.cuda.Stream()
            st["plan"].capture(st["stream"])
        elif case.get("align"):
            st["alignments"] = _zeros(_room(case), B.ALIGN_BYTES)
    elif kind in ("ungapped", "align"):
        b1, b2 = _pair(case, seed)
        st.update(g1=_indexed(b1), g2=_indexed(b2))
        if kind == "align":
            st["records"] = B.plast_search(st["g1"], st["g2"], st["params"])
            st["alignments"] = _zeros(_room(case), B.ALIGN_BYTES)
        else:
            st["out"] = _zeros(_room(case, hits=True), B.HIT_BYTES)
    elif kind == "extend":
        n1 = 30 + int(math.sqrt(case["hits"] / 0.2))
        b1, b2 = _pair({"n1": n1, "n2": 10 * n1, "planted": 0.05}, seed)
        st.update(g1=_indexed(b1), g2=_indexed(b2))
        st["hits"] = B.plast_ungapped(st["g1"], st["g2"])[:case["hits"]].clone()
        st["out"] = _zeros(case["hits"], B.GAPPED_BYTES)
    else:
        rng = np.random.default_rng(seed)
        src = synth.protein_bank(rng, case["n1"])
        longest = min(100000, case["nt"] // 4)
        dna = synth.dna_bank(rng, case["nt"], proteins=src, n_planted=max(1, case["nt"] // 25000), max_contig=longest)
        st["dna"] = _codes(dna)
        st["aa"] = _zeros(2 * (case["nt"] + longest), 1).view(torch.int8)
        if case.get("both"):
            nt = max(3000, case["n1"] * 1024)
            st["dna_q"] = _codes(synth.dna_bank(rng, nt, proteins=src, n_planted=max(1, case["n1"] // 5),
                                                min_contig=600, max_contig=1450))
        else:
            st["q"] = _codes(src)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _translated_bank(dna):
    codes, off = dna
    aa, seq_off, _ = B.plast_translate6(codes.view(torch.uint8), off)
    return B.plast_index_bank(aa, seq_off), aa


def _aligned(st, g1, g2, records):
    alignments, extended = B.plast_full_gapped(g1, g2, records, st["params"])
    st["alignments"][:alignments.numel()].copy_(alignments.view(-1))
    return {"alignments": st["alignments"], "kept": len(alignments), "extended": extended}


def run(st):
    case, prm = st["case"], st["params"]
    kind = case["kind"]
    if kind == "compare":
        g1, g2 = B.plast_index_bank(*st["q"]), B.plast_index_bank(*st["t"])
        records, hits = B.plast_search_ex(g1, g2, prm, s0=case.get("s0", 0), out=st["out"])
        return {"records": st["out"], "kept": len(records), "hits": hits}
    if kind in ("query", "load"):
        bank = B.plast_index_bank(*st["t"]) if kind == "load" else st["bank"]
        q = B.plast_index_bank(*st["q"])
        records = B.plast_search(q, bank, prm, out=st["out"])
        got = {"records": st["out"], "kept": len(records)}
        return {**got, **_aligned(st, q, bank, records)} if case.get("align") else got
    if kind == "plan":
        st["plan"].launch(st["stream"])
        records, hits = st["plan"].result(st["stream"])
        return {"records": st["plan"].records, "kept": len(records), "hits": hits}
    if kind == "ungapped":
        hits = B.plast_ungapped(st["g1"], st["g2"], prm, out=st["out"])
        return {"hits": st["out"], "kept": len(hits)}
    if kind == "extend":
        if case["fixed"]:
            records = B.plast_small_gapped_noalloc(st["g1"], st["g2"], st["hits"], st["out"], prm)
        else:
            records = B.plast_small_gapped(st["g1"], st["g2"], st["hits"], prm, out=st["out"])
        return {"records": st["out"], "kept": len(records)}
    if kind == "align":
        return _aligned(st, st["g1"], st["g2"], st["records"])
    bank, aa = _translated_bank(st["dna"])
    q = _translated_bank(st["dna_q"])[0] if case.get("both") else B.plast_index_bank(*st["q"])
    records = B.plast_search(q, bank, prm, out=st["out"])
    st["aa"][:aa.numel()].copy_(aa)
    return {"records": st["out"], "kept": len(records), "aa": st["aa"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
UNGAPPED_OPS = 48 * 2               # per pair: an add and a maximum per cell of the window
SMALL_OPS = 2 * 64 * 17 * 5         # per hit: two sides of 64 rows x 17 band cells, three maxima and two adds each
FULL_OPS = 6450 * 5                 # per record: the mean cells of its two sides


def work(case):
    kind = case["kind"]
    if kind == "extend":
        hits = case["hits"]
        return {"bytes": hits * (B.HIT_BYTES + 2 * 145 + 0.2 * B.GAPPED_BYTES), "flops": hits * SMALL_OPS}
    r1, r2 = _residues(case)
    pairs = PAIR_RATE * r1 * r2
    hits = pairs * (LOW_HIT_RATE if case.get("lowc") else HIT_RATE)
    records = hits * (0.9 if case.get("lowc") else 0.13)
    if kind == "align":
        return {"bytes": r1 + r2 + records * (B.GAPPED_BYTES + 0.65 * B.ALIGN_BYTES), "flops": records * FULL_OPS}
    codes = r1 + r2
    if kind == "translated":
        codes = r1 + case["nt"] + r2
    elif kind in ("query", "plan"):  # of the resident bank, the words whose key the query has
        codes = r1 + r2 * (1.0 - math.exp(-r1 / B.NKEYS))
    flops = pairs * UNGAPPED_OPS
    if kind == "ungapped":
        return {"bytes": codes + hits * B.HIT_BYTES, "flops": flops}
    flops += hits * SMALL_OPS
    out = records * B.GAPPED_BYTES
    if case.get("align"):
        flops += records * FULL_OPS
        out += records * 0.65 * B.ALIGN_BYTES
    return {"bytes": codes + out, "flops": flops}
