"""Performance cases of the overlap-and-layout path: what a user of the package has it do, through
its public entry points, from the smallest read sets to the largest.

A case names one operation and a read set (genome length, coverage, read lengths, errors, repeats)
with the parameters of the call. Inputs are drawn on the GPU from the seed, with the same recipe as
the repository's synthetic workloads: uniform genomes with optional diverged repeat families, long
reads of lognormal length from both strands with insertions, deletions and substitutions (3:2:1),
and an overlap graph R built from the reads' true coordinates. The sizes of a case's outputs are
the case's own: its genome and reads are drawn once from the case, and the seed decides which of
their many equivalent forms is the input -- the order of the reads, the strand each was read from
and the naming of the bases -- so that every read id, k-mer code, position and edge differs between
seeds. Every output is a whole number, so there is nothing to approximate: results are compared
for equality.
"""
import math
import random
import zlib

import numpy as np
import torch

import paper_2010_10055_gb300 as sg

ASCII = (65, 67, 71, 84)  # A C G T


# ------------------------------------------------------------------------------------ cases
def _case(name, op, G, coverage, mean, err, k=17, hi=20, t=2, seeds=2, fuzz=1000, min_overlap=1000, mode=0,
          repeats="none", **more):
    c = dict(op=op, G=int(G), coverage=float(coverage), mean=float(mean), sd=0.4 * float(mean), err=float(err), k=k,
             lo=2, hi=hi, min_shared=t, max_seeds=seeds, fuzz=fuzz, min_overlap=min_overlap, mode=mode,
             repeats=repeats, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest read set of the repository: a plasmid-sized genome, all three operations.
        # Nothing here is large; calls, launches and read-backs are what it costs.
        _case("step-50kbp-10x", "step", 50_000, 10, 2000, 0.12, hi=8, fuzz=0, min_overlap=1),
        # Reads -> A, At for one bacterial genome at 30x with noisy long reads.
        _case("kmer-5Mbp-30x", "kmer", 5_000_000, 30, 10000, 0.15, hi=20, repeats="bacterial"),
        # The same call on accurate reads with long k-mers: most windows recur, and the code fills
        # a 64-bit word on its own.
        _case("kmer-12Mbp-25x-k31", "kmer", 12_000_000, 25, 10000, 0.01, k=31, hi=50, repeats="bacterial"),
        # C = A At for the bacterial genome, A and At already there (a parameter sweep over
        # min_shared, or k-mers selected elsewhere).
        _case("overlap-5Mbp-30x", "overlap", 5_000_000, 30, 10000, 0.15, hi=20, repeats="bacterial"),
        # C = A At for a small eukaryote, where chance k-mers and repeat copies outnumber true overlaps.
        _case("overlap-25Mbp-40x", "overlap", 25_000_000, 40, 10000, 0.15, hi=30, repeats="eukaryote"),
        # Transitive reduction of a bacterial overlap graph (about 0.6 M edges).
        _case("reduce-5Mbp-30x", "reduce", 5_000_000, 30, 10000, 0.15),
        # Transitive reduction of the overlap graph of a 100 Mbp genome (about 22 M edges).
        _case("reduce-100Mbp-40x", "reduce", 100_000_000, 40, 10000, 0.15),
        # Overlap graph estimated from C's seeds, then reduced in the other modes: drifting
        # offsets and false overlaps, more rounds.
        _case("seeds-5Mbp-30x", "seeds", 5_000_000, 30, 10000, 0.15, hi=20, repeats="bacterial", mode=3),
        # Many independent read sets (20 kbp to 2 Mbp genomes) in one batched call.
        _case("batch-64-sets", "batch", 2_000_000, 25, 6000, 0.135, min_overlap=500, count=64, G_min=20_000),
        # The whole path from host buffers to host buffers, as a program with reads from a file runs it.
        _case("host-5Mbp-30x", "host", 5_000_000, 30, 10000, 0.15, hi=20, repeats="bacterial"),
        # The largest single-GPU read set: a 100 Mbp genome at 40x (4.1 Gbp of reads), all three operations.
        _case("step-100Mbp-40x", "step", 100_000_000, 40, 10000, 0.15, hi=30, repeats="eukaryote"),
    ]


def draw(rng: random.Random):
    """One more case: an operation on a genome of any length up to the listed ones' largest, with
    coverage, read length, errors and call parameters of the batched and served workloads."""
    op = rng.choice(["step", "kmer", "kmer", "overlap", "overlap", "reduce", "seeds", "batch", "host"])
    top = dict(step=100e6, kmer=100e6, overlap=25e6, reduce=100e6, seeds=5e6, batch=2e6, host=5e6)[op]
    low = 2e5 if op == "batch" else 5e4
    G = int(math.exp(rng.uniform(math.log(low), math.log(top))))
    coverage = round(rng.uniform(10, 40), 2)
    mean = round(rng.uniform(2000, 10000))
    k = rng.choice([17, 17, 17, 17, 15, 19, 21, 31]) if G > 1_000_000 else rng.choice([17, 17, 15, 21, 31])
    err = round(rng.uniform(0.12, 0.15) if k <= 19 else rng.uniform(0.005, 0.03), 4)
    more = dict(count=rng.randint(8, 64), G_min=20_000) if op == "batch" else {}
    if op == "batch":
        k = 17
        err = round(rng.uniform(0.12, 0.15), 4)
    return _case(None, op, G, coverage, mean, err, k=k, hi=max(8, round((0.75 if k <= 19 else 2.0) * coverage)),
                 t=rng.choice([2, 2, 2, 3]), seeds=rng.choice([2, 2, 2, 1, 3]), fuzz=rng.choice([0, 500, 1000, 1000]),
                 min_overlap=rng.choice([500, 1000]), mode=rng.choice([0, 0, 1, 2, 3]),
                 repeats=rng.choice(["none", "bacterial", "eukaryote"]) if op != "batch" else "none", **more)


# ----------------------------------------------------------------------------------- inputs
def _genome(gen, pyr, G, repeats):
    """2-bit codes of a uniform genome with its repeat families: 'bacterial' 2 families of 5 copies
    per Mbp (5-8 kbp, 1 % divergence); 'eukaryote' 2 % of the genome in families of 2-200 copies
    (1-10 kbp, 0.5-3 %)."""
    dev = gen.device
    g = torch.randint(0, 4, (G,), dtype=torch.uint8, device=dev, generator=gen)
    want = {"none": 0, "bacterial": int(0.065 * G), "eukaryote": int(0.02 * G)}[repeats]
    done = 0
    while done < want:
        if repeats == "bacterial":
            length, copies, div = pyr.randint(5000, 8000), 5, 0.01
        else:
            length = pyr.randint(1000, 10000)
            copies = int(math.exp(pyr.uniform(math.log(2), math.log(200))))
            div = pyr.uniform(0.005, 0.03)
        if length * 2 > G:
            break
        copies = max(2, min(copies, (want - done) // length + 1))
        fam = torch.randint(0, 4, (length,), dtype=torch.uint8, device=dev, generator=gen)
        for _ in range(copies):
            at = pyr.randint(0, G - length)
            sub = torch.rand(length, device=dev, generator=gen) < div
            alt = (fam + torch.randint(1, 4, (length,), dtype=torch.uint8, device=dev, generator=gen)) & 3
            copy = torch.where(sub, alt, fam)
            g[at:at + length] = copy if pyr.random() < 0.5 else 3 - copy.flip(0)
        done += length * copies
    return g


def _coordinates(gen, G, coverage, mean, sd):
    """Template intervals and strands of the reads: lognormal lengths of at least 500 bases."""
    dev = gen.device
    n = max(4, round(coverage * G / mean))
    s2 = math.log(1 + (sd / mean) ** 2)
    z = torch.randn(n, dtype=torch.float64, device=dev, generator=gen)
    length = torch.exp(math.log(mean) - s2 / 2 + math.sqrt(s2) * z).long().clamp(min(500, G), G)
    start = (torch.rand(n, dtype=torch.float64, device=dev, generator=gen) * (G - length + 1)).long()
    strand = torch.randint(0, 2, (n,), dtype=torch.int64, device=dev, generator=gen)
    return start, start + length, strand


def _reads(gen, g, start, end, strand, err):
    """ASCII bases and offsets of the reads: each template base is deleted (err / 3), substituted
    (err / 6) or copied, then a random base is inserted (err / 2)."""
    dev = g.device
    ascii_ = torch.tensor(ASCII, dtype=torch.uint8, device=dev)
    p_ins, p_del, p_sub = err / 2, err / 3, err / 6
    length = end - start
    total = torch.cumsum(length, 0).cpu().numpy()
    parts, sizes, i0 = [], [], 0
    while i0 < length.numel():  # about 128 M template bases at a time
        done = int(total[i0 - 1]) if i0 else 0
        i1 = max(i0 + 1, int(np.searchsorted(total, done + (1 << 27), side="right")))
        L = length[i0:i1]
        N = int(total[i1 - 1]) - done
        base = torch.cumsum(L, 0) - L
        r = torch.repeat_interleave(torch.arange(i1 - i0, device=dev), L, output_size=N)
        local = torch.arange(N, device=dev) - base[r]
        rev = strand[i0:i1][r] == 1
        b = g[torch.where(rev, end[i0:i1][r] - 1 - local, start[i0:i1][r] + local)]
        b = torch.where(rev, 3 - b, b)
        u = torch.rand(N, device=dev, generator=gen)
        b = torch.where((u >= p_del) & (u < p_del + p_sub),
                        (b + torch.randint(1, 4, (N,), dtype=torch.uint8, device=dev, generator=gen)) & 3, b)
        keep = u >= p_del
        ins = torch.rand(N, device=dev, generator=gen) < p_ins
        cnt = keep.to(torch.uint8) + ins.to(torch.uint8)
        to = torch.cumsum(cnt, 0, dtype=torch.int64)
        out = ascii_[torch.randint(0, 4, (int(to[-1]),), device=dev, generator=gen)]
        first = to - cnt
        out[first[keep]] = ascii_[b[keep].long()]
        ends = to[base + L - 1]
        sizes.append(torch.diff(ends, prepend=torch.zeros(1, dtype=torch.int64, device=dev)))
        parts.append(out)
        i0 = i1
    off = torch.zeros(length.numel() + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(sizes), 0, out=off[1:])
    return (torch.cat(parts) if len(parts) > 1 else parts[0]), off


def _overlap_graph(start, end, strand, min_overlap):
    """R from true coordinates: every pair overlapping by min_overlap or more, neither contained in
    the other; for a starting first, R_ab = (e_b - e_a, 2 s_a + s_b) and
    R_ba = (s_b - s_a, 2 (1 - s_b) + (1 - s_a))."""
    dev, n = start.device, start.numel()
    order = torch.argsort(start, stable=True)
    s, e = start[order], end[order]
    hi = torch.searchsorted(s, e - min_overlap, right=True)
    cnt = (hi - torch.arange(n, device=dev) - 1).clamp(min=0)
    a = torch.repeat_interleave(torch.arange(n, device=dev), cnt)
    b = a + 1 + torch.arange(a.numel(), device=dev) - (torch.cumsum(cnt, 0) - cnt)[a]
    ok = (s[b] > s[a]) & (e[b] > e[a])
    a, b = order[a[ok]], order[b[ok]]
    row, col = torch.cat([a, b]), torch.cat([b, a])
    suffix = torch.cat([end[b] - end[a], start[b] - start[a]])
    d = torch.cat([2 * strand[a] + strand[b], 2 * (1 - strand[b]) + (1 - strand[a])])
    by = torch.argsort(row * n + col)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.bincount(row, minlength=n), 0, out=rp[1:])
    return sg.DeviceGraph(n, rp, col[by].int(), suffix[by].int(), d[by].to(torch.uint8))


def _reordered(seq, off, perm, flip, table):
    """Read perm[i] of (seq, off) as read i, reverse-complemented where flip[i], bases renamed by table."""
    dev = seq.device
    length = (off[1:] - off[:-1])[perm]
    new = torch.zeros_like(off)
    torch.cumsum(length, 0, out=new[1:])
    lut = torch.zeros(2, 256, dtype=torch.uint8, device=dev)
    for x in range(4):  # table[3 - x] == 3 - table[x]: complements stay complements
        lut[0, ASCII[x]] = ASCII[table[x]]
        lut[1, ASCII[x]] = ASCII[3 - table[x]]
    lut = lut.reshape(-1)
    out = torch.empty_like(seq)
    ends, i0, n = new[1:].cpu().numpy(), 0, perm.numel()
    while i0 < n:
        done = int(ends[i0 - 1]) if i0 else 0
        i1 = max(i0 + 1, int(np.searchsorted(ends, done + (1 << 27), side="right")))
        N = int(ends[i1 - 1]) - done
        r = i0 + torch.repeat_interleave(torch.arange(i1 - i0, device=dev), length[i0:i1], output_size=N)
        local = torch.arange(done, done + N, device=dev) - new[r]
        at = off[perm[r]] + torch.where(flip[r] == 1, length[r] - 1 - local, local)
        out[done:done + N] = lut[seq[at].long() + 256 * flip[r]]
        i0 = i1
    return out, new


def _read_set(case, G, seed, reads=True, graph=True):
    shape = [case["op"] == "seeds", G, case["repeats"]] + [case[k] for k in ("coverage", "mean", "sd", "err")]
    own = zlib.crc32(repr(shape).encode())
    gen = torch.Generator(device="cuda")
    gen.manual_seed(own)
    start, end, strand = _coordinates(gen, G, case["coverage"], case["mean"], case["sd"])
    if reads:
        g = _genome(gen, random.Random(own), G, case["repeats"])
        seq, off = _reads(gen, g, start, end, strand, case["err"])
    gen.manual_seed(seed)
    perm = torch.randperm(start.numel(), device="cuda", generator=gen)
    # which seed of a pair comes first depends on the naming: where R is estimated from it, the
    # reads are only reordered
    fixed = case["op"] == "seeds"
    flip = torch.randint(0, 1 if fixed else 2, perm.shape, device="cuda", generator=gen)
    pyr = random.Random(seed)
    first = 0 if fixed else pyr.randrange(4)
    second = 1 if fixed else pyr.choice([x for x in range(4) if x not in (first, 3 - first)])
    start, end, strand = start[perm], end[perm], strand[perm] ^ flip
    out = {}
    if graph:
        out["R"] = _overlap_graph(start, end, strand, case["min_overlap"])
    if reads:
        out["seq"], out["off"] = _reordered(seq, off, perm, flip, (first, second, 3 - second, 3 - first))
    return out


def prepare(case, seed):
    op, G, base = case["op"], case["G"], int(seed) * 1009 + 17
    c = dict(case)
    if op == "batch":
        pyr = random.Random(zlib.crc32(repr([case["count"], G, case["G_min"]]).encode()))
        items = []
        for b in range(case["count"]):  # sets of the case, each in the form of this seed
            Gb = int(math.exp(pyr.uniform(math.log(case["G_min"]), math.log(G))))
            cov, mean = pyr.uniform(10, 40), pyr.uniform(2000, 10000)
            d = _read_set(dict(c, coverage=cov, mean=mean, sd=0.4 * mean), Gb, base + 1 + b)
            items.append(dict(seq=d["seq"], offsets=d["off"], lo=2, hi=max(8, round(0.75 * cov)), R=d["R"]))
        return dict(case=c, items=items)
    d = _read_set(c, G, base, reads=op != "reduce", graph=op in ("reduce", "step", "host"))
    if op == "host":
        R = {k: getattr(d["R"], k).cpu().numpy() for k in ("row_ptr", "col", "suffix", "dir")}
        params = type("Params", (), {p: case[p] for p in ("k", "lo", "hi", "min_shared", "max_seeds", "fuzz")})
        return dict(case=c, seq=d["seq"].cpu().numpy(), off=d["off"].cpu().numpy(), R=dict(R, n=d["R"].n),
                    params=params, pipeline=sg.HostPipeline())
    if op in ("overlap", "seeds"):
        km = sg.build_kmer_matrix(d["seq"], d["off"], case["k"], case["lo"], case["hi"])
        if op == "overlap":
            return dict(case=c, km=km)
        C = sg.overlap_spgemm(km, case["min_shared"], case["max_seeds"])
        return dict(case=c, C=C, off=d["off"])
    return dict(case=c, **d)


# -------------------------------------------------------------------------------------- run
class _Array:
    """A device array of a batch's result (the struct's pointer) as a tensor; keeps the result alive."""

    def __init__(self, ptr, n, kind, owner):
        self.__cuda_array_interface__ = dict(shape=(int(n),), typestr=kind, data=(int(ptr), False), version=3)
        self.owner = owner


def _batch_tensors(res):
    r = res.r

    def view(ptr, n, kind):
        return torch.as_tensor(_Array(ptr, n, kind, res), device="cuda") if n else torch.empty(0, device="cuda")

    def csr(m):
        return [view(m.row_ptr, m.n_rows + 1, "<i8"), view(m.col, m.nnz, "<i4"), view(m.val, m.nnz, "<i4")]

    C, S = r.C, r.S
    return dict(A=csr(r.A), At=csr(r.At), codes=view(r.d_kmer_codes, r.A.n_cols, "<i8"),
                C=[view(C.row_ptr, C.n + 1, "<i8"), view(C.col, C.nnz, "<i4"), view(C.count, C.nnz, "<i4"),
                   view(C.seed_i, C.max_seeds * C.nnz, "<i4"), view(C.seed_k, C.max_seeds * C.nnz, "<i4")],
                S=[view(S.row_ptr, S.n + 1, "<i8"), view(S.col, S.nnz, "<i4"), view(S.suffix, S.nnz, "<i4"),
                   view(S.dir, S.nnz, "|u1")],
                read_off=res.read_off, col_off=res.col_off, iterations=res.iterations)


def run(state):
    c, op = state["case"], state["case"]["op"]
    if op == "batch":
        return _batch_tensors(sg.run_batch(state["items"], c["k"], c["min_shared"], c["max_seeds"], c["fuzz"], c["mode"]))
    if op == "host":
        return state["pipeline"].run(state["seq"], state["off"], state["params"], state["R"], c["mode"])
    if op == "reduce":
        S, rounds = sg.transitive_reduce(state["R"], c["fuzz"], c["mode"])
        return dict(S=S.tensors(), rounds=rounds)
    if op == "overlap":
        return dict(C=sg.overlap_spgemm(state["km"], c["min_shared"], c["max_seeds"]).tensors())
    if op == "seeds":
        R = sg.overlap_graph_from_seeds(state["C"], state["off"], c["k"], c["min_overlap"])
        S, rounds = sg.transitive_reduce(R, c["fuzz"], c["mode"])
        return dict(R=R.tensors(), S=S.tensors(), rounds=rounds)
    km = sg.build_kmer_matrix(state["seq"], state["off"], c["k"], c["lo"], c["hi"])
    out = dict(A=km.A.tensors(), At=km.At.tensors(), codes=km.codes())
    if op == "step":
        out["C"] = sg.overlap_spgemm(km, c["min_shared"], c["max_seeds"]).tensors()
        S, rounds = sg.transitive_reduce(state["R"], c["fuzz"], c["mode"])
        out.update(S=S.tensors(), rounds=rounds)
    return out


# ------------------------------------------------------------------------------------- work
def _sizes(c, G, coverage, mean):
    """Expected sizes of one read set: reads, bases, nnz(A), columns, nnz(C), nnz(R), nnz(S)."""
    total = coverage * G * (1 + c["err"] / 2 - c["err"] / 3)
    n = coverage * G / mean
    right = (1 - c["err"]) ** c["k"]          # windows without an error
    true = coverage * right                    # occurrences of a genome k-mer
    chance = total / (4.0 ** c["k"] / 2)       # occurrences of any other code
    nnz = total * (right * (1 - math.exp(-true)) + (1 - right) * (1 - math.exp(-chance)))
    m = (G * max(0.0, 1 - (1 + true) * math.exp(-true))
         + 4.0 ** c["k"] / 2 * max(0.0, 1 - (1 + chance) * math.exp(-chance)))
    m = min(m, nnz / 2)
    # overlapping reads; repeats of up to 200 copies add the reads of the other copies
    nnz_c = n * 2 * coverage * (1 if c["repeats"] != "eukaryote" else 5)
    nnz_r = n * coverage * max(0.1, 1 - c["min_overlap"] / mean) * 0.65
    return dict(total=total, n=n, nnz=nnz, m=m, nnz_c=nnz_c, nnz_r=nnz_r, nnz_s=min(nnz_r, 6 * n))


def work(case):
    """Bytes of each input read once and each output written once. Integer work: no flops."""
    op = case["op"]
    if op == "batch":  # genomes log-uniform in [G_min, G], coverage 10-40, reads 2-10 kbp
        lo, hi = case["G_min"], case["G"]
        z = _sizes(case, (hi - lo) / math.log(hi / lo), 25.0, 5000.0)
        z = {k: v * case["count"] for k, v in z.items()}
    else:
        z = _sizes(case, case["G"], case["coverage"], case["mean"])
    reads = z["total"] + 8 * z["n"]
    a_at = 16 * z["nnz"] + 8 * z["n"] + 16 * z["m"]         # A and At (col, val), row pointers, codes
    c = (8 + 8 * case["max_seeds"]) * z["nnz_c"] + 8 * z["n"]
    r, s = 9 * z["nnz_r"] + 8 * z["n"], 9 * z["nnz_s"] + 8 * z["n"]
    if op == "seeds":  # C's columns and first seeds in, R out; R in, S out
        b = 12 * z["nnz_c"] + 16 * z["n"] + 2 * r + s
    else:
        b = {"kmer": reads + a_at, "overlap": a_at - 8 * z["m"] + c, "reduce": r + s, "host": reads + r + c + s,
             "step": reads + a_at + (a_at - 8 * z["m"]) + c + r + s,
             "batch": reads + a_at + (a_at - 8 * z["m"]) + c + r + s}[op]
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """Every output is a whole number: there is no rounding to measure."""
    return None
