"""The bucketed k-mer form and A = At transposed at the sizes where they can go wrong, bit for bit
against the oracle: one and two grouping levels, one- and two-word records, buckets larger than a
block's shared memory (skewed and constant sequences), reads shorter than a window, empty reads,
more read sets than prefixes, reliable ranges around the form's limit; and the general form, which
takes over past those limits."""
import numpy as np
import pytest

import oracle
import paper_2010_10055_gb300 as sg
import synth
from tests.gpu_util import assert_csr_equal, assert_kmer_equal, dev, gpu_kmer

pytestmark = pytest.mark.gpu


def _cat(parts):
    off = np.cumsum([0] + [len(p) for p in parts]).astype(np.int64)
    return np.frombuffer(b"".join(parts), np.uint8).copy(), off


def _sampled(seed, G, coverage, mean, probs=None, err=0.02):
    rng = np.random.default_rng(seed)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), size=G, p=probs)
    rd = synth.reads(g, coverage, mean, 0.4 * mean, 1, err, err, err, seed)
    return rd["seq"], rd["offsets"]


def _check(seq, off, k, lo, hi):
    exp = oracle.build_kmer_matrix(seq, off, k, lo, hi)
    _, got = gpu_kmer(seq, off, k, lo, hi)
    assert_kmer_equal(got, exp)
    return exp


# 7,400 records of 8 bytes (3,700 of 16) to a bucket and 1,024 prefixes: one level to 3.8 M windows
# (1.9 M), then two; total 33 .. 5.5 M
@pytest.mark.parametrize("k,G,coverage,mean", [(17, 40, 1, 33), (17, 3000, 3, 300), (11, 90000, 20, 700),
                                               (21, 150000, 20, 4000), (31, 60000, 12, 5000), (31, 260000, 10, 3000),
                                               (17, 550000, 10, 6000), (27, 500000, 9, 2500)])
@pytest.mark.parametrize("lo,hi", [(2, 40), (1, 6)])
def test_sizes(k, G, coverage, mean, lo, hi):
    seq, off = _sampled(k + G, G, coverage, mean)
    seq[::1013] = ord("N")
    _check(seq, off, k, lo, hi)


@pytest.mark.parametrize("k,n", [(17, 12), (31, 400)])
def test_long_rows(k, n):
    """Rows of A longer than a block holds (8,192 entries), between short ones."""
    rng = np.random.default_rng(n)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), size=60000).tobytes()
    parts = []
    for i in range(n):
        L = 45000 if i % 5 == 0 else int(rng.integers(20, 9000))
        a = int(rng.integers(0, 60000 - L))
        parts.append(g[a:a + L])
    exp = _check(*_cat(parts), k, 2, 600)
    assert np.diff(exp["A"]["row_ptr"]).max() > 16384


def test_short_and_empty_reads():
    rng = np.random.default_rng(3)
    g = rng.choice(np.frombuffer(b"ACGT", np.uint8), size=5000).tobytes()
    parts = []
    for i in range(60000):
        L = int(rng.choice([0, 0, 0, 1, 10, 16, 17, 18, 31, 40]))
        a = int(rng.integers(0, 4900))
        parts.append(g[a:a + L])
    seq, off = _cat(parts + [b""] * 5000)
    for k in (17, 31):
        _check(seq, off, k, 2, 1000)


def test_skewed_and_constant_sequences():
    # four fifths A and T: the buckets of low codes hold many times their share, refined in place
    seq, off = _sampled(5, 200000, 24, 3000, probs=[0.4, 0.1, 0.1, 0.4], err=0.05)
    _check(seq, off, 17, 2, 60)
    # one code with far more records than a bucket holds, beside ordinary ones
    seq2, off2 = _sampled(6, 60000, 10, 2000)
    parts = [b"A" * 30000, b"ACACACACAC" * 3000, seq2.tobytes(), b"T" * 500]
    s, o = _cat(parts)
    _check(s, np.concatenate([o[:3], o[2] + off2[1:], [o[-1]]]), 17, 2, 50)
    for k in (17, 31):
        _check(np.full(50000, ord("A"), np.uint8), np.array([0, 20000, 50000]), k, 1, 20)


@pytest.mark.parametrize("hi", [1024, 1025, 1 << 30])
def test_reliable_range_limit(hi):
    # 1,200 copies of one 200-base stretch, each in a read of its own: above 1,024 the general form runs
    rng = np.random.default_rng(9)
    unit = rng.choice(np.frombuffer(b"ACGT", np.uint8), size=200).tobytes()
    parts = [unit] * 1200 + [unit[:100]] * 400
    seq, off = _cat(parts)
    _check(seq, off, 17, 2, hi)
    _check(seq, off, 17, 1100, max(hi, 1100))


@pytest.mark.parametrize("nsets", [3, 700])
def test_batch_prefixes(nsets):
    """Set ids above the code bits: fewer and more sets than prefixes, sizes 0 to 60 kbp."""
    rng = np.random.default_rng(nsets)
    sets, items = [], []
    for b in range(nsets):
        G = int(rng.choice([0, 30, 400, 3000])) if nsets > 3 else [0, 60000, 2500][b]
        seq, off = _sampled(100 + b, G, 8, 500) if G > 200 else (np.zeros(0, np.uint8), np.zeros(2, np.int64))
        sets.append((seq, off, 2 + b % 2, 9 + b % 5))
        items.append(dict(seq=dev(seq, np.uint8), offsets=dev(off, np.int64), lo=2 + b % 2, hi=9 + b % 5))
    res = sg.run_batch(items, 17, 2, 2)
    for b in range(0, nsets, 1 if nsets < 10 else 23):
        exp = oracle.build_kmer_matrix(sets[b][0], sets[b][1], 17, sets[b][2], sets[b][3])
        got = res.item(b)
        assert np.array_equal(got["codes"], exp["codes"]), b
        assert_csr_equal(got["A"], exp["A"], f"A {b}")
        assert_csr_equal(got["At"], exp["At"], f"At {b}")


@pytest.mark.parametrize("cfg", [{}, {"bloom_binned": 0, "bloom_slice_mb": 1}, {"bloom_scatter_levels": 2, "bloom_bin_kb": 16},
                                 {"kmer_direct_seg": 0}, {"kmer_direct_seg": 0, "kmer_sort_buckets": 0}],
                         ids=lambda c: ",".join(f"{k}={v}" for k, v in c.items()) or "defaults")
@pytest.mark.parametrize("k", [17, 31])
def test_general_form(k, cfg):
    """The filters and radix sort, which run where the bucketed form does not."""
    seq, off = _sampled(31 + k, 60000, 10, 2000)
    saved = sg.tunables()
    try:
        for name, v in dict(cfg, kmer_bucketed=0).items():
            sg.tune(name, v)
        _check(seq, off, k, 2, 14)
    finally:
        for name, v in saved.items():
            sg.tune(name, v)
