"""Buckets whose records crowd into few slots, which the finishing pass sorts instead of ranking them slot by
slot: codes of high frequency under a high hi, satellites of codes far above hi that share slots with others
(k = 31), and dense rows of A among empty ones. Bit for bit against the general form (radix sorts) or a plain
sort, in about its time."""
import pytest
import torch

import paper_2010_10055_gb300 as sg
from tests.test_gpu_oversized_buckets import _ascii, _both_forms, _gen, _random, _rows_match

pytestmark = pytest.mark.gpu


def _reads_of(g, n, L, seed, err):
    at = torch.randint(0, g.numel() - L + 1, (n,), device="cuda", generator=_gen(seed))
    x = g[(at[:, None] + torch.arange(L, device="cuda")[None, :]).reshape(-1)]
    x = torch.where(torch.rand(x.numel(), device="cuda", generator=_gen(seed + 1)) < err, _random(seed + 2, x.numel()), x)
    return _ascii(x), torch.arange(0, n * L + 1, L, device="cuda")


# frequencies of 130 to 900: slots a warp still ranks, slots that are sorted
@pytest.mark.parametrize("k", [17, 21, 31])
@pytest.mark.parametrize("coverage", [130, 300, 900])
def test_deep_coverage(k, coverage):
    G, L = 24_000_000 // coverage, 2000
    seq, off = _reads_of(_random(coverage, G), 24_000_000 // L, L, 11, 0.003)
    t1, t0 = _both_forms(seq, off, k, 2, 1000)
    assert t1 < 1.2 * t0 + 1e-3, (t1, t0)


@pytest.mark.parametrize("k", [17, 31])
def test_satellites(k):
    """30 % of a genome is one repeat of 171 bases, 5,000 copies at 10x."""
    g = _random(21, 2_850_000)
    g[1_000_000:1_855_000] = _random(22, 171).repeat(5000)
    seq, off = _reads_of(g, 5700, 5000, 23, 0.002)
    t1, t0 = _both_forms(seq, off, k, 2, 40)
    assert t1 < 1.2 * t0 + 1e-3, (t1, t0)


@pytest.mark.parametrize("every,length", [(4000, 6000), (1, 4), (9000, 1500)])
def test_dense_rows_among_empty_ones(every, length):
    """A million reads, all but every 4,000th or 9,000th empty: a group of rows has a slot for each, and the
    entries of a dense row share a few."""
    n = 1 << 20
    dense = torch.arange(17, n, every, device="cuda")[:260]
    lens = torch.zeros(n, dtype=torch.int64, device="cuda")
    lens[dense] = length if length > 17 else 400
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(lens, 0)])
    half = _random(31, int(off[-1]) // 2 + 1)
    seq = _ascii(torch.cat([half, half])[:int(off[-1])].contiguous())
    km = sg.build_kmer_matrix(seq, off, 17, 2, 60)
    assert km.A.nnz > 50_000
    _rows_match(km, n)
