"""Rows of C at the edges of the compact tables: kept partners that crowd into few of the bins that order them
(reads in genome order, with far partners through a repeat), and rows of A of 65,534 to 65,538 entries, around
the 16-bit indices' limit. Bit for bit against the two-pass form or the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2010_10055_gb300 as sg
from tests.gpu_util import assert_overlap_equal, gpu_kmer
from tests.test_gpu_oversized_buckets import _ascii, _gen, _random

pytestmark = pytest.mark.gpu

BIN_LIMIT = 48  # partners of one bin ranked against each other; above, the row's partners are sorted


def _crowded_rows(C):
    """Rows whose partners after them fill a bin of the counting order beyond its limit."""
    rp, col = C["row_ptr"].cpu().numpy(), C["col"].cpu().numpy()
    n = 0
    for i in range(rp.size - 1):
        k = col[rp[i]:rp[i + 1]]
        k = k[k > i]
        if k.size <= BIN_LIMIT:
            continue
        nb = max(32, 1 << int(k.size - 1).bit_length())
        n += np.bincount((k - k[0]) * nb // (k[-1] - k[0] + 1)).max() > BIN_LIMIT + 1
    return n


@pytest.mark.parametrize("max_seeds", [0, 1, 2])
def test_reads_in_genome_order(max_seeds):
    G, L, n = 400_000, 800, 40_000  # 80x
    g = _random(1, G)
    g[380_000:383_000] = g[20_000:23_000]  # a repeat at either end
    at = torch.sort(torch.randint(0, G - L, (n,), device="cuda", generator=_gen(2)))[0]
    x = g[(at[:, None] + torch.arange(L, device="cuda")[None, :]).reshape(-1)]
    x = torch.where(torch.rand(x.numel(), device="cuda", generator=_gen(3)) < 0.02, _random(4, x.numel()), x)
    km = sg.build_kmer_matrix(_ascii(x), torch.arange(0, n * L + 1, L, device="cuda"), 17, 2, 300)
    got = sg.overlap_spgemm(km, 2, max_seeds).tensors()
    saved = sg.tunables()["spgemm_fused"]
    try:
        sg.tune("spgemm_fused", 0)
        exp = sg.overlap_spgemm(km, 2, max_seeds).tensors()
    finally:
        sg.tune("spgemm_fused", saved)
    assert all(torch.equal(got[key], exp[key]) for key in exp)
    assert _crowded_rows(got) > 50


@pytest.fixture(scope="module")
def long_rows():
    rng = np.random.default_rng(5)
    g = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 120_000)]
    lens = [65534 + 30 + d for d in range(5)] * 2 + [65000, 66000] + [3000] * 60 + [90_000]
    at = [int(rng.integers(0, g.size - m + 1)) for m in lens]
    order = rng.permutation(len(lens))
    parts = [g[at[i]:at[i] + lens[i]] for i in order]
    off = np.concatenate([[0], np.cumsum([p.size for p in parts])]).astype(np.int64)
    km, host = gpu_kmer(np.concatenate(parts), off, 31, 1, 200)  # 31-mers of a random genome are distinct
    rows = np.diff(host["A"]["row_ptr"])
    assert {65534, 65535, 65536, 65537} <= set(rows.tolist()), sorted(rows)[-14:]
    return km, host


@pytest.mark.parametrize("max_seeds", [0, 1, 2, 3])
@pytest.mark.parametrize("upper", [1, 0])
def test_rows_around_the_index_limit(long_rows, max_seeds, upper):
    km, host = long_rows
    saved = sg.tunables()["spgemm_upper"]
    try:
        sg.tune("spgemm_upper", upper)
        C = sg.overlap_spgemm(km, 2, max_seeds)
    finally:
        sg.tune("spgemm_upper", saved)
    assert_overlap_equal(C.to_numpy(), oracle.overlap_spgemm(host["A"], host["At"], 2, max_seeds))
