"""The concatenation of a batch's read sets at every alignment of source and destination and at lengths
around its 16-byte steps, and prefix counts of groups of 32 bases that hold several sets: the batch
against each set alone, by the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2010_10055_gb300 as sg
from tests.gpu_util import assert_csr_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [[1, 2, 3, 5, 15, 16, 17, 18, 19, 20, 21, 31, 32, 33, 47, 48, 49, 63, 64, 65, 80],
                                  [4099, 8, 515, 16, 3, 1025, 7, 999, 64, 30, 2050, 31],
                                  [70001, 69999, 1, 70003]])
@pytest.mark.parametrize("shift", [0, 1, 2, 3, 9, 15])
def test_any_alignment(lens, shift):
    rng = np.random.default_rng(len(lens) * 16 + shift)
    pool = torch.zeros(sum(lens) + 32 * len(lens) + 64, dtype=torch.uint8, device="cuda")
    sets, items, at = [], [], shift
    for n in lens:
        g = rng.choice(np.frombuffer(b"ACGT", np.uint8), size=max(1, n // 3))
        seq = np.resize(g, n).copy()  # each set repeats itself: columns with several reads
        off = np.unique(np.concatenate([[0, n], np.arange(0, n, 150)])).astype(np.int64)
        view = pool[at:at + n]
        view.copy_(torch.from_numpy(seq))
        at += n + int(rng.integers(0, 20))
        sets.append((seq, off))
        items.append(dict(seq=view, offsets=torch.from_numpy(off).cuda(), lo=1, hi=12))
    res = sg.run_batch(items, k=11, min_shared=1, max_seeds=2, fuzz=0)
    for b, (seq, off) in enumerate(sets):
        km = oracle.build_kmer_matrix(seq, off, 11, 1, 12)
        got = res.item(b)
        assert np.array_equal(got["codes"], km["codes"]), b
        assert_csr_equal(got["A"], km["A"], f"A[{b}]")
