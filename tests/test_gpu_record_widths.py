"""One-word records that fill all 64 bits (code below the prefix, read, position, strand), with prefixes that
are not split any further, and prefixes lengthened so that one word does; bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2010_10055_gb300 as sg
from tests.gpu_util import assert_kmer_equal, gpu_kmer

pytestmark = pytest.mark.gpu


def _reads(n, longest, total, seed):
    """n reads of one genome, the first of `longest` bases, about `total` bases in all."""
    rng = np.random.default_rng(seed)
    g = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, total // 8)]
    lens = rng.integers(1, 2 * (total - longest) // n, n)
    lens[0] = longest
    at = rng.integers(0, g.size - lens)
    seq = np.concatenate([g[a:a + m] for a, m in zip(at, lens)])
    return seq, np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


# k = 21: 42 code bits; more than 3.9 M windows: two levels and 6 bits of prefix. 10 bits of read, 17 of
# position, 1 of strand and 42 - 6 of code make 64; 12 bits of read need a prefix of 8. With 6 or 8 bits of
# prefix the highest ones hold about a thousand records (both strands' codes are that high): not split.
@pytest.mark.parametrize("n,pb1", [(1000, 6), (4000, 8)])
def test_full_words(n, pb1):
    seq, off = _reads(n, 100_000, 4_400_000, n)
    assert off[-1] * 2 >> 10 > 7447 and n > 1 << (9 if pb1 == 6 else 11)
    exp = oracle.build_kmer_matrix(seq, off, 21, 2, 20)
    km, got = gpu_kmer(seq, off, 21, 2, 20)
    st = sg.last_kmer_stats()
    assert st["sort_key_bytes"] == 8 and st["sort_passes"] == 0  # one word, bucketed
    assert_kmer_equal(got, exp)
