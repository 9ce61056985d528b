"""Rows of C whose guessed tables differ by orders of magnitude and share launches: read sets of very
different depth in one input, with tables guessed too small (redone in the same launch, in the next
one, in global memory), about right and too large, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2010_10055_gb300 as sg
import synth
from tests.gpu_util import assert_overlap_equal, gpu_kmer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def depths():
    seqs, lens = [], []
    for i, (G, coverage) in enumerate([(30000, 5.0), (15000, 50.0), (3000, 250.0), (600, 1.0)]):
        g = np.random.default_rng(7 + i).choice(np.frombuffer(b"ACGT", np.uint8), size=G)
        rd = synth.reads(g, coverage, 600.0, 250.0, 1, 0.01, 0.01, 0.01, 7 + i)
        seqs.append(rd["seq"])
        lens.append(np.diff(rd["offsets"]))
    seq = np.concatenate(seqs)
    off = np.concatenate([[0], np.cumsum(np.concatenate(lens))]).astype(np.int64)
    km, host = gpu_kmer(seq, off, 17, 2, 300)
    return km, host


@pytest.fixture(scope="module")
def expected(depths):
    return {S: oracle.overlap_spgemm(depths[1]["A"], depths[1]["At"], 2, S) for S in (0, 1, 2)}


@pytest.mark.parametrize("S", [0, 1, 2])
@pytest.mark.parametrize("guess,escalate", [(1, 0), (1, 1), (1, 2), (20, 2), (60, 1), (180, 2), (2000, 2)])
@pytest.mark.parametrize("upper", [0, 1])
def test_grouped_tables(depths, expected, S, guess, escalate, upper):
    cfg = {"spgemm_guess_pct": guess, "spgemm_escalate": escalate, "spgemm_upper": upper}
    saved = {k: sg.tunables()[k] for k in cfg}
    try:
        for k, v in cfg.items():
            sg.tune(k, v)
        C = sg.overlap_spgemm(depths[0], 2, S)
        assert_overlap_equal(C.to_numpy(), expected[S])
    finally:
        for k, v in saved.items():
            sg.tune(k, v)
