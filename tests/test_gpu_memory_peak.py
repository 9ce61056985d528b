"""The peak that sg_memory_stats reports is one that device memory reached: what both pools (temporaries,
outputs) hold at one time, not the sum of two peaks that do not coincide."""
import gc

import numpy as np
import pytest
import torch

import paper_2010_10055_gb300 as sg
import synth
from tests.gpu_util import dev
from tests.test_gpu_kmer_memory import _Limited

pytestmark = pytest.mark.gpu


def test_peak_of_both_pools_together():
    d = synth.make(synth.BACTERIAL.scaled(0.05))
    seq, off = dev(d["seq"], np.uint8), dev(d["offsets"], np.int64)

    def step():  # temporaries peak in the k-mer stage, while few outputs exist; outputs with C
        km = sg.build_kmer_matrix(seq, off, 17, 2, 20)
        cs = [sg.overlap_spgemm(km, 2, 2) for _ in range(40)]
        for x in [km] + cs:
            x.free()

    step()
    torch.cuda.synchronize()
    gc.collect()
    with _Limited(1 << 40) as a:  # the same calls, every block counted by the caller
        step()
    base = sg.memory_stats()[1]
    sg.memory_reset_peak()
    assert sg.memory_stats()[2] == base
    step()
    torch.cuda.synchronize()
    reserved, in_use, peak = sg.memory_stats()
    assert in_use == base and peak <= reserved
    # the library rounds a block up to 512 bytes
    assert a.peak <= peak - base <= a.peak + 512 * 1000, (a.peak, peak - base)
    sg.memory_reset_peak()
    assert sg.memory_stats()[2] == sg.memory_stats()[1]
