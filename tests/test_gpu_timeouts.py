"""Bounded waits that run out in scans and radix sorts whose outputs later kernels of the call use as
indices, without faulting the GPU: nothing may work on them once a wait has given up. With the test hook on,
the call ends in SG_ERR_TIMEOUT; the same call is right again afterwards."""
import numpy as np
import pytest
import torch

import paper_2010_10055_gb300 as sg
import synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


def _bases(seed, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")[
        torch.randint(0, 4, (n,), device="cuda", generator=g)]


def _tensors(km):
    return [t.clone() for m in (km.A, km.At) for t in m.tensors().values()] + [km.codes().clone()]


def _stalled_then_exact(call):
    before = call()
    sg.debug_stall_lookback(True)
    try:
        with pytest.raises(sg.SgError) as e:
            call()
        assert e.value.status == sg.SG_ERR_TIMEOUT
    finally:
        sg.debug_stall_lookback(False)
    after = call()
    assert all(torch.equal(a, b) for a, b in zip(before, after))


@pytest.mark.parametrize("k", [17, 31])
def test_bucket_ranges(k):
    """More than 4,096 buckets (one tile of the scan) in the second grouping level of the windows, of
    one- and two-word records."""
    seq = _bases(1, 20_000_000)
    seq[10_000_000:] = seq[:10_000_000].clone()  # every window twice
    off = torch.arange(0, 20_000_001, 5000, device="cuda")
    _stalled_then_exact(lambda: _tensors(sg.build_kmer_matrix(seq, off, k, 2, 8)))


def test_bucket_ranges_of_rows():
    """The same scan in the transposition: more than 2^23 reads, nearly all empty, make more than 4,096 buckets of
    rows while the windows' own stage has a single level."""
    total, n = 400_000, (1 << 23) + 1000
    seq = _bases(2, total // 2).repeat(2)
    off = torch.full((n + 1,), total, dtype=torch.int64, device="cuda")
    off[:401] = torch.arange(0, total + 1, 1000, device="cuda")
    _stalled_then_exact(lambda: _tensors(sg.build_kmer_matrix(seq, off, 17, 2, 8)))


@pytest.fixture
def tuned():
    saved = sg.tunables()
    yield lambda **kw: [sg.tune(name, v) for name, v in kw.items()]
    for name, v in saved.items():
        sg.tune(name, v)


# sorted windows by position, by index and in pairs; segments from the sorted keys, from unpacked ones and
# (hi beyond the walk bound) without the packed flags
@pytest.mark.parametrize("k,hi,cfg", [(17, 8, {}), (17, 8, {"kmer_direct_seg": 0}), (17, 5000, {}), (31, 8, {}),
                                      (23, 8, {"kmer_sort_buckets": 0}), (23, 5000, {"kmer_sort_buckets": 0})])
def test_radix_of_windows(tuned, k, hi, cfg):
    tuned(kmer_bucketed=0, **cfg)
    seq = _bases(3, 100_000).repeat(2)
    off = torch.arange(0, 200_001, 2000, device="cuda")
    _stalled_then_exact(lambda: _tensors(sg.build_kmer_matrix(seq, off, k, 2, hi)))


@pytest.mark.parametrize("rec", [0, 1])
def test_radix_of_the_mirror(tuned, rec):
    """Fewer than 4,096 reads (single-tile scans), more than 4,096 mirrored entries."""
    tuned(spgemm_mirror_rec=rec)
    d = synth.make(synth.BACTERIAL.scaled(0.1))
    km = sg.build_kmer_matrix(dev(d["seq"], np.uint8), dev(d["offsets"], np.int64), 17, 2, 20)
    assert km.A.shape[0] < 4096 and sg.overlap_spgemm(km, 2, 2).nnz > 3 * 4096
    _stalled_then_exact(lambda: [t.clone() for t in sg.overlap_spgemm(km, 2, 2).tensors().values()])
