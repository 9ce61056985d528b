"""C for read sets whose rows are of different kinds: many short rows with many partners per entry (reads of low
complexity) beside long rows with few. The sampled guess of tables and of the region for the result has to hold
for both, so that no row is computed a second time in global memory; bit for bit against the two-pass form."""
import pytest
import torch

import paper_2010_10055_gb300 as sg
from tests.test_gpu_crowded_slots import _reads_of
from tests.test_gpu_oversized_buckets import _ascii, _random

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tails", [5000, 20000])
@pytest.mark.parametrize("max_seeds", [2, 3])
def test_short_rows_of_many_partners(tails, max_seeds):
    a, off = _reads_of(_random(41, 400_000), 2160, 5000, 42, 0.15)  # 27x
    b = _ascii(_random(45, tails * 1000, 0.8))  # 85 % A
    seq = torch.cat([a, b])
    off = torch.cat([off, off[-1] + 1000 * torch.arange(1, tails + 1, device="cuda")])
    km = sg.build_kmer_matrix(seq, off, 17, 2, 20)
    sg.prof_reset()
    sg.prof_enable(True)
    C = sg.overlap_spgemm(km, 2, max_seeds)
    torch.cuda.synchronize()
    sg.prof_enable(False)
    launches = {name: n for name, (n, _) in sg.prof_collect().items()}
    saved = sg.tunables()["spgemm_fused"]
    try:
        sg.tune("spgemm_fused", 0)
        E = sg.overlap_spgemm(km, 2, max_seeds)
    finally:
        sg.tune("spgemm_fused", saved)
    got, exp = C.tensors(), E.tensors()
    assert all(torch.equal(got[key], exp[key]) for key in exp)
    assert any(name.startswith("spgemm_numeric_t") for name in launches)
    if max_seeds == 2:
        assert "spgemm_numeric_gmem" not in launches, launches
