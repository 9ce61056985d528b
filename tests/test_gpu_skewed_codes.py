"""Genomes of unequal base composition: the split of the prefixes grows with the skew of the codes, and from
about three quarters A and T on short k-mers take the general form. Bit for bit against the general form, and
in no more than about its time, from one level of buckets to two with the counts on the host."""
import pytest
import torch

import paper_2010_10055_gb300 as sg
from tests.test_gpu_crowded_slots import _gen
from tests.test_gpu_oversized_buckets import _ascii, _both_forms, _build, _random

pytestmark = pytest.mark.gpu


def _composed(seed, n, at):
    u = torch.rand(n, device="cuda", generator=_gen(seed))
    cuts = torch.tensor([at / 2, 0.5, 1 - at / 2], device="cuda")
    return torch.bucketize(u, cuts).to(torch.uint8)


def _reads(G, total, at, err):
    g, L = _composed(1, G, at), 2000
    n = total // L
    start = torch.randint(0, G - L, (n,), device="cuda", generator=_gen(2))
    x = g[(start[:, None] + torch.arange(L, device="cuda")[None, :]).reshape(-1)]
    rev = torch.rand(n, device="cuda", generator=_gen(3)) < 0.5
    x = x.view(n, L)
    x = torch.where(rev[:, None], 3 - x.flip(1), x).reshape(-1)
    x = torch.where(torch.rand(x.numel(), device="cuda", generator=_gen(4)) < err, _random(5, x.numel()), x)
    return _ascii(x), torch.arange(0, n * L + 1, L, device="cuda")


# one level of buckets (3 M windows), two with the skew found on the device (9 M) and on the host (40 M)
@pytest.mark.parametrize("k,err", [(17, 0.1), (21, 0.02), (31, 0.01)])
@pytest.mark.parametrize("total", [1_500_000, 3_000_000, 9_000_000, 40_000_000])
@pytest.mark.parametrize("at", [0.5, 0.6, 0.7, 0.82, 0.25])
def test_composition(at, total, k, err):
    seq, off = _reads(total // 25, total, at, err)
    t1, t0 = _both_forms(seq, off, k, 2, 50)
    assert t1 < 1.3 * t0 + 3e-4, (t1, t0)
    _, stats = _build(seq, off, k, 2, 50)
    if k <= 19 and total > 1 << 21 and at == 0.82:
        assert stats["sort_passes"] > 0, stats
    if at in (0.5, 0.6):  # (elsewhere a bucket may be too large for the form)
        assert stats["sort_passes"] == 0, stats


def test_invalid_offsets_of_two_levels():
    """Offsets are validated beside the first passes: nothing behind them may use records that no pass wrote."""
    seq, off = _reads(200_000, 9_000_000, 0.5, 0.01)
    bad = off.clone()
    bad[7] = bad[9]
    for o in (bad, off[:-1].clone(), off + 1):
        with pytest.raises(sg.SgError) as e:
            sg.build_kmer_matrix(seq, o, 17, 2, 50)
        assert e.value.status == sg.SG_ERR_INVALID
    _both_forms(seq, off, 17, 2, 50)
