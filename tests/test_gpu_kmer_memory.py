"""Device memory that the bucketed k-mer form cannot have: the call goes on in the general form (or, for A, by a
sort) with that memory given back, and is right. Injected failures at every allocation, and an allocator
with a limit between the two forms' needs."""
import ctypes
import gc

import numpy as np
import pytest
import torch

import paper_2010_10055_gb300 as sg
import synth
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


def _tensors(km):
    return [t.clone() for m in (km.A, km.At) for t in m.tensors().values()] + [km.codes().clone()]


def _equal(a, b):
    return len(a) == len(b) and all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.fixture(scope="module")
def reads():
    d = synth.make(synth.BACTERIAL.scaled(0.02))
    return dev(d["seq"], np.uint8), dev(d["offsets"], np.int64)


def _settled():
    torch.cuda.synchronize()
    gc.collect()
    return sg.memory_stats()[1]


@pytest.mark.parametrize("k", [17, 31])
def test_every_allocation_failing_once(reads, k):
    call = lambda: sg.build_kmer_matrix(*reads, k, 2, 20)
    km = call()
    exp = _tensors(km)
    km.free()
    held, general, failed = _settled(), 0, 0
    for nth in range(1, 60):
        sg.debug_fail_alloc_after(nth)
        try:
            km = call()
        except sg.SgError as e:
            assert e.status == sg.SG_ERR_OOM
            failed += 1
        else:
            general += sg.last_kmer_stats()["sort_passes"] > 0
            assert _equal(_tensors(km), exp), nth
            km.free()
        finally:
            sg.debug_fail_alloc_after(0)
        assert _settled() == held, nth
    # what both forms need ends the call: the error words and A's own arrays
    assert general >= 8 and 1 <= failed <= 6, (general, failed)


def test_batch_with_a_failing_allocation(reads):
    """The batch's column counts per set are counted once, not by both forms."""
    seq, off = reads
    items = [dict(seq=seq, offsets=off, lo=2, hi=20)] * 3
    view = lambda r: [(r.item(b)["codes"], r.item(b)["At"]["col"], r.item(b)["A"]["val"]) for b in range(3)]
    exp = view(sg.run_batch(items, k=17))
    seen = 0
    for nth in range(2, 40):
        sg.debug_fail_alloc_after(nth)
        try:
            res = sg.run_batch(items, k=17)
        except sg.SgError as e:
            assert e.status == sg.SG_ERR_OOM
            continue
        finally:
            sg.debug_fail_alloc_after(0)
        seen += sg.last_kmer_stats()["sort_passes"] > 0
        for a, b in zip(view(res), exp):
            assert all(np.array_equal(x, y) for x, y in zip(a, b)), nth
    assert seen >= 5, seen


class _Limited:
    """sg_set_allocator callbacks over PyTorch's allocator that refuse to hold more than `limit` bytes."""

    def __init__(self, limit):
        self.limit, self.held, self.peak, self.sizes, self.refused = limit, 0, 0, {}, 0
        self.alloc = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)(self._alloc)
        self.free = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)(self._free)

    def _alloc(self, n, stream, ctx):
        if self.held + n > self.limit:
            self.refused += 1
            return None
        p = torch.cuda.caching_allocator_alloc(n)
        self.sizes[p] = n
        self.held += n
        self.peak = max(self.peak, self.held)
        return p

    def _free(self, p, stream, ctx):
        self.held -= self.sizes.pop(p)
        torch.cuda.caching_allocator_delete(p)

    def __enter__(self):
        L = sg.lib()
        L.sg_set_allocator.argtypes = [ctypes.c_void_p] * 3
        torch.cuda.synchronize()
        L.sg_set_allocator(ctypes.cast(self.alloc, ctypes.c_void_p), ctypes.cast(self.free, ctypes.c_void_p), None)
        return self

    def __exit__(self, *_):
        torch.cuda.synchronize()
        sg.lib().sg_set_allocator(None, None, None)


def test_allocator_with_a_limit(reads):
    def once(limit, form):
        sg.tune("kmer_bucketed", form)
        with _Limited(limit) as a:
            km = sg.build_kmer_matrix(*reads, 17, 2, 20)
            out, passes = _tensors(km), sg.last_kmer_stats()["sort_passes"]
            km.free()
            torch.cuda.synchronize()
            assert a.held == 0
        return out, passes, a

    saved = sg.tunables()["kmer_bucketed"]
    try:
        exp, passes, general = once(1 << 40, 0)
        assert passes > 0
        _, passes, bucketed = once(1 << 40, 1)
        assert passes == 0 and bucketed.peak > general.peak
        got, passes, a = once((general.peak + bucketed.peak) // 2, 1)
        assert a.refused and passes > 0 and _equal(got, exp)
    finally:
        sg.tune("kmer_bucketed", saved)
