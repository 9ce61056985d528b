"""The transitive reduction at the degrees where a row changes its kernel or its table size, in
every mode, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2010_10055_gb300 as sg
from tests.gpu_util import assert_graph_equal

pytestmark = pytest.mark.gpu

# a warp's row holds up to 128 entries (tables of 64 to 256 slots, 32 entries per register), a
# block's hashed row up to 2,048
DEGREES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 200, 2047, 2048, 2049, 2600]


def _graph(seed, n=2700, max_suffix=1000):
    rng = np.random.default_rng(seed)
    rows = [np.zeros(0, np.int64)] * n
    where = rng.permutation(n)
    for i in range(n):
        deg = DEGREES[i] if i < len(DEGREES) else int(rng.integers(0, 24))
        r = int(where[i])
        rows[r] = np.sort(rng.choice(np.delete(np.arange(n), r), size=deg, replace=False))
    rp = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int64)
    nnz = int(rp[-1])
    return dict(n=n, row_ptr=rp, col=np.concatenate(rows).astype(np.int32),
                suffix=rng.integers(0, max_suffix, nnz).astype(np.uint32), dir=rng.integers(0, 4, nnz).astype(np.uint8))


@pytest.mark.parametrize("warp_rows", [1, 0])
@pytest.mark.parametrize("mode,fuzz,max_suffix", [(0, 0, 1000), (1, 300, 1000), (2, 1000, 1 << 30), (3, 0, 50),
                                                  (0, (1 << 30) - 1, 1 << 30)])
def test_every_row_form(mode, fuzz, max_suffix, warp_rows):
    R = _graph(7 + mode, max_suffix=max_suffix)
    assert set(DEGREES) <= set(np.diff(R["row_ptr"]).tolist())
    D = sg.DeviceGraph.from_numpy(R)
    saved = sg.tunables()["tr_warp_rows"]
    try:
        sg.tune("tr_warp_rows", warp_rows)
        N, Nd = sg.minplus_square(D, mode & 1)
        eN, eNd = oracle.minplus(R, mode & 1)
        assert np.array_equal(N.cpu().numpy().view(np.uint32), eN)
        assert np.array_equal(Nd.cpu().numpy(), eNd)
        S, it = sg.transitive_reduce(D, fuzz=fuzz, mode=mode)
        eS, eit = oracle.transitive_reduce(R, fuzz, mode)
        assert_graph_equal(S.to_numpy(), eS)
        assert it == eit
    finally:
        sg.tune("tr_warp_rows", saved)
