"""The record of which table handled each row of C (the hook that the stratified full-size sample uses) with
rows that are redone in place, in a larger table of the same launch: a row's recorded table can hold its
partners, and a row redone is recorded as such."""
import numpy as np
import pytest

import oracle
import paper_2010_10055_gb300 as sg
from tests.gpu_util import assert_overlap_equal
from tests.test_gpu_table_groups import depths  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("guess,escalate", [(10, 2), (20, 1), (60, 2), (180, 2)])
def test_recorded_tables_hold_their_rows(depths, guess, escalate):  # noqa: F811
    km, host = depths
    every = oracle.overlap_spgemm(host["A"], host["At"], 1, 0)
    rows = np.repeat(np.arange(host["A"]["n_rows"]), np.diff(every["row_ptr"]))
    partners = np.bincount(rows[every["col"] > rows], minlength=host["A"]["n_rows"])  # of the upper form
    saved = sg.tunables()
    try:
        sg.tune("spgemm_guess_pct", guess)
        sg.tune("spgemm_escalate", escalate)
        sg.debug_record_classes(True)
        C = sg.overlap_spgemm(km, 2, 2)
        codes = sg.debug_spgemm_classes(km.A.shape[0])
    finally:
        sg.debug_record_classes(False)
        for name, v in saved.items():
            sg.tune(name, v)
    assert_overlap_equal(C.to_numpy(), oracle.overlap_spgemm(host["A"], host["At"], 2, 2))
    shared = ((codes >= 6) & (codes <= 14)) | ((codes >= 102) & (codes <= 110))
    log2 = np.where(codes >= 96, codes - 96, codes)
    assert shared.sum() > 100
    assert (partners[shared] <= 0.75 * 2.0 ** log2[shared]).all()
    if guess < 100:
        assert ((codes >= 103) & (codes <= 110)).sum() > 100
