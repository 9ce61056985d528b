"""The autotuner and the two forms of the k-mer stage, on the CPU with a fake step: the switch between the
forms is tried, parameters of the general form are tried only where that form runs, and times that differ by
noise change nothing."""
import pytest

import paper_2010_10055_gb300 as sg
from paper_2010_10055_gb300 import autotune


@pytest.fixture(autouse=True)
def restore_tunables():
    saved = sg.tunables()
    yield
    for k, v in saved.items():
        sg.tune(k, v)


def run(cost, **kw):
    """Every setting timed, and the result; the general form runs where kmer_bucketed is 0."""
    seen = []

    def timer(step, reps):
        seen.append(dict(sg.tunables()))
        return cost(seen[-1], len(seen))

    general = lambda: seen[-1]["kmer_bucketed"] == 0
    res = autotune.autotune(lambda: None, timer=timer, general=general, **kw)
    start = sg.tunables() if not seen else seen[0]
    tried = {k for t in seen for k in t if t[k] != start[k]}
    return res, tried


def test_bucketed_step_leaves_the_general_form_alone():
    res, tried = run(lambda t, i: 10.0 + 5.0 * (t["kmer_bucketed"] == 0))
    assert "kmer_bucketed" in tried and res["params"]["kmer_bucketed"] == 1
    assert not tried & set(autotune.GENERAL_FORM)
    assert tried >= {"spgemm_guess_pct", "tr_blocks_per_sm"}


def test_general_form_is_tuned_where_it_runs():
    # the general form wins, and then its filter is worth tuning
    res, tried = run(lambda t, i: 10.0 - 3.0 * (t["kmer_bucketed"] == 0) * (1 + 0.1 * (t["bloom_bits"] == 12)))
    assert res["params"]["kmer_bucketed"] == 0 and res["params"]["bloom_bits"] == 12
    assert tried >= set(autotune.GENERAL_FORM)


def test_noise_adopts_nothing():
    before = sg.tunables()
    res, _ = run(lambda t, i: 10.0 - 0.04 * (i % 7) / 6.0)  # 0.4 % from run to run
    assert res["params"] == before


def test_given_spaces_are_searched_as_they_are():
    _, tried = run(lambda t, i: 10.0, space={"bloom_bits": [6, 8, 10]})
    assert tried == {"bloom_bits"}
