"""The tuner keeps the library's own choice unless a candidate is faster by more than its repeats scatter and 1 %, and
the committed table holds nothing else (host only)."""
from paper_2311_12134_gb300 import autotune as at

DEFAULT = at.label(at.DEFAULTS)
TWO = at.label({"solve_steps": 0, "streams": 2})


def test_noise_keeps_the_defaults():
    assert at.choose({DEFAULT: [79.66, 79.46, 79.52], TWO: [79.31, 79.36, 79.5]}) == at.DEFAULTS
    assert at.choose({DEFAULT: [79.5, 79.5, 79.5], TWO: [70.0, 78.0, 86.0]}) == at.DEFAULTS
    assert at.choose({DEFAULT: [79.6, 79.5, 79.5], TWO: [77.0, 77.3, 77.1]}) == {"solve_steps": 0, "streams": 2}
    assert at.choose({DEFAULT: [1277.6, 1277.7, 1277.6], TWO: [1276.9, 1277.0, 1277.1]}) == at.DEFAULTS
    assert at.choose({TWO: [2.0], at.label({"solve_steps": 1, "streams": 2}): [3.0]}) == {"solve_steps": 0, "streams": 2}


def test_committed_table_is_borne_out_by_its_times():
    table = at.load_table()
    assert table
    for entry in table.values():
        assert all(len(v) >= 3 for v in entry["ms_per_step"].values())
        assert entry["settings"] == at.choose(entry["ms_per_step"])
