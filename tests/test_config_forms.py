"""A configuration's tables may be anything that gives a value for an index."""
from collections import deque

import numpy as np
import pytest

import paper_1909_08665_gb300 as pkg
import workload

TABLES = ("conn_prob", "w_mean", "w_sd", "proj_scale")
ROWS = ("pop_sizes", "pop_exc", "d_mean", "d_sd", "k_ext", "i_dc")


@pytest.mark.parametrize("row", [list, tuple, deque, np.array, lambda v: dict(enumerate(v)),
                                 lambda v: list(v) + [7] * 3])
def test_rows_of_any_kind(row):
    cfg = workload.microcircuit(0.1)
    want = bytes(pkg.make_config(cfg))
    other = dict(cfg)
    for key in ROWS[1:]:
        other[key] = row(cfg[key])
    for key in TABLES:
        other[key] = [row(r) for r in cfg[key]]
    assert bytes(pkg.make_config(other)) == want


def test_rows_too_short_are_refused():
    cfg = workload.microcircuit(0.1)
    for key in ROWS[1:]:
        with pytest.raises((IndexError, ValueError)):
            pkg.make_config(dict(cfg, **{key: list(cfg[key])[:-1]}))
