"""The oracle's assign rounds the square and the sum of a squared distance once: pinned to exact rational
arithmetic on records that the rule with two roundings decides differently."""
import numpy as np
import pytest

import near_ties
import oracle
from synth.workloads import F32, I32, Section


@pytest.mark.parametrize("d,K,pair", [(2, 2, (0, 1)), (7, 3, (0, 2)), (32, 5, (3, 4)), (9, 8, (2, 7))])
def test_assign_rounds_square_and_sum_once(d, K, pair):
    x, cent, want = near_ties.records(d, K, pair, 12, seed=d)
    sec = Section("assign", (d, K), frozenset(range(d)), frozenset([d]), table=tuple(float(v) for v in cent.reshape(-1)))
    fields = [np.ascontiguousarray(x[:, j]) for j in range(d)] + [np.zeros(len(x), np.int32)]
    oracle.section(sec, [F32] * d + [I32], fields)
    assert np.array_equal(fields[d], want)
