"""Marshalling of a batch's inputs: the rows by column are those of one value after the other, and every input
that the value-by-value form takes or refuses is taken or refused alike."""
import collections

import numpy as np
import pytest

from paper_2204_11404_gb300 import capi
from paper_2204_11404_gb300.simulator import BatchSimulator

F = capi.NOISE_FIELDS


def by_value(n, noise):
    nz = np.zeros((max(n, 1), len(F)))
    for i, d in enumerate(noise):
        for j, f in enumerate(F):
            nz[i, j] = float(d.get(f, 0.0))
    return nz


def rows(n, noise):
    return BatchSimulator._inputs(range(n), ["c128"] * n, noise)[3]


SAME = [dict(p1=0.1 * i, theta_rx=np.float32(0.01) * i, twirl=i % 2) for i in range(5)]


@pytest.mark.parametrize("n,noise", [
    (5, SAME), (5, tuple(SAME)), (5, SAME[:3]), (5, []), (1, [{}]), (0, []), (0, [dict(p1=0.5)]),
    (5, SAME[:4] + [dict(p2=1, theta_rz=2, round_rx=3)]), (2, [dict(p1="0.25"), dict(p1=np.array(0.5))]),
    (2, [dict(p1=0.1, other=3), dict(p1=0.2, other="x")]), (2, [dict(p1=True), dict(p1=np.int64(1))]),
    (2, [collections.defaultdict(lambda: 9.0, p1=0.1), collections.defaultdict(lambda: 9.0, p2=0.2)]),
])
def test_rows(n, noise):
    assert np.array_equal(rows(n, noise), by_value(n, noise))


def test_any_iterable():
    assert np.array_equal(rows(5, (d for d in SAME)), by_value(5, SAME))
    assert np.array_equal(rows(5, iter(SAME)), by_value(5, SAME))
    assert BatchSimulator._inputs(range(3), iter(["c64", "c128u", 3]), [{}] * 3)[2].tolist() == [1, 2, 3]


@pytest.mark.parametrize("error,n,noise", [
    (TypeError, 2, [dict(p1=None)] * 2), (TypeError, 2, [dict(p1=1j)] * 2), (ValueError, 1, [dict(p1="a")]),
    (IndexError, 2, SAME), (AttributeError, 1, [3]), (TypeError, 1, None),
])
def test_refused(error, n, noise):
    with pytest.raises(error):
        by_value(n, noise)
    with pytest.raises(error):
        rows(n, noise)
