"""The packed-copy sizes that the benchmark's elastic lines report: the units counted one by one, for one block
size (a number that json.dumps accepts) and for an array of them."""
import json

import numpy as np

import bench


def _count(m):
    nb = -(-m // 16)
    return sum(1 for i in range(nb) for _ in range(i, nb))


def test_sym_units():
    ms = [1, 16, 17, 30, 36, 72, 120, 180]
    assert json.loads(json.dumps([bench.sym_units(m) * 256 for m in ms])) == [_count(m) * 256 for m in ms]
    assert np.array_equal(bench.sym_units(np.array(ms)), [_count(m) for m in ms])
