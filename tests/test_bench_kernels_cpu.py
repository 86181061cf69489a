"""bench.py's claims about a pass: its kernels and the bytes it must move."""
import argparse

import numpy as np
import pytest

import bench
import synth


def code(mb, nb, entries):
    row, col, shift = (np.array(v, np.int32) for v in zip(*entries))
    return dict(mb=mb, nb=nb, Z=8, row=row, col=col, shift=shift)


# rows 0 and 1 meet columns 0 and 1 once each; row 2 meets column 0 twice;
# columns 2 and 3 have degree 1, on rows 0 and 2
SMALL = code(3, 4, [(0, 0, 0), (0, 1, 1), (0, 2, 0), (1, 0, 2), (1, 1, 3), (2, 0, 4), (2, 0, 5), (2, 1, 0), (2, 3, 0)])


def test_layered_kernels_of_a_hand_made_code():
    # each row a group: rows 0 and 1 update in their check pass, row 2 in a pass of its own
    assert bench.layered_launches(SMALL, 3) == 2 + 1 + 1 + 2
    # two groups, rows {0, 1} and {2}: rows 0 and 1 meet the same columns
    assert bench.layered_launches(SMALL, 2) == 2 + 2 + 2
    # five heavy circulants are no exact shape
    five = code(1, 6, [(0, c, 0) for c in range(5)] + [(0, c, 1) for c in range(5)])
    assert bench.layered_launches(five, 1) == 2 + 2


@pytest.mark.parametrize("schedule, layers, vn_pass, kernels", [
    ("flooding", 0, "accumulate", 2), ("flooding", 0, "separate", 3),
    ("layered", 0, "accumulate", 2 + 30 + 2 * 19), ("layered", 7, "accumulate", 2 + 2 * 7),
])
def test_kernels_of_a_pass_on_the_rate_002_code(schedule, layers, vn_pass, kernels):
    """30 of its 49 rows meet each heavy column once; the others have two
    circulants in one."""
    args = argparse.Namespace(schedule=schedule, layers=layers, vn_pass=vn_pass)
    assert bench.kernels_per_pass(args, synth.rate002_code(64)) == kernels


def test_syndrome_bytes_count_the_rows_that_read_it():
    # rows 0 and 2 have one degree-1 node each, row 1 has none
    assert bench.syndrome_rows(SMALL) == 1
    d = synth.rate002_code(20000)
    assert bench.syndrome_rows(d) == 1
    shape = dict(Z=20000, n_h=119, n_d1=48, n_hcols=2, syn_rows=1)
    cn, vn = bench.pass_bytes(**shape)
    assert cn == 8 * 119 * 20000 + 4 * 50 * 20000 + (1 + 2 * 48) * 20000 / 8 == 23282500
    assert vn == 28 * 2 * 20000
    assert bench.iteration_bytes(**shape) == 8 * 119 * 20000 + 4 * 48 * 20000 + 24 * 20000 + 97 * 20000 / 8
