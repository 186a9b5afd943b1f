"""The loops of the 8-bit levels, played on the host with a warp's lanes in several orders between two votes: nothing but
a vote keeps lanes together, so the marks must not depend on the order.  CTAs with fewer sub-blocks than a warp has lanes
are the delicate ones: some lanes have no sub-block of their own."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1912_04050_b200 import build, inputs

HERE = os.path.dirname(os.path.abspath(__file__))
N, MARK_STRIDE = 256, 136


@pytest.fixture(scope="module")
def lanes(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("lanes") / "loop_lanes.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-fno-strict-aliasing", "-I", build.CSRC,
                           "-o", so, os.path.join(HERE, "host", "loop_lanes.cpp")])
    return ctypes.CDLL(so)


def permutation(kind, rng):
    if kind == "random":
        return rng.permutation(N)
    p = inputs.structured_perms(8)[kind].astype(np.int64)
    a, b = rng.integers(0, N, 2)                             # (two outputs swapped: no two sub-blocks alike)
    p[[a, b]] = p[[b, a]]
    return p


def play(lanes, perms, order, valid=None):
    """The marks as the lanes leave them, one row per sub-block, and the number of votes."""
    succ = np.empty((len(perms), N), np.uint8)
    j = np.arange(N)
    for r, p in enumerate(perms):
        inv = np.empty(N, np.int64)
        inv[p] = j
        succ[r] = inv[p[j ^ 1] ^ 1]
    marks = np.zeros((len(perms), MARK_STRIDE), np.uint8)
    ptr = [a.ctypes.data_as(ctypes.c_void_p) for a in (succ, marks)]
    votes = lanes.play_loop_marks(len(perms), len(perms) if valid is None else valid, *ptr, order)
    assert votes > 0
    return marks[:, :N // 2], votes


def marks_wanted(p):
    words = oracle.route(p.astype(np.uint32), 8)[14]          # the output side of the first level
    return 2 + ((np.repeat(words, 32) >> np.tile(np.arange(32, dtype=np.uint32), 4)) & 1)


@pytest.mark.parametrize("kind", ["random", "identity", "shift1", "transpose", "sattolo"])
@pytest.mark.parametrize("regions", [4, 8, 16, 32])
def test_marks_of_sub_blocks_do_not_depend_on_the_order_of_the_lanes(lanes, regions, kind):
    """Lanes ascending, descending, and shuffled at every vote.  (Where lanes without a sub-block repeated the last one's
    walk, about one shuffled round of random permutations in fifty came out wrong.)"""
    rng = np.random.default_rng(regions)
    for order in range(400 if kind == "random" else 40):
        perms = [permutation(kind, rng) for _ in range(regions)]
        marks, _ = play(lanes, perms, order)
        for r, p in enumerate(perms):
            assert np.array_equal(marks[r], marks_wanted(p)), (kind, r, order)


@pytest.mark.parametrize("regions,valid", [(16, 1), (16, 5), (16, 16), (32, 31)])
def test_padding_gets_no_marks_and_takes_no_rounds(lanes, regions, valid):
    """Sub-blocks of padding, the identity, beside random ones: 128 loops of one switch each would keep the others waiting."""
    rng = np.random.default_rng(100 * regions + valid)
    perms = [rng.permutation(N) for _ in range(valid)] + [np.arange(N)] * (regions - valid)
    marks, votes = play(lanes, perms, 2, valid)
    for r in range(valid):
        assert np.array_equal(marks[r], marks_wanted(perms[r])), r
    assert not marks[valid:].any()
    assert votes == play(lanes, perms[:valid], 2)[1]


@pytest.mark.parametrize("short,kind,most", [(1, "identity", 64), (5, "identity", 64), (15, "identity", 64),
                                             (9, "transpose", 64), (15, "bitrev", 64)])
def test_sub_blocks_of_short_loops_beside_random_ones(lanes, short, kind, most):
    """A lane whose loops all end within a round keeps the others waiting: loops of one switch are marked without walks
    however few such lanes there are, loops of two where most are such.  (Round by round they take 128 and 70 votes; a
    random permutation has 128 hops, three to a round, a hop or two of every loop lost: 48 to 60.)"""
    rng = np.random.default_rng(short)
    perms = [rng.permutation(N) for _ in range(16)]
    for r in rng.permutation(16)[:short]:
        perms[r] = inputs.structured_perms(8)[kind].astype(np.int64)
    marks, votes = play(lanes, perms, 2)
    for r, p in enumerate(perms):
        assert np.array_equal(marks[r], marks_wanted(p)), r
    assert votes <= most, votes

