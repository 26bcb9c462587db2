"""Packing of gate lists (sv.pack_gates): the fields of every gate are its own, whatever the gates beside it hold."""
import itertools
from collections import namedtuple

import numpy as np
import pytest

from paper_2308_01999_gb300 import sv

G = namedtuple("G", "targets matrix controls control_values")
X = np.array([[0, 1], [1, 0]], dtype=complex)


def unpack(rec):
    return [(tuple(int(q) for q in r["targets"][:r["n_targets"]]), tuple(int(q) for q in r["controls"][:r["n_controls"]]),
             tuple(int(q) for q in r["control_values"][:r["n_controls"]])) for r in rec]


@pytest.mark.parametrize("square", [False, True])
def test_longer_control_values_stay_with_their_gate(square):
    """Values beyond a gate's controls are ignored, as the C call ignores them; they never reach the next gate."""
    gates = [G((0,), X, (1, 2), (0, 1, 1)), G((3,), X, (4, 5), (1, 0)), G((6,), X, (7, 8), ()),
             G([0], X, np.array([1, 2]), (0, 0, 0, 1))]
    rec, _ = sv.pack_gates(gates, square)
    assert unpack(rec) == [((0,), (1, 2), (0, 1)), ((3,), (4, 5), (1, 0)), ((6,), (7, 8), (1, 1)), ((0,), (1, 2), (0, 0))]


@pytest.mark.parametrize("lengths", [p for n in (2, 3) for p in itertools.product((1, 2, 3), repeat=n) if 1 in p])
def test_missing_control_values_are_an_error(lengths):
    """Also where the lengths of a group add up to the right total (3 and 1 for two gates of two controls)."""
    gates = [G((0,), X, (1, 2), (0, 1, 0)[:k]) for k in lengths]
    with pytest.raises((IndexError, ValueError)):
        sv.pack_gates(gates)
    with pytest.raises((IndexError, ValueError)):
        sv.sv_fuse_plan(gates, 4, 2)


def test_too_many_targets_is_an_index_error():
    """Not an attempt to allocate 4^k entries."""
    with pytest.raises(IndexError):
        sv.pack_gates([G(tuple(range(24)), X, (), ())])


def test_missing_control_values_in_the_direct_call():
    with pytest.raises(ValueError):
        sv.sv_apply_matrix(0, (0,), X, (1, 2), (1,))
