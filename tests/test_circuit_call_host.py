"""StateVector.apply_circuit hands a list of gates to one native call; whatever else yields gates goes through
apply_gate one by one, each gate asked for after the one before it has been applied (no GPU needed: the calls
are recorded)."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen
from paper_2308_01999_gb300 import sv

X = gen.gate_x()


@pytest.fixture
def state(monkeypatch):
    s = sv.StateVector.__new__(sv.StateVector)
    s.handle = None
    s.log = []
    monkeypatch.setattr(sv, "sv_apply_matrix", lambda h, t, m, c=(), cv=None, adjoint=False: s.log.append(("apply", tuple(t))))
    return s


def test_generator_sees_the_gates_before_it(state):
    """A program may choose the next gate by what it measures on the state so far."""
    def program():
        for q in range(3):
            state.log.append(("ask", q))
            yield gen.Gate((q,), X)

    state.apply_circuit(program())
    assert state.log == [(what, q) for k in range(3) for what, q in (("ask", k), ("apply", (k,)))]


def test_iterable_object_is_walked_in_step(state):
    class Program:
        def __iter__(self):
            for q in range(2):
                state.log.append(("ask", q))
                yield gen.Gate((q,), X)

    state.apply_circuit(Program())
    assert state.log == [("ask", 0), ("apply", (0,)), ("ask", 1), ("apply", (1,))]


@pytest.mark.parametrize("bad", [gen.Gate((1 << 40,), X), gen.Gate((0,) * 24, X), gen.Gate((0,), X, (1, 2), (1,)),
                                 gen.Gate((0,), "no matrix")])
def test_gates_before_one_that_cannot_be_packed(state, bad):
    state.apply_circuit([gen.Gate((2,), X), bad])
    assert state.log[0] == ("apply", (2,))


def test_overridden_apply_gate_is_called(state):
    class Counting(sv.StateVector):
        def apply_gate(self, g, adjoint=False):
            self.log.append(g.targets)

    state.__class__ = Counting
    state.apply_circuit([gen.Gate((0,), X), gen.Gate((1,), np.eye(2))])
    assert state.log == [(0,), (1,)]


def test_long_lists_are_packed_in_parts(state, monkeypatch):
    """The packed copies of the matrices stay bounded, whatever the circuit's length; the order is kept."""
    calls = []

    class Lib:
        @staticmethod
        def sv_apply_circuit(h, gates, n):
            calls.append([gates[i].targets[0] for i in range(n)])
            return 0

    monkeypatch.setattr(sv, "lib", lambda: Lib)
    order = [i % 7 for i in range(10001)]
    state.apply_circuit([gen.Gate((q,), X) for q in order])
    assert sum(calls, []) == order
    assert max(map(len, calls)) <= 4096
    wide = gen.Gate(tuple(range(6)), np.eye(64))
    calls.clear()
    state.apply_circuit((wide,) * 600)
    assert sum(map(len, calls)) == 600 and max(map(len, calls)) * 64 * 64 * 16 <= 1 << 25


def test_gate_that_cannot_be_packed_in_a_later_part(state, monkeypatch):
    class Lib:
        @staticmethod
        def sv_apply_circuit(h, gates, n):
            state.log.extend(("apply", (gates[i].targets[0],)) for i in range(n))
            return 0

    monkeypatch.setattr(sv, "lib", lambda: Lib)
    gates = [gen.Gate((i % 5,), X) for i in range(5000)]
    state.apply_circuit(gates + [gen.Gate((0,) * 24, X), gen.Gate((3,), X)])   # the recorder takes everything
    assert [t for _, t in state.log[:5000]] == [g.targets for g in gates] and len(state.log) == 5002
