"""A circuit in one call equals its gates one by one, bit for bit, also where the kernels overlap their launches
(small states) and where a gate in the middle is rejected."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [2, 5, 11, 16])
def test_circuit_equals_gates(name, n):
    import torch
    from paper_2308_01999_gb300 import sv
    rng = gen.rng_for(n)
    gates = gen.layered_random_circuit(n, 6, n, ("cz", "cnot", "crz"))
    for k in range(1, min(n, 6) + 1):
        t = tuple(int(q) for q in rng.choice(n, k, replace=False))
        gates += [gen.Gate(t, gen.random_gate_dense(rng, k), (), ()), gen.Gate(t, np.diag(np.exp(1j * np.arange(1 << k))), (), ())]
    gates.append(gen.Gate((0,), gen.gate_ry(0.3), (1,), (0,)))
    gates.append(gen.Gate((1,), [[0, 1], [1, 0]], (), ()))           # a matrix that is not an array yet
    out = []
    for how in ("circuit", "circuit", "gates"):
        psi = torch.zeros(1 << n, dtype=getattr(torch, name), device="cuda")
        s = sv.StateVector(psi)
        s.set_basis_state(1)
        if how == "circuit":
            s.apply_circuit(gates)
        else:
            for g in gates:
                s.apply_gate(g)
                torch.cuda.synchronize()
        out.append(psi.cpu())
        s.close()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


@pytest.mark.parametrize("bad", [gen.Gate((7,), gen.gate_x()), gen.Gate((0,), np.eye(4)), gen.Gate((0,), gen.gate_x(), (0,)),
                                 gen.Gate((0,) * 7, np.eye(128))])
def test_rejected_gate_ends_the_circuit(bad):
    import torch
    from paper_2308_01999_gb300 import sv
    psi = torch.zeros(1 << 4, dtype=torch.complex64, device="cuda")
    s = sv.StateVector(psi)
    s.set_basis_state(0)
    with pytest.raises((sv.SvError, ValueError)):
        s.apply_circuit([gen.Gate((2,), gen.gate_x()), bad, gen.Gate((3,), gen.gate_x())])
    assert abs(complex(psi[4])) == 1                                  # the first gate applied, the third did not
    s.close()
