"""Many Pauli strings in few passes (csrc/k_pauli.cu), and rotations, where the mask space can go wrong: small
states, dependent and low masks, more strings than a pass holds, against a plain FP64 reference."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def apply_string(v, codes):
    i = np.arange(v.size)
    for q, c in enumerate(codes):
        if c == 1:
            v = v[i ^ (1 << q)]
        elif c == 2:
            v = np.where((i >> q) & 1, 1j, -1j) * v[i ^ (1 << q)]
        elif c == 3:
            v = np.where((i >> q) & 1, -1, 1) * v
    return v


def strings(n, rng):
    some = rng.integers(0, 4, size=(37, n))
    z_only = 3 * rng.integers(0, 2, size=(19, n))
    low = rng.integers(0, 4, size=(9, n)) * (np.arange(n) < 3)
    same_mask = np.where(rng.integers(0, 2, size=(20, n)), 1, 2) * (np.arange(n) % 2) + 3 * (np.arange(n) % 2 == 0) * rng.integers(0, 2, size=(20, n))
    return [some, z_only, low, same_mask, np.concatenate([some[:5], z_only[:18], low, same_mask[:3]]), some[:1], some[:2],
            np.zeros((2, n), int)]


@pytest.mark.parametrize("name", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 11, 17])
def test_strings_against_fp64(name, n):
    import torch
    from paper_2308_01999_gb300 import sv
    rng = gen.rng_for(n)
    psi = torch.from_numpy(gen.random_state(n, 5)).to(getattr(torch, name)).cuda()
    v = psi.cpu().numpy().astype(np.complex128)
    s = sv.StateVector(psi)
    code = sv.SV_C64 if name == "complex64" else sv.SV_C128
    # complex64: 2u per product, 6u along the tree, 2u compensated, of sum |w_i| <= 1 (u = 2^-24)
    tol = 10 * 2.0 ** -24 if name == "complex64" else (n + 40) * 2.0 ** -53
    for p in strings(n, rng):
        p = p.astype(np.int32)
        sites = np.tile(np.arange(n, dtype=np.int32), (len(p), 1))
        want = np.array([np.vdot(v, apply_string(v, c)).real for c in p])
        assert np.max(np.abs(s.expectation_pauli(p, sites) - want)) <= tol
        got = sv.sv_expectation_pauli_noalloc(n, code, psi.data_ptr(), s.stream.cuda_stream, p, sites)
        assert np.max(np.abs(got - want)) <= tol
    s.close()


@pytest.mark.parametrize("name", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [1, 2, 3, 9, 14])
def test_rotations_against_fp64(name, n):
    import torch
    from paper_2308_01999_gb300 import sv
    rng = gen.rng_for(100 + n)
    psi = torch.from_numpy(gen.random_state(n, 6)).to(getattr(torch, name)).cuda()
    want = psi.cpu().numpy().astype(np.complex128)
    s = sv.StateVector(psi)
    count = 0
    for p in strings(n, rng)[:3]:
        for c in p[:8]:
            theta = rng.uniform(-3, 3)
            s.pauli_rotation(theta, c, range(n))
            want = np.cos(theta) * want + 1j * np.sin(theta) * apply_string(want, c)
            count += 1
    # per rotation: cos and sin rounded (u each), product and sum (u each)
    u = 2.0 ** -24 if name == "complex64" else 2.0 ** -53
    got = psi.cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(got - want) <= 4 * count * u + 8 * count * 2.0 ** -53
    s.close()
