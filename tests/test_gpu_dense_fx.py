"""complex128 dense gates in block fixed point (csrc/k_dense_fx.cu) against extended precision.

Every output amplitude of a dense gate in FP64 is within (2 * 2^k + 2) u sum_l |m_l| |x_l| of the exact
product (u = 2^-53; 2 * 2^k roundings of a real sum, two more for the parts); the tests hold each amplitude,
however small beside the others, to twice that: once for the kernel, once for margin between a complex
modulus and its parts.
"""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def exact_and_bound(v, targets, m, controls=()):
    """m on the targets in extended precision, and sum |m||x| for every amplitude (0 where the gate does nothing)."""
    n, k = v.size.bit_length() - 1, len(targets)
    idx = np.arange(v.size)
    first = np.ones(v.size, bool)
    for q in targets:
        first &= (idx >> q) & 1 == 0
    for c in controls:
        first &= (idx >> c) & 1 == 1
    base = idx[first]
    offs = np.array([sum(((j >> t) & 1) << q for t, q in enumerate(targets)) for j in range(1 << k)])
    at = base[None, :] + offs[:, None]
    x = v[at].astype(np.clongdouble)
    out, bound = v.astype(np.clongdouble), np.zeros(v.size)
    out[at] = m.astype(np.clongdouble) @ x
    bound[at] = (np.abs(m) @ np.abs(x).astype(np.float64))
    return out, bound


def apply(v, targets, m, controls=()):
    import torch
    from paper_2308_01999_gb300 import sv
    psi = torch.from_numpy(v.copy()).cuda()
    s = sv.StateVector(psi)
    s.apply(targets, m, controls)
    out = psi.cpu().numpy()
    s.close()
    return out


def check(v, targets, m, controls=()):
    want, bound = exact_and_bound(v, targets, m, controls)
    got = apply(v, targets, m, controls).astype(np.clongdouble)
    tol = 2 * (2 * m.shape[0] + 2) * U * bound + 1e-320
    err = np.abs(got - want).astype(np.float64)
    assert np.all(err <= tol), f"worst {np.max(err / tol)} of the bound"


def states(n, rng):
    v = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    yield "normal", v
    yield "graded", v * 2.0 ** rng.uniform(-40, 0, v.size)
    yield "mixed groups", v * 2.0 ** rng.uniform(-8, 0, v.size)
    yield "sparse", np.where(rng.random(v.size) < 0.7, 0, v)
    yield "small parts", v.real + 1e-12j * v.imag
    yield "tiny", v * 1e-290
    yield "denormal", v * 2.0 ** rng.uniform(-1070, -1000, v.size)
    yield "huge", v * 1e250
    basis = np.zeros(1 << n, complex)
    basis[5 % v.size] = 1
    yield "basis", basis


@pytest.mark.parametrize("targets", [(0,), (3,), (0, 1), (5, 2), (0, 4, 7), (8, 1, 3), (0, 1, 2, 3), (7, 3, 8, 5),
                                     (0, 1, 2, 3, 4), (8, 2, 6, 3, 5)])
def test_dense_matches_extended_precision(targets):
    rng = gen.rng_for(7 + len(targets))
    k = len(targets)
    m = gen.random_gate_dense(rng, k)
    near_identity = np.eye(1 << k) + 1e-4 * m          # entries of very different sizes
    sparse = m.copy()
    sparse[rng.random(m.shape) < 0.3] = 0
    sparse[0, 0], sparse[0, -1] = 1, 0.5
    level = np.exp(2j * np.pi * rng.random(m.shape))   # every entry as large as the largest: full sums
    edge = level.copy()
    edge[0, 1], edge[-1, 0] = 2.0 ** -5 * (1 + 1j), 1e-3
    for matrix in (m, level, edge, near_identity, sparse, 1e30 * m, np.full(m.shape, -1.0 + 1.0j), m.real + 0j):
        for _, v in states(9, rng):
            with np.errstate(all="ignore"):
                check(v.astype(np.complex128), targets, matrix.astype(np.complex128))


@pytest.mark.parametrize("n,targets,controls", [(1, (0,), ()), (2, (1, 0), ()), (3, (0, 2), (1,)), (4, (3, 0, 1, 2), ()),
                                                (6, (4, 2, 5), (0, 3)), (13, (12,), (0,)), (13, (0, 6, 11, 12), (3,)), (4, (2, 0, 3), ()), (5, (1, 4, 2), ()),
                                                (5, (0, 1, 2, 3, 4), ()), (7, (6, 0, 2, 5, 3), ()), (8, (1, 7, 4), (0, 2, 5)),
                                                (15, (0, 9, 14, 3), ())])
def test_dense_small_states_and_controls(n, targets, controls):
    rng = gen.rng_for(n)
    m = gen.random_gate_dense(rng, len(targets))
    check(gen.random_state(n, 3), targets, m, controls)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_dense_nonfinite_groups_only(k, bad):
    """A non-finite amplitude spoils its own group, as in FP64, and no other."""
    rng = gen.rng_for(k)
    m = gen.random_gate_dense(rng, k)
    v = gen.random_state(8, 1)
    targets = tuple(range(1, k + 1))
    want, bound = exact_and_bound(v, targets, m)
    w = v.copy()
    w[200] = complex(bad, 1.0)
    got = apply(w, targets, m)
    group = (np.arange(w.size) & ~sum(1 << q for q in targets)) == (200 & ~sum(1 << q for q in targets))
    assert not np.any(np.isfinite(got[group]))
    assert np.all(np.abs(got - want)[~group] <= 2 * (2 * m.shape[0] + 2) * U * bound[~group])
