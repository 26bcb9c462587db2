"""complex64 dense gates on 5 and 6 targets on the tensor cores at FP32's accuracy (csrc/k_tc_x3.cu).

Bound per amplitude, u = 2^-24 and X at most twice the largest real of the group and of the group sharing its 16-byte
chunk (taken over the whole state here): the digits leave out u X / 2 of every x, the second accumulator (2^-6 of the
sum |m||x|, 36 additions) and the closing additions round to a few u of sum |m||x|:
|err| <= u (8 sum |m||x| + X sum |m|)."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu
# every copy order (qubit 0 a target, lowest target 1 to 3, 4 and above) and place of a 5-target gate's extra qubit
CASES = [(23, t) for t in [(0, 1, 2, 3, 4), (18, 19, 20, 21, 22), (22, 0, 7, 3, 5), (1, 0, 8, 4, 6), (2, 9, 3, 6, 11),
                           (15, 9, 1, 6, 22), (3, 5, 14, 6, 9), (4, 9, 12, 6, 11)]] + \
        [(n, t) for n, t in [(22, (0, 1, 2, 3, 4, 5)), (22, (1, 2, 3, 4, 5, 6)), (22, (7, 0, 3, 5, 2, 21)), (23, (3, 4, 5, 6, 7, 8)),
                             (22, (4, 9, 12, 6, 11, 5)), (22, (21, 20, 19, 18, 17, 16)), (22, (2, 9, 3, 6, 11, 13)),
                             (23, (15, 9, 1, 6, 22, 3)), (22, (1, 12, 14, 8, 9, 16))]]


def groups(n, targets):
    idx = np.arange(1 << n)
    first = np.ones(1 << n, bool)
    for q in targets:
        first &= (idx >> q) & 1 == 0
    offs = np.array([sum(((j >> t) & 1) << q for t, q in enumerate(targets)) for j in range(1 << len(targets))])
    return idx[first][None, :] + offs[:, None]


def apply(v, targets, m):
    import torch
    from paper_2308_01999_gb300 import sv
    psi = torch.from_numpy(v.copy()).cuda()
    s = sv.StateVector(psi)
    s.apply(targets, m)
    s.check()
    out = psi.cpu().numpy()
    s.close()
    return out


def check(v, targets, m):
    n = v.size.bit_length() - 1
    at = groups(n, targets)
    want, tol = np.zeros(v.size, complex), np.zeros(v.size)
    want[at] = m @ v[at].astype(complex)
    top = 2 * max(np.max(np.abs(v.real)), np.max(np.abs(v.imag))).astype(float)
    tol[at] = 2.0 ** -24 * (8 * (np.abs(m) @ np.abs(v[at]).astype(float)) + top * np.abs(m).sum(1)[:, None]) + 1e-44
    got = apply(v, targets, m).astype(complex)
    err = np.abs(got - want)
    assert np.all(err <= tol), np.max(err / tol)
    return np.linalg.norm(got - want) / np.linalg.norm(want)


@pytest.mark.parametrize("n,targets", CASES)
def test_against_fp64(n, targets):
    m = gen.random_gate_dense(gen.rng_for(n + len(targets)), len(targets))
    rel = check(gen.random_state(n, 3).astype(np.complex64), targets, m)
    print(f"rel {rel:.2e}")
    assert rel <= 1.5e-7         # the FP32 chains of k_dense5 / k_dense6: 1.5e-7


@pytest.mark.parametrize("k", [5, 6])
def test_scales(k):
    rng = gen.rng_for(k)
    n, targets = 23, tuple(int(q) for q in rng.choice(23, k, replace=False))
    m = gen.random_gate_dense(rng, k)
    v = gen.random_state(n, 4) * 64
    at = groups(n, targets)
    graded = v.copy()
    graded[at] *= 2.0 ** rng.uniform(-30, 0, at.shape[1])[None, :]      # groups of very different sizes
    basis = np.zeros(1 << n, complex)
    basis[77] = 1
    for w in (v * 1e-25, v * 1e30, v * 1e36, graded, basis):
        check(w.astype(np.complex64), targets, m)
    assert not apply((0 * v).astype(np.complex64), targets, m).any()


@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("targets", [(0, 3, 5, 8, 9, 11), (1, 3, 5, 8, 9, 11), (5, 4, 6, 8, 9, 11)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite_groups_only(k, targets, bad):
    n, targets = 23, targets[:k]
    m = gen.random_gate_dense(gen.rng_for(k), k)
    v = gen.random_state(n, 1).astype(np.complex64)
    clean = apply(v, targets, m)
    w = v.copy()
    w[1234] = complex(1.0, bad)
    got = apply(w, targets, m)
    mask = ~sum(1 << q for q in targets)
    group = (np.arange(w.size) & mask) == (1234 & mask)
    assert not np.any(np.isfinite(got[group]))
    assert np.allclose(got[~group], clean[~group], rtol=0, atol=2.0 ** -26)
