"""complex64 dense gates on 5 and 6 targets in native precision, held to each group's own scale.

A group is the 2^k amplitudes that a gate mixes; nothing outside it may enter its result's error. With
u = 2^-24, the closing additions round to about 4 u sum |m||x| per amplitude. The digits leave out at most
2^-34 of the group's largest part and of the row's largest entry per product; over 128 products of random sign
(rms a third of the most, 4.5 standard deviations) that is 2^-31 of both, 8 u sum |m||x| at a row spread
of 2^10 (an entry 2^-10 of the row's largest that meets the one large amplitude).
Tolerance per amplitude: 12 u sum |m||x| over the group, and 10 u of the norm per group; matrices of a wider spread are
held to what FP32 chains have (or left to them), whose 2 * 2^k partial sums (each at most sum |m||x|) round by u / sqrt(3) rms: 4.5 deviations are
4.5 sqrt(2 * 2^k / 3) u per amplitude. Where the entries' spread is what is tested, the worst amplitude of 4096 groups
is also held to twice that of such a chain on the same groups."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen
from tests.test_gpu_tc_x3 import apply, groups

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
TARGETS = [(23, (0, 3, 5, 8, 9)), (23, (1, 3, 5, 8, 9)), (23, (22, 4, 6, 8, 9)), (22, (0, 1, 2, 3, 4, 5)),
           (22, (1, 2, 4, 9, 12, 21)), (22, (4, 9, 12, 6, 11, 5))]


def check(v, targets, m, parts=False, limit=12):
    n = v.size.bit_length() - 1
    v = v.astype(np.complex64)
    at = groups(n, targets)
    x = v[at].astype(complex)
    want = m @ x
    got = apply(v, targets, m).astype(complex)[at]
    err = np.abs(got - want)
    worst = np.max(err / (U * (np.abs(m) @ np.abs(x)) + 1e-40))
    norm = np.linalg.norm(want, axis=0)
    group = np.max(np.linalg.norm(err, axis=0) / (norm + 1e-35))
    print(f"worst {worst:.2f} u, group {group:.2e}")
    assert worst <= limit
    assert group <= 10 * U or limit > 12
    if parts:
        for a, b in ((got.real - want.real, np.abs(x.real)), (got.imag - want.imag, np.abs(x.imag))):
            assert np.all(np.abs(a) <= 12 * U * (np.abs(m.real) @ b) + 1e-40)
    return x, want, got


def chain(k):
    return 4.5 * (2 * 2 ** k / 3) ** 0.5


def fp32_chain(m, x):
    """The product as one chain of FP32 multiply-adds per part, members in order."""
    m, x = m.astype(np.complex64), x.astype(np.complex64)

    def fma(a, b, c):
        return (a.astype(float) * b.astype(float) + c).astype(np.float32)

    re = im = np.zeros((m.shape[0], x.shape[1]), np.float32)
    for a, b in zip(m.T[:, :, None], x[:, None, :]):
        re = fma(-a.imag, b.imag, fma(a.real, b.real, re))
        im = fma(a.imag, b.real, fma(a.real, b.imag, im))
    return re.astype(float) + 1j * im


def lowest_free(targets):
    return next(q for q in range(8) if q not in targets)


@pytest.mark.parametrize("n,targets", TARGETS)
@pytest.mark.parametrize("ratio", [2.0 ** -4, 2.0 ** -8, 2.0 ** -16, 2.0 ** -24])
def test_small_group_beside_a_large_one(n, targets, ratio):
    """Groups that differ in the lowest qubit that is no target share 16-byte chunks."""
    m = gen.random_gate_dense(gen.rng_for(n), len(targets))
    v = gen.random_state(n, 5) * 32
    bit = (np.arange(v.size) >> lowest_free(targets)) & 1
    check(np.where(bit == 1, ratio, 1.0) * v, targets, m)


@pytest.mark.parametrize("n,targets", TARGETS)
def test_groups_over_many_orders(n, targets):
    m = gen.random_gate_dense(gen.rng_for(n + 1), len(targets))
    v = gen.random_state(n, 6) * 64
    at = groups(n, targets)
    v[at] *= 2.0 ** gen.rng_for(n).uniform(-30, 0, at.shape[1])[None, :]
    check(v, targets, m)


def limit_matrix(k, spread):
    """Rows whose entry of column 3 is 2^-spread of the row's largest, every other entry at least that."""
    m = gen.random_gate_dense(gen.rng_for(k), k)
    top = np.abs(m).max(1, keepdims=True)
    m = m * np.maximum(1.0, top * 2.0 ** -spread / np.abs(m))
    m[:, 3] *= top[:, 0] * 2.0 ** -spread / np.abs(m[:, 3])
    return m


@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("spread", [0, 4, 8, 9.999, 10.9, 11, 13])
def test_one_large_amplitude_meets_the_small_entries(k, spread):
    n, targets = 23, (2, 5, 6, 11, 13, 17)[:k]
    m = gen.random_gate_dense(gen.rng_for(k), k) if spread == 0 else limit_matrix(k, spread)
    at = groups(n, targets)
    for depth in (8, 12, 16, 20):
        v = gen.random_state(n, depth) * 2.0 ** (n / 2 - depth)
        v[at[3]] = np.exp(1j * np.arange(at.shape[1]))
        x, want, got = (a[:, :4096] for a in check(v, targets, m, limit=12 if spread <= 10 else chain(k)))
        scale = np.abs(m) @ np.abs(x)
        assert np.max(np.abs(got - want) / scale) <= 2 * np.max(np.abs(fp32_chain(m, x) - want) / scale)


@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("angle", [0.01, 0.3])
def test_near_identity(k, angle):
    """exp(-i angle H) for a Hermitian H without zero entries, on groups with one large amplitude."""
    n, targets = 23, (0, 5, 6, 11, 13, 17)[:k]
    a = gen.random_gate_dense(gen.rng_for(k), k)
    w, q = np.linalg.eigh(a + a.conj().T)
    m = (q * np.exp(-1j * angle * w)) @ q.conj().T
    v = gen.random_state(n, 2) * 2.0 ** (n / 2 - 12)
    v[groups(n, targets)[1]] = 1
    check(v, targets, m, limit=chain(k))


@pytest.mark.parametrize("k", [5, 6])
def test_real_gate_keeps_small_parts(k):
    """A real matrix does not mix real and imaginary parts: each is held to its own scale."""
    n, targets = 23, (1, 5, 6, 11, 13, 17)[:k]
    rng = gen.rng_for(k)
    q = np.linalg.qr(rng.standard_normal((1 << k, 1 << k)))[0]
    q = np.where(np.abs(q) < 2.0 ** -9, 2.0 ** -9, q) + 0j
    v = gen.random_state(n, 7)
    check(v.real + 1j * 2.0 ** -18 * v.imag, targets, q, parts=True)
    check(2.0 ** -25 * v.real + 1j * v.imag, targets, q, parts=True)
