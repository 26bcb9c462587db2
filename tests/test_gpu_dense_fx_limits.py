"""complex128 dense gates in block fixed point (csrc/k_dense_fx.cu) where their ranges end.

Spread: matrices whose small entries meet the large amplitudes of a group are held, amplitude by amplitude, to 1.25
times the worst error of the FP64 chain that the kernel stands in for, on the same groups (both as multiples of
u sum |m||x|, u = 2^-53; the quarter is for the maximum of a few thousand groups being itself a random number), and
never below 3 u for the closing roundings.
Full sums: largest digits of one sign, whose sums come near 2^24 units, stay within 2 u, and cancel where half of them
change sign, to what the kernel states that it leaves out (2^-65 of the sum of magnitudes; a sum of digits that is off
by one unit would show as 2^-50).
Parts: a matrix whose entries are all real, or that becomes so when some rows and columns are multiplied by i, adds
nothing from one half of a group's parts to the other. Each part is held to 2 (2 * 2^k + 2) u of its own sum."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen
from tests.test_gpu_dense_fx import U, apply

pytestmark = pytest.mark.gpu
LD = np.longdouble


def chain(m, x):
    """One chain of FP64 multiply-adds per part, members in order."""
    def fma(a, b, c):
        return (a.astype(LD) * b.astype(LD) + c.astype(LD)).astype(np.float64)

    re = im = np.zeros(x.shape)
    for a, b in zip(m.T[:, :, None], x[:, None, :]):
        re = fma(-a.imag, b.imag, fma(a.real, b.real, re))
        im = fma(a.imag, b.real, fma(a.real, b.imag, im))
    return re, im


def exact(m, x):
    mr, mi, a, b = (p.astype(LD) for p in (m.real, m.imag, x.real, x.imag))
    return mr @ a - mi @ b, mr @ b + mi @ a


def run(m, x):
    """m on the groups x (members x groups): targets are the lowest qubits, so that column g is group g."""
    k = m.shape[0].bit_length() - 1
    out = apply(np.ascontiguousarray(x.T).reshape(-1), tuple(range(k)), m).reshape(-1, 1 << k).T
    return out.real, out.imag


def worst(got, want, scale):
    err = np.hypot(*(np.abs(g - w).astype(float) for g, w in zip(got, want)))
    return np.max(err / scale) / U


def spread_matrix(rng, k, dm, small):
    """Entries near the largest, but the first `small` columns' exponents dm below it."""
    d = 1 << k
    m = rng.uniform(.5, 1, (d, d)) * rng.choice([-1, 1], (d, d)) + 1j * rng.uniform(.5, 1, (d, d)) * rng.choice([-1, 1], (d, d))
    m[:, :small] = (0.5 + 0.02 * rng.random((d, small))) * 2.0 ** -dm * (1 + 1j * rng.uniform(-1, 1, (d, small)))
    return m


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dm", [4, 5, 6, 7, 8, 11, 12, 17])
@pytest.mark.parametrize("depth", [3, 9, 14, 30, 2000])
def test_small_entries_meet_large_amplitudes(k, dm, depth):
    rng = gen.rng_for(100 * k + dm)
    d, count = 1 << k, 4096 >> max(0, k - 3)
    for small in sorted({1, d // 2}):
        m = spread_matrix(rng, k, dm, small)
        for large in sorted({1, small, min(small + 1, d)}):
            x = (rng.standard_normal((d, count)) + 1j * rng.standard_normal((d, count))) * 2.0 ** -depth
            x[:large] = rng.uniform(.5, 1, (large, count)) + 1j * rng.uniform(-1, 1, (large, count))
            want, scale = exact(m, x), np.abs(m) @ np.abs(x)
            here, fp64 = worst(run(m, x), want, scale), worst(chain(m, x), want, scale)
            print(f"small {small}, large {large}: {here:.2f} u, FP64 {fp64:.2f} u")
            assert here <= 1.25 * max(fp64, 2.4), (small, large, here, fp64)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dm", [7, 8, 9, 10, 11])
@pytest.mark.parametrize("real", [False, True])
def test_small_entries_anywhere(k, dm, real):
    """Small entries in any places, and groups with any of their amplitudes large, the others small or zero."""
    rng = gen.rng_for(1000 * k + dm + real)
    d, count = 1 << k, 4096 >> max(0, k - 3)
    m = spread_matrix(rng, k, dm, 0)
    m = np.where(rng.random((d, d)) < 0.3, 2.0 ** -dm * rng.uniform(0.9, 1, (d, d)), 1) * m
    if real:
        m = m.real + 0j
    x = rng.uniform(.5, 1, (d, count)) + 1j * rng.uniform(-1, 1, (d, count))
    x *= np.where(rng.random((d, count)) < rng.uniform(0, 1, count), 1, 2.0 ** -rng.choice([3, 14, 30, 2000], count).astype(float))
    x[0, ~x.any(axis=0)] = 1
    want, scale = exact(m, x), np.abs(m) @ np.abs(x)
    here, fp64 = worst(run(m, x), want, scale), worst(chain(m, x), want, scale)
    print(f"dm {dm}, real {real}: {here:.2f} u, FP64 {fp64:.2f} u")
    assert here <= 1.25 * max(fp64, 2.4)


@pytest.mark.parametrize("k", [3, 4, 5])
@pytest.mark.parametrize("digit", [8, 9])
def test_full_sums_of_digits(k, digit):
    d = 1 << k
    bits = "1" * (digit - 2)                                            # the top digit, then digits of all ones below their sign
    while len(bits) < 53:
        bits += "0" + "1" * (digit - 1)
    a = int(bits[:53], 2) * 2.0 ** -53
    m = np.full((d, d), a - 1j * a)
    m[1::2] = a + 1j * a                                                # these rows' imaginary parts add up, the others' real parts
    x = np.full((d, 8), a + 1j * a)
    x[d // 2:, 1::2] *= -1
    want, got = exact(m, x), run(m, x)
    left_out = 2.0 ** -65 * (np.abs(m) @ np.abs(x))
    for w, g in zip(want, got):
        assert np.all(np.abs(g - w).astype(float) <= 2 * U * np.abs(w).astype(float) + left_out)


def real_like(rng, k):
    """Real matrices, the same under multiplications of rows and columns by i, and with zero entries; and the phases of
    the columns."""
    d = 1 << k
    phase = np.array([1, 1j])
    h = np.array([[1.0]])
    for _ in range(k):
        h = np.kron(h, np.array([[1, 1], [1, -1]]) / np.sqrt(2))
    for real in (h, np.linalg.qr(rng.standard_normal((d, d)))[0] + 0.3):
        zero = real * (rng.random((d, d)) < 0.8)
        zero[0] = real[0]
        rows, cols = phase[rng.integers(0, 2, d)][:, None], phase[rng.integers(0, 2, d)]
        one = np.ones(d)
        yield real + 0j, one
        yield 1j * real, one
        yield rows * real * cols, cols
        yield rows * zero * cols, cols


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_real_gates_keep_small_parts(k):
    rng = gen.rng_for(k)
    d = 1 << k
    a, b = rng.standard_normal((d, 256)), rng.standard_normal((d, 256))
    for m, phase in real_like(rng, k):
        for v in (a + 1e-8j * b, 1e-8 * a + 0.6j * b, 0 * a + 1j * b, a + 0j, a + 1e-40j * b, a + 1e-300j * b):
            for x in (v, phase[:, None] * v):
                want = exact(m, x)
                sums = (np.abs(m.real) @ np.abs(x.real) + np.abs(m.imag) @ np.abs(x.imag),
                        np.abs(m.real) @ np.abs(x.imag) + np.abs(m.imag) @ np.abs(x.real))
                for g, w, s in zip(run(m, x), want, sums):
                    assert np.all(np.abs(g - w).astype(float) <= 2 * (2 * d + 2) * U * s + 1e-320)
