"""complex128 dense gates in block fixed point (csrc/k_dense_fx.cu) where its groups are uneven (u = 2^-53).

Parts: a matrix whose entries are all real, or that becomes so when some rows and columns are multiplied by i, adds
nothing from one half of a group's parts to the other. Each part is held to 2 (2 * 2^k + 2) u of its own sum."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen
from tests.test_gpu_dense_fx import U, apply

pytestmark = pytest.mark.gpu
LD = np.longdouble


def exact(m, x):
    mr, mi, a, b = (p.astype(LD) for p in (m.real, m.imag, x.real, x.imag))
    return mr @ a - mi @ b, mr @ b + mi @ a


def run(m, x):
    """m on the groups x (members x groups): targets are the lowest qubits, so that column g is group g."""
    k = m.shape[0].bit_length() - 1
    out = apply(np.ascontiguousarray(x.T).reshape(-1), tuple(range(k)), m).reshape(-1, 1 << k).T
    return out.real, out.imag


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
