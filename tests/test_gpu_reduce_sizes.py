"""<Z_q>, samples and collapse at the sizes where their kernels split the work differently (csrc/k_reduce.cu)."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def make(n, name, seed, sparse=False):
    import torch
    from paper_2308_01999_gb300 import sv
    g = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float32 if name == "complex64" else torch.float64
    v = torch.randn((1 << n, 2), generator=g, device="cuda", dtype=real)
    if sparse:
        v *= (torch.rand(1 << n, generator=g, device="cuda") < 0.01)[:, None]
        v[(1 << n) // 3] = 1
    v /= torch.linalg.vector_norm(v)
    psi = torch.view_as_complex(v)
    return psi, sv.StateVector(psi)


@pytest.mark.parametrize("name,n", [("complex64", n) for n in (3, 8, 12, 14, 15, 24, 25, 27, 28, 29)] +
                         [("complex128", n) for n in (3, 11, 13, 14, 23, 26, 27)])
def test_z_of_every_qubit(name, n):
    import torch
    psi, s = make(n, name, n)
    got = s.expectation_z_all()
    p = torch.view_as_real(psi).double().square_().sum(1)
    want = np.array([float((p.view(-1, 2, 1 << q).sum((0, 2)) * torch.tensor([1.0, -1.0], device="cuda", dtype=p.dtype)).sum())
                     for q in range(n)])
    # complex64: 2u per square, 4u per tree, 8u over the iterations; FP64 (n + 20) u
    tol = 14 * 2.0 ** -24 if name == "complex64" else (n + 20) * 2.0 ** -53
    assert np.max(np.abs(got - want)) <= tol
    s.close()


@pytest.mark.parametrize("name", ["complex64", "complex128"])
@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 9, 11, 12, 13, 20, 25])
def test_samples_bracket_their_random_numbers(name, sparse, n):
    import torch
    psi, s = make(n, name, 50 + n, sparse)
    r = np.sort(np.concatenate([gen.rng_for(n).random(2000), [0.0, np.nextafter(1.0, 0.0)]]))
    got = s.sample(r)
    p = torch.view_as_real(psi).double().square().sum(1)
    cum = torch.cumsum(p, 0).cpu().numpy()
    p = p.cpu().numpy()
    eps = 1e-6 if name == "complex64" else 1e-12      # the segment sums' FP32 runs, as for a probability
    t = r * cum[-1]
    assert np.all(p[got] > 0) and np.all(np.diff(got) >= 0)
    assert np.all(cum[got] - p[got] <= t + eps) and np.all(t <= cum[got] + eps)
    s.close()


@pytest.mark.parametrize("name", ["complex64", "complex128"])
@pytest.mark.parametrize("n,qubits", [(1, [0]), (2, [1]), (5, [0, 3]), (12, [0]), (12, [1, 2]), (13, [4, 11, 0, 7])])
def test_collapse_keeps_one_branch(name, n, qubits):
    import torch
    for parity in (0, 1):
        psi, s = make(n, name, n)
        before = psi.clone()
        s.collapse(qubits, parity, 0.25)
        i = torch.arange(1 << n, device="cuda")
        odd = sum((i >> q) & 1 for q in qubits) % 2
        want = torch.where(odd == parity, before * 2, torch.zeros_like(before))
        assert torch.equal(psi, want)
        s.close()
