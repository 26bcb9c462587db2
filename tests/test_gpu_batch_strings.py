"""Expectation sums of the batched engine where strings share passes: dependent, equal and empty masks, every group
size, small and split states, against a plain FP64 reference of the same circuit's state."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def expect(v, codes):
    i, w = np.arange(v.size), v
    for q, c in enumerate(codes):
        if c == 1:
            w = w[i ^ (1 << q)]
        elif c == 2:
            w = np.where((i >> q) & 1, 1j, -1j) * w[i ^ (1 << q)]
        elif c == 3:
            w = np.where((i >> q) & 1, -1, 1) * w
    return np.vdot(v, w).real


def strings(n, rng):
    a, b, c = (rng.integers(0, 4, size=n) for _ in range(3))
    z = 3 * rng.integers(0, 2, size=n)
    ab = np.where((a % 3 != 0) != (b % 3 != 0), 1, 0)                 # X/Y mask = mask(a) ^ mask(b)
    low = rng.integers(0, 4, size=n) * (np.arange(n) < 2)
    return [[a], [a, b], [a, a, b], [a, b, ab], [a, b, c], [z, a, b, c, z], [a, z, b], [low, a, b, c], [np.zeros(n, int), z, low, a],
            [a, b, c, b, a, ab, c, z]]


@pytest.mark.parametrize("n", [2, 3, 4, 5, 9, 14, 15, 18, 19])
def test_strings_in_groups(n):
    import torch
    from paper_2308_01999_gb300 import sv
    rng = gen.rng_for(n)
    lists = strings(n, rng)
    states = [(n, gen.ansatz_circuit(n, 2, gen.rng_for(7)), np.array(p, dtype=np.int32)) for p in lists]
    b = sv.Batch(torch.cuda.current_stream())
    b.compile(states)
    buf = torch.empty(b.state_amps, dtype=torch.complex64, device="cuda")
    b.launch(buf, keep_states=True)
    res = b.results()
    for (off, m, _, _), p, got in zip(b.offsets, lists, res):
        v = buf[off:off + (1 << m)].cpu().numpy().astype(np.complex128)
        want = [expect(v, c) for c in p]
        # 2u per product, 3u per tree (8u for a single string's runs), 2u compensated, factor 2, sum |w| <= 1
        assert np.max(np.abs(got - want)) <= 24 * 2.0 ** -24
    b.close()
