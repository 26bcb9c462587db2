"""Expectation sums of the batched engine whose terms overflow FP32: an infinite sum stays infinite, with its sign, for
strings that share a pass as for a string on its own."""
import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 9, 14, 15])
@pytest.mark.parametrize("count", [1, 2, 3, 6])
def test_infinite_terms(n, count):
    import torch
    from paper_2308_01999_gb300 import sv
    h = np.array([[1, 1], [1, -1]]) / np.sqrt(2)
    gates = [gen.Gate((q,), h * (1e25 if q == 0 else 1)) for q in range(n)]        # amplitudes 1e25 2^(-n/2), all alike
    paulis = np.zeros((count, n), np.int32)
    for s in range(count):
        paulis[s, s % n] = 1                                                         # X: every pair's term is +infinity
    b = sv.Batch(torch.cuda.current_stream())
    b.compile([(n, gates, paulis)])
    buf = torch.empty(b.state_amps, dtype=torch.complex64, device="cuda")
    b.launch(buf)
    assert np.all(b.results()[0] == np.inf)
    b.close()
