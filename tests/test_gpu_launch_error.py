"""A launch that the runtime refuses is reported by its own call and by no later one.

The refusal here: a kernel on the legacy stream while a stream that waits for it is being captured (an error code of the
launch; nothing reaches the GPU)."""
import ctypes as C

import numpy as np
import pytest

from paper_2308_01999_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("matrix", [gen.gate_ry(0.3), np.diag([1, 1j]), gen.gate_x()], ids=["dense", "diagonal", "permutation"])
def test_refused_launch_leaves_no_error_behind(matrix):
    import torch
    from paper_2308_01999_gb300 import sv
    psi = torch.zeros(1 << 6, dtype=torch.complex64, device="cuda")
    s = sv.StateVector(psi)
    s.set_basis_state(0)
    torch.cuda.synchronize()
    cuda = C.CDLL("libcuda.so.1")
    stream, graph = C.c_void_p(), C.c_void_p()
    assert cuda.cuStreamCreate(C.byref(stream), 0) == 0
    assert cuda.cuStreamBeginCapture_v2(stream, 0) == 0
    try:
        with pytest.raises(sv.SvError):
            s.apply((2,), matrix)
    finally:
        cuda.cuStreamEndCapture(stream, C.byref(graph))
    s.pauli_rotation(0.2, [1], [0])                       # a plain launch, which asks for the last error
    assert abs(s.norm2() - 1) < 1e-6
    assert cuda.cuStreamDestroy_v2(stream) == 0
    s.close()
