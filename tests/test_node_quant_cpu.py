"""Box quantisation at the ends of FP32: trees over quads of extreme size,
offset or flatness keep their invariants (every dequantised child box contains
the exact one), host-built and by the host run of the linear builder."""
import ctypes as C

import numpy as np
import pytest

from paper_2001_02620_gb300 import build as B
from paper_2001_02620_gb300 import inputs as I


@pytest.fixture(scope="module")
def native():
    B.build()
    from paper_2001_02620_gb300 import _native as N
    return N


@pytest.mark.parametrize("builder", [0, 2])
@pytest.mark.parametrize("scale,offset,flat", [
    (1.0, 0.0, False), (1.0, 0.0, True), (1e-3, 1e6, False), (1.0, 3.0e7, False), (1e-38, 0.0, False),
    (1e-44, 0.0, False), (1e30, 0.0, True), (3.0e38, 0.0, False), (1e-30, -1e-3, False)])
def test_extreme_boxes(native, builder, scale, offset, flat):
    v, q = I.tiny_mesh()
    v = v.astype(np.float64)
    if flat:
        v[:, 2] = 0.25
    v = np.clip(v * scale + offset, -3.3e38, 3.3e38).astype(np.float32)
    q = np.ascontiguousarray(q[:900])
    m = native.qrt_mesh(v.ctypes.data_as(C.POINTER(C.c_float)), v.shape[0],
                        q.ctypes.data_as(C.POINTER(C.c_uint32)), q.shape[0])
    o = native.qrt_build_opts()
    o.blas_builder = builder
    nn, d = C.c_uint64(), C.c_uint32()
    rc = native.lib().qrt_blases_build_check((native.qrt_mesh * 1)(m), 1, C.byref(o), C.byref(nn), C.byref(d))
    assert rc == 0, native.lib().qrt_last_error()
    assert nn.value > 0
