"""Network prediction where page-locked memory is not to be had: the library's
network compiled with an allocation that fails (the runtime's typed
cudaMallocHost calls cudaHostAlloc), against the library itself."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1204_4098_gb300 import build, lbm, warmstart

pytestmark = pytest.mark.gpu

STUB = r"""
#include <cuda_runtime.h>
extern "C" cudaError_t no_page_locked_memory(void**, size_t, unsigned) {
  return cudaErrorMemoryAllocation;
}
namespace lbm { void count_launches(unsigned long long) {} }
"""


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    d = tmp_path_factory.mktemp("mlp")
    (d / "stub.cu").write_text(STUB)
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    for src, extra, obj in ((os.path.join(build.CSRC, "lbm_mlp.cu"),
                             ["-DcudaHostAlloc=no_page_locked_memory"], "mlp.o"),
                            (str(d / "stub.cu"), [], "stub.o")):
        subprocess.run([build._nvcc(), *build.ARCH, *flags, *extra, "-c", src, "-o",
                        str(d / obj)], check=True, capture_output=True, text=True)
    subprocess.run([build._nvcc(), *build.ARCH, "-shared", "-o", str(d / "mlp.so"),
                    str(d / "mlp.o"), str(d / "stub.o")], check=True, capture_output=True,
                   text=True)
    return ctypes.CDLL(str(d / "mlp.so"))


def test_small_predictions_go_through_device_memory(L):
    P = ctypes.c_void_p
    params = warmstart.glorot_params(3)
    rng = np.random.default_rng(1)
    m = P()
    assert L.lbm_mlp_create(0, None, ctypes.byref(m)) == lbm.LBM_OK
    assert L.lbm_mlp_set_params(m, P(params.ctypes.data)) == lbm.LBM_OK
    want = lbm.MLP(params)
    for n in (1, 256, 4096, 300):
        X = rng.uniform(-1, 1, (n, 4)).astype(np.float32)
        Y = np.zeros((n, 3), dtype=np.float32)
        assert L.lbm_mlp_predict(m, P(X.ctypes.data), n, P(Y.ctypes.data)) == lbm.LBM_OK
        assert np.array_equal(Y, want.predict(X))
    L.lbm_mlp_destroy(m)
