"""The table logarithm of the FP64 tree walks against CUDA's log, over the whole range of normal numbers
and around 1, and the arguments that it hands to the library.

Tolerance: two units in the last place: half a unit from the table's last addition, a quarter from log 2
rounded, a quarter from the table and the series, and what the library's own result (documented: one unit)
is off.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pp_log.cuh"
__global__ void both(const double* x, double* a, double* b, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = pp::log_table(x[i]), b[i] = log(x[i]);
}
extern "C" int run(const double* x, double* a, double* b, int n) {
    both<<<(n + 255) / 256, 256>>>(x, a, b, n);
    return int(cudaDeviceSynchronize());
}
"""


def test_log_table(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_04398_gb300 import _build
    src, lib = tmp_path / "log.cu", tmp_path / "liblog.so"
    src.write_text(SOURCE)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", "-o", str(lib), str(src)],
                   check=True)
    rng = np.random.default_rng(0)
    near_one = 1.0 + np.concatenate([s * 2.0 ** -np.arange(1, 53.0) for s in (1.0, -0.5)])
    bins = 1.0 + np.arange(257) / 256
    x = np.concatenate([np.exp(rng.uniform(-700, 700, 100000)), np.exp(rng.uniform(-20, 20, 200000)),
                        1.0 + rng.uniform(-0.02, 0.02, 200000), near_one, bins, np.nextafter(bins, 0),
                        np.array([2.0 ** -1022, np.finfo(float).max, 1.0, 5e-324, 0.0, -1.0, np.inf, np.nan])])
    t = torch.tensor(x, device="cuda")
    a, b = torch.empty_like(t), torch.empty_like(t)
    dll = ctypes.CDLL(os.fspath(lib))
    assert dll.run(*(ctypes.c_void_p(v.data_ptr()) for v in (t, a, b)), ctypes.c_int(len(x))) == 0
    a, b = a.cpu().numpy(), b.cpu().numpy()
    special = ~np.isfinite(b)
    assert np.array_equal(a[special], b[special], equal_nan=True)
    x, a, b = x[~special], a[~special], b[~special]
    err, allowed = np.abs(a - b), 2 * np.spacing(np.abs(b))
    assert (err <= allowed).all(), (x[np.argmax(err / allowed)], np.max(err / allowed))
    assert (a[x == 1.0] == 0.0).all()
