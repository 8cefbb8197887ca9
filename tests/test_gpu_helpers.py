"""The fast reciprocal and the small-angle arctangent that the projector kernels
share (ct_device.cuh), swept over the depths and slopes a geometry can have
and compared with 64-bit values.  The kernel is compiled here from that header."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

KERNEL = """
#include "ct_device.cuh"
__global__ void sweep(const float *x, const float *num, const float *den, float *r, float *s, int n) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    r[t] = ctp::rcp_newton(x[t]);
    s[t] = ctp::slope_angle(num[t], den[t]);
}
extern "C" int run(const float *x, const float *num, const float *den, float *r, float *s, int n) {
    sweep<<<(n + 255) / 256, 256>>>(x, num, den, r, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def swept(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_16741_gb300 import build
    d = tmp_path_factory.mktemp("helpers")
    (d / "h.cu").write_text(KERNEL)
    so = str(d / "h.so")
    subprocess.run([build.nvcc(), "-shared", "-o", so, str(d / "h.cu"), "-I" + build.CSRC] + build.ARCH + build.NVCC_FLAGS,
                   check=True, capture_output=True)
    rng = np.random.default_rng(0)
    n = 1 << 20
    x = np.exp(rng.uniform(np.log(1e-3), np.log(1e6), n)) * rng.choice([-1.0, 1.0], n)  # depths in any unit, and their negatives
    den = np.exp(rng.uniform(np.log(1e-2), np.log(1e8), n))
    slope = np.exp(rng.uniform(np.log(1e-7), np.log(4.0), n))
    slope[: n // 4] = rng.uniform(0.9 / 16, 1.1 / 16, n // 4)  # both sides of the switch to the library
    num = den * slope * rng.choice([-1.0, 1.0], n)
    dev = [torch.as_tensor(a.astype(np.float32)).cuda() for a in (x, num, den)]
    out = [torch.empty_like(dev[0]) for _ in range(2)]
    torch.cuda.synchronize()
    assert C.CDLL(os.path.abspath(so)).run(*[C.c_void_p(t.data_ptr()) for t in dev + out], n) == 0
    return [t.double().cpu().numpy() for t in dev + out]


def test_reciprocal_is_good_to_an_ulp(swept, report):
    """A Newton step squares the fast division's 2 ulp; its last operation rounds once more, so the result is the
    correctly rounded one or its neighbour."""
    x, _, _, r, _ = swept
    exact = 1.0 / x
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64)
    err = np.abs(r - exact) / ulp
    report(f"reciprocal: at most {err.max():.3f} ulp")
    assert err.max() <= 1.0


def test_slope_angle_on_both_sides_of_its_switch(swept, report):
    """Below 1/16 the quotient's 2 ulp, the series' product rounded twice and 2.6e-11 of truncation: under 4 ulp;
    above, the library's bound of 3 ulp."""
    _, num, den, _, s = swept
    exact = np.arctan2(num, den)
    err = np.abs(s - exact) / np.abs(exact)
    small = np.abs(num / den) < 1.0 / 16
    report(f"slope angle: relative error at most {err[small].max():.2e} below 1/16, {err[~small].max():.2e} above")
    assert err.max() <= 4 * 2.0 ** -23
