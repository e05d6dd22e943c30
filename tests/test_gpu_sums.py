"""The sums of the Krylov reductions: site sums of products in FP32 (SiteNorm, SiteDot) and pairs of floats above
them (RunSum<float>, cta_sum_run), compiled from the header into a small library of their own."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1211_1214_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "blas.cuh"
using namespace ddrw;
__global__ void __launch_bounds__(256) k_sums(long n, const float2 *a, const float2 *b, float *site, double *total)
{
    __shared__ float2 sm[8][3], tot[3];
    RunSum<float> run[3];
    for (long j = threadIdx.x; j < n; j += 256) {
        SiteNorm<float> nn;
        SiteDot<float> dd;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            const cpx<float> x = {a[12 * j + k].x, a[12 * j + k].y}, y = {b[12 * j + k].x, b[12 * j + k].y};
            nn.add(k, x);
            dd.add(k, x, y);
        }
        const float v[3] = {nn.total(), dd.total().re, dd.total().im};
        for (int q = 0; q < 3; q++) {
            site[3 * j + q] = v[q];
            run[q].add(v[q]);
        }
    }
    cta_sum_run<3, 256, float>(run, sm, tot);
    __syncthreads();
    if (threadIdx.x < 3) {
        RunSum<float> r;
        r.join(tot[threadIdx.x]);
        total[threadIdx.x] = r.value();
    }
}
extern "C" int sums(long n, const float2 *a, const float2 *b, float *site, double *total)
{
    k_sums<<<1, 256>>>(n, a, b, site, total);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(SOURCE)
    cmd = [build.NVCC] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", "-o", str(d / "sums.so"), str(d / "sums.cu")]
    subprocess.run(cmd, check=True, cwd=os.path.dirname(build.CSRC))
    return ctypes.CDLL(str(d / "sums.so"))


@pytest.mark.parametrize("n", [1, 255, 20000])
def test_site_sums_and_pair_sums(lib, n):
    rng = np.random.default_rng(n)
    a, b = (rng.standard_normal((n, 12, 2)).astype(np.float32) for _ in range(2))
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    site = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    total = torch.zeros(3, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.sums(ctypes.c_long(n), *(ctypes.c_void_p(t.data_ptr()) for t in (da, db, site, total))) == 0
    site, total = site.cpu().numpy().astype(np.float64), total.cpu().numpy()
    # pairs: each of the at most 80 + 8 additions on the way of a term loses less than 2^-45 of the sums so far
    assert np.all(np.abs(total - site.sum(0)) <= 96 * 2.0**-45 * np.abs(site).sum(0))
    # site sums: no further from 64 bits than adding up the components one by one, each product sum
    # rounded to FP32 (rms over the sites; the margin is the scatter of 20000 of them)
    A, B = a.astype(np.float64), b.astype(np.float64)
    x, y, u, v = A[..., 0], A[..., 1], B[..., 0], B[..., 1]
    f32 = lambda z: z.astype(np.float32).astype(np.float64)
    terms = [(x, x, y, y), (x, u, y, v), (x, v, -y, u)]
    for q, (p, r, s, t) in enumerate(terms):
        want = (p * r + s * t).sum(1)
        old = np.zeros(n)
        for k in range(12):
            old = f32(old + f32(p[:, k] * r[:, k] + f32(s[:, k] * t[:, k])))
        err, was = np.sqrt(np.mean((site[:, q] - want) ** 2)), np.sqrt(np.mean((old - want) ** 2))
        assert err <= (1.0 if n > 1000 else 2.0) * was + (0 if n > 1 else 1e-6 * np.abs(want).max() + 1e-6)
