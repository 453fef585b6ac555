"""Device functions of the exact paths on their own, in a small kernel compiled
against the library's headers: the reciprocal of the error model, the truncated
64-bit product, and the eight-copy form of the FP32 inverse-Normal table that the
corrections read, against the one-copy form of the exact kernels."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "exact64.cuh"
using namespace mlmc;
__global__ void k_reciprocal(const double *x, double *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = reciprocal(x[i]);
}
__global__ void k_mulhi(const uint64_t *a, const uint64_t *b, uint64_t *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = mulhi64_3(a[i], b[i]);
}
__global__ void k_normal(const uint32_t *J, float *one, float *eight, int n) {
  __shared__ float4 t0[PhiTable<0>::SIZE], t4[PhiTable<4>::SIZE];
  PhiTable<0>::stage(t0);
  PhiTable<4>::stage(t4);
  copies_done();
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    one[i] = exact_normal_f32<0>(J[i], t0, PhiTable<0>::lane());
    eight[i] = exact_normal_f32<4>(J[i], t4, PhiTable<4>::lane());
  }
}
static int done() { return cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess; }
extern "C" int reciprocals(const double *x, double *y, int n) {
  k_reciprocal<<<(n + 127) / 128, 128>>>(x, y, n);
  return done();
}
extern "C" int mulhis(const uint64_t *a, const uint64_t *b, uint64_t *y, int n) {
  k_mulhi<<<(n + 127) / 128, 128>>>(a, b, y, n);
  return done();
}
extern "C" int normals(const uint32_t *J, float *one, float *eight, int n) {
  k_normal<<<(n + 127) / 128, 128>>>(J, one, eight, n);
  return done();
}
"""


@pytest.fixture(scope="module")
def f(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07123_gb300 import build
    d = tmp_path_factory.mktemp("device_functions")
    (d / "f.cu").write_text(SOURCE)
    r = subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-shared", "-o", str(d / "f.so"), str(d / "f.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(d / "f.so"))

    def call(name, outs, *ins):
        dev = [torch.from_numpy(x.view(s)).cuda() for x, s in ins]
        res = [torch.zeros(len(ins[0][0]), dtype=t, device="cuda") for t in outs]
        torch.cuda.synchronize()
        assert getattr(lib, name)(*(ctypes.c_void_p(x.data_ptr()) for x in dev + res), len(ins[0][0])) == 0
        return [x.cpu().numpy() for x in res]

    call.torch = torch
    return call


def test_reciprocal(f):
    """[2^-100, 2^100): r (1 + e + e^2) misses 1/x by e^3 (2^-63 of it), the last rounding is half a unit; so at most
    one unit in the last place.  Elsewhere it is the division."""
    rng = np.random.default_rng(3)
    p2 = 2.0 ** np.arange(-103, 104)
    x = np.concatenate([p2, np.nextafter(p2, 0), np.nextafter(p2, np.inf), p2 * (1 + 2.0 ** -24),
                        (1 + rng.random(400_000)) * 2.0 ** rng.integers(-100, 100, 400_000), 1 + 4 * rng.random(400_000)])
    x = np.concatenate([x, -x, [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1.7e308, 2.0 ** -1022]])
    y, = f("reciprocals", [f.torch.float64], (x, np.float64))
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    fast = (np.abs(x) >= 2.0 ** -100) & (np.abs(x) < 2.0 ** 100)
    assert np.all(np.abs(y[fast] - want[fast]) <= np.spacing(np.abs(want[fast])))
    assert np.array_equal(y[~fast], want[~fast], equal_nan=True)


def test_truncated_product(f):
    """At most 3 units low for high words that add to less than 2^32, up to that edge and at the largest factors that
    exact64_consts allows."""
    rng = np.random.default_rng(4)
    top = 1 << 32
    a, b = [], []
    for h in [0, 1, top // 2 - 1, top // 2, top - 2, top - 1] + [int(v) for v in rng.integers(0, top, 3000)]:
        g = top - 1 - h
        for g2 in (g, int(rng.integers(0, g + 1))):
            for lo in ((0xFFFFFFFF, 0xFFFFFFFF), (0, 0xFFFFFFFF), tuple(int(v) for v in rng.integers(0, top, 2))):
                a.append(h << 32 | lo[0])
                b.append(g2 << 32 | lo[1])
    y = int(6.34 * 2 ** 60)
    for c in (int(2.0 ** 65 / 6.4), int(2.0 ** 69 / 43), y):
        a.append(c)
        b.append(y if c != int(2.0 ** 69 / 43) else y * y >> 64)
        assert (a[-1] >> 32) + (b[-1] >> 32) < top
    got, = f("mulhis", [f.torch.int64], (np.array(a, dtype=np.uint64), np.int64), (np.array(b, dtype=np.uint64), np.int64))
    for i, j, g in zip(a, b, got.view(np.uint64)):
        assert 0 <= (i * j >> 64) - int(g) <= 3, (hex(i), hex(j))


def test_copied_inverse_normal_table(f):
    """Both forms of the table give the same bits: at and beside every part's ends, at u = 1/2 (the last part), and
    over random words, each by every lane of a copy group."""
    ends = np.concatenate([(16 + np.arange(17)) * 2.0 ** (e - 4) for e in range(0, 31)]).astype(np.int64)
    J = np.concatenate([ends + k for k in range(-3, 4)] + [np.arange(2 ** 31 - 300, 2 ** 31), np.arange(0, 300),
                                                           np.random.default_rng(5).integers(0, 2 ** 31, 500_000)])
    J = J[(J >= 0) & (J < 2 ** 31)]
    J = np.concatenate([J, 2 ** 32 - 1 - J]).astype(np.uint32)
    J = np.concatenate([np.roll(J, s) for s in range(8)])
    one, eight = f("normals", [f.torch.float32, f.torch.float32], (J, np.int32))
    assert np.array_equal(one.view(np.uint32), eight.view(np.uint32))
    assert np.all(np.isfinite(one)) and np.abs(one).max() < 6.5
