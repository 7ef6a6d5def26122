"""The FP64 roots and reciprocals of the factorisation kernels (fp64_scalar.cuh)
against CUDA's sqrt and division and against the host's long double, over their ranges.

A small program of its own includes the header.  The bounds are the header's: a last step
whose error before rounding is below 2^-70 / 2^-53 ulp leaves 0.5 ulp and, on one random
value in 2^16 at most, the neighbour of CUDA's correctly rounded result (short mantissas may
lie as near a tie as that)."""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>
#include "fp64_scalar.cuh"

__device__ unsigned long long mix(unsigned long long z) {   // splitmix64
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
// mantissa: random, or (odd i, one in eight) a few bits set or cleared at either end
__device__ double sample(unsigned long long i, int emin, int emax) {
  unsigned long long m = mix(3 * i), e = mix(3 * i + 1), k = mix(3 * i + 2);
  if ((i & 1) && (k & 7) == 0) {
    m = 1ull << (k >> 3) % 52;
    if (k >> 20 & 1) m = (1ull << 52) - m;
    if (k >> 21 & 1) m = k >> 22 & 3;
  }
  const unsigned long long x = (m & ((1ull << 52) - 1)) | (unsigned long long)(1023 + emin + (long long)(e % (emax - emin + 1))) << 52;
  return __longlong_as_double((long long)x);
}
__device__ int apart(double a, double b) {
  const long long d = __double_as_longlong(a) - __double_as_longlong(b);
  return d > 1 || d < -1 ? 2 : d != 0;
}
struct Out { double x, root, inv, y, rec; };
__global__ void run(Out* out, int kept, unsigned long long n, unsigned long long* count) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step) {
    Out o;
    o.x = sample(i, -930, 930);
    zolo::root_pair(o.x, &o.root, &o.inv);
    o.y = sample(i + n, -1020, 1020);
    o.rec = zolo::reciprocal(o.y);
    const int d[2] = {apart(o.root, sqrt(o.x)), apart(o.rec, 1.0 / o.y)};
    for (int q = 0; q < 2; ++q)
      if (d[q] > 1 || (d[q] && !(i & 1))) atomicAdd(&count[2 * q + (d[q] > 1)], 1ull);
    if (i < (unsigned long long)kept) out[i] = o;
  }
}
int main() {
  const int kept = 200000;
  const unsigned long long n = 1ull << 24;
  Out* d;
  unsigned long long *c, h[4];
  if (cudaMalloc(&d, sizeof(Out) * kept) != cudaSuccess || cudaMalloc(&c, sizeof(h)) != cudaSuccess) return 2;
  cudaMemset(c, 0, sizeof(h));
  run<<<1024, 256>>>(d, kept, n, c);
  std::vector<Out> o(kept);
  if (cudaMemcpy(o.data(), d, sizeof(Out) * kept, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  cudaMemcpy(h, c, sizeof(h), cudaMemcpyDeviceToHost);
  long double root = 0, inv = 0, rec = 0;
  auto ulps = [](double got, long double want) {
    int e;
    frexp((double)want, &e);
    return fabsl(got - want) / ldexpl(1.0L, e - 53);
  };
  for (const Out& q : o) {
    const long double s = sqrtl((long double)q.x);
    root = fmaxl(root, ulps(q.root, s));
    inv = fmaxl(inv, fabsl((long double)q.inv * s - 1.0L) * ldexpl(1.0L, 53));
    rec = fmaxl(rec, ulps(q.rec, 1.0L / q.y));
  }
  printf("%Lf %Lf %Lf %llu", root, inv, rec, n);
  for (int q = 0; q < 4; ++q) printf(" %llu", h[q]);
  printf("\n");
  return 0;
}
"""


def test_roots_and_reciprocals(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06204_gb300 import build
    src, exe = tmp_path / "scalar.cu", tmp_path / "scalar"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I" + build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    root, inv, rec = map(float, out[:3])
    n = int(out[3])
    counts = list(map(int, out[4:]))
    print(out)
    assert root <= 0.501 and rec <= 0.501     # ulp
    assert inv <= 1.51                        # units of 2^-53, relative
    for q in range(2):
        assert counts[2 * q] <= n / 2 / 2 ** 16 and counts[2 * q + 1] == 0
