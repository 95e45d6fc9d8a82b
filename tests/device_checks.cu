// Test kernels: device functions of the library compared over whole ranges of patterns with the instructions or the longer arithmetic
// they stand for.  Each counts its mismatches.
#include "../paper_2605_14929_b200/csrc/sop_device.cuh"

namespace {

// The quotient dot / sqrt(x) of the fast steps against square root and division rounded to nearest, for the patterns x0 .. x0 + n - 1
// and every dot given.  bad[0]: mismatches where the root is not all ones, bad[1]: where it is, bad[2]: such x, [3]: all_ones_root that
// disagrees with the root itself.
__global__ void cosine_kernel(unsigned x0, unsigned n, const float* dots, int n_dots, unsigned long long* bad) {
  unsigned long long b0 = 0, b1 = 0, ones = 0, wrong = 0;
  const unsigned long long total = (unsigned long long)n * (unsigned)n_dots, stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const unsigned at = (unsigned)(i / (unsigned)n_dots), d = (unsigned)(i - (unsigned long long)at * (unsigned)n_dots);
    const float x = __uint_as_float(x0 + at), dot = dots[d], root = __fsqrt_rn(x), want = __fdiv_rn(dot, root);
    const bool all = (__float_as_uint(root) & 0x7FFFFFu) == 0x7FFFFFu;
    if (d == 0) {
      ones += all ? 1 : 0;
      wrong += all != (sop::all_ones_root(x) == 0u) || all != (sop::all_ones_root(-x) == 0u) ? 1 : 0;
    }
    const float2 two = sop::cosine_pair(make_float2(-x, -x), make_float2(dot, -dot));
    const bool differs = __float_as_uint(want) != __float_as_uint(two.x) || __float_as_uint(-want) != __float_as_uint(two.y) ||
                         __float_as_uint(want) != __float_as_uint(sop::cosine_one(-x, dot));
    if (differs) { if (all) ++b1; else ++b0; }
  }
  if (b0) atomicAdd(&bad[0], b0);
  if (b1) atomicAdd(&bad[1], b1);
  if (ones) atomicAdd(&bad[2], ones);
  if (wrong) atomicAdd(&bad[3], wrong);
}

}  // namespace

extern "C" int check_cosine(unsigned x0, unsigned n, const float* dots, int n_dots, unsigned long long* bad) {
  cosine_kernel<<<1184, 256>>>(x0, n, dots, n_dots, bad);
  return (int)cudaDeviceSynchronize();
}
