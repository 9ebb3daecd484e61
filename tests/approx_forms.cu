// Compares the library's hardware forms (lanes.cuh, f64_2state.cuh) with the CUDA
// functions they stand for, and prints the number of differences, and of rsqrt64
// the largest relative error in units of 2^-53 (test_approx_forms_gpu.py).
#include <cstdio>

#include "f64_2state.cuh"
#include "lanes.cuh"

using namespace qcl;

struct Result {
  unsigned long long rsqrt, div, rcp, pairs;
  unsigned long long err;  // bits of the largest error (positive doubles order as integers)
};

__global__ void check_rsqrt(Result* r) {  // every positive normal float
  unsigned long long bad = 0;
  for (uint32_t b = 0x00800000u + blockIdx.x * blockDim.x + threadIdx.x; b < 0x7f800000u;
       b += gridDim.x * blockDim.x)
    bad += __float_as_uint(rsqrt_normal(__uint_as_float(b))) !=
           __float_as_uint(rsqrtf(__uint_as_float(b)));
  if (bad) atomicAdd(&r->rsqrt, bad);
}

__global__ void check_rcp(Result* r) {  // every integer from 1 to 2^24
  unsigned long long bad = 0;
  for (uint32_t d = 1 + blockIdx.x * blockDim.x + threadIdx.x; d <= 1u << 24;
       d += gridDim.x * blockDim.x)
    bad += __float_as_uint(rcp_integer((float)d)) != __float_as_uint(__frcp_rn((float)d));
  if (bad) atomicAdd(&r->rcp, bad);
}

// 2^30 pairs of normal floats of either sign with |b| <= 2^126 and a normal quotient
__global__ void check_div(Result* r) {
  unsigned long long bad = 0, seen = 0;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < 1u << 29; k += gridDim.x * blockDim.x) {
    const u4 w = philox_draw(3, k, 0, 6u);
    for (int h = 0; h < 2; ++h) {
      const float a = __uint_as_float(h ? w.z : w.x), b = __uint_as_float(h ? w.w : w.y);
      const float q = a / b;
      if (!(fabsf(a) >= 0x1p-126f && fabsf(a) <= 0x1p127f && fabsf(b) >= 0x1p-126f &&
            fabsf(b) <= 0x1p126f && fabsf(q) >= 0x1p-125f && fabsf(q) <= 0x1p126f))
        continue;
      ++seen;
      bad += __float_as_uint(div_normal(a, b)) != __float_as_uint(__fdividef(a, b));
    }
  }
  if (bad) atomicAdd(&r->div, bad);
  atomicAdd(&r->pairs, seen);
}

// y = rsqrt64(x): 1 - x y^2 from exact products is twice its relative error; x of
// every exponent from -500 to 500
__global__ void check_rsqrt64(Result* r) {
  double worst = 0.0;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < 1u << 26; k += gridDim.x * blockDim.x) {
    const u4 w = philox_draw(4, k, 0, 6u);
    const int ex = 1023 - 500 + (int)(w.x % 1001u);
    const double x = __hiloint2double((ex << 20) | (int)(w.y >> 12), (int)w.z);
    const double y = rsqrt64(x);
    const double p = __dmul_rn(y, y), pl = __fma_rn(y, y, -p);
    const double q = __dmul_rn(x, p), ql = __fma_rn(x, pl, __fma_rn(x, p, -q));
    const double e = fabs(__dsub_rn(__dsub_rn(1.0, q), ql)) * 0.5;
    worst = fmax(worst, e);
  }
  atomicMax(&r->err, (unsigned long long)__double_as_longlong(worst));
}

int main() {
  Result *d = nullptr, h{};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 1;
  cudaMemset(d, 0, sizeof(h));
  check_rsqrt<<<1216, 256>>>(d);
  check_rcp<<<1216, 256>>>(d);
  check_div<<<1216, 256>>>(d);
  check_rsqrt64<<<1216, 256>>>(d);
  if (cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  cudaFree(d);
  double err;
  memcpy(&err, &h.err, sizeof(err));
  printf("%llu %llu %llu %llu %.6f\n", h.rsqrt, h.rcp, h.div, h.pairs, err * 0x1p53);
  return 0;
}
