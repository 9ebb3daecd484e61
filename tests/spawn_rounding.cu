// Evaluates the FP32 spawning test and its child on pseudo-random walkers and
// writes the results to the standard output: built with and without multiply-add
// contraction, the bytes are the same (test_spawn_rounding_gpu.py).
#include <cstdio>
#include <vector>

#include "bulk2.cuh"

using namespace qcl;

struct Out {
  uint32_t T, ev, deg;
  float fac, hi, lo, ph;
  int32_t e;
};

__device__ float draw(uint32_t i, uint32_t k, float lo, float hi) {
  const u4 w = philox_draw(17, k, i, 5u);
  return __fmaf_rn(__uint2float_rn(w.x >> 8), __fmul_rn(0x1p-24f, __fsub_rn(hi, lo)), lo);
}

template <int KIND, bool DIA>
__global__ void evaluate(const BulkParams bp, int n, Out* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Scal z;
  z.A = draw(i, 0, -3.0f, 3.0f);
  z.B = KIND == 1 ? draw(i, 1, -3.0f, 3.0f) : bp.b0;
  const float Av = draw(i, 2, -4.0f, 4.0f), Bv = KIND == 1 ? draw(i, 3, -4.0f, 4.0f) : 0.0f;
  closed_form(z);
  z.sa = (i & 1) ? 1.0f : -1.0f;
  z.sb = (i & 2) ? 1.0f : -1.0f;
  z.q = DIA ? (i >> 2) & 3 : 0;
  z.m = {draw(i, 4, 1.0f, 2.0f), draw(i, 5, -0x1p-25f, 0x1p-25f)};
  z.mexp = 3;
  z.ph = {draw(i, 6, -9.0f, 9.0f), 0.0f};
  Out o{};
  o.ev = spawn_event<KIND, DIA>(z, draw(i, 7, 0.0f, 3.0f), Av, DIA ? z.B : Bv,
                                philox_draw(17, 8, i, 5u).x, bp, o.deg, o.T, o.fac);
  o.ph = z.ph.lo;
  if (o.ev) spawn_child<DIA>(z, o.ev, o.T, o.fac);
  renorm(z.m, z.mexp);
  o.hi = z.m.hi;
  o.lo = z.m.lo;
  o.e = z.mexp;
  out[i] = o;
}

int main() {
  const int n = 1 << 18;
  BulkParams bp{};
  bp.b0 = 0.37f;
  bp.hdt_hbar = 0.0123f;
  bp.amp = 0.0217f;
  bp.kamp = 20.0f * bp.amp;
  bp.tmax = 1u << 23;
  Out* dev = nullptr;
  if (cudaMalloc(&dev, sizeof(Out) * n) != cudaSuccess) return 1;
  std::vector<Out> host(n);
  auto run = [&](auto kernel) {
    kernel<<<n / 256, 256>>>(bp, n, dev);
    if (cudaMemcpy(host.data(), dev, sizeof(Out) * n, cudaMemcpyDeviceToHost) != cudaSuccess)
      return false;
    return fwrite(host.data(), sizeof(Out), n, stdout) == (size_t)n;
  };
  const bool ok = run(evaluate<0, false>) && run(evaluate<1, false>) && run(evaluate<0, true>) &&
                  run(evaluate<1, true>);
  cudaFree(dev);
  return ok ? 0 : 2;
}
