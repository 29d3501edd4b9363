// Small contractions in one launch: both operands read in their stored layouts,
// the output written in the order the caller wants.
//
// Most steps of a contraction path are tiny (gate-sized tensors): their cost is
// launches and dependent latencies, not bytes or flops.  A permute per operand,
// a tiled GEMM and a permute of the output were up to four launches of 6 to
// 14 us.  Here every output element is a dot product whose operand offsets are
// bit deposits of its index; operands sit in L1/L2.
#include <algorithm>

#include "kernels.cuh"

namespace tnq {

namespace {

constexpr int SM_THREADS = 128;

__device__ __forceinline__ float2 tf32_rna2(float2 v) {
  return make_float2(__uint_as_float((__float_as_uint(v.x) + 0x1000u) & 0xffffe000u),
                     __uint_as_float((__float_as_uint(v.y) + 0x1000u) & 0xffffe000u));
}

// 2^log_l lanes share an output element (each takes every 2^log_l-th K value;
// their sums meet by shuffles), so that few outputs with a longer K still fill
// warps.  Offsets of the K values are tabulated in shared memory.
__global__ void __launch_bounds__(SM_THREADS) cgemm_small_kernel(const __grid_constant__ SmallOp op) {
  __shared__ uint2 ktab[1 << SMALL_MAX_K];
  __shared__ uint3 otab[32];
  const int t = threadIdx.x;
  for (int k = t; k < 1 << op.nk; k += SM_THREADS) {
    uint32_t a = 0, b = 0;
    for (int j = 0; j < op.nk; ++j)
      if ((k >> j) & 1) {
        a |= 1u << op.ka[j];
        b |= 1u << op.kb[j];
      }
    ktab[k] = make_uint2(a, b);
  }
  if (t < op.n_out) {
    auto bit = [](int p) { return p < 0 ? 0u : 1u << p; };
    otab[t] = make_uint3(bit(op.pa[t]), bit(op.pb[t]), bit(op.pc[t]));
  }
  __syncthreads();
  const uint32_t idx = blockIdx.x * SM_THREADS + t;
  const uint32_t o = idx >> op.log_l, L = 1u << op.log_l;
  const bool live = o < 1u << op.n_out;
  uint32_t oa = 0, ob = 0, oc = 0;
  for (int j = 0; j < op.n_out; ++j) {
    const uint3 w = otab[j];
    if ((o >> j) & 1) {
      oa |= w.x;
      ob |= w.y;
      oc |= w.z;
    }
  }
  float re = 0.f, im = 0.f;
  if (live) {
    const float2* A = op.A + oa;
    const float2* B = op.B + ob;
#pragma unroll 8
    for (uint32_t k = idx & (L - 1); k < 1u << op.nk; k += L) {
      const uint2 q = ktab[k];
      float2 a = __ldg(A + q.x), b = __ldg(B + q.y);
      if (op.round_tf32) {
        a = tf32_rna2(a);
        b = tf32_rna2(b);
      }
      re = fmaf(a.x, b.x, re);
      re = fmaf(-a.y, b.y, re);
      im = fmaf(a.x, b.y, im);
      im = fmaf(a.y, b.x, im);
    }
  }
  for (uint32_t d = 1; d < L; d <<= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, d);
    im += __shfl_xor_sync(0xffffffffu, im, d);
  }
  if (live && (idx & (L - 1)) == 0) {
    if (op.acc) {
      double2 v = op.acc[oc];
      v.x += re;
      v.y += im;
      op.acc[oc] = v;
    } else {
      op.C[oc] = make_float2(re, im);
    }
  }
}

}  // namespace

int small_lanes_log2(int n_out, int nk) {
  // enough threads to fill the chip (2^16) while lanes have a K value each
  return std::max(0, std::min({5, nk, 16 - n_out}));
}

cudaError_t launch_cgemm_small(const SmallOp& op, cudaStream_t st) {
  if (op.n_out < 0 || op.n_out > 24 || op.nk < 0 || op.nk > SMALL_MAX_K || op.log_l < 0 || op.log_l > 5)
    return cudaErrorInvalidConfiguration;
  const long long threads = 1ll << (op.n_out + op.log_l);
  cgemm_small_kernel<<<unsigned((threads + SM_THREADS - 1) / SM_THREADS), SM_THREADS, 0, st>>>(op);
  return cudaGetLastError();
}

}  // namespace tnq
