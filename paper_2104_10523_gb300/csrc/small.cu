// Small contractions in one launch: both operands read in their stored layouts,
// the output written in the order the caller wants.
//
// Most steps of a contraction path are tiny (gate-sized tensors): their cost is
// launches and dependent latencies, not bytes or flops.  A permute per operand,
// a tiled GEMM and a permute of the output were up to four launches of 6 to
// 14 us (64 x 64 x 64: 45 us on the device, 66 a call).  Here every output element
// is a dot product whose operand offsets are bit deposits of its index; operands
// sit in L1/L2 (one launch of 4 us, 17 a call).
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
// warps.  Offsets of the K values are tabulated in shared memory, 2^SMALL_TAB_K
// at a time.  The grid's y cuts the K range into splits whose sums go to part.
constexpr int SMALL_TAB_K = 10;

__global__ void __launch_bounds__(SM_THREADS) cgemm_small_kernel(const __grid_constant__ SmallOp op,
                                                                 float2* __restrict__ part) {
  __shared__ uint2 ktab[1 << SMALL_TAB_K];
  __shared__ uint3 otab[32];
  const int t = threadIdx.x;
  const uint32_t K = 1u << op.nk, kchunk = K / gridDim.y, kbeg = blockIdx.y * kchunk;
  if (t < op.n_out) {
    auto bit = [](int p) { return p < 0 ? 0u : 1u << p; };
    otab[t] = make_uint3(bit(op.pa[t]), bit(op.pb[t]), bit(op.pc[t]));
  }
  const uint32_t idx = blockIdx.x * SM_THREADS + t;
  const uint32_t o = idx >> op.log_l, L = 1u << op.log_l;
  const bool live = o < 1u << op.n_out;
  uint32_t oa = 0, ob = 0, oc = 0;
  float re = 0.f, im = 0.f;
  for (uint32_t k0 = 0; k0 < kchunk; k0 += 1u << SMALL_TAB_K) {
    const uint32_t kn = min(kchunk - k0, 1u << SMALL_TAB_K);
    if (k0) __syncthreads();
    for (uint32_t k = t; k < kn; k += SM_THREADS) {
      const uint32_t kk = kbeg + k0 + k;
      uint32_t a = 0, b = 0;
      for (int j = 0; j < op.nk; ++j)
        if ((kk >> j) & 1) {
          a |= 1u << op.ka[j];
          b |= 1u << op.kb[j];
        }
      ktab[k] = make_uint2(a, b);
    }
    __syncthreads();
    if (!k0) {
      for (int j = 0; j < op.n_out; ++j) {
        const uint3 w = otab[j];
        if ((o >> j) & 1) {
          oa |= w.x;
          ob |= w.y;
          oc |= w.z;
        }
      }
    }
    if (live) {
      const float2* A = op.A + oa;
      const float2* B = op.B + ob;
#pragma unroll 8
      for (uint32_t k = idx & (L - 1); k < kn; k += L) {
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
  }
  for (uint32_t d = 1; d < L; d <<= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, d);
    im += __shfl_xor_sync(0xffffffffu, im, d);
  }
  if (live && (idx & (L - 1)) == 0) {
    if (part) {
      part[(size_t(blockIdx.y) << op.n_out) + oc] = make_float2(re, im);
    } else if (op.acc) {
      double2 v = op.acc[oc];
      v.x += re;
      v.y += im;
      op.acc[oc] = v;
    } else {
      op.C[oc] = make_float2(re, im);
    }
  }
}

// The same sums, in the same order, where one lane an output (log_l = 0) leaves the
// chip idle: a warp an output, whose lanes load 32 K values at once, then all add them
// up in ascending K, each taken from its lane by shuffles.  One lane alone waits for a
// few uncoalesced loads at a time.
__global__ void __launch_bounds__(SM_THREADS) cgemm_small_ordered_kernel(const __grid_constant__ SmallOp op,
                                                                         float2* __restrict__ part) {
  const int lane = threadIdx.x & 31;
  const uint32_t o = (blockIdx.x * SM_THREADS + threadIdx.x) >> 5;
  if (o >> op.n_out) return;  // whole warps
  const uint32_t kchunk = (1u << op.nk) / gridDim.y, kbeg = blockIdx.y * kchunk;
  uint32_t oa = 0, ob = 0, oc = 0;
  for (int j = 0; j < op.n_out; ++j)
    if ((o >> j) & 1) {
      oa |= op.pa[j] < 0 ? 0u : 1u << op.pa[j];
      ob |= op.pb[j] < 0 ? 0u : 1u << op.pb[j];
      oc |= 1u << op.pc[j];
    }
  for (int j = 0; j < 5; ++j)
    if ((lane >> j) & 1) {  // nk >= 5: the low K bits are the lane's
      oa |= 1u << op.ka[j];
      ob |= 1u << op.kb[j];
    }
  auto load = [&](uint32_t k, float2* a, float2* b) {
    uint32_t qa = oa, qb = ob;
    for (int j = 5; j < op.nk; ++j)
      if ((k >> j) & 1) {
        qa |= 1u << op.ka[j];
        qb |= 1u << op.kb[j];
      }
    *a = __ldg(op.A + qa);
    *b = __ldg(op.B + qb);
  };
  float re = 0.f, im = 0.f;
  float2 a, b, an, bn;
  load(kbeg, &a, &b);
  for (uint32_t k0 = 0; k0 < kchunk; k0 += 32, a = an, b = bn) {
    if (k0 + 32 < kchunk) load(kbeg + k0 + 32, &an, &bn);
    if (op.round_tf32) {
      a = tf32_rna2(a);
      b = tf32_rna2(b);
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const float ax = __shfl_sync(0xffffffffu, a.x, i), ay = __shfl_sync(0xffffffffu, a.y, i);
      const float bx = __shfl_sync(0xffffffffu, b.x, i), by = __shfl_sync(0xffffffffu, b.y, i);
      re = fmaf(ax, bx, re);
      re = fmaf(-ay, by, re);
      im = fmaf(ax, by, im);
      im = fmaf(ay, bx, im);
    }
  }
  if (lane) return;
  if (part) {
    part[(size_t(blockIdx.y) << op.n_out) + oc] = make_float2(re, im);
  } else if (op.acc) {
    double2 v = op.acc[oc];
    v.x += re;
    v.y += im;
    op.acc[oc] = v;
  } else {
    op.C[oc] = make_float2(re, im);
  }
}

// ------------------------------------------------------------------ step program
// A run of small steps in one launch: one cluster (the grid) of CTAs walks the steps level
// by level, a cluster barrier between levels (the barrier's release and acquire
// order the intermediates, which stay in L2).  Each step alone is a launch whose
// 2 to 3 us are latency; a level costs about one, whatever its number of steps.
// The records of the steps are copied to shared memory first; a warp finds its
// step by its place among the level's warp-sized units.
// The cluster grows with the largest level: one CTA for at most 2^10 outputs (a
// block barrier is cheaper than a cluster's), eight of 16 warps for at most 2^13,
// sixteen of 32 warps above (eight where a cluster of sixteen cannot be placed).
// A 4x5 noisy pass, whose levels hold many steps of 2^14 outputs, took 132 us with
// eight of 16 warps and 48 with sixteen of 32; a 3x4 batch loses 5 us to the
// wider launch.
constexpr int PROG_CTAS = 16, PROG_CTAS_PORTABLE = 8, PROG_THREADS = 1024;

struct ProgLevels {
  int n;
  short begin[PROG_MAX_OPS + 1];
};

__global__ void __launch_bounds__(PROG_THREADS)
    prog_kernel(const ProgOp* __restrict__ gops, const __grid_constant__ ProgLevels lv, int n_ops, int n_slices, int slice_id) {
  extern __shared__ __align__(16) unsigned char prog_raw[];
  ProgOp* ops = reinterpret_cast<ProgOp*>(prog_raw);
  const int t = threadIdx.x, lane = t & 31;
  {
    const uint4* src = reinterpret_cast<const uint4*>(gops);
    uint4* dst = reinterpret_cast<uint4*>(prog_raw);
    for (int i = t; i < n_ops * int(sizeof(ProgOp) / 16); i += blockDim.x) dst[i] = __ldg(src + i);
  }
  __syncthreads();
  for (int i = t; i < n_ops; i += blockDim.x) {
    unsigned long long a = 0, b = 0;
    for (int j = 0; j < n_slices; ++j)
      if ((slice_id >> j) & 1) {
        if (ops[i].sa[j] >= 0) a |= 8ull << ops[i].sa[j];
        if (ops[i].sb[j] >= 0) b |= 8ull << ops[i].sb[j];
      }
    ops[i].a += a;
    ops[i].b += b;
  }
  __syncthreads();
  const uint32_t per = blockDim.x >> 5, warp = blockIdx.x * per + (t >> 5), warps = gridDim.x * per;
  for (int l = 0; l < lv.n; ++l) {
    const int o0 = lv.begin[l], o1 = lv.begin[l + 1];
    const ProgOp& last = ops[o1 - 1];
    const int lt = last.n_out + last.log_l;
    const uint32_t units = last.warp_begin + (lt > 5 ? 1u << (lt - 5) : 1u);
    for (uint32_t u = warp; u < units; u += warps) {
      int at = o0 - 1;  // the last step of the level that begins at or before u
      for (int q = o0; q < o1; q += 32) {
        const unsigned m = __ballot_sync(0xffffffffu, q + lane < o1 && ops[q + lane].warp_begin <= u);
        at += __popc(m);
      }
      const ProgOp& op = ops[at];
      // Output index o = idx >> log_l: its bits above the lanes' are the same for
      // the whole warp, so lane j contributes bit j's offsets and the warp ORs them;
      // the lanes' own bits are at most five.  (A loop over the record's bits in
      // every lane was a chain of shared-memory reads, most of a level's time.)
      const int n_out = op.n_out, log_l = op.log_l, nk = op.nk, lane_bits = 5 - log_l;
      const uint32_t idx = (u - op.warp_begin) * 32 + lane, L = 1u << log_l;
      const uint32_t o = idx >> log_l;
      const bool live = o < 1u << n_out;
      uint32_t oa = 0, ob = 0, oc = 0;
      if (lane >= lane_bits && lane < n_out && ((o >> lane) & 1)) {
        const uint4 w = op.bit[lane];
        oa = w.x;
        ob = w.y;
        oc = w.z;
      }
      oa = __reduce_or_sync(0xffffffffu, oa);
      ob = __reduce_or_sync(0xffffffffu, ob);
      oc = __reduce_or_sync(0xffffffffu, oc);
#pragma unroll
      for (int j = 0; j < 5; ++j)
        if (j < lane_bits && j < n_out && ((o >> j) & 1)) {
          const uint4 w = op.bit[j];
          oa |= w.x;
          ob |= w.y;
          oc |= w.z;
        }
      // K index: its low log_l bits are the lane's, the others count the
      // iterations; lane q holds the offsets of iteration q (of 32 at a time)
#pragma unroll
      for (int j = 0; j < 5; ++j)
        if (j < log_l && ((idx >> j) & 1)) {
          const uint2 w = op.kbit[j];
          oa |= w.x;
          ob |= w.y;
        }
      const float2* A = reinterpret_cast<const float2*>(op.a) + (live ? oa : 0);
      const float2* B = reinterpret_cast<const float2*>(op.b) + (live ? ob : 0);
      const int kb_iter = nk - log_l, iters = 1 << kb_iter;
      float re = 0.f, im = 0.f;
      for (int i0 = 0; i0 < iters; i0 += 32) {
        uint32_t qa = 0, qb = 0;
#pragma unroll
        for (int j = 0; j < PROG_MAX_K; ++j)
          if (j < kb_iter && (((i0 + lane) >> j) & 1)) {
            const uint2 w = op.kbit[log_l + j];
            qa |= w.x;
            qb |= w.y;
          }
        const int n = min(32, iters - i0);
#pragma unroll 4
        for (int i = 0; i < n; ++i) {
          const uint32_t ka = __shfl_sync(0xffffffffu, qa, i), kb = __shfl_sync(0xffffffffu, qb, i);
          // plain loads: earlier levels of this launch may have written them
          if (live) {
            const float2 a = A[ka], b = B[kb];
            re = fmaf(a.x, b.x, re);
            re = fmaf(-a.y, b.y, re);
            im = fmaf(a.x, b.y, im);
            im = fmaf(a.y, b.x, im);
          }
        }
      }
      for (uint32_t d = 1; d < L; d <<= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, d);
        im += __shfl_xor_sync(0xffffffffu, im, d);
      }
      if (live && (idx & (L - 1)) == 0) {
        if (op.acc) {
          double2* p = reinterpret_cast<double2*>(op.c) + oc;
          double2 v = *p;
          v.x += re;
          v.y += im;
          *p = v;
        } else {
          reinterpret_cast<float2*>(op.c)[oc] = make_float2(re, im);
        }
      }
    }
    if (l + 1 < lv.n && gridDim.x == 1) {
      __syncthreads();
    } else if (l + 1 < lv.n) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
}

}  // namespace

int prog_lanes_log2(int n_out, int nk) {
  // two K values a lane while the step stays within the cluster's threads
  return std::max(0, std::min({5, nk - 1, 12 - n_out}));
}

cudaError_t launch_prog(const ProgOp* ops, const int* levels, int n_levels, int n_ops, int max_units, int n_slices,
                        int slice_id, cudaStream_t st) {
  if (n_ops < 1 || n_ops > PROG_MAX_OPS || n_levels < 1 || n_levels > n_ops || n_slices > 32)
    return cudaErrorInvalidConfiguration;
  ProgLevels lv;
  lv.n = n_levels;
  for (int i = 0; i <= n_levels; ++i) lv.begin[i] = short(levels[i]);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto shape = [&](int ctas, int threads, size_t smem) {
    cfg.blockDim = dim3(unsigned(threads));
    attr[0].val.clusterDim.x = unsigned(ctas);
    cfg.gridDim = dim3(unsigned(ctas));
    cfg.dynamicSmemBytes = smem;
  };
  static std::atomic<uint64_t> done{0};
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(prog_kernel), int(PROG_MAX_OPS * sizeof(ProgOp)), &done);
  if (e != cudaSuccess) return e;
  const size_t smem = size_t(n_ops) * sizeof(ProgOp);
  if (max_units > 256) {
    // a cluster of sixteen is beyond the portable size: asked for on each launch's
    // device, and only where it can be placed
    static std::atomic<uint64_t> wide{0}, narrow{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (!((wide.load() | narrow.load()) & bit) || !bit) {
      int n = 0;
      shape(PROG_CTAS, PROG_THREADS, PROG_MAX_OPS * sizeof(ProgOp));
      const bool fits = cudaFuncSetAttribute(prog_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                        cudaOccupancyMaxActiveClusters(&n, prog_kernel, &cfg) == cudaSuccess && n >= 1;
      if (!fits) cudaGetLastError();
      if (bit) (fits ? wide : narrow).fetch_or(bit);
      shape(fits ? PROG_CTAS : PROG_CTAS_PORTABLE, PROG_THREADS, smem);
    } else {
      shape(wide.load() & bit ? PROG_CTAS : PROG_CTAS_PORTABLE, PROG_THREADS, smem);
    }
  } else if (max_units > 32) {
    shape(PROG_CTAS_PORTABLE, PROG_THREADS / 2, smem);
  } else {
    shape(1, PROG_THREADS, smem);
  }
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, prog_kernel, ops, lv, n_ops, n_slices, slice_id);
}

int small_lanes_log2(int n_out, int nk) {
  // enough threads to fill the chip (2^16) while lanes have a K value each
  return std::max(0, std::min({5, nk, 16 - n_out}));
}

// Whether a warp an output is faster than a lane an output: up to 2^12 sums (outputs
// x splits) of at least 64 values.  Calls in us, lane and warp: 2^8 sums of 2^10 134
// and 45, 2^12 of 2^8 54 and 35, 2^12 of 2^6 29 and 22; 2^13 level (34 and 34 at
// 2^7), 2^14 of 2^8 52 and 83.
static bool small_ordered_warps(int n_out, int nk, int splits) {
  int ls = 0;
  while ((1 << ls) < splits) ++ls;
  return nk - ls >= 6 && n_out + ls <= 12;
}

cudaError_t launch_cgemm_small(const SmallOp& op, void* part, int splits, cudaStream_t st) {
  if (op.n_out < 0 || op.n_out > SMALL_MAX_OUT || op.nk < 0 || op.nk > 31 || op.log_l < 0 || op.log_l > 5 ||
      splits < 1 || splits > 65535 || (splits & (splits - 1)) || splits > (1 << std::min(op.nk, 16)) ||
      (splits > 1 && !part))
    return cudaErrorInvalidConfiguration;
  float2* const parts = splits > 1 ? reinterpret_cast<float2*>(part) : nullptr;
  if (op.log_l == 0 && small_ordered_warps(op.n_out, op.nk, splits)) {
    const dim3 grid{unsigned(((32ll << op.n_out) + SM_THREADS - 1) / SM_THREADS), unsigned(splits), 1u};
    cgemm_small_ordered_kernel<<<grid, SM_THREADS, 0, st>>>(op, parts);
    return cudaGetLastError();
  }
  const long long threads = 1ll << (op.n_out + op.log_l);
  const dim3 grid{unsigned((threads + SM_THREADS - 1) / SM_THREADS), unsigned(splits), 1u};
  cgemm_small_kernel<<<grid, SM_THREADS, 0, st>>>(op, parts);
  return cudaGetLastError();
}

}  // namespace tnq
