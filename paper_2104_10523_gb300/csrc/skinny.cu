// Bandwidth-oriented complex GEMMs for skinny contraction steps.
//
// Many steps of a contraction path have a tiny side: few output rows (a small
// operand meeting a large one).  Their cost is reading the large operand once
// and writing the output once; a tiled GEMM would leave most lanes idle.
//
//   C[h][s][g] = sum_k S[h][s][k] G[h][g][k] for a small side of at most 128
//   rows and K of at most 32: each thread loads its rows of the large operand,
//   in their stored bit layout, into registers (gather kernel).  Many rows of a
//   longer K, up to 32 of them on the small side: a thread per row of the large
//   operand, both operands staged from [row][K] order (rows kernel).
#include <algorithm>

#include "kernels.cuh"

namespace tnq {

namespace {

constexpr int GATHER_SMAX = 128;  // small-operand rows of the gather kernel
constexpr int GATHER_REPS = 4;    // row blocks of a CTA

// CTAs an SM the register allocation leaves room for: without the bound the
// compiler unrolls into 80 registers at K = 8 and a quarter of the warps goes
// (8 x 2^23 x 8 176 -> 192 us a call).
constexpr int gather_min_ctas(int K, int rows) {
  return K <= 2 ? (rows == 2 ? 8 : 6) : K == 4 ? 6 : K == 8 ? 4 : K == 16 ? (rows == 2 ? 5 : 4) : rows == 2 ? 3 : 2;
}

// Nearest TF32 value, ties away from zero (finite inputs).
__device__ __forceinline__ float2 tf32_rna2(float2 v) {
  return make_float2(__uint_as_float((__float_as_uint(v.x) + 0x1000u) & 0xffffe000u),
                     __uint_as_float((__float_as_uint(v.y) + 0x1000u) & 0xffffe000u));
}

// Short-K rows kernel reading the large operand in its stored bit layout (no
// separate permute): row R of the (g bits, then batch bits) row index starts at
// the source offset sum_j bit_j(R) << rowpos[j], and element k of a row is
// dep(k, kpos) further on.  One thread owns ROWS rows, held in registers; a CTA
// owns cta_rows consecutive rows of the batch-major row index, so with short
// rows (ng < cta_rows) it serves several batch entries, whose S rows it stages
// together, gathered from their stored layout (one 16-byte pad per entry spreads
// the entries over the banks); with ROWS = 2 a CTA stays within one entry.  A CTA
// of a single entry walks
// reps blocks of rows, so that staging S (a dependent gather before the first
// row can be used) is paid once for all of them.
// ROUND rounds both operands to TF32 first (the products are then exact in
// FP32: the arithmetic of the plain TF32 mode on the CUDA cores).
//
// Bound: HBM while 4 FFMA per (s, k) of a row stay below the 8 (K + ns) bytes
// it moves, then the shared-memory reads of S (16 bytes to 32 lanes take four
// cycles of the one port), which ROWS = 2 halves: 16 x 2^23 x 16 466 -> 392 us,
// 8 x 2^23 x 32 545 -> 463 (from K = 16 on in CTAs of 128 threads, whose load and
// compute phases overlap better, five of them an SM at K = 16).  8 x 2^25 x 8
// moves 6.8 TB/s.  One launch for every batch entry: 4096 entries of 4 x 2^12 x 8
// took 33.5 ms as one tensor-core launch each (8 us a launch).
template <int K, int ROWS, bool ROUND, int T>
__global__ void __launch_bounds__(T, gather_min_ctas(K, ROWS))
    cgemm_rows_gather_kernel(const float2* __restrict__ S, const __grid_constant__ SmallDesc sd,
                             const float2* __restrict__ G, const __grid_constant__ GatherDesc gd,
                             float2* __restrict__ C, double2* __restrict__ acc, int ns, int log_per, int log_ng,
                             int cta_rows, int reps, int entries, int slice_id) {
  extern __shared__ __align__(16) float2 Ss[];  // [entries][ns * K + 2]
  __shared__ unsigned long long blk_base[GATHER_REPS];
  const int t = threadIdx.x;
  const long long C0 = (long long)blockIdx.x * reps * cta_rows;  // the CTA's first row
  const int h0 = int(C0 >> log_ng);
  const int per = ns * K, pitch = per + 2;
  if (t < reps) {
    const long long R0 = C0 + (long long)t * cta_rows;
    unsigned long long o = 0;
    for (int j = 0; j < gd.n_slice; ++j)
      if (gd.slice_src[j] >= 0 && ((slice_id >> j) & 1)) o |= 1ull << gd.slice_src[j];
    for (int j = 0; j < gd.nrow; ++j)
      if ((R0 >> j) & 1) o |= 1ull << gd.rowpos[j];
    blk_base[t] = o;
  }
  for (int i = t; i < entries * per; i += T) {
    const float2 v = __ldg(S + small_dep(sd, (uint32_t(h0) << log_per) + i));
    Ss[i + 2 * (i >> log_per)] = ROUND ? tf32_rna2(v) : v;
  }
  size_t lo = 0;
#pragma unroll
  for (int j = 0; (1 << j) < T; ++j)
    if (j < gd.nrow && ((t >> j) & 1)) lo |= size_t(1) << gd.rowpos[j];
  __syncthreads();
  const bool pairs = K > 1 && gd.pairs;
  for (int it = 0; it < reps; ++it) {
    const long long R0 = C0 + (long long)it * cta_rows;
    bool live[ROWS];
    float2 gv[ROWS][K];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      live[r] = r * T + t < cta_rows;
      size_t base = size_t(blk_base[it]) | lo;
      if (r) base |= size_t(1) << gd.rowpos[T == 256 ? 8 : 7];  // ROWS <= 2: the row bit above the thread bits
#pragma unroll
      for (int kk = 0; kk < K; ++kk) gv[r][kk] = make_float2(0.f, 0.f);
      if (live[r]) {
        const float2* p = G + base;
        if (pairs) {
          // the lowest K bit is the stored layout's stride-1 bit: pairs (k, k+1) are
          // adjacent and 16-byte aligned (every other offset bit is >= 1)
#pragma unroll
          for (int kk = 0; kk + 1 < K; kk += 2) {
            uint32_t ko = 0;
#pragma unroll
            for (int j = 1; (1 << j) < K; ++j)
              if ((kk >> j) & 1) ko |= 1u << gd.kpos[j];
            const float4 v = __ldg(reinterpret_cast<const float4*>(p + ko));
            gv[r][kk] = make_float2(v.x, v.y);
            gv[r][kk + 1] = make_float2(v.z, v.w);
          }
        } else {
#pragma unroll
          for (int kk = 0; kk < K; ++kk) {
            uint32_t ko = 0;
#pragma unroll
            for (int j = 0; (1 << j) < K; ++j)
              if ((kk >> j) & 1) ko |= 1u << gd.kpos[j];
            gv[r][kk] = __ldg(p + ko);
          }
        }
      }
      if (ROUND) {
#pragma unroll
        for (int kk = 0; kk < K; ++kk) gv[r][kk] = tf32_rna2(gv[r][kk]);
      }
    }
    // output [h][s][g]: the row's batch entry and g
    size_t obase[ROWS];
    const float2* Sr = Ss;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const long long R = R0 + (live[r] ? r * T + t : 0);
      const size_t h = size_t(R >> log_ng);
      obase[r] = ((h * size_t(ns)) << log_ng) + size_t(R & ((1ll << log_ng) - 1));
      if (ROWS == 1) Sr = Ss + (int(h) - h0) * pitch;
    }
#pragma unroll 4
    for (int s = 0; s < ns; ++s) {
      float ar[ROWS], ai[ROWS];
#pragma unroll
      for (int r = 0; r < ROWS; ++r) ar[r] = ai[r] = 0.f;
      if constexpr (K == 1) {
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
          const float2 a = Sr[s], b = gv[r][0];
          ar[r] = fmaf(-a.y, b.y, a.x * b.x);
          ai[r] = fmaf(a.y, b.x, a.x * b.y);
        }
      } else {
#pragma unroll
        for (int kk = 0; kk < K; kk += 2) {
          const float4 a2 = *reinterpret_cast<const float4*>(Sr + s * K + kk);
#pragma unroll
          for (int r = 0; r < ROWS; ++r) {
            const float2 b0 = gv[r][kk], b1 = gv[r][kk + 1];
            ar[r] = fmaf(a2.x, b0.x, ar[r]);
            ar[r] = fmaf(-a2.y, b0.y, ar[r]);
            ai[r] = fmaf(a2.x, b0.y, ai[r]);
            ai[r] = fmaf(a2.y, b0.x, ai[r]);
            ar[r] = fmaf(a2.z, b1.x, ar[r]);
            ar[r] = fmaf(-a2.w, b1.y, ar[r]);
            ai[r] = fmaf(a2.z, b1.y, ai[r]);
            ai[r] = fmaf(a2.w, b1.x, ai[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        if (!live[r]) continue;
        const size_t o = obase[r] + (size_t(s) << log_ng);
        if (acc) {
          double2 v = acc[o];
          v.x += ar[r];
          v.y += ai[r];
          acc[o] = v;
        } else {
          C[o] = make_float2(ar[r], ai[r]);
        }
      }
    }
  }
}

// ------------------------------------------------------------------ rows kernel
// C[h][s][g] = sum_k S[h][s][k] G[h][g][k] for K of 64 and more, at most 32 rows of
// S: a CTA owns 128 rows of G, one a thread, and walks K (or its share of it) 32
// values at a time, which it stages in shared memory by coalesced loads.  Every
// output is one sum in ascending K.
//
// Bound: HBM while few rows of S meet G, the FFMA pipe at 32.  8 x 2^20 x 64 takes 467
// us a call with G in this order and 655 after a permute of G (long-K kernel: 1394
// and 1434); 32 x 2^20 x 64 522 (1336).  It needs G with K
// lowest, a permute where G is stored otherwise; beside the long-K kernel, which
// reads any order but spends a CTA's table set-up on 16 or 32 rows, it wins where
// rows are many and K is short, see rows_faster().
constexpr int RW_THREADS = 128;  // rows of G per CTA
constexpr int RW_KC = 32;        // K values staged per iteration
constexpr int RW_SMAX = 32;

__global__ void __launch_bounds__(RW_THREADS) cgemm_rows_kernel(const float2* __restrict__ S,
                                                                const float2* __restrict__ G, float2* __restrict__ C,
                                                                double2* __restrict__ acc, float2* __restrict__ part,
                                                                int ns, int ng, int K, int batch, int kchunk,
                                                                int tiles_g) {
  __shared__ float2 Gs[RW_THREADS][RW_KC + 1];
  __shared__ float2 Ss[RW_SMAX][RW_KC + 1];
  const int t = threadIdx.x;
  const int g0 = int(blockIdx.x % tiles_g) * RW_THREADS, h = int(blockIdx.x / tiles_g);
  const int kbeg = int(blockIdx.y) * kchunk, kend = min(K, kbeg + kchunk);
  const float2* Sh = S + size_t(h) * ns * K;
  const float2* Gh = G + size_t(h) * ng * K;
  float ar[RW_SMAX], ai[RW_SMAX];
#pragma unroll
  for (int s = 0; s < RW_SMAX; ++s) ar[s] = ai[s] = 0.f;
  for (int k0 = kbeg; k0 < kend; k0 += RW_KC) {
    const int kc = min(RW_KC, kend - k0);
    for (int idx = t; idx < RW_THREADS * RW_KC; idx += RW_THREADS) {
      const int r = idx / RW_KC, kk = idx % RW_KC;
      Gs[r][kk] = g0 + r < ng && kk < kc ? Gh[size_t(g0 + r) * K + k0 + kk] : make_float2(0.f, 0.f);
    }
    for (int idx = t; idx < RW_SMAX * RW_KC; idx += RW_THREADS) {
      const int r = idx / RW_KC, kk = idx % RW_KC;
      Ss[r][kk] = r < ns && kk < kc ? Sh[size_t(r) * K + k0 + kk] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int kk = 0; kk < kc; ++kk) {
      const float2 g = Gs[t][kk];
#pragma unroll
      for (int s = 0; s < RW_SMAX; ++s) {
        if (s < ns) {
          const float2 a = Ss[s][kk];
          ar[s] = fmaf(a.x, g.x, ar[s]);
          ar[s] = fmaf(-a.y, g.y, ar[s]);
          ai[s] = fmaf(a.x, g.y, ai[s]);
          ai[s] = fmaf(a.y, g.x, ai[s]);
        }
      }
    }
    __syncthreads();
  }
  if (g0 + t >= ng) return;
  const size_t base = size_t(h) * ns * ng + size_t(g0 + t);
#pragma unroll
  for (int s = 0; s < RW_SMAX; ++s) {
    if (s < ns) {
      const size_t o = base + size_t(s) * ng;
      if (part) {
        part[size_t(blockIdx.y) * batch * ns * ng + o] = make_float2(ar[s], ai[s]);
      } else if (acc) {
        double2 v = acc[o];
        v.x += ar[s];
        v.y += ai[s];
        acc[o] = v;
      } else {
        C[o] = make_float2(ar[s], ai[s]);
      }
    }
  }
}

}  // namespace

cudaError_t launch_cgemm_rows(const void* S, const void* G, void* C, void* acc, void* part, int splits, int ns, int ng,
                              int K, int batch, cudaStream_t st) {
  if (ns < 1 || ns > RW_SMAX || splits < 1 || splits > 65535 || (splits > 1 && !part))
    return cudaErrorInvalidConfiguration;
  const long long tiles_g = (ng + RW_THREADS - 1) / RW_THREADS;
  if (tiles_g * batch > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  const int kchunk = ((K + splits - 1) / splits + RW_KC - 1) / RW_KC * RW_KC;
  if ((long long)kchunk * (splits - 1) >= K) return cudaErrorInvalidConfiguration;  // an empty split
  const dim3 grid{unsigned(tiles_g * batch), unsigned(splits), 1u};
  cgemm_rows_kernel<<<grid, RW_THREADS, 0, st>>>(
      reinterpret_cast<const float2*>(S), reinterpret_cast<const float2*>(G), reinterpret_cast<float2*>(C),
      reinterpret_cast<double2*>(acc), splits > 1 ? reinterpret_cast<float2*>(part) : nullptr, ns, ng, K, batch, kchunk,
      int(tiles_g));
  return cudaGetLastError();
}

cudaError_t launch_cgemm_rows_gather(const void* Ssmall, const SmallDesc& sd, const void* Gsrc, const GatherDesc& gd,
                                     void* C, void* acc,
                                     int ns, int ng, int K, int batch, int slice_id, bool round_tf32, int sm_count,
                                     cudaStream_t st) {
  if (ns < 1 || ns > GATHER_SMAX || K < 1 || K > 32 || gd.nrow > 32 || gd.nk > 5 || (1 << gd.nk) != K || (ng & (ng - 1)))
    return cudaErrorInvalidConfiguration;
  if (ns & (ns - 1)) return cudaErrorInvalidConfiguration;
  int log_ng = 0, log_per = 0;
  while ((1 << log_per) < ns * K) ++log_per;
  while ((1 << log_ng) < ng) ++log_ng;
  const long long total = (long long)ng * batch;
  if (total != 1ll << gd.nrow) return cudaErrorInvalidConfiguration;
  // two rows a thread (each S value read serves both) while registers allow
  // and the halved grid still covers the chip
  const int rows = ng >= 512 && total >= 512ll * 4 * std::max(1, sm_count) ? 2 : 1;
  const int threads = K >= 16 && rows == 2 ? 128 : 256;
  long long cta_rows = std::min<long long>(total, threads * rows);
  const long long entry_bytes = 8ll * (ns * K + 2);
  // S rows of every entry of the CTA within 32 KB: fewer rows where many entries meet
  while (cta_rows > ng && (cta_rows / ng) * entry_bytes > 32 * 1024) cta_rows /= 2;
  const int entries = int(std::max<long long>(1, cta_rows / ng));
  const size_t smem = size_t(entries) * size_t(entry_bytes);
  if (smem > 48 * 1024 || total / cta_rows > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // several row blocks a CTA while the grid still makes a few waves
  int reps = 1;
  while (reps < GATHER_REPS && 2 * reps * cta_rows <= ng && total / (2 * reps * cta_rows) >= 16ll * std::max(1, sm_count))
    reps *= 2;
  const unsigned grid = unsigned(total / (cta_rows * reps));
  GatherDesc g = gd;
  g.pairs = gd.nk >= 1 && gd.kpos[0] == 0 && (reinterpret_cast<uintptr_t>(Gsrc) & 15) == 0;
  const float2* Sp = reinterpret_cast<const float2*>(Ssmall);
  const float2* Gp = reinterpret_cast<const float2*>(Gsrc);
  float2* Cp = reinterpret_cast<float2*>(C);
  double2* Ap = reinterpret_cast<double2*>(acc);
#define TNQ_GATHER1(K_, R_, T_) \
  cgemm_rows_gather_kernel<K_, R_, T_, (K_ >= 16 && R_ == 2 ? 128 : 256)><<<grid, threads, smem, st>>>(       \
      Sp, sd, Gp, g, Cp, Ap, ns, log_per, log_ng, int(cta_rows), reps, entries, slice_id)
#define TNQ_GATHER(K_, R_)                   \
  do {                                       \
    if (round_tf32) TNQ_GATHER1(K_, R_, true); \
    else TNQ_GATHER1(K_, R_, false);         \
  } while (0)
#define TNQ_GATHER12(K_)           \
  do {                             \
    if (rows == 2) TNQ_GATHER(K_, 2); \
    else TNQ_GATHER(K_, 1);        \
  } while (0)
  switch (K) {
    case 1: TNQ_GATHER12(1); break;
    case 2: TNQ_GATHER12(2); break;
    case 4: TNQ_GATHER12(4); break;
    case 8: TNQ_GATHER12(8); break;
    case 16: TNQ_GATHER12(16); break;
    default: TNQ_GATHER12(32);
  }
#undef TNQ_GATHER12
#undef TNQ_GATHER
#undef TNQ_GATHER1
  return cudaGetLastError();
}

}  // namespace tnq
