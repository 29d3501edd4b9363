// Bandwidth-oriented complex GEMMs for skinny contraction steps.
//
// Many steps of a contraction path have a tiny side: few output rows (a small
// operand meeting a large one) or a tiny output with a long contracted
// dimension (the inner products that close a network).  Their cost is reading
// the large operand once; a tiled GEMM would leave most lanes idle.
//
//   rows kernel:  C[h][s][g] = sum_k S[h][s][k] G[h][g][k] for a small side of
//                 at most 32 rows: each thread owns one row g of the large
//                 operand, the small operand and a K slice of G are staged in
//                 shared memory by coalesced loads;
//   gather kernel: short K (<= 32), each thread loads its rows of the large
//                 operand, in their stored bit layout, into registers;
//   dot kernel:   M, N <= 8 and long K: every thread walks its own part of K
//                 with 16-byte loads and keeps the M x N sums in registers; the
//                 CTA reduces them and writes one partial per CTA.
#include <algorithm>

#include "kernels.cuh"

namespace tnq {

namespace {

constexpr int RW_THREADS = 128;  // rows of the large operand per CTA
constexpr int RW_KC = 32;        // K elements staged per iteration
constexpr int RW_SMAX = 32;
constexpr int GATHER_SMAX = 128;  // small-operand rows of the gather kernel
constexpr int GATHER_REPS = 4;    // row blocks of a CTA

__global__ void __launch_bounds__(RW_THREADS) cgemm_rows_kernel(
    const float2* __restrict__ S, const float2* __restrict__ G, float2* __restrict__ C, double2* __restrict__ acc,
    float2* __restrict__ part, int ns, int ng, int K, int batch, int kchunk, int tiles_g) {
  __shared__ float2 Gs[RW_THREADS][RW_KC + 1];
  __shared__ float2 Ss[RW_SMAX][RW_KC + 1];
  const int t = threadIdx.x;
  const int tile = int(blockIdx.x % tiles_g);
  const int h = int(blockIdx.x / tiles_g);
  const int g0 = tile * RW_THREADS;
  const int split = blockIdx.y;
  const int kbeg = split * kchunk, kend = min(K, kbeg + kchunk);
  const float2* Sh = S + size_t(h) * ns * K;
  const float2* Gh = G + size_t(h) * ng * K;
  float ar[RW_SMAX], ai[RW_SMAX];
#pragma unroll
  for (int s = 0; s < RW_SMAX; ++s) ar[s] = ai[s] = 0.f;
  for (int k0 = kbeg; k0 < kend; k0 += RW_KC) {
    const int kc = min(RW_KC, kend - k0);
    // stage G[g0 .. g0+127][k0 .. k0+kc): row segments are contiguous in K
    for (int idx = t; idx < RW_THREADS * RW_KC; idx += RW_THREADS) {
      const int r = idx / RW_KC, kk = idx % RW_KC;
      float2 v = make_float2(0.f, 0.f);
      if (g0 + r < ng && kk < kc) v = Gh[size_t(g0 + r) * K + k0 + kk];
      Gs[r][kk] = v;
    }
    for (int idx = t; idx < RW_SMAX * RW_KC; idx += RW_THREADS) {
      const int r = idx / RW_KC, kk = idx % RW_KC;
      float2 v = make_float2(0.f, 0.f);
      if (r < ns && kk < kc) v = Sh[size_t(r) * K + k0 + kk];
      Ss[r][kk] = v;
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
  const int g = g0 + t;
  if (g >= ng) return;
  const size_t hbase = size_t(h) * ns * ng;
#pragma unroll
  for (int s = 0; s < RW_SMAX; ++s) {
    if (s < ns) {
      const size_t o = hbase + size_t(s) * ng + g;
      if (part) {
        part[size_t(split) * batch * ns * ng + o] = make_float2(ar[s], ai[s]);
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

constexpr int DOT_THREADS = 256;

// Dot products for M, N <= 8: the M x N outputs form (M / TM) x (N / TN) <= 4
// blocks of TM x TN (TM = min(M, 4), TN = min(N, 4)); the block index sits in
// the low bits of the thread index, so the lanes of one warp that share a row
// read it in the same 16-byte load instruction and every loaded value serves
// TN (or TM) complex multiply-adds from registers.  Each thread keeps two
// K-pairs in flight per iteration; per-CTA partials go to part[split][batch][M][N].
//
// Each operand is addressed as row base + K offset, both bit deposits of the
// row index (row bits, then batch bits) and of k into the operand's stored bit
// positions (DotOp): a contiguous [batch][rows][K] operand has K in the low
// bits; an operand read in place (its permute fused) has them where it stores
// them, in increasing positions.  A thread advances its K offset by adding in
// the deposited domain: dep(k + d) = ((dep(k) | ~mask) + dep(d)) & mask, the
// carries running through the non-K positions.
__device__ __forceinline__ size_t dot_dep(long long v, const signed char* pos, int n) {
  size_t o = 0;
  for (int j = 0; j < n; ++j)
    if ((v >> j) & 1) o |= size_t(1) << pos[j];
  return o;
}

__device__ __forceinline__ size_t dep_add(size_t x, size_t inc, size_t mask) { return ((x | ~mask) + inc) & mask; }

template <int R>
__device__ __forceinline__ void cdot_load(const float2* __restrict__ p, const size_t (&row)[R], size_t koff, bool in,
                                          float4 (&v)[R]) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) v[i] = *reinterpret_cast<const float4*>(p + row[i] + koff);
  }
}

template <int TM, int TN>
__device__ __forceinline__ void cdot_fma(const float4 (&a)[TM], const float4 (&b)[TN], float (&cr)[TM][TN],
                                         float (&ci)[TM][TN]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      cr[i][j] = fmaf(a[i].x, b[j].x, cr[i][j]);
      cr[i][j] = fmaf(-a[i].y, b[j].y, cr[i][j]);
      ci[i][j] = fmaf(a[i].x, b[j].y, ci[i][j]);
      ci[i][j] = fmaf(a[i].y, b[j].x, ci[i][j]);
      cr[i][j] = fmaf(a[i].z, b[j].z, cr[i][j]);
      cr[i][j] = fmaf(-a[i].w, b[j].w, cr[i][j]);
      ci[i][j] = fmaf(a[i].z, b[j].w, ci[i][j]);
      ci[i][j] = fmaf(a[i].w, b[j].z, ci[i][j]);
    }
}

template <int TM, int TN>
__global__ void __launch_bounds__(DOT_THREADS, 2) cdot_blk_kernel(const __grid_constant__ DotOp A,
                                                                  const __grid_constant__ DotOp B,
                                                                  float2* __restrict__ part, int M, int N, int K,
                                                                  int kchunk) {
  __shared__ float red[DOT_THREADS / 32][2 * 64];
  const int split = blockIdx.x, h = blockIdx.y;
  const int kbeg = split * kchunk, kend = min(K, kbeg + kchunk);
  const int nbj = N / TN, nb = (M / TM) * nbj;  // nb in {1, 2, 4}
  const int blk = threadIdx.x & (nb - 1), kq = threadIdx.x / nb;
  const int bi = blk / nbj, bj = blk % nbj;
  const int step = 2 * (DOT_THREADS / nb);  // K values one CTA iteration covers
  size_t ra[TM], rb[TN];
#pragma unroll
  for (int i = 0; i < TM; ++i) ra[i] = dot_dep((long long)h * M + bi * TM + i, A.rowpos, A.nrow);
#pragma unroll
  for (int j = 0; j < TN; ++j) rb[j] = dot_dep((long long)h * N + bj * TN + j, B.rowpos, B.nrow);
  const size_t ma = A.kmask, mb = B.kmask;
  const size_t a_step = dot_dep(step, A.kpos, A.nk), b_step = dot_dep(step, B.kpos, B.nk);
  const size_t a_2step = dot_dep(2 * step, A.kpos, A.nk), b_2step = dot_dep(2 * step, B.kpos, B.nk);
  float cr[TM][TN], ci[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) cr[i][j] = ci[i][j] = 0.f;
  // k is even and K bit 0 is stored bit 0 of both operands, so (k, k+1) is one
  // aligned 16-byte pair; kend is even
  int k = kbeg + 2 * kq;
  size_t ka = dot_dep(k, A.kpos, A.nk), kb = dot_dep(k, B.kpos, B.nk);
  for (; k < kend; k += 2 * step) {
    float4 a0[TM], b0[TN], a1[TM], b1[TN];
    const bool in1 = k + step < kend;
    cdot_load<TM>(A.p, ra, ka, true, a0);
    cdot_load<TN>(B.p, rb, kb, true, b0);
    cdot_load<TM>(A.p, ra, dep_add(ka, a_step, ma), in1, a1);
    cdot_load<TN>(B.p, rb, dep_add(kb, b_step, mb), in1, b1);
    cdot_fma<TM, TN>(a0, b0, cr, ci);
    cdot_fma<TM, TN>(a1, b1, cr, ci);
    ka = dep_add(ka, a_2step, ma);
    kb = dep_add(kb, b_2step, mb);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      float r = cr[i][j], im = ci[i][j];
      // sum over the lanes of the same block (lane bits above the block bits)
      for (int off = 16; off >= nb; off >>= 1) {
        r += __shfl_xor_sync(0xffffffffu, r, off);
        im += __shfl_xor_sync(0xffffffffu, im, off);
      }
      if (lane < nb) {
        red[warp][2 * (lane * TM * TN + i * TN + j)] = r;
        red[warp][2 * (lane * TM * TN + i * TN + j) + 1] = im;
      }
    }
  __syncthreads();
  for (int q = threadIdx.x; q < 2 * M * N; q += DOT_THREADS) {
    float v = 0.f;
    for (int w = 0; w < DOT_THREADS / 32; ++w) v += red[w][q];
    const int b = q / (2 * TM * TN), ij = (q % (2 * TM * TN)) >> 1;
    const int i = (b / nbj) * TM + ij / TN, j = (b % nbj) * TN + ij % TN;
    float* dst = reinterpret_cast<float*>(part + (size_t(split) * gridDim.y + h) * M * N + size_t(i) * N + j);
    dst[q & 1] = v;
  }
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
// together, gathered from their stored layout (one 16-byte pad per entry spreads the entries over the banks);
// with ROWS = 2 a CTA stays within one entry.  A CTA of a single entry walks
// reps blocks of rows, so that staging S (a dependent gather before the first
// row can be used) is paid once for all of them.
// ROUND rounds both operands to TF32 first (the products are then exact in
// FP32: the arithmetic of the plain TF32 mode on the CUDA cores).
//
// Bound: HBM while 4 FFMA per (s, k) of a row stay below the 8 (K + ns) bytes
// it moves.  One launch for every batch entry: 4096 entries of 4 x 2^12 x 8
// took 33.5 ms as one tensor-core launch each (8 us a launch).
template <int K, int ROWS, bool ROUND>
__global__ void __launch_bounds__(256) cgemm_rows_gather_kernel(const float2* __restrict__ S,
                                                                const __grid_constant__ SmallDesc sd,
                                                                const float2* __restrict__ G,
                                                                const __grid_constant__ GatherDesc gd,
                                                                float2* __restrict__ C, double2* __restrict__ acc,
                                                                int ns, int log_per, int log_ng, int cta_rows,
                                                                int reps, int entries, int slice_id) {
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
  for (int i = t; i < entries * per; i += 256) {
    const float2 v = __ldg(S + small_dep(sd, (uint32_t(h0) << log_per) + i));
    Ss[i + 2 * (i >> log_per)] = ROUND ? tf32_rna2(v) : v;
  }
  size_t lo = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < gd.nrow && ((t >> j) & 1)) lo |= size_t(1) << gd.rowpos[j];
  __syncthreads();
  const bool pairs = K > 1 && gd.kpos[0] == 0;
  for (int it = 0; it < reps; ++it) {
    const long long R0 = C0 + (long long)it * cta_rows;
    bool live[ROWS];
    float2 gv[ROWS][K];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      live[r] = r * 256 + t < cta_rows;
      size_t base = size_t(blk_base[it]) | lo;
      if (r) base |= size_t(1) << gd.rowpos[8];  // ROWS <= 2: the row bit above the thread bits
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
      const long long R = R0 + (live[r] ? r * 256 + t : 0);
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

}  // namespace

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
  const int rows = K <= 8 && ng >= 512 && total >= 512ll * 4 * std::max(1, sm_count) ? 2 : 1;
  long long cta_rows = std::min<long long>(total, 256 * rows);
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
  const float2* Sp = reinterpret_cast<const float2*>(Ssmall);
  const float2* Gp = reinterpret_cast<const float2*>(Gsrc);
  float2* Cp = reinterpret_cast<float2*>(C);
  double2* Ap = reinterpret_cast<double2*>(acc);
#define TNQ_GATHER1(K_, R_, T_) \
  cgemm_rows_gather_kernel<K_, R_, T_><<<grid, 256, smem, st>>>(Sp, sd, Gp, gd, Cp, Ap, ns, log_per, log_ng, int(cta_rows), reps, entries, \
                                                      slice_id)
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
    case 16: TNQ_GATHER(16, 1); break;
    default: TNQ_GATHER(32, 1);
  }
#undef TNQ_GATHER12
#undef TNQ_GATHER
#undef TNQ_GATHER1
  return cudaGetLastError();
}

cudaError_t launch_cgemm_rows(const void* Ssmall, const void* Gbig, void* C, void* acc, void* part, int splits,
                              int ns, int ng, int K, int batch, cudaStream_t st) {
  if (ns < 1 || ns > RW_SMAX || splits < 1 || splits > 65535) return cudaErrorInvalidConfiguration;
  const long long tiles_g = (ng + RW_THREADS - 1) / RW_THREADS;
  if (tiles_g * batch > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  int kchunk = ((K + splits - 1) / splits + RW_KC - 1) / RW_KC * RW_KC;
  dim3 grid{unsigned(tiles_g * batch), unsigned(splits), 1u};
  cgemm_rows_kernel<<<grid, RW_THREADS, 0, st>>>(
      reinterpret_cast<const float2*>(Ssmall), reinterpret_cast<const float2*>(Gbig), reinterpret_cast<float2*>(C),
      reinterpret_cast<double2*>(acc), splits > 1 ? reinterpret_cast<float2*>(part) : nullptr, ns, ng, K, batch,
      kchunk, int(tiles_g));
  return cudaGetLastError();
}

DotOp dot_contiguous(const void* p, int rows, int K, int batch) {
  // [batch][rows][K]: K bits lowest, then the row bits, then the batch bits
  DotOp d{};
  d.p = reinterpret_cast<const float2*>(p);
  int nk = 0, nr = 0, nh = 0;
  while ((1 << nk) < K) ++nk;
  while ((1 << nr) < rows) ++nr;
  while ((1 << nh) < batch) ++nh;
  d.nk = nk;
  for (int j = 0; j < nk; ++j) d.kpos[j] = (signed char)j;
  d.nrow = nr + nh;
  for (int j = 0; j < nr + nh; ++j) d.rowpos[j] = (signed char)(nk + j);
  d.kmask = (nk >= 64) ? ~0ull : ((1ull << nk) - 1);
  return d;
}

cudaError_t launch_cdot_ops(const DotOp& A, const DotOp& B, void* part, int splits, int M, int N, int K, int batch,
                            cudaStream_t st) {
  if (M < 1 || M > 8 || N < 1 || N > 8 || splits < 1 || batch > 65535) return cudaErrorInvalidConfiguration;
  // M, N and K are powers of two (all-dim-2 tensors); K bit 0 must be stored
  // bit 0 of both operands for the 16-byte pair loads
  if ((M & (M - 1)) || (N & (N - 1)) || (K & (K - 1)) || K < 2) return cudaErrorInvalidConfiguration;
  if (A.nk < 1 || B.nk < 1 || A.kpos[0] != 0 || B.kpos[0] != 0 || A.nk > 40 || B.nk > 40 || A.nrow > 24 ||
      B.nrow > 24)
    return cudaErrorInvalidConfiguration;
  // K offsets advance by carry-through-mask addition: positions must increase
  for (int j = 1; j < A.nk; ++j)
    if (A.kpos[j] <= A.kpos[j - 1]) return cudaErrorInvalidConfiguration;
  for (int j = 1; j < B.nk; ++j)
    if (B.kpos[j] <= B.kpos[j - 1]) return cudaErrorInvalidConfiguration;
  int kchunk = (K + splits - 1) / splits;
  kchunk = (kchunk + 1) & ~1;
  dim3 grid{unsigned(splits), unsigned(batch), 1u};
  float2* Pp = reinterpret_cast<float2*>(part);
  const int tm = M < 4 ? M : 4, tn = N < 4 ? N : 4;
#define TNQ_DOT(TM_, TN_) \
  if (tm == TM_ && tn == TN_) cdot_blk_kernel<TM_, TN_><<<grid, DOT_THREADS, 0, st>>>(A, B, Pp, M, N, K, kchunk)
  TNQ_DOT(1, 1); else TNQ_DOT(1, 2); else TNQ_DOT(1, 4); else TNQ_DOT(2, 1); else TNQ_DOT(2, 2);
  else TNQ_DOT(2, 4); else TNQ_DOT(4, 1); else TNQ_DOT(4, 2); else TNQ_DOT(4, 4);
#undef TNQ_DOT
  return cudaGetLastError();
}

cudaError_t launch_cdot(const void* A, const void* B, void* part, int splits, int M, int N, int K, int batch,
                        cudaStream_t st) {
  return launch_cdot_ops(dot_contiguous(A, M, K, batch), dot_contiguous(B, N, K, batch), part, splits, M, N, K, batch,
                         st);
}

}  // namespace tnq
