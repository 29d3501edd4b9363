// Long-K contractions with a small side (M <= 32): operands staged tile by tile
// from their stored layouts.
//
// These steps (the inner products that close a network, long-K rows) read both
// operands once and do few flops per byte.  Permuting an operand first costs a
// read and a write of it, so here a CTA stages tiles of both in shared memory
// straight from the stored order: a tile holds all M indices, up to 32 N values
// and the K indices among the lowest stored bits of either operand, so that the
// reads of both run along contiguous memory whatever the orders are.  Tiles are
// double-buffered (cp.async of 8 bytes: any index may be the stride-1 one).
//
// M = 4, N = 8, K = 2^20 with scattered indices (100 MB): two permutes (63 us)
// and the dot kernel with its reduction (76 us) before, 37 and 3 us now.  What
// bounds it is the latency of the shared-memory reads (short scoreboard) with 16
// warps an SM, not memory (2.8 TB/s); deeper unrolling and smaller tiles measured
// the same.
#include <algorithm>
#include <vector>

#include "kernels.cuh"
#include "splitk.h"

namespace tnq {

namespace {

constexpr int KD_THREADS = 256;

__device__ __forceinline__ void cp_async8(uint32_t smem_dst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_dst), "l"(gsrc) : "memory");
}

__device__ __forceinline__ uint32_t dep8(uint32_t v, const signed char* pos, int n) {
  uint32_t o = 0;
  for (int j = 0; j < n; ++j)
    if ((v >> j) & 1) o |= 1u << pos[j];
  return o;
}

// Block (bi, bj) of TM x TN outputs: rows bi + nbi * i, columns bj + nbj * j
// (neighbouring blocks read neighbouring rows of the odd-pitched tiles).  The
// block index sits in the low bits of the thread index, the other bits take
// every 2^kg-th K value of a tile.
template <int TM, int TN>
__global__ void __launch_bounds__(KD_THREADS, 2) cgemm_kdot_kernel(const __grid_constant__ KdotDesc d,
                                                                   const float2* __restrict__ A,
                                                                   const float2* __restrict__ B,
                                                                   float2* __restrict__ C, double2* __restrict__ acc,
                                                                   float2* __restrict__ part, int splits) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ uint2 hi_a[32], hi_b[32];       // (source, tile) offsets of element block i (256 elements each)
  __shared__ uint2 kdig[KD_DIGITS][16];      // (A, B) offsets of a 4-bit digit of the K tile index
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int pitch = (1 << d.tk) + 1;
  const int ea = 1 << d.na, eb = 1 << d.nb;  // elements of the A and B tiles
  const int rows_a = 1 << d.tm;
  const int buf_elems = (rows_a + (1 << d.tn)) * pitch;
  auto tile_off = [&](uint32_t e, const signed char* pos, const signed char* to, int n) {
    uint32_t src = 0, dst = 0;
    for (int j = 0; j < n; ++j)
      if ((e >> j) & 1) {
        src |= 1u << pos[j];
        // to >= 0: K bit of the tile; else row bit -1 - to
        dst += to[j] >= 0 ? 1u << to[j] : uint32_t(pitch) << (-1 - to[j]);
      }
    return make_uint2(src, dst);
  };
  if (t < 32) {
    if (t * KD_THREADS < ea) hi_a[t] = tile_off(t * KD_THREADS, d.a_pos, d.a_to, d.na);
    if (t * KD_THREADS < eb) hi_b[t] = tile_off(t * KD_THREADS, d.b_pos, d.b_to, d.nb);
  }
  const int ndig = (d.nko + 3) / 4;
  for (int e = t; e < ndig * 16; e += KD_THREADS) {
    const int g = e >> 4, n = min(4, d.nko - 4 * g);
    kdig[g][e & 15] = make_uint2(dep8(e & 15, d.ko_a + 4 * g, n), dep8(e & 15, d.ko_b + 4 * g, n));
  }
  const uint2 lo_a = tile_off(t, d.a_pos, d.a_to, min(d.na, 8)), lo_b = tile_off(t, d.b_pos, d.b_to, min(d.nb, 8));
  // unit: batch bits lowest (neighbouring CTAs then read neighbouring memory
  // where a batch index is the stride-1 one), then the N bits outside the tile
  const uint32_t unit = blockIdx.x, split = blockIdx.y;
  const float2* Au = A + dep8(unit, d.u_a, d.nh);
  const float2* Bu = B + dep8(unit, d.u_b, d.nu);
  __syncthreads();
  const uint32_t tiles = 1u << d.nko;
  const uint32_t t0 = uint32_t(uint64_t(tiles) * split / splits), t1 = uint32_t(uint64_t(tiles) * (split + 1) / splits);
  const uint32_t sbase = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  auto issue = [&](uint32_t kt, int b) {
    uint32_t ka = 0, kb = 0;
    for (int g = 0; g < ndig; ++g) {
      const uint2 q = kdig[g][(kt >> (4 * g)) & 15];
      ka |= q.x;
      kb |= q.y;
    }
    const uint32_t base = sbase + uint32_t(b * buf_elems) * 8u;
    const float2* Ap = Au + (ka | lo_a.x);
    const float2* Bp = Bu + (kb | lo_b.x);
    if (t < ea)
      for (int i = 0; i * KD_THREADS < ea; ++i) cp_async8(base + (lo_a.y + hi_a[i].y) * 8u, Ap + hi_a[i].x);
    if (t < eb) {
      const uint32_t bb = base + uint32_t(rows_a * pitch) * 8u;
      for (int i = 0; i * KD_THREADS < eb; ++i) cp_async8(bb + (lo_b.y + hi_b[i].y) * 8u, Bp + hi_b[i].x);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int nbi = rows_a / TM, nbj = (1 << d.tn) / TN, nblk = nbi * nbj;
  const int blk = t & (nblk - 1), kq = t / nblk, kg = KD_THREADS / nblk;
  const int bi = blk / nbj, bj = blk % nbj;
  float cr[TM][TN], ci[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) cr[i][j] = ci[i][j] = 0.f;
  if (t0 < t1) issue(t0, 0);
  int b = 0;
  for (uint32_t kt = t0; kt < t1; ++kt) {
    if (kt + 1 < t1) issue(kt + 1, b ^ 1);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const float2* as = smem + b * buf_elems + bi * pitch;
    const float2* bs = smem + b * buf_elems + (rows_a + bj) * pitch;
#pragma unroll 2
    for (int k = kq; k < 1 << d.tk; k += kg) {
      float2 a[TM], v[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = as[i * nbi * pitch + k];
#pragma unroll
      for (int j = 0; j < TN; ++j) v[j] = bs[j * nbj * pitch + k];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          cr[i][j] = fmaf(a[i].x, v[j].x, cr[i][j]);
          cr[i][j] = fmaf(-a[i].y, v[j].y, cr[i][j]);
          ci[i][j] = fmaf(a[i].x, v[j].y, ci[i][j]);
          ci[i][j] = fmaf(a[i].y, v[j].x, ci[i][j]);
        }
    }
    __syncthreads();  // buffer b is refilled by the next iteration
    b ^= 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // sum over the K groups: lanes of a block by shuffles, then the warps in order
  const int per_warp = min(nblk, 32);
  float2* red = smem;  // [warp][block of the warp][TM * TN], at most 32 KB
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      float r = cr[i][j], m = ci[i][j];
      for (int off = 16; off >= nblk; off >>= 1) {
        r += __shfl_xor_sync(0xffffffffu, r, off);
        m += __shfl_xor_sync(0xffffffffu, m, off);
      }
      if (lane < per_warp) red[(warp * per_warp + lane) * (TM * TN) + i * TN + j] = make_float2(r, m);
    }
  __syncthreads();
  const uint32_t out0 = dep8(unit, d.u_c, d.nu);
  for (int q = t; q < nblk * TM * TN; q += KD_THREADS) {
    const int ob = q / (TM * TN), ij = q % (TM * TN);
    const int wstep = max(1, nblk / 32), w0 = ob / 32, l = ob % 32;
    float r = 0.f, m = 0.f;
    for (int w = nblk > 32 ? w0 : 0; w < KD_THREADS / 32; w += wstep) {
      const float2 v = red[(w * per_warp + l) * (TM * TN) + ij];
      r += v.x;
      m += v.y;
    }
    const uint32_t mi = ob / nbj + nbi * (ij / TN), ni = ob % nbj + nbj * (ij % TN);
    const uint32_t o = out0 | dep8(mi, d.m_c, d.tm) | dep8(ni, d.n_c, d.tn);
    if (part) {
      part[(size_t(split) << d.nc) + o] = make_float2(r, m);
    } else if (acc) {
      double2 v = acc[o];
      v.x += r;
      v.y += m;
      acc[o] = v;
    } else {
      C[o] = make_float2(r, m);
    }
  }
}

}  // namespace

bool build_kdot(int nM, int nN, int nK, int nH, const signed char* pos_a, const signed char* pos_b,
                const signed char* pos_c, KdotDesc* d) {
  if (!use_kdot(nM, nN, nK) || nM + nN + nH > 31) return false;
  *d = KdotDesc{};
  d->nc = nM + nN + nH;
  d->nh = nH;
  d->tm = nM;
  kdot_tile(nM, nN, nK, &d->tn, &d->tk);
  // N indices of the tile: the lowest stored ones of B
  std::vector<int> nord(nN), kord;
  for (int j = 0; j < nN; ++j) nord[j] = j;
  std::sort(nord.begin(), nord.end(), [&](int x, int y) { return pos_b[nK + x] < pos_b[nK + y]; });
  // K indices of the tile: the lowest of A and the lowest of B in turn
  std::vector<int> ka(nK), kb(nK);
  for (int j = 0; j < nK; ++j) ka[j] = kb[j] = j;
  std::sort(ka.begin(), ka.end(), [&](int x, int y) { return pos_a[x] < pos_a[y]; });
  std::sort(kb.begin(), kb.end(), [&](int x, int y) { return pos_b[x] < pos_b[y]; });
  std::vector<char> in(nK, 0);
  for (int i = 0; i < nK; ++i)
    for (int c : {ka[i], kb[i]})
      if (!in[c]) {
        in[c] = 1;
        kord.push_back(c);
      }
  struct Bit {
    int pos, to;
  };
  std::vector<Bit> ab, bb;
  for (int i = 0; i < d->tk; ++i) {
    ab.push_back({pos_a[kord[i]], i});
    bb.push_back({pos_b[kord[i]], i});
  }
  for (int i = 0; i < nM; ++i) {
    ab.push_back({pos_a[nK + i], -1 - i});
    d->m_c[i] = pos_c[nN + i];
  }
  for (int i = 0; i < d->tn; ++i) {
    bb.push_back({pos_b[nK + nord[i]], -1 - i});
    d->n_c[i] = pos_c[nord[i]];
  }
  auto by_pos = [](const Bit& x, const Bit& y) { return x.pos < y.pos; };
  std::sort(ab.begin(), ab.end(), by_pos);
  std::sort(bb.begin(), bb.end(), by_pos);
  d->na = (int)ab.size();
  d->nb = (int)bb.size();
  for (int i = 0; i < d->na; ++i) {
    d->a_pos[i] = (signed char)ab[i].pos;
    d->a_to[i] = (signed char)ab[i].to;
  }
  for (int i = 0; i < d->nb; ++i) {
    d->b_pos[i] = (signed char)bb[i].pos;
    d->b_to[i] = (signed char)bb[i].to;
  }
  d->nko = nK - d->tk;
  for (int i = 0; i < d->nko; ++i) {
    d->ko_a[i] = pos_a[kord[d->tk + i]];
    d->ko_b[i] = pos_b[kord[d->tk + i]];
  }
  for (int i = 0; i < nH; ++i) {
    d->u_a[i] = pos_a[nK + nM + i];
    d->u_b[i] = pos_b[nK + nN + i];
    d->u_c[i] = pos_c[nN + nM + i];
  }
  d->nu = nH;
  for (int i = d->tn; i < nN; ++i, ++d->nu) {
    d->u_b[d->nu] = pos_b[nK + nord[i]];
    d->u_c[d->nu] = pos_c[nord[i]];
  }
  return d->nko <= 4 * KD_DIGITS;
}

cudaError_t launch_cgemm_kdot(const KdotDesc& d, const void* A, const void* B, void* C, void* acc, void* part,
                              int splits, cudaStream_t st) {
  if (splits < 1 || splits > 65535 || splits > (1 << d.nko) || d.nu > 30 || (splits > 1 && !part))
    return cudaErrorInvalidConfiguration;
  const int pitch = (1 << d.tk) + 1;
  const size_t smem = std::max<size_t>(size_t(2) * ((1 << d.tm) + (1 << d.tn)) * pitch * sizeof(float2), 32 * 1024);
  const dim3 grid{1u << d.nu, unsigned(splits), 1u};
  const float2* Ap = reinterpret_cast<const float2*>(A);
  const float2* Bp = reinterpret_cast<const float2*>(B);
  float2* Pp = splits > 1 ? reinterpret_cast<float2*>(part) : nullptr;
  const int tm = std::min(1 << d.tm, 4), tn = std::min(1 << d.tn, 4);
  cudaError_t e = cudaErrorInvalidConfiguration;
#define TNQ_KD(TM_, TN_)                                                                                         \
  if (tm == TM_ && tn == TN_) {                                                                                  \
    static std::atomic<uint64_t> done{0};                                                                        \
    e = allow_smem(reinterpret_cast<const void*>(cgemm_kdot_kernel<TM_, TN_>), 2 * (kKdotTileElems + 64) * 8, &done); \
    if (e != cudaSuccess) return e;                                                                              \
    cgemm_kdot_kernel<TM_, TN_><<<grid, KD_THREADS, smem, st>>>(d, Ap, Bp, reinterpret_cast<float2*>(C),         \
                                                                reinterpret_cast<double2*>(acc), Pp, splits);    \
    e = cudaGetLastError();                                                                                      \
  }
  TNQ_KD(1, 1) TNQ_KD(1, 2) TNQ_KD(1, 4) TNQ_KD(2, 1) TNQ_KD(2, 2) TNQ_KD(2, 4) TNQ_KD(4, 1) TNQ_KD(4, 2) TNQ_KD(4, 4)
#undef TNQ_KD
  return e;
}

}  // namespace tnq
