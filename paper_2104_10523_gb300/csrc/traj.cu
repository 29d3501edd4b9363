// Kraus-trajectory sampler (builds trajectory leaves on the GPU) and the FP64
// reductions of noisy bitstring probabilities.  See traj.cuh.
#include <algorithm>

#include "traj.cuh"

namespace tnq {

namespace {

// SplitMix64 (Steele, Lea & Flood 2014): the i-th output of the generator
// started at `seed` is mix(seed + i * golden_gamma).
__device__ __forceinline__ double draw_uniform(uint64_t seed, uint64_t traj, uint64_t chan) {
  const uint64_t i = (traj << 32) + chan + 1;
  uint64_t z = seed + i * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return double(z >> 11) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// Index of the operator factor F applies in trajectory (term) tau of the pass.
__device__ __forceinline__ int pick_of(const TrajFactor& F, long long tau, uint64_t seed, uint64_t traj_base,
                                       const double* __restrict__ cumq, const int8_t* __restrict__ picks, int n_sel,
                                       int64_t n_terms) {
  if (F.channel == 2 || (F.channel == 1 && picks)) {
    // pick table: per term (observables) or per distinct trajectory (noise)
    const int64_t term = int64_t(traj_base) + tau;
    return term < n_terms ? int(picks[term * n_sel + F.chan_index]) : 0;
  }
  if (!F.channel) return 0;
  const double u = draw_uniform(seed, traj_base + uint64_t(tau), uint64_t(F.chan_index));
  int k = F.n_ops - 1;
  for (int j = 0; j < F.n_ops; ++j)
    if (u < cumq[F.cum_off + j]) {
      k = j;
      break;
    }
  return k;
}

// A CTA builds one leaf for a block of trajectories.  Most of them pick operator
// 0 of every channel of the leaf: that product is computed once and copied, and
// only the others (listed in shared memory) are multiplied up, 16 lanes to a
// 4x4 product (FP64 runs at a small fraction of the FP32 rate, and a thread
// holding whole matrices indexes local memory).  256 trajectories of 78 leaves
// with about 8 factors each took 411 us a pass, one thread per matrix.
constexpr int TL_THREADS = 256;

__global__ void __launch_bounds__(TL_THREADS) traj_leaf_kernel(
    const TrajLeafDesc* __restrict__ leaves, const TrajFactor* __restrict__ factors, const double2* __restrict__ mats,
    const double* __restrict__ cumq, char* ws, uint64_t seed, uint64_t traj_base, int traj_log2,
    const int8_t* __restrict__ picks, int n_sel, int64_t n_terms) {
  __shared__ double2 prod[TL_THREADS / 16][16];  // running product of a half-warp
  __shared__ float2 def[16];                     // product of picks 0, as stored
  __shared__ unsigned short todo[TL_THREADS];
  __shared__ int n_todo;
  const int t = threadIdx.x, hw = t >> 4, e = t & 15;
  const long long T = 1ll << traj_log2, tau0 = (long long)blockIdx.y * TL_THREADS;
  const TrajLeafDesc L = leaves[blockIdx.x];
  const int ns = L.n_slots, D = 1 << ns, rank_op = L.nfree + ns, n_out = 1 << rank_op;
  if (t == 0) n_todo = 0;
  __syncthreads();
  const long long tau = tau0 + t;
  bool plain = true;
  if (tau < T)
    for (int f = 0; f < L.n_factors && plain; ++f)
      plain = pick_of(factors[L.factor_off + f], tau, seed, traj_base, cumq, picks, n_sel, n_terms) == 0;
  if (tau < T && !plain) todo[atomicAdd(&n_todo, 1)] = (unsigned short)t;
  // product for trajectory `tt` (picks 0 when tt < 0) by the 16 lanes of a
  // half-warp, lane e holding entry e; stored entries (rows x free-input
  // columns, closed inputs take column entry 0) go to `out`
  auto build = [&](long long tt, float2* out) {
    double2(&M)[16] = prod[hw];
    const unsigned mask = 0xffffu << (t & 16);
    const bool on = e < D * D;
    const int r = e / D, c = e % D;
    M[e] = make_double2(on && r == c ? 1.0 : 0.0, 0.0);
    __syncwarp(mask);
    for (int f = 0; f < L.n_factors; ++f) {
      const TrajFactor F = factors[L.factor_off + f];
      const int k = tt < 0 ? 0 : pick_of(F, tt, seed, traj_base, cumq, picks, n_sel, n_terms);
      const double2* U = mats + size_t(F.mat_off + k) * 16;
      double2 s = make_double2(0.0, 0.0);
      if (on) {
        if (ns == 1) {  // 2x2 group, one-qubit op
          s = cadd(cmul(U[r * 2 + 0], M[0 * 2 + c]), cmul(U[r * 2 + 1], M[1 * 2 + c]));
        } else if (F.arity == 2) {  // 4x4 op on both slots (indices swapped if listed reversed)
          const int rr = F.swap ? (((r & 1) << 1) | (r >> 1)) : r;
          for (int k2 = 0; k2 < 4; ++k2) {
            const int kk = F.swap ? (((k2 & 1) << 1) | (k2 >> 1)) : k2;
            s = cadd(s, cmul(U[rr * 4 + kk], M[k2 * 4 + c]));
          }
        } else {  // one-qubit op on slot 0 (most significant) or slot 1
          const int a = r >> 1, b = r & 1;
          if (F.slot_mask == 1)
            s = cadd(cmul(U[a * 2 + 0], M[b * 4 + c]), cmul(U[a * 2 + 1], M[(2 | b) * 4 + c]));
          else
            s = cadd(cmul(U[b * 2 + 0], M[(a << 1) * 4 + c]), cmul(U[b * 2 + 1], M[(a << 1 | 1) * 4 + c]));
        }
      }
      __syncwarp(mask);
      if (on) M[e] = s;
      __syncwarp(mask);
    }
    if (e < n_out) {
      const int row = e >> L.nfree, cf = e & ((1 << L.nfree) - 1);
      int col = 0, bit = 0;
      for (int s = ns - 1; s >= 0; --s) {
        if ((L.in_fixed_mask >> s) & 1) continue;
        col |= ((cf >> bit) & 1) << (ns - 1 - s);
        ++bit;
      }
      const double2 v = M[row * D + col];
      out[e] = make_float2(float(v.x), float(v.y));
    }
    __syncwarp(mask);
  };
  if (hw == 0) build(-1, def);
  __syncthreads();
  float2* out = reinterpret_cast<float2*>(ws + L.out_offset) + (size_t(tau0) << rank_op);
  for (int i = hw; i < n_todo; i += TL_THREADS / 16) build(tau0 + todo[i], out + (size_t(todo[i]) << rank_op));
  if (tau < T && plain)
    for (int j = 0; j < n_out; ++j) out[(size_t(t) << rank_op) + j] = def[j];
}

struct Pos {
  int n;
  int p[32];
};

__device__ __forceinline__ size_t scatter(long long v, const Pos& P) {
  size_t r = 0;
  for (int j = 0; j < P.n; ++j)
    if ((v >> j) & 1) r |= size_t(1) << P.p[j];
  return r;
}

// A CTA per bitstring: its threads share the trajectories out and meet in a
// fixed tree.  (16 bitstrings of a pass used 16 threads, each a chain of 256
// dependent sums: 182 us.)
constexpr int NA_THREADS = 256;

__global__ void __launch_bounds__(NA_THREADS) noisy_accumulate_kernel(const double2* __restrict__ acc, int64_t nb,
                                                                      int64_t nt, Pos bp, Pos tp, double* psum,
                                                                      double* p2sum,
                                                                      const double* __restrict__ weights) {
  __shared__ double sh[2][NA_THREADS / 32];
  for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
    const size_t base = scatter(b, bp);
    double s = 0.0, s2 = 0.0;
    for (int64_t t = threadIdx.x; t < nt; t += NA_THREADS) {
      const double2 a = acc[base | scatter(t, tp)];
      const double p = a.x * a.x + a.y * a.y;
      const double w = weights ? weights[t] : 1.0;
      s += w * p;
      s2 += w * p * p;
    }
    for (int d = 16; d; d >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, d);
      s2 += __shfl_xor_sync(0xffffffffu, s2, d);
    }
    if ((threadIdx.x & 31) == 0) {
      sh[0][threadIdx.x >> 5] = s;
      sh[1][threadIdx.x >> 5] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double u = 0.0, u2 = 0.0;
      for (int w = 0; w < NA_THREADS / 32; ++w) {
        u += sh[0][w];
        u2 += sh[1][w];
      }
      psum[b] += u;
      p2sum[b] += u2;
    }
    __syncthreads();
  }
}

__global__ void noisy_finalize_kernel(const double* psum, const double* p2sum, int64_t nb, int64_t n, double* p,
                                      double* se) {
  for (int64_t b = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; b < nb; b += int64_t(gridDim.x) * blockDim.x) {
    const double m = psum[b] / double(n);
    p[b] = m;
    if (se) {
      const double var = fmax(p2sum[b] / double(n) - m * m, 0.0);
      se[b] = n > 1 ? sqrt(var / double(n - 1)) : 0.0;
    }
  }
}

__global__ void traj_amp_out_kernel(const double2* __restrict__ acc, int64_t nb, int64_t t0, int64_t nt, Pos bp,
                                    Pos tp, double2* out, int64_t stride) {
  const int64_t total = nb * nt;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t t = i / nb, b = i % nb;
    out[t * stride + b] = acc[scatter(b, bp) | scatter(t0 + t, tp)];
  }
}

Pos make_pos(const int* p, int n) {
  Pos P;
  P.n = n;
  for (int j = 0; j < n && j < 32; ++j) P.p[j] = p[j];
  return P;
}

unsigned blocks_for(int64_t n) { return unsigned(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096))); }

}  // namespace

cudaError_t launch_traj_leaves(const TrajLeafDesc* leaves, int n_leaves, const TrajFactor* factors,
                               const double2* mats, const double* cumq, char* ws, uint64_t seed,
                               uint64_t traj_base, int traj_log2, cudaStream_t st, const int8_t* picks, int n_sel,
                               int64_t n_terms) {
  if (n_leaves == 0) return cudaSuccess;
  const long long blocks = ((1ll << traj_log2) + TL_THREADS - 1) / TL_THREADS;
  traj_leaf_kernel<<<dim3(unsigned(n_leaves), unsigned(blocks), 1u), TL_THREADS, 0, st>>>(
      leaves, factors, mats, cumq, ws, seed, traj_base, traj_log2, picks, n_sel, n_terms);
  return cudaGetLastError();
}

cudaError_t launch_noisy_accumulate(const void* acc, int64_t nb, int64_t nt, const int* bpos, int nbpos,
                                    const int* tpos, int ntpos, double* psum, double* p2sum, cudaStream_t st,
                                    const double* weights) {
  const unsigned grid = unsigned(std::max<int64_t>(1, std::min<int64_t>(nb, 65535)));
  noisy_accumulate_kernel<<<grid, NA_THREADS, 0, st>>>(reinterpret_cast<const double2*>(acc), nb, nt,
                                                       make_pos(bpos, nbpos), make_pos(tpos, ntpos), psum, p2sum,
                                                       weights);
  return cudaGetLastError();
}

cudaError_t launch_noisy_finalize(const double* psum, const double* p2sum, int64_t nb, int64_t n_traj, double* p,
                                  double* se, cudaStream_t st) {
  noisy_finalize_kernel<<<blocks_for(nb), 256, 0, st>>>(psum, p2sum, nb, n_traj, p, se);
  return cudaGetLastError();
}

cudaError_t launch_traj_amplitudes_out(const void* acc, int64_t nb, int64_t t0, int64_t nt, const int* bpos,
                                       int nbpos, const int* tpos, int ntpos, double2* out, int64_t out_stride,
                                       cudaStream_t st) {
  traj_amp_out_kernel<<<blocks_for(nb * nt), 256, 0, st>>>(reinterpret_cast<const double2*>(acc), nb, t0, nt,
                                                           make_pos(bpos, nbpos), make_pos(tpos, ntpos), out,
                                                           out_stride);
  return cudaGetLastError();
}

}  // namespace tnq
