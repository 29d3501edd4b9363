// Device kernels and their launch descriptors (shared by the executor and the
// pairwise-contraction entry point).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace tnq {

// Calls set() once on every device that is current when this runs; `done` (one per
// use) remembers the devices where it succeeded.
template <typename Set>
cudaError_t once_per_device(std::atomic<uint64_t>* done, Set set) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? 1ull << dev : 0;
  if (done->load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = set();
  if (e == cudaSuccess) done->fetch_or(bit, std::memory_order_release);
  return e;
}

// Lets kernel f use `bytes` of dynamic shared memory, always the same number (a
// limit set for one launch could be lowered by another thread before it), on the
// current device.
inline cudaError_t allow_smem(const void* f, int bytes, std::atomic<uint64_t>* done) {
  return once_per_device(done,
                         [&] { return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

// Operand formats written by the permute kernel.
enum PermMode {
  PM_C64 = 0,          // complex64 copy in the new order
  PM_AEXP_F32 = 1,     // A' = [[re,-im],[im,re]] real expansion, FP32 (2 rows x 2K floats per complex row)
  PM_AEXP_TF32 = 2,    // as above, rounded to TF32
  PM_AEXP_TF32X3 = 3,  // as above, hi/lo TF32 split into dst0/dst1
  PM_AEXP_BF16X3 = 4,  // as above, hi/lo BF16 split
  PM_B_TF32 = 5,       // complex64 rounded to TF32
  PM_B_TF32X3 = 6,     // complex64 hi/lo TF32 split
  PM_B_BF16X3 = 7      // complex pairs as bf16x2, hi/lo split
};

struct PermDesc {
  int r;                       // destination rank
  int u;                       // bits staged per tile
  int n_outer;                 // r - u
  int kbits;                   // A' expansion: number of K bits (lowest destination bits)
  int mode;
  int n_slice;                 // slice-id bits
  int tile_src[16];            // i-th tile bit (source order): its source bit position
  int tile_dst_sorted[16];     // tile bits in destination order: destination bit position
  int tile_srcidx_of_dst[16];  // j-th tile bit in destination order -> its source-order index
  int outer_src[32];
  int outer_dst[32];
  int slice_src[32];           // source bit of slice bit j, or -1
};

void build_perm_desc(const int* src_labels, int src_rank, const int* dst_labels, int dst_rank,
                     const int* slice_labels, int n_slice, int mode, int kbits, PermDesc* d);

cudaError_t launch_permute(const PermDesc& d, const void* src, void* dst0, void* dst1, int slice_id,
                           int sm_count, cudaStream_t st);

// C[h][m][n] = sum_k A[h][m][k] * B[h][n][k] (complex64, FP32 FFMA); with acc
// non-null the result is added in FP64 to acc (same layout) instead of stored.
// With splits > 1 the K range is cut into `splits` parts whose FP32 partial
// products go to part[s][h][m][n]; launch_reduce_splits then forms C or acc.
cudaError_t launch_cgemm_simt(const void* A, const void* B, void* C, void* acc, void* part, int splits, int M,
                              int N, int K, int batch, cudaStream_t st);
// in_order: the splits of an output are always added one after the other
cudaError_t launch_reduce_splits(const void* part, int splits, size_t n, void* C, void* acc, int sm_count,
                                 cudaStream_t st, bool in_order = false);

// Long-K step with at most 32 rows on its small side (see kdot.cu).  The tile
// lists hold its stored bits in increasing position with their place in the
// tile (K bit i of the tile, or -1 - i for row bit i); ko: K bits outside the
// tile; u: batch bits (nh of them), then N bits outside the tile.
constexpr int KD_DIGITS = 7;  // 4-bit digits of a K tile index
struct KdotDesc {
  int na, nb;          // tile bits of A and B
  int tm, tn, tk;      // log2 of M rows, N rows and K values of a tile
  int nko, nh, nu;
  int nc;              // log2 of the output elements (stride of a split's partials)
  signed char a_pos[16], a_to[16], b_pos[16], b_to[16];
  signed char ko_a[28], ko_b[28];
  signed char u_a[32], u_b[32], u_c[32];
  signed char m_c[8], n_c[8];
};
// pos_a / pos_b: stored positions of [K][M][H] and [K][N][H]; pos_c: positions
// in C of the output bits [N][M][H].
bool build_kdot(int nM, int nN, int nK, int nH, const signed char* pos_a, const signed char* pos_b,
                const signed char* pos_c, KdotDesc* d);
cudaError_t launch_cgemm_kdot(const KdotDesc& d, const void* A, const void* B, void* C, void* acc, void* part,
                              int splits, cudaStream_t st);

// Bit positions (in the large operand's stored layout) of its row index (the
// N or M bits, then the batch bits) and of its K bits, plus sliced labels.
struct GatherDesc {
  int nrow;
  int rowpos[32];
  int nk;
  int kpos[8];
  int n_slice;
  int slice_src[32];
  int pairs;  // set by launch_cgemm_rows_gather: K bit 0 is stored bit 0 of a 16-byte aligned operand
};
// Small operand read in place: bit j of its [K][rows][batch] index (K bits
// lowest) sits at stored position pos[j].
struct SmallDesc {
  int n;
  signed char pos[32];
};
__device__ __forceinline__ uint32_t small_dep(const SmallDesc& d, uint32_t v) {
  uint32_t o = 0;
  for (int j = 0; j < d.n && (v >> j); ++j)
    if ((v >> j) & 1) o |= 1u << d.pos[j];
  return o;
}
// rows kernel with K <= 32 and ns <= 128 reading the large operand in place
// (fused permute), the small one as well; output [batch][ns][ng].  round_tf32: both operands are
// rounded to TF32 first.
cudaError_t launch_cgemm_rows_gather(const void* Ssmall, const SmallDesc& sd, const void* Gsrc, const GatherDesc& gd,
                                     void* C, void* acc,
                                     int ns, int ng, int K, int batch, int slice_id, bool round_tf32, int sm_count,
                                     cudaStream_t st);

// rows kernel (see skinny.cu): S [batch][ns][K], G [batch][ng][K], output [batch][ns][ng],
// ns <= 32; splits > 1 leaves FP32 sums of equal K ranges in part.
cudaError_t launch_cgemm_rows(const void* S, const void* G, void* C, void* acc, void* part, int splits, int ns, int ng,
                              int K, int batch, cudaStream_t st);

// One small contraction reading both operands in place (see small.cu): bit j of
// an output index (2^n_out of them) sits at stored position pa[j] of A, pb[j]
// of B (-1: not an index of that operand) and pc[j] of C; bit j of the
// contracted index at ka[j], kb[j].  With acc the result is added in FP64.
constexpr int SMALL_MAX_K = 10;    // log2 of the longest contracted extent taken for latency's sake
constexpr int SMALL_MAX_OUT = 30;  // log2 of the most output elements
struct SmallOp {
  const float2* A;   // slice offsets already added
  const float2* B;
  float2* C;
  double2* acc;
  int n_out, nk;
  int log_l;         // log2 of the lanes sharing an output (small_lanes_log2)
  int round_tf32;    // round the operands to TF32 first
  signed char pa[32], pb[32], pc[32];
  signed char ka[32], kb[32];
};
// A step of a step program: operands and output by byte address, index bits as
// element offsets.  An output bit's entry holds its offset in A, B and C (0:
// not an index of that tensor).
constexpr int PROG_MAX_OUT = 14;   // log2 of the largest output of a program step
constexpr int PROG_MAX_K = 10;     // log2 of its longest contracted extent
constexpr int PROG_MAX_WORK = 15;  // log2 of its complex multiply-adds (2^18 made a 3x4 batch 72 us, from 66)
constexpr int PROG_MAX_OPS = 160;  // steps per launch (their records sit in shared memory)
struct ProgOp {
  unsigned long long a, b, c;      // byte addresses (c of the FP64 accumulator when acc is set)
  uint32_t warp_begin;             // first warp-sized unit of the step within its level
  uint32_t pad0;
  short n_out, nk, log_l;
  short acc;                       // add in FP64
  short pad[4];
  uint4 bit[PROG_MAX_OUT];
  uint2 kbit[PROG_MAX_K];          // (A, B) offset of a contracted index's bit
  signed char sa[32], sb[32];      // stored positions of the sliced labels the slice id fixes (-1: none)
};
static_assert(sizeof(ProgOp) % 16 == 0, "records are copied 16 bytes at a time");
// Runs ops[0 .. n_ops) of a program, level by level: level l is ops
// [levels[l], levels[l + 1]), whose steps depend on earlier levels only.
// max_units: warp-sized units of the largest level.
cudaError_t launch_prog(const ProgOp* ops, const int* levels, int n_levels, int n_ops, int max_units, int n_slices,
                        int slice_id, cudaStream_t st);
int prog_lanes_log2(int n_out, int nk);
int small_lanes_log2(int n_out, int nk);
// splits > 1 (a power of two): FP32 sums of equal K ranges go to part[split][2^n_out].
cudaError_t launch_cgemm_small(const SmallOp& op, void* part, int splits, cudaStream_t st);

// Projection leaves j < n_proj at leaves_base + j * stride_bytes:
// P_j[(b << 1) | x] = [bits[b * row_len + tab[j]] == x] for b < n_valid, else 0.
// tab (device) also lists, after the n_proj entries, the n_open row entries
// that must hold -1 (open qubits).  Entries of another value set *err_flag.
cudaError_t launch_proj_fill(void* leaves_base, size_t stride_bytes, int n_proj, int n_open, const int* tab,
                             int row_len, int batch_log2, const int8_t* bits, int64_t n_valid, int* err_flag,
                             cudaStream_t st);

// out[b * 2^n_open + o] = acc[root_index(b, o)] for b < n_valid (complex128;
// only the real part, as one double, when real_only), where root_index =
// sum_j bit_j(b) << pos[j] + sum_i bit_(n_open-1-i)(o) << open_pos[i].
cudaError_t launch_finalize(const void* acc, void* out, int64_t n_valid, const int* pos_table, int n_pos,
                            const int* open_pos, int n_open, bool real_only, cudaStream_t st);

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st);

}  // namespace tnq
