// libmulo: kernels and C ABI of the MuLo-SD draft-and-verify round (sm_100a).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/mulo.h"
#include "mulo_dense.cuh"
#include "mulo_islands.cuh"
#include "mulo_resident.cuh"
#include "mulo_full.cuh"
#include "mulo_redraw.cuh"
#include "mulo_rows.cuh"
#include "mulo_stream.cuh"

using namespace mulo;

// ============================================================== row kernels

struct RowKernelArgs {
  DevParams P;
  const char* cond;
  const char* uncond;
  const char* draft;
  const int32_t* draft_tok_lo;   // fused / upsample: [B,h,w]
  const int32_t* draft_tok_hi;   // unfused verify / resample: [B,H,W]
  const float* stats_in;         // unfused: [B,h,w,4]
  const uint16_t* nn;
  const uint32_t* reject_bits;   // resample stage
  const uint32_t* expand_bits;   // resample stage
  // outputs
  float* p_tok;
  float* q_tok;
  float* accept_prob;
  uint8_t* flags;                // workspace: 1 = rejected
  int32_t* cand_res;             // workspace
  int32_t* cand_tgt;             // workspace
  int32_t* out_tok;              // resample stage
  int32_t* tok_hi_out;           // upsample stage
  float* stats_out;              // upsample stage
  float* q_tok_hi_out;           // upsample stage
  uint32_t* dev_status;
};

__device__ __forceinline__ RowSrc target_row(const RowKernelArgs& a, size_t row) {
  const size_t bytes = (size_t)a.P.V * (a.P.bf16 ? 2 : 4);
  RowSrc r;
  r.cond = a.cond + row * bytes;
  r.uncond = a.uncond ? a.uncond + row * bytes : nullptr;
  r.s = a.P.cfg_scale;
  r.invT = a.P.invT;
  r.V = a.P.V;
  r.bf16 = a.P.bf16;
  return r;
}
__device__ __forceinline__ RowSrc draft_row(const RowKernelArgs& a, size_t cell) {
  const size_t bytes = (size_t)a.P.V * (a.P.bf16 ? 2 : 4);
  RowSrc r;
  r.cond = a.draft + cell * bytes;
  r.uncond = nullptr;
  r.s = 0.f;
  r.invT = a.P.invT;
  r.V = a.P.V;
  r.bf16 = a.P.bf16;
  return r;
}

__device__ __forceinline__ PoolSmem carve_pool(const DevParams& P, unsigned char* dyn) {
  PoolSmem ps;
  ps.pn = reinterpret_cast<double*>(dyn);
  ps.bitmap = reinterpret_cast<uint32_t*>(dyn + (size_t)max(P.pool_k, 1) * sizeof(double));
  return ps;
}

// The kernels of the general path come in two versions: RES for vocabularies whose rows stay in shared memory, and
// the one that reads the row from L1/L2 again and again (V > 49152).  The latter wants as many thread blocks per SM as its
// registers allow: compiled for two, the draft's kernels lost a tenth to a third (4096 rows of 4096 ids: 34 us, 42 us).
template <bool RES>
using GeneralScratch = std::conditional_t<RES, ResScratch, BlockScratch>;

__device__ __forceinline__ void round_z(double& Z) {   // Z_q as the stages hand it on: an fp32 (hi, lo) pair
  const float hi = (float)Z, lo = (float)(Z - (double)hi);
  Z = (double)hi + (double)lo;
}

// mulo_upsample_pool: one CTA per low-res cell.
template <bool RES>
__device__ __forceinline__ void upsample_cell(const RowKernelArgs& a, int cell, GeneralScratch<RES>& sc, unsigned char* dyn) {
  const DevParams& P = a.P;
  const int b = cell / (P.h * P.w), rem = cell % (P.h * P.w), ca = rem / P.w, cc = rem % P.w;
  RowSrc qr = draft_row(a, cell);
  const int tok = checked_token(a.draft_tok_lo[cell], P.V, a.dev_status);
  RowStats sq;
  float zq;
  if constexpr (RES) {
    int calls = 0;
    res_row_stats(ResRow(reinterpret_cast<float*>(dyn), P.V), qr, P.top_k, sc, calls, tok, zq, sq);
  } else {
    dense_row_stats(qr, P.top_k, sc, sq.theta, sq.m, sq.Z);
    zq = load1(qr, tok);
  }
  if (threadIdx.x == 0) {
    const float Zhi = (float)sq.Z, Zlo = (float)(sq.Z - (double)Zhi);
    a.stats_out[(size_t)cell * 4 + 0] = sq.theta;
    a.stats_out[(size_t)cell * 4 + 1] = sq.m;
    a.stats_out[(size_t)cell * 4 + 2] = Zhi;
    a.stats_out[(size_t)cell * 4 + 3] = Zlo;
    double q = (zq >= sq.theta) ? exp((double)zq - (double)sq.m) / ((double)Zhi + (double)Zlo) : 0.0;
    for (int di = 0; di < P.r; ++di)
      for (int dj = 0; dj < P.r; ++dj) {
        size_t t = ((size_t)b * P.H + (size_t)ca * P.r + di) * P.W + (size_t)cc * P.r + dj;
        a.tok_hi_out[t] = a.draft_tok_lo[cell];
        a.q_tok_hi_out[t] = (float)q;
      }
  }
}
template <bool RES>
__global__ void __launch_bounds__(kThreads, RES ? 2 : 4) k_upsample_pool(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  upsample_cell<RES>(a, blockIdx.x, sc, dyn);   // b*h*w + ca*w + cc
}
// Second launch of its fast path: the cells the fast kernel marked.
template <bool RES>
__global__ void __launch_bounds__(kThreads, RES ? 2 : 4) k_upsample_failed(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  __shared__ unsigned found[kWarps];
  let_next_begin();
  wait_for_previous();
  const int total = a.P.B * a.P.h * a.P.w;
  for (int c0 = (int)blockIdx.x * kThreads; c0 < total; c0 += (int)gridDim.x * kThreads) {
    const int cell = c0 + (int)threadIdx.x;
    const bool mine = cell < total && __float_as_uint(a.stats_out[(size_t)cell * 4]) == kStatsLeft;
    const unsigned word = __ballot_sync(kFull, mine);
    if ((threadIdx.x & 31) == 0) found[threadIdx.x >> 5] = word;
    if (!__syncthreads_or(mine)) continue;
    for (int w = 0; w < kWarps; ++w)
      for (unsigned left = found[w]; left; left &= left - 1u) {   // (block-uniform)
        upsample_cell<RES>(a, c0 + w * 32 + __ffs(left) - 1, sc, dyn);
        __syncthreads();
      }
    __syncthreads();
  }
}

// The inverse-CDF draw of uniform u from softmax(topk(row / T)); one thread writes the token to *out (-1: no mass, a row
// whose largest logit mixes to +inf).
template <bool RES>
__device__ __forceinline__ void draw_row(const RowSrc& src, int top_k, double u, GeneralScratch<RES>& sc, unsigned char* dyn,
                                         int32_t* out) {
  RowStats st;
  if constexpr (RES) {
    const ResRow row(reinterpret_cast<float*>(dyn), src.V);
    int calls = 0;
    float unused;
    const ResSums sums = res_row_stats(row, src, top_k, sc, calls, -1, unused, st);
    res_pick(row, sums, u, [&](int x) -> double { return (double)row.at(x); }, out);
    if (!(sums.total > 0.0) && threadIdx.x == 0) *out = -1;
  } else {
    dense_row_stats(src, top_k, sc, st.theta, st.m, st.Z);
    __syncthreads();
    const float invZ = (float)(1.0 / st.Z);
    // lambda = 0 and no special token: the weights are the probabilities themselves
    const int tok = dense_draw(src, src, st, st, invZ, invZ, 0.0f, -1, 0.0, nullptr, u, sc);
    if (threadIdx.x == 0) *out = tok;
  }
}

// The drafter's own draw (Sec. 3.2 Step 1) for one low-res cell by the general routines:
// q = softmax(topk(l_q / T)), inverse CDF with word 0 of the tag-1 Philox stream.
template <bool RES>
__device__ __forceinline__ void sample_cell(const RowKernelArgs& a, int cell, GeneralScratch<RES>& sc, unsigned char* dyn) {
  const DevParams& P = a.P;
  const int b = cell / (P.h * P.w), rem = cell % (P.h * P.w);
  const uint4 rnd = philox4x32_10(make_uint4((uint32_t)rem, (uint32_t)b + P.image_offset, P.round, 1u),
                                  make_uint2(P.seed_lo, P.seed_hi));
  draw_row<RES>(draft_row(a, cell), P.top_k, uniform24(rnd.x), sc, dyn, a.out_tok + cell);
}

// mulo_sample_draft, general path: one CTA per low-res cell.
template <bool RES>
__global__ void __launch_bounds__(kThreads, RES ? 2 : 3) k_sample_draft(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  sample_cell<RES>(a, blockIdx.x, sc, dyn);
}

// Second launch of mulo_sample_draft's fast path: the cells the fast kernel put on its list.
template <bool RES>
__global__ void __launch_bounds__(kThreads, RES ? 2 : 3) k_sample_failed(RowKernelArgs a, const int32_t* fail_list,
                                                            const uint32_t* fail_count) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  let_next_begin();
  wait_for_previous();
  const size_t total = (size_t)a.P.B * a.P.h * a.P.w;
  const size_t n = min((size_t)*fail_count, total);
  for (size_t idx = blockIdx.x; idx < n; idx += gridDim.x) {
    const size_t cell = (size_t)fail_list[idx];
    if (cell < total) sample_cell<RES>(a, (int)cell, sc, dyn);
    __syncthreads();
  }
}

// ---- the redraw of R_X, one launch per sequential step (Sec. 3.4, Algorithm 1 Step 6)
// Plan: the positions sorted by their step -- count, scan, fill.  offsets[s] is where step s starts in
// pos_list (s = 1 .. max_step, offsets[max_step + 1] the end); the cursors live behind the offsets.
constexpr int kScanThreads = 1024;

__global__ void __launch_bounds__(256) k_redraw_count(const int32_t* __restrict__ step, int n, int max_step,
                                                      int32_t* cursor) {
  let_next_begin();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int s = step[i];
    if (s >= 1 && s <= max_step) atomicAdd(&cursor[s], 1);
  }
}

__global__ void __launch_bounds__(kScanThreads) k_redraw_scan(int max_step, int32_t* offsets, int32_t* cursor) {
  __shared__ int warp_tot[kScanThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  let_next_begin();
  wait_for_previous();
  const int n = max_step + 1;                       // entries 0 .. max_step (entry 0 counts nothing)
  const int per = (n + kScanThreads - 1) / kScanThreads;
  const int beg = min(n, tid * per), end = min(n, beg + per);
  int mine = 0;
  for (int i = beg; i < end; ++i) mine += i == 0 ? 0 : cursor[i];
  int inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) warp_tot[warp] = inc;
  __syncthreads();
  int pre = 0;
  for (int w = 0; w < warp; ++w) pre += warp_tot[w];
  int run = pre + inc - mine;                        // positions with a step below this thread's first
  for (int i = beg; i < end; ++i) {
    const int c = i == 0 ? 0 : cursor[i];
    offsets[i] = run;
    cursor[i] = run;
    run += c;
  }
  if (tid == kScanThreads - 1) offsets[max_step + 1] = pre + inc;   // (the last thread's inclusive sum: the total)
}

__global__ void __launch_bounds__(256) k_redraw_fill(const int32_t* __restrict__ step, int n, int max_step,
                                                     int32_t* cursor, int32_t* pos_list) {
  wait_for_previous();   // (the first step is not let in early: its list is being written)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int s = step[i];
    if (s >= 1 && s <= max_step) pos_list[atomicAdd(&cursor[s], 1)] = i;
  }
}

// mulo_downsample: one thread per low-res cell; the most frequent token of its r x r block,
// ties to the one that comes first in raster order of the block (Step 7 stand-in).
__global__ void __launch_bounds__(256) k_downsample(const int32_t* x, int32_t* y,
                                                    int cells, int h, int w, int W, int r) {
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  let_next_begin();
  wait_for_previous();
  if (cell >= cells) return;
  const int b = cell / (h * w), rem = cell % (h * w), ca = rem / w, cc = rem % w;
  const int32_t* blk = x + ((size_t)b * h * r + (size_t)ca * r) * W + (size_t)cc * r;
  int best_tok = -1, best_count = 0;
  for (int s1 = 0; s1 < r * r; ++s1) {
    const int tok = blk[(size_t)(s1 / r) * W + s1 % r];
    int count = 0;
    for (int s2 = 0; s2 < r * r; ++s2) count += blk[(size_t)(s2 / r) * W + s2 % r] == tok;
    if (count > best_count) {
      best_count = count;
      best_tok = tok;
    }
  }
  y[cell] = best_tok;
}

// Statistics of a draft row by the general routines, Z_q rounded as the stages hand it on.
template <bool RES>
__device__ __forceinline__ void general_draft_stats(const DevParams& P, const RowSrc& qr, GeneralScratch<RES>& sc, unsigned char* dyn,
                                                    RowStats& sq) {
  if constexpr (RES) {
    int calls = 0;
    float unused;
    res_row_stats(ResRow(reinterpret_cast<float*>(dyn), P.V), qr, P.top_k, sc, calls, -1, unused, sq);
    __syncthreads();   // the row's memory is free again
  } else {
    dense_row_stats(qr, P.top_k, sc, sq.theta, sq.m, sq.Z);
  }
  round_z(sq.Z);
}
// One position by the general routines (its results are valid in thread 0).
template <bool RES, class WantDraws>
__device__ __forceinline__ void general_position(const RowKernelArgs& a, const RowSrc& tr, const RowSrc& qr, const RowStats& sq,
                                                 int tok, uint32_t image, uint32_t t, bool decide, int given_accept,
                                                 WantDraws want, GeneralScratch<RES>& sc, unsigned char* dyn, PositionOut& o) {
  const DevParams& P = a.P;
  if constexpr (RES) {
    int calls = 0;
    res_position(P, ResRow(reinterpret_cast<float*>(dyn), P.V), tr, qr, sq, tok, a.nn, image, t, decide, given_accept, want, sc,
                 calls, a.dev_status, o);
  } else {
    dense_position(P, tr, qr, sq, tok, a.nn, image, t, decide, given_accept, want, sc, carve_pool(P, dyn), a.dev_status, o);
  }
}
__device__ __forceinline__ void store_position(const RowKernelArgs& a, size_t g, const PositionOut& o) {   // one thread
  a.flags[g] = o.accepted ? 0 : 1;
  a.cand_res[g] = o.tok_residual;
  a.cand_tgt[g] = o.tok_target;
  if (a.p_tok) a.p_tok[g] = o.p_tok;
  if (a.q_tok) a.q_tok[g] = o.q_tok;
  if (a.accept_prob) a.accept_prob[g] = o.accept_prob;
}
__device__ __forceinline__ RowStats given_stats(const RowKernelArgs& a, size_t cell) {
  RowStats sq;
  sq.theta = a.stats_in[cell * 4 + 0];
  sq.m = a.stats_in[cell * 4 + 1];
  sq.Z = (double)a.stats_in[cell * 4 + 2] + (double)a.stats_in[cell * 4 + 3];
  return sq;
}

// One position of mulo_verify: draft statistics given.
template <bool RES>
__device__ __forceinline__ void verify_position(const RowKernelArgs& a, size_t g, GeneralScratch<RES>& sc, unsigned char* dyn) {
  const DevParams& P = a.P;
  const int N = P.H * P.W;
  const int b = (int)(g / N), t = (int)(g % N), i = t / P.W, j = t % P.W;
  const size_t cell = ((size_t)b * P.h + i / P.r) * P.w + j / P.r;
  const RowStats sq = given_stats(a, cell);
  const int tok = checked_token(a.draft_tok_hi[g], P.V, a.dev_status);
  PositionOut o;
  general_position<RES>(a, target_row(a, g), draft_row(a, cell), sq, tok, (uint32_t)b + P.image_offset, (uint32_t)t, true, 0,
                        [](int) { return (int)kDrawNone; }, sc, dyn, o);
  if (threadIdx.x == 0) {
    a.flags[g] = o.accepted ? 0 : 1;
    a.p_tok[g] = o.p_tok;
    a.q_tok[g] = o.q_tok;
    a.accept_prob[g] = o.accept_prob;
  }
}

// mulo_verify (FUSED = false): one CTA per target position, draft statistics given.
// mulo_round  (FUSED = true):  one CTA per low-res cell: draft statistics, then its
// r*r children; accept flags and candidate draws go to the workspace.
template <bool FUSED, bool RES>
__global__ void __launch_bounds__(kThreads, 2) k_verify_rows(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  const DevParams& P = a.P;
  const int N = P.H * P.W;
  if (FUSED) {
    const int cell = blockIdx.x;
    const int b = cell / (P.h * P.w), rem = cell % (P.h * P.w), ca = rem / P.w, cc = rem % P.w;
    RowSrc qr = draft_row(a, cell);
    RowStats sq;
    general_draft_stats<RES>(P, qr, sc, dyn, sq);
    const int tok = checked_token(a.draft_tok_lo[cell], P.V, a.dev_status);
    for (int di = 0; di < P.r; ++di)
      for (int dj = 0; dj < P.r; ++dj) {
        const int t = (ca * P.r + di) * P.W + cc * P.r + dj;
        const size_t g = (size_t)b * N + t;
        PositionOut o;
        const int mode = P.resample_mode;
        general_position<RES>(a, target_row(a, g), qr, sq, tok, (uint32_t)b + P.image_offset, (uint32_t)t, true, 0,
                              [mode](int acc) { return draws_for(mode, acc); }, sc, dyn, o);
        if (threadIdx.x == 0) store_position(a, g, o);
        __syncthreads();
      }
  } else {
    verify_position<RES>(a, blockIdx.x, sc, dyn);
  }
}

// Second launch of mulo_verify's fast path: the positions the fast kernel put on its list.
template <bool RES>
__global__ void __launch_bounds__(kThreads, 2) k_verify_left(RowKernelArgs a, const int32_t* fail_list, const uint32_t* fail_count) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  let_next_begin();
  wait_for_previous();
  const size_t total = (size_t)a.P.B * a.P.H * a.P.W, n = min((size_t)*fail_count, total);
  for (size_t idx = blockIdx.x; idx < n; idx += gridDim.x) {
    const size_t g = (size_t)fail_list[idx];
    if (g < total) verify_position<RES>(a, g, sc, dyn);
    __syncthreads();
  }
}

// Second launch of mulo_round's fast paths: the positions the fast kernel put on its
// list (rows whose prediction failed), done by the general routines, one CTA at a time.
template <bool RES>
__global__ void __launch_bounds__(kThreads, 2) k_verify_failed(RowKernelArgs a, const int32_t* fail_list,
                                                            const uint32_t* fail_count) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  let_next_begin();
  wait_for_previous();
  const DevParams& P = a.P;
  const int N = P.H * P.W;
  const size_t total = (size_t)P.B * N;
  const size_t n = min((size_t)*fail_count, total);
  for (size_t idx = blockIdx.x; idx < n; idx += gridDim.x) {
    const size_t g = (size_t)fail_list[idx];
    if (g >= total) continue;
    const int b = (int)(g / N), t = (int)(g % N), i = t / P.W, j = t % P.W;
    const size_t cell = ((size_t)b * P.h + i / P.r) * P.w + j / P.r;
    RowSrc qr = draft_row(a, cell);
    RowStats sq;
    general_draft_stats<RES>(P, qr, sc, dyn, sq);
    const int tok = checked_token(a.draft_tok_lo[cell], P.V, a.dev_status);
    PositionOut o;
    const int mode = P.resample_mode;
    general_position<RES>(a, target_row(a, g), qr, sq, tok, (uint32_t)b + P.image_offset, (uint32_t)t, true, 0,
                          [mode](int acc) { return draws_for(mode, acc); }, sc, dyn, o);
    if (threadIdx.x == 0) store_position(a, g, o);
    __syncthreads();
  }
}

__device__ __forceinline__ int get_bit(const uint32_t* bits, int Ww, int H, int b, int i, int j) {
  return (bits[((size_t)b * H + i) * Ww + (j >> 5)] >> (j & 31)) & 1u;
}

// Would position (i,j), if it had been accepted, have been swept into R_X by
// another rejection?  (some other rejected position within radius l, and -- with
// clipping -- (i,j) is not the image's first rejection)
__device__ __forceinline__ bool covered_by_other(const uint32_t* rej, int Ww, int H, int W, int b, int i,
                                                 int j, int l, int clip, int t0) {
  if (clip && i * W + j == t0) return false;
  for (int ii = max(0, i - l); ii <= min(H - 1, i + l); ++ii)
    for (int jj = max(0, j - l); jj <= min(W - 1, j + l); ++jj)
      if ((ii != i || jj != j) && get_bit(rej, Ww, H, b, ii, jj)) return true;
  return false;
}

// One position of mulo_resample; positions outside R_X copy x~.
template <bool RES>
__device__ __forceinline__ void resample_position(const RowKernelArgs& a, size_t g, GeneralScratch<RES>& sc, unsigned char* dyn) {
  const DevParams& P = a.P;
  const int N = P.H * P.W, Ww = (P.W + 31) / 32;
  const int b = (int)(g / N), t = (int)(g % N), i = t / P.W, j = t % P.W;
  const int tok_raw = a.draft_tok_hi[g];
  if (!get_bit(a.expand_bits, Ww, P.H, b, i, j)) {
    if (threadIdx.x == 0) a.out_tok[g] = tok_raw;
    return;
  }
  const int rejected = get_bit(a.reject_bits, Ww, P.H, b, i, j);
  int use_res;
  if (P.resample_mode == MULO_RESAMPLE_RESIDUAL_ALL) use_res = 1;
  else if (P.resample_mode == MULO_RESAMPLE_TARGET_ALL) use_res = 0;
  else if (P.resample_mode == MULO_RESAMPLE_ISOLATED_RESIDUAL) {
    use_res = rejected;
    if (rejected) {
      // first rejection of the image: scan the words of image b (uniform across the CTA)
      int t0 = N;
      for (int w = 0; w < P.H * Ww && t0 == N; ++w) {
        uint32_t v = a.reject_bits[(size_t)b * P.H * Ww + w];
        if (v) t0 = (w / Ww) * P.W + (w % Ww) * 32 + __ffs(v) - 1;
      }
      if (covered_by_other(a.reject_bits, Ww, P.H, P.W, b, i, j, P.radius, P.clip, t0)) use_res = 0;
    }
  } else use_res = rejected;
  const size_t cell = ((size_t)b * P.h + i / P.r) * P.w + j / P.r;
  const RowStats sq = given_stats(a, cell);
  const int tok = checked_token(tok_raw, P.V, a.dev_status);
  PositionOut o;
  const int draw = use_res ? kDrawResidual : kDrawTarget;
  general_position<RES>(a, target_row(a, g), draft_row(a, cell), sq, tok, (uint32_t)b + P.image_offset, (uint32_t)t, false,
                        !rejected, [draw](int) { return draw; }, sc, dyn, o);
  if (threadIdx.x == 0) a.out_tok[g] = use_res ? o.tok_residual : o.tok_target;
}
// mulo_resample: one CTA per target position.
template <bool RES>
__global__ void __launch_bounds__(kThreads, 2) k_resample_rows(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  resample_position<RES>(a, blockIdx.x, sc, dyn);
}
// Second launch of its fast path: the positions the fast kernel marked.
template <bool RES>
__global__ void __launch_bounds__(kThreads, 2) k_resample_left(RowKernelArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GeneralScratch<RES> sc;
  __shared__ unsigned found[kWarps];
  let_next_begin();
  wait_for_previous();
  const size_t total = (size_t)a.P.B * a.P.H * a.P.W;
  for (size_t g0 = (size_t)blockIdx.x * kThreads; g0 < total; g0 += (size_t)gridDim.x * kThreads) {
    const size_t g = g0 + threadIdx.x;
    const bool mine = g < total && a.out_tok[g] == kPickLeft;   // (x~ of such a value: it is copied once more)
    const unsigned word = __ballot_sync(kFull, mine);
    if ((threadIdx.x & 31) == 0) found[threadIdx.x >> 5] = word;
    if (!__syncthreads_or(mine)) continue;
    for (int w = 0; w < kWarps; ++w)
      for (unsigned left = found[w]; left; left &= left - 1u) {   // (block-uniform)
        resample_position<RES>(a, g0 + w * 32 + __ffs(left) - 1, sc, dyn);
        __syncthreads();
      }
    __syncthreads();
  }
}

// ============================================================= mask kernel
// One CTA per image, warps over 32-position tiles: ballot packs accept flags
// into row words, ffs/popc give t_0 and the counts, funnel shifts dilate.

struct MaskArgs {
  int H, W, r, radius, clip, resample_mode;
  const uint8_t* flags;          // [B,H,W] 1 = rejected           (MODE 0, 2)
  const uint32_t* reject_in;     // [B,H,Ww]                        (MODE 1)
  const int32_t* first_in;       // [B]                             (MODE 1)
  uint32_t* reject_bits;         // out (MODE 0, 2)
  uint32_t* expand_bits;         // out (MODE 1, 2)
  int32_t* n_reject;             // out (MODE 0, 2), may be null
  int32_t* first_reject;         // out (MODE 0, 2), may be null
  int32_t* n_expand;             // out (MODE 1, 2), may be null
  const int32_t* cand_res;       // MODE 2
  const int32_t* cand_tgt;       // MODE 2
  const int32_t* draft_tok_lo;   // MODE 2: [B,h,w]
  int32_t* out_tok;              // MODE 2
};

constexpr int kMaskThreads = 256;

// MODE 0: flags -> reject bits, counts, t_0            (tail of mulo_verify)
// MODE 1: reject bits -> expand bits, count            (mulo_local_reject_expand)
// MODE 2: flags -> both masks, counts, output tokens   (tail of mulo_round)
template <int MODE>
__global__ void __launch_bounds__(kMaskThreads) k_mask(MaskArgs a) {
  extern __shared__ uint32_t words[];
  const int H = a.H, W = a.W, Ww = (W + 31) / 32, nw = H * Ww, N = H * W;
  uint32_t* rej = words;
  uint32_t* hd = words + nw;
  uint32_t* ex = words + 2 * nw;
  __shared__ int s_nrej, s_first, s_nexp;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_previous();
  if (tid == 0) {
    s_nrej = 0;
    s_first = N;
    s_nexp = 0;
  }
  __syncthreads();
  if (MODE == 1) {
    for (int w = tid; w < nw; w += kMaskThreads) rej[w] = a.reject_in[(size_t)b * nw + w];
    if (tid == 0) s_first = a.first_in[b];
  } else {
    for (int w = warp; w < nw; w += kMaskThreads / 32) {
      const int i = w / Ww, j = (w % Ww) * 32 + lane;
      const bool r = j < W && a.flags[(size_t)b * N + (size_t)i * W + j] != 0;
      const uint32_t word = __ballot_sync(kFull, r);
      if (lane == 0) {
        rej[w] = word;
        if (word) {
          atomicAdd(&s_nrej, __popc(word));
          atomicMin(&s_first, i * W + (w % Ww) * 32 + __ffs(word) - 1);
        }
      }
    }
  }
  __syncthreads();
  const int t0 = s_first;
  if (MODE != 1) {
    for (int w = tid; w < nw; w += kMaskThreads) a.reject_bits[(size_t)b * nw + w] = rej[w];
    if (tid == 0) {
      if (a.n_reject) a.n_reject[b] = s_nrej;
      if (a.first_reject) a.first_reject[b] = t0;
    }
  }
  if (MODE == 0) return;

  // horizontal dilation by l: OR of the row shifted by -l..l, with carries
  // across word boundaries (l <= 31, so only the two adjacent words matter)
  const int l = a.radius;
  for (int w = tid; w < nw; w += kMaskThreads) {
    const int wj = w % Ww;
    const uint32_t cur = rej[w];
    const uint32_t prev = wj > 0 ? rej[w - 1] : 0u;
    const uint32_t next = wj + 1 < Ww ? rej[w + 1] : 0u;
    uint32_t acc = cur;
    for (int s = 1; s <= l; ++s) {
      acc |= __funnelshift_l(prev, cur, s);   // bits moved towards higher j
      acc |= __funnelshift_r(cur, next, s);   // bits moved towards lower j
    }
    if (wj == Ww - 1 && (W & 31)) acc &= (1u << (W & 31)) - 1u;
    hd[w] = acc;
  }
  __syncthreads();
  // vertical dilation, then Eq. 6's clause u >= t_0
  for (int w = tid; w < nw; w += kMaskThreads) {
    const int i = w / Ww, wj = w % Ww;
    uint32_t acc = 0u;
    for (int ii = max(0, i - l); ii <= min(H - 1, i + l); ++ii) acc |= hd[ii * Ww + wj];
    if (a.clip) {
      const int i0 = t0 / W, j0 = t0 % W;
      if (t0 >= N || i < i0) acc = (t0 >= N) ? acc : 0u;
      else if (i == i0) {
        const int lo = j0 - wj * 32;   // first kept bit of this word
        if (lo >= 32) acc = 0u;
        else if (lo > 0) acc &= ~((1u << lo) - 1u);
      }
    }
    ex[w] = acc;
    a.expand_bits[(size_t)b * nw + w] = acc;
    if (acc) atomicAdd(&s_nexp, __popc(acc));
  }
  __syncthreads();
  if (tid == 0 && a.n_expand) a.n_expand[b] = s_nexp;
  if (MODE != 2) return;

  // output assembly: x~ outside R_X, the position's draw inside
  const int h = H / a.r, w_lo = W / a.r;
  for (int t = tid; t < N; t += kMaskThreads) {
    const int i = t / W, j = t % W;
    const size_t g = (size_t)b * N + t;
    int tok = a.draft_tok_lo[((size_t)b * h + i / a.r) * w_lo + j / a.r];
    if ((ex[i * Ww + (j >> 5)] >> (j & 31)) & 1u) {
      const int rejected = (rej[i * Ww + (j >> 5)] >> (j & 31)) & 1u;
      int use_res;
      if (a.resample_mode == MULO_RESAMPLE_RESIDUAL_ALL) use_res = 1;
      else if (a.resample_mode == MULO_RESAMPLE_TARGET_ALL) use_res = 0;
      else if (a.resample_mode == MULO_RESAMPLE_ISOLATED_RESIDUAL)
        use_res = rejected && !covered_by_other(rej, Ww, H, W, 0, i, j, l, a.clip, t0);
      else use_res = rejected;
      tok = use_res ? a.cand_res[g] : a.cand_tgt[g];
    }
    a.out_tok[g] = tok;
  }
}

// ================================================================ host side

struct mulo_ctx {
  int device;
  int sm_count;
  int smem_optin;
  void* ws;
  size_t ws_bytes;
  uint64_t launches;
  std::vector<cudaEvent_t> ev;   // start/stop pairs around the fused row kernel
  size_t ev_used;
  int force_dense;               // diagnostics: never take the fast top-k path
  struct Ready { const void* kernel; size_t dyn; int per_sm; };
  // Kernels whose shared-memory cap is raised, and the CTAs of them an SM holds.  A fixed table (nothing on the way to a
  // launch may throw) whose entries stay as they are once counted: calls from several threads read it without a lock.
  Ready ready[64];
  std::atomic<int> n_ready;
  std::mutex ready_mutex;        // for adding an entry
};

static const size_t kStatusBytes = 256;

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static mulo_status validate(const mulo_params* p) {
  if (!p) return MULO_ERR_INVALID_ARG;
  if (p->B < 0 || p->H <= 0 || p->W <= 0 || p->r <= 0) return MULO_ERR_INVALID_ARG;
  if (p->H % p->r || p->W % p->r) return MULO_ERR_INVALID_ARG;
  if (p->V <= 0 || p->V % 8) return MULO_ERR_INVALID_ARG;
  if (p->logit_dtype != MULO_F32 && p->logit_dtype != MULO_BF16) return MULO_ERR_INVALID_ARG;
  if (!(p->temperature > 0.0f) || !isfinite(p->temperature)) return MULO_ERR_INVALID_ARG;
  if (!isfinite(p->cfg_scale)) return MULO_ERR_INVALID_ARG;
  if (p->accept_mode != MULO_ACCEPT_RATIO && p->accept_mode != MULO_ACCEPT_THRESHOLD) return MULO_ERR_INVALID_ARG;
  if (p->resample_mode < 0 || p->resample_mode > MULO_RESAMPLE_ISOLATED_RESIDUAL) return MULO_ERR_INVALID_ARG;
  if (p->radius < 0) return MULO_ERR_INVALID_ARG;
  if (p->pool_k > 1 && !(p->pool_delta >= 0.0f)) return MULO_ERR_INVALID_ARG;
  if (p->V > 65536) return MULO_ERR_UNSUPPORTED;
  if (p->radius > 31) return MULO_ERR_UNSUPPORTED;
  if (p->pool_k > 2048 || p->pool_k > p->V) return MULO_ERR_UNSUPPORTED;
  if ((size_t)p->H * ((p->W + 31) / 32) > 4000) return MULO_ERR_UNSUPPORTED;
  if ((double)p->B * p->H * p->W > 2.0e9) return MULO_ERR_UNSUPPORTED;
  return MULO_OK;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// Kernels are launched on the calling thread's current device, while limits, workspace and the
// built-in scratch array belong to the context's device: the two must be the same.
static mulo_status on_context_device(const mulo_ctx* ctx) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess) {
    cudaGetLastError();
    return MULO_ERR_CUDA;
  }
  return cur == ctx->device ? MULO_OK : MULO_ERR_INVALID_ARG;
}

static DevParams to_dev(const mulo_params* p) {
  DevParams d;
  d.B = p->B; d.H = p->H; d.W = p->W; d.V = p->V; d.r = p->r;
  d.h = p->H / p->r; d.w = p->W / p->r;
  d.bf16 = p->logit_dtype == MULO_BF16;
  d.invT = 1.0f / p->temperature;
  d.cfg_scale = p->cfg_scale;
  d.top_k = (p->top_k > 0 && p->top_k < p->V) ? p->top_k : 0;
  d.accept_mode = p->accept_mode;
  d.tau = (double)p->tau;
  d.pool_k = p->pool_k > 1 ? p->pool_k : 1;
  d.pool_delta = (double)p->pool_delta;
  d.radius = p->radius; d.clip = p->clip_before_first != 0; d.resample_mode = p->resample_mode;
  d.seed_lo = (uint32_t)(p->seed & 0xffffffffu); d.seed_hi = (uint32_t)(p->seed >> 32);
  d.round = p->round; d.image_offset = p->image_offset;
  return d;
}

static size_t pool_smem_bytes(const DevParams& d) {
  if (d.pool_k <= 1) return 0;
  return (size_t)d.pool_k * sizeof(double) + (size_t)((d.V + 31) / 32) * 4;
}

struct Workspace {
  uint32_t* status;
  uint8_t* flags;
  int32_t* cand_res;
  int32_t* cand_tgt;
  int32_t* fail_list;   // positions the streaming kernel leaves to the dense routines
  size_t bytes;
};

static Workspace carve_ws(void* base, const mulo_params* p) {
  const size_t n = (size_t)p->B * p->H * p->W;
  Workspace w;
  char* c = (char*)base;
  size_t off = 0;
  w.status = (uint32_t*)(c + off); off += kStatusBytes;
  w.flags = (uint8_t*)(c + off); off += align_up(n, 256);
  w.cand_res = (int32_t*)(c + off); off += align_up(n * 4, 256);
  w.cand_tgt = (int32_t*)(c + off); off += align_up(n * 4, 256);
  w.fail_list = (int32_t*)(c + off); off += align_up(n * 4, 256);
  w.bytes = off;
  return w;
}

extern "C" {

const char* mulo_status_string(mulo_status s) {
  switch (s) {
    case MULO_OK: return "ok";
    case MULO_ERR_INVALID_ARG: return "invalid argument";
    case MULO_ERR_UNSUPPORTED: return "unsupported size or parameter";
    case MULO_ERR_WORKSPACE: return "workspace missing or too small";
    case MULO_ERR_CUDA: return "CUDA runtime error";
    case MULO_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

mulo_status mulo_create(mulo_ctx** out, int device) {
  if (!out) return MULO_ERR_INVALID_ARG;
  *out = nullptr;
  // (two attributes: the whole property struct takes the driver 2 to 40 ms)
  int sm_count = 0, smem_optin = 0;
  if (cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess) {
    cudaGetLastError();
    return MULO_ERR_CUDA;
  }
  if (cudaSetDevice(device) != cudaSuccess) return MULO_ERR_CUDA;
  mulo_ctx* c = new (std::nothrow) mulo_ctx();
  if (!c) return MULO_ERR_INVALID_ARG;
  c->device = device;
  c->sm_count = sm_count;
  c->smem_optin = smem_optin;
  c->ws = nullptr;
  c->ws_bytes = 0;
  c->launches = 0;
  c->ev_used = 0;
  c->force_dense = 0;
  c->n_ready = 0;
  *out = c;
  return MULO_OK;
}

void mulo_destroy(mulo_ctx* ctx) {
  if (!ctx) return;
  for (cudaEvent_t e : ctx->ev) cudaEventDestroy(e);
  delete ctx;
}

mulo_status mulo_set_general_path_only(mulo_ctx* ctx, int on) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  ctx->force_dense = on != 0;
  return MULO_OK;
}

mulo_status mulo_set_timing(mulo_ctx* ctx, int max_launches) {
  if (!ctx || max_launches < 0 || max_launches > 4096) return MULO_ERR_INVALID_ARG;
  for (cudaEvent_t e : ctx->ev) cudaEventDestroy(e);
  ctx->ev.clear();
  ctx->ev_used = 0;
  for (int i = 0; i < 2 * max_launches; ++i) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return MULO_ERR_CUDA;
    ctx->ev.push_back(e);
  }
  return MULO_OK;
}

mulo_status mulo_read_timing(mulo_ctx* ctx, double* row_kernel_ms, uint64_t* row_kernel_launches) {
  if (!ctx || !row_kernel_ms || !row_kernel_launches) return MULO_ERR_INVALID_ARG;
  double total = 0.0;
  for (size_t i = 0; i + 1 < ctx->ev_used; i += 2) {
    if (cudaEventSynchronize(ctx->ev[i + 1]) != cudaSuccess) return MULO_ERR_CUDA;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, ctx->ev[i], ctx->ev[i + 1]) != cudaSuccess) return MULO_ERR_CUDA;
    total += ms;
  }
  *row_kernel_ms = total;
  *row_kernel_launches = ctx->ev_used / 2;
  ctx->ev_used = 0;
  return MULO_OK;
}

mulo_status mulo_workspace_bytes(const mulo_params* p, size_t* bytes) {
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!bytes) return MULO_ERR_INVALID_ARG;
  *bytes = carve_ws(nullptr, p).bytes;
  return MULO_OK;
}

mulo_status mulo_set_workspace(mulo_ctx* ctx, void* dev_ptr, size_t bytes) {
  if (!ctx || !dev_ptr || ((uintptr_t)dev_ptr & 255u) || bytes < kStatusBytes) return MULO_ERR_INVALID_ARG;
  if (cudaMemset(dev_ptr, 0, kStatusBytes) != cudaSuccess) return MULO_ERR_CUDA;
  ctx->ws = dev_ptr;
  ctx->ws_bytes = bytes;
  return MULO_OK;
}

mulo_status mulo_status_of_device_flags(uint32_t flags) {
  return (flags & MULO_DEV_TIMEOUT) ? MULO_ERR_TIMEOUT : MULO_OK;
}

mulo_status mulo_poll_device_status(mulo_ctx* ctx, void* stream, uint32_t* flags) {
  if (!ctx || !flags) return MULO_ERR_INVALID_ARG;
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(flags, ctx->ws, sizeof(uint32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess) return MULO_ERR_CUDA;
  if (cudaMemsetAsync(ctx->ws, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return MULO_ERR_CUDA;
  return mulo_status_of_device_flags(*flags);
}

mulo_status mulo_poll_fallback_counts(mulo_ctx* ctx, void* stream, uint32_t counts[5]) {
  if (!ctx || !counts) return MULO_ERR_INVALID_ARG;
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* src = (char*)ctx->ws + sizeof(uint32_t);
  if (cudaMemcpyAsync(counts, src, 5 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess) return MULO_ERR_CUDA;
  if (cudaMemsetAsync(src, 0, 5 * sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return MULO_ERR_CUDA;
  return MULO_OK;
}

mulo_status mulo_kernel_launches(const mulo_ctx* ctx, uint64_t* count) {
  if (!ctx || !count) return MULO_ERR_INVALID_ARG;
  *count = ctx->launches;
  return MULO_OK;
}

}  // extern "C"

static mulo_status check_ws(mulo_ctx* ctx, const mulo_params* p, Workspace* w) {
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  *w = carve_ws(ctx->ws, p);
  if (w->bytes > ctx->ws_bytes) return MULO_ERR_WORKSPACE;
  return MULO_OK;
}

static mulo_status launched(mulo_ctx* ctx, int n) {
  if (cudaGetLastError() != cudaSuccess) return MULO_ERR_CUDA;
  ctx->launches += (uint64_t)n;
  return MULO_OK;
}

// Dynamic shared memory of the general path's kernels.
static size_t general_smem(const DevParams& d, bool pooling) {
  if (resident_fits(d.V)) return resident_bytes(d.V);
  return pooling ? pool_smem_bytes(d) : 0;
}

// CTAs of `threads` with `dyn` bytes of dynamic shared memory that an SM holds; 0 if the kernel cannot run so.  The
// kernel's shared-memory cap is raised on the way -- always to all that the device allows, so that contexts and threads
// that set it for the same kernel agree.  Asked once per context, kernel and size.
template <class K>
static int ctas_per_sm(mulo_ctx* ctx, K kernel, int threads, size_t dyn) {
  const void* const key = (const void*)kernel;
  const int n = ctx->n_ready.load(std::memory_order_acquire);
  for (int i = 0; i < n; ++i)
    if (ctx->ready[i].kernel == key && ctx->ready[i].dyn == dyn) return ctx->ready[i].per_sm;
  cudaFuncAttributes fa;
  int per_sm = 0;
  if (cudaFuncGetAttributes(&fa, key) != cudaSuccess || dyn + fa.sharedSizeBytes > (size_t)ctx->smem_optin ||
      cudaFuncSetAttribute(key, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - (int)fa.sharedSizeBytes) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, dyn) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lock(ctx->ready_mutex);
  const int at = ctx->n_ready.load(std::memory_order_relaxed);
  if (at < (int)(sizeof ctx->ready / sizeof ctx->ready[0])) {   // (full: asked again on each call)
    ctx->ready[at] = {key, dyn, per_sm};
    ctx->n_ready.store(at + 1, std::memory_order_release);
  }
  return per_sm;
}

// Launches a kernel that may begin while the one before it in the stream still runs (it waits for it itself: wait_for_previous).
template <class... P, class... A>
static bool launch_after(void (*kernel)(P...), unsigned grid, int threads, size_t dyn, cudaStream_t st, const A&... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kernel, P(args)...) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

// Launches one of the general path's kernels in the version for this vocabulary; false if it cannot run.
#define MULO_LAUNCH_GENERAL(KERNEL, grid, dyn, st, ...)                                     \
  (resident_fits(a.P.V)                                                                     \
       ? launch_general(ctx, KERNEL(true), (unsigned)(grid), dyn, st, __VA_ARGS__)          \
       : launch_general(ctx, KERNEL(false), (unsigned)(grid), dyn, st, __VA_ARGS__))
template <class K, class... A>
static bool launch_general(mulo_ctx* ctx, K kernel, unsigned grid, size_t dyn, cudaStream_t st, const A&... args) {
  if (ctas_per_sm(ctx, kernel, kThreads, dyn) < 1) return false;
  kernel<<<grid, kThreads, dyn, st>>>(args...);
  return true;
}
// ... for the rows that a fast kernel left, after it.
#define MULO_LAUNCH_LEFT(KERNEL, dyn, st, ...) \
  (resident_fits(a.P.V) ? launch_left(ctx, KERNEL(true), dyn, st, __VA_ARGS__) : launch_left(ctx, KERNEL(false), dyn, st, __VA_ARGS__))
template <class K, class... A>
static bool launch_left(mulo_ctx* ctx, K kernel, size_t dyn, cudaStream_t st, const A&... args) {
  return ctas_per_sm(ctx, kernel, kThreads, dyn) >= 1 && launch_after(kernel, 2u * (unsigned)ctx->sm_count, kThreads, dyn, st, args...);
}
#define K_UPSAMPLE(RES) k_upsample_pool<RES>
#define K_UPSAMPLE_FAILED(RES) k_upsample_failed<RES>
#define K_VERIFY_LEFT(RES) k_verify_left<RES>
#define K_RESAMPLE_LEFT(RES) k_resample_left<RES>
#define K_SAMPLE(RES) k_sample_draft<RES>
#define K_SAMPLE_FAILED(RES) k_sample_failed<RES>
#define K_VERIFY(RES) k_verify_rows<false, RES>
#define K_ROUND(RES) k_verify_rows<true, RES>
#define K_ROUND_FAILED(RES) k_verify_failed<RES>
#define K_RESAMPLE(RES) k_resample_rows<RES>

// ---- the fast top-k path of mulo_round -------------------------------------------------

// inverse of the standard normal CDF by bisection (host, set-up only)
static double inv_norm_cdf(double p) {
  double lo = -12.0, hi = 12.0;
  for (int i = 0; i < 200; ++i) {
    const double mid = 0.5 * (lo + hi);
    if (0.5 * erfc(-mid / sqrt(2.0)) < p) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}

// Fills `s` and returns the dynamic shared memory the streaming kernel needs, or 0 if these
// parameters are not eligible (then the general kernel runs).
static size_t plan_stream(const mulo_ctx* ctx, const DevParams& d, StreamArgs* s) {
  if (d.top_k <= 0) return 0;
  // pooling keeps a bitmap of the pooled token ids in the row's selection scratch (2 KB)
  if (d.pool_k > 1 && d.V > 16384) return 0;
  const int V = d.V, k = d.top_k;
  if (V < 1024 || 1 + d.r * d.r > kMaxRowsPerParent) return 0;
  // candidates aimed for beyond k: about six standard deviations of the count of entries
  // above a fixed value near the k-th largest
  const int margin = (int)fmax(64.0, 6.0 * sqrt((double)k));
  const int margin_boot = margin + 3 * margin / 4;   // rows without a prediction: the pivot comes from one chunk's statistics
  if ((double)(k + margin_boot) > 0.5 * V) return 0;
  const int esz = d.bf16 ? 2 : 4;
  const int epl = 16 / esz, piece = 32 * epl;
  s->chunk = kChunkPieces * piece;
  s->n_chunks = (V + s->chunk - 1) / s->chunk;
  if (s->n_chunks > 255) return 0;
  s->n_seg = s->n_chunks * kSWarps;
  // capacity of a row's candidate array: the bootstrap density's mean plus six standard
  // deviations of a binomial(V, density) count, rounded up to a multiple of 64
  const double pb = (double)(k + margin_boot) / V;
  int cap = (int)ceil(V * pb + 6.0 * sqrt(V * pb * (1.0 - pb)));
  cap += s->n_seg;              // every segment's run is rounded up to an even length
  {   // a segment of the draft row may hold at most 255 candidates (8-bit offsets in its look-up table)
    const double seg_mean = (double)kPPW * piece * pb;
    if (seg_mean + 6.0 * sqrt(seg_mean * (1.0 - pb)) > 255.0) return 0;
  }
  cap = (cap + 63) / 64 * 64;
  if (cap > 65535) return 0;
  s->cap = cap;
  s->margin = margin;
  s->a_theta = (float)inv_norm_cdf(1.0 - (double)k / V);
  s->a_boot = (float)inv_norm_cdf(1.0 - (double)(k + margin_boot) / V);
  const size_t dyn = stream_layout(*s, esz);
  const size_t fixed = sizeof(StreamSmem) + 1024;
  if (dyn + fixed > (size_t)ctx->smem_optin) return 0;
  return dyn;
}

template <bool BF16, bool HAS_U, bool SAMPLE = false, bool POOL = false>
static bool launch_stream_t(mulo_ctx* ctx, const StreamArgs& s, size_t dyn, cudaStream_t st) {
  auto kern = k_round_stream<BF16, HAS_U, SAMPLE, POOL>;
  const int per_sm = ctas_per_sm(ctx, kern, kSThreads, dyn);
  if (per_sm < 1) return false;
  int grid = ctx->sm_count * per_sm;
  if (grid > s.n_parents) grid = s.n_parents;
  kern<<<grid, kSThreads, dyn, st>>>(s);
  return true;
}

static bool launch_stream(mulo_ctx* ctx, const StreamArgs& s, size_t dyn, cudaStream_t st) {
  const bool hu = s.uncond != nullptr;
  if (s.P.pool_k > 1) {
    if (s.P.bf16)
      return hu ? launch_stream_t<true, true, false, true>(ctx, s, dyn, st)
                : launch_stream_t<true, false, false, true>(ctx, s, dyn, st);
    return hu ? launch_stream_t<false, true, false, true>(ctx, s, dyn, st)
              : launch_stream_t<false, false, false, true>(ctx, s, dyn, st);
  }
  if (s.P.bf16) return hu ? launch_stream_t<true, true>(ctx, s, dyn, st) : launch_stream_t<true, false>(ctx, s, dyn, st);
  return hu ? launch_stream_t<false, true>(ctx, s, dyn, st) : launch_stream_t<false, false>(ctx, s, dyn, st);
}

// ---- rows with a top-k cut, NW warps per row (mulo_rows.cuh) ----------------------------

// Fills `s` and returns the dynamic shared memory of a CTA of nw warps, or 0 if these parameters are not eligible.
static size_t plan_rows_nw(const mulo_ctx* ctx, const DevParams& d, int kind, int nw, RowsArgs* s) {
  if (d.top_k <= 0) return 0;
  const int V = d.V, k = d.top_k;
  if (V < 1024) return 0;
  const int esz = d.bf16 ? 2 : 4, ids = 16 / esz;
  // Candidates aimed for beyond k: 3.5 standard deviations of the count of entries above a fixed value near the
  // k-th largest (a row that misses, about one in two thousand, is streamed again); more for rows without a
  // prediction.
  const double p = (double)k / V;
  const int margin = (int)fmax(48.0, 3.5 * sqrt(k * (1.0 - p)));
  const int margin_boot = margin + 3 * margin / 4;
  if ((double)(k + margin_boot) > 0.5 * V) return 0;
  s->row_bytes = (uint32_t)(V * esz);
  const int pieces = (int)((s->row_bytes + kRPieceBytes - 1) / kRPieceBytes);
  s->ppg = (pieces + 4 * nw - 1) / (4 * nw);
  s->n_words = (s->ppg + 3) / 4;
  // A list column holds the candidates of two threads: their share plus 3.6 standard deviations of that
  // binomial count (3 for a row without prediction); a thread's own at most 64.
  auto rows_for = [&](int count, double threads, double dev) {
    const double pc = (double)count / V, mu = threads * s->ppg * ids * pc;
    return mu + dev * sqrt(mu * (1.0 - pc));
  };
  if (rows_for(k + margin, 1.0, 4.5) > 64.0) return 0;
  s->R = (int)ceil(fmax(rows_for(k + margin, 2.0, 3.6), rows_for(k + margin_boot, 2.0, 3.0))) + 1 + kRSlack;
  if (s->R < 32) s->R = 32;
  s->margin = margin;
  const size_t dyn = rows_layout(*s, nw, d.bf16, kind);
  if (2 * (dyn + sizeof(RowsSmem<4, true>) + 1024) > (size_t)ctx->smem_optin) return 0;   // too few rows in flight per SM
  return dyn;
}

// Two warps per row where their lists hold the candidates (k / V up to about 0.13 here), else four.  Two is the faster one
// wherever both do: what every warp of a row repeats (bin search, ranking, decision) is a third of the instructions.
// 8192 rows of V = 16384, k / V = 0.02, 0.05, 0.1: 248, 255, 269 us with two, 273, 290, 302 with four.  Above, four against the
// chunked kernel (mulo_stream.cuh): 315 and 585 us at 0.15, 344 and 706 at 0.3.
// ... unless the lists of a two-warp CTA (fp32: those of the draft row are twice as long in bytes) leave room for fewer than
// seven of them per SM.  4608 rows, guidance, k = V / 8: V = 16384 fp32 (five) 279 us with two, 210 with four; 12288 fp32 (six)
// 6 to 22 % for four; 16384 bf16 (seven) 5 % for two, 8192 fp32 (eight) 10 % for two.
static size_t plan_rows(const mulo_ctx* ctx, const DevParams& d, int kind, RowsArgs* s, int* nw) {
  *nw = 2;
  size_t dyn = plan_rows_nw(ctx, d, kind, 2, s);
  if (!dyn || ((kind == kRowsRound || kind == kRowsResample) && 7 * (dyn + sizeof(RowsSmem<2, false>) + 1024) > (size_t)ctx->smem_optin + 1024)) {
    RowsArgs four = *s;
    if (const size_t dyn4 = plan_rows_nw(ctx, d, kind, 4, &four)) {
      *s = four;
      *nw = 4;
      dyn = dyn4;
    }
  }
  if (!dyn) return 0;
  const int k_boot = d.top_k + s->margin + 3 * s->margin / 4;
  s->a_theta = (float)inv_norm_cdf(1.0 - (double)d.top_k / d.V);
  s->a_boot = (float)inv_norm_cdf(1.0 - (double)k_boot / d.V);
  s->a_max = (float)inv_norm_cdf(1.0 - 0.5 / d.V);
  return dyn;
}

template <bool BF16, bool HAS_U, int KIND, bool POOL, bool PLAIN, int NW>
static bool launch_rows_p(mulo_ctx* ctx, const RowsArgs& s, size_t dyn, cudaStream_t st) {
  auto kern = k_round_rows<BF16, HAS_U, KIND, POOL, PLAIN, NW>;
  const int per_sm = ctas_per_sm(ctx, kern, NW * 32, dyn);
  if (per_sm < 1) return false;
  int grid = ctx->sm_count * per_sm;
  if (grid > s.n_units) grid = s.n_units;
  kern<<<grid, NW * 32, dyn, st>>>(s);
  return true;
}

template <bool BF16, bool HAS_U, int KIND, int NW>
static bool launch_rows_t(mulo_ctx* ctx, const RowsArgs& s, size_t dyn, cudaStream_t st) {
  const bool plain = s.P.invT == 1.0f && s.row_bytes % (16u * kRPieceBytes * NW) == 0;
  if constexpr (KIND == kRowsRound)
    if (s.P.pool_k > 1)
      return plain ? launch_rows_p<BF16, HAS_U, KIND, true, true, NW>(ctx, s, dyn, st)
                   : launch_rows_p<BF16, HAS_U, KIND, true, false, NW>(ctx, s, dyn, st);
  return plain ? launch_rows_p<BF16, HAS_U, KIND, false, true, NW>(ctx, s, dyn, st)
               : launch_rows_p<BF16, HAS_U, KIND, false, false, NW>(ctx, s, dyn, st);
}

template <int KIND, int NW>
static bool launch_rows_nw(mulo_ctx* ctx, const RowsArgs& s, size_t dyn, cudaStream_t st) {
  if constexpr (KIND == kRowsRound || KIND == kRowsVerify || KIND == kRowsResample)
    if (s.uncond) return s.P.bf16 ? launch_rows_t<true, true, KIND, NW>(ctx, s, dyn, st) : launch_rows_t<false, true, KIND, NW>(ctx, s, dyn, st);
  return s.P.bf16 ? launch_rows_t<true, false, KIND, NW>(ctx, s, dyn, st) : launch_rows_t<false, false, KIND, NW>(ctx, s, dyn, st);
}

template <int KIND>
static bool launch_rows(mulo_ctx* ctx, const RowsArgs& s, int nw, size_t dyn, cudaStream_t st) {
  return nw == 2 ? launch_rows_nw<KIND, 2>(ctx, s, dyn, st) : launch_rows_nw<KIND, 4>(ctx, s, dyn, st);
}

// ---- rows without a top-k cut (mulo_full.cuh, mulo_flat.cuh) ------------------------------
static bool round_needs_q(const DevParams& d) {
  return !(d.accept_mode == MULO_ACCEPT_THRESHOLD && d.resample_mode == MULO_RESAMPLE_TARGET_ALL);
}

// Pooled rows without residual redraws, V = 256 W with W a multiple of the ids in 16 bytes, and the rows of one position
// (draft row if q is needed, conditional, unconditional) within a CTA's shared memory.  (64 x 64, 16 images, lists of 1000:
// 1240 us here, 1280 on mulo_flat.cuh's kernel; with residual redraws, 4 images, it is 566 to 388 the other way round.)
static size_t plan_full(const mulo_ctx* ctx, const DevParams& d, bool has_u, FullArgs* s) {
  if (d.top_k > 0 && d.top_k < d.V) return 0;
  if (d.pool_k <= 1 || d.resample_mode != MULO_RESAMPLE_TARGET_ALL) return 0;
  const int esz = d.bf16 ? 2 : 4, n = 16 / esz;
  if (d.V % (kFThreads * n) != 0) return 0;
  const int need_q = round_needs_q(d) ? 1 : 0;
  const size_t rows = (size_t)need_q + 1 + (has_u ? 1 : 0);
  const size_t dyn = rows * (size_t)d.V * esz + (size_t)d.V / 8 + (size_t)kFThreads * 8;
  if (dyn + sizeof(FullSmem) + 1024 > (size_t)ctx->smem_optin) return 0;
  s->W = d.V / kFThreads;
  s->need_q = need_q;
  return dyn;
}

template <bool BF16, bool HAS_U>
static bool launch_full_t(mulo_ctx* ctx, const FullArgs& s, size_t dyn, cudaStream_t st) {
  auto kern = k_round_full<BF16, HAS_U>;
  const int per_sm = ctas_per_sm(ctx, kern, kFThreads, dyn);
  if (per_sm < 1) return false;
  int grid = ctx->sm_count * per_sm;
  if (grid > s.n_units) grid = s.n_units;
  kern<<<grid, kFThreads, dyn, st>>>(s);
  return true;
}

static bool launch_full(mulo_ctx* ctx, const FullArgs& s, size_t dyn, cudaStream_t st) {
  const bool hu = s.uncond != nullptr;
  if (s.P.bf16) return hu ? launch_full_t<true, true>(ctx, s, dyn, st) : launch_full_t<true, false>(ctx, s, dyn, st);
  return hu ? launch_full_t<false, true>(ctx, s, dyn, st) : launch_full_t<false, false>(ctx, s, dyn, st);
}


// Fills `s` and returns the dynamic shared memory of a CTA, or 0 if these parameters are not eligible.
static size_t plan_flat(const mulo_ctx* ctx, const DevParams& d, bool sample, FlatArgs* s, bool* res) {
  if (d.top_k > 0 && d.top_k < d.V) return 0;
  if (!sample && d.r > kFlatMaxRatio) return 0;
  *res = !sample && (d.pool_k > 1 || d.resample_mode != MULO_RESAMPLE_TARGET_ALL);   // a row is needed a second time
  const int nw = *res ? kFlatResWarps : kFlatWarps;
  s->P = d;
  s->row_bytes = (uint32_t)(d.V * (d.bf16 ? 2 : 4));
  const int pieces = (int)((s->row_bytes + kRPieceBytes - 1) / kRPieceBytes);
  s->ppg = (pieces + 4 * nw - 1) / (4 * nw);
  s->n_words = (s->ppg + 3) / 4;
  s->need_q = !sample && round_needs_q(d) ? 1 : 0;
  const size_t dyn = flat_smem(*s, nw, *res);
  if (dyn + sizeof(FlatSmem<kFlatResWarps>) + 1024 > (size_t)ctx->smem_optin) return 0;
  return dyn;
}

template <bool BF16, bool HAS_U, bool SAMPLE, bool POOL, bool RES>
static bool launch_flat_p(mulo_ctx* ctx, const FlatArgs& s, size_t dyn, cudaStream_t st) {
  constexpr int nw = RES ? kFlatResWarps : kFlatWarps;
  const bool even = s.row_bytes % (16u * kRPieceBytes * nw) == 0;
  auto kern = !even ? k_round_flat<BF16, HAS_U, SAMPLE, POOL, RES, false, true>
              : s.P.invT != 1.0f ? k_round_flat<BF16, HAS_U, SAMPLE, POOL, RES, true, true>
                                 : k_round_flat<BF16, HAS_U, SAMPLE, POOL, RES, true, false>;
  const int per_sm = ctas_per_sm(ctx, kern, nw * 32, dyn);
  if (per_sm < 1) return false;
  int grid = ctx->sm_count * per_sm;
  if (grid > s.n_units) grid = s.n_units;
  kern<<<grid, nw * 32, dyn, st>>>(s);
  return true;
}

template <bool BF16, bool HAS_U, bool SAMPLE>
static bool launch_flat_t(mulo_ctx* ctx, const FlatArgs& s, bool res, size_t dyn, cudaStream_t st) {
  if constexpr (!SAMPLE) {
    if (s.P.pool_k > 1) return launch_flat_p<BF16, HAS_U, false, true, true>(ctx, s, dyn, st);
    if (res) return launch_flat_p<BF16, HAS_U, false, false, true>(ctx, s, dyn, st);
  }
  return launch_flat_p<BF16, HAS_U, SAMPLE, false, false>(ctx, s, dyn, st);
}

static bool launch_flat(mulo_ctx* ctx, const FlatArgs& s, bool sample, bool res, size_t dyn, cudaStream_t st) {
  const bool hu = s.uncond != nullptr;
  if (sample)
    return s.P.bf16 ? launch_flat_t<true, false, true>(ctx, s, res, dyn, st) : launch_flat_t<false, false, true>(ctx, s, res, dyn, st);
  if (s.P.bf16)
    return hu ? launch_flat_t<true, true, false>(ctx, s, res, dyn, st) : launch_flat_t<true, false, false>(ctx, s, res, dyn, st);
  return hu ? launch_flat_t<false, true, false>(ctx, s, res, dyn, st) : launch_flat_t<false, false, false>(ctx, s, res, dyn, st);
}

// Are there enough rows with a cut for the stages to stream them (two warps each) instead of keeping each in one CTA's shared
// memory?  That CTA is the sooner done with a row.  us streamed / kept: draft rows, 1024 of 16384 ids: 31 / 45, of 4096: 34 / 25, 576 of 16384:
// 28 / 28; verified, 784 rows of 16384: 38 / 43, of 4096: 37 / 29, of 8192 fp32: 39 / 36, 1296 rows: 44 / 68, 39 / 41, 38 / 54.
// How many positions are redrawn is not known here, and few of them are sooner done by a CTA each: all of the grid / 30 / 10 / 3 %
// of it, 2500 positions of 16384 ids: 128 / 173, 60 / 72, 48 / 43, 46 / 35, of 4096: 69 / 96, 36 / 43, 34 / 31, 34 / 25, of 8192 fp32: 101 / 129,
// 50 / 55, 44 / 36, 38 / 29; 1296 of 16384: 81 / 100, 48 / 47, 46 / 31, 40 / 29.  So the line lies where 10 % are nearly as quick either way.
static bool many_rows(const mulo_ctx* ctx, int kind, int V, long long rows) {
  const int per_sm = kind == kRowsResample ? 16 : kind == kRowsStats ? (V > 4096 ? 4 : 16) : V >= 12288 ? 4 : 8;
  return !ctx->force_dense && rows > (long long)per_sm * ctx->sm_count;
}

static size_t mask_smem(const mulo_params* p) { return (size_t)3 * p->H * ((p->W + 31) / 32) * 4; }

// Everything mulo_round can refuse without touching the device.
static mulo_status check_round_args(const mulo_ctx* ctx, const mulo_params* p, const void* tgt_cond,
                                    const void* tgt_uncond, const void* draft_logits_lo, const int32_t* draft_tok_lo,
                                    const uint16_t* nn, const int32_t* out_tok, const uint32_t* reject_bits,
                                    const uint32_t* expand_bits) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!tgt_cond || !draft_logits_lo || !draft_tok_lo || !out_tok || !reject_bits || !expand_bits)
    return MULO_ERR_INVALID_ARG;
  if (p->pool_k > 1 && !nn) return MULO_ERR_INVALID_ARG;
  if (!aligned16(tgt_cond) || !aligned16(tgt_uncond) || !aligned16(draft_logits_lo)) return MULO_ERR_INVALID_ARG;
  return on_context_device(ctx);
}

extern "C" {

mulo_status mulo_upsample_pool(mulo_ctx* ctx, const mulo_params* p, const void* draft_logits_lo,
                               const int32_t* draft_tok_lo, const uint16_t* nn, int32_t* draft_tok_hi,
                               float* draft_stats_lo, float* q_tok_hi, void* stream) {
  (void)nn;
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!draft_logits_lo || !draft_tok_lo || !draft_tok_hi || !draft_stats_lo || !q_tok_hi) return MULO_ERR_INVALID_ARG;
  if (!aligned16(draft_logits_lo)) return MULO_ERR_INVALID_ARG;
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  RowKernelArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.draft = (const char*)draft_logits_lo;
  a.draft_tok_lo = draft_tok_lo;
  a.tok_hi_out = draft_tok_hi;
  a.stats_out = draft_stats_lo;
  a.q_tok_hi_out = q_tok_hi;
  a.dev_status = (uint32_t*)ctx->ws;
  // Without a cut there is nothing to search: many rows (more than four per SM) are read twice from L1 / L2 by four thread
  // blocks per SM instead of kept in shared memory by two -- 4096 rows of 1024, 4096, 16392, 49152 bf16 ids: 26, 34, 81, 206 us,
  // 38, 47, 106, 346 us resident; fp32 up to 8192 ids likewise (56, 71 us), above it the row no longer stays in L1 (16384 ids:
  // 148, 106 us).  64 rows: 14 to 17 us, 9 to 14 us resident.
  const int cells = p->B * a.P.h * a.P.w;
  const cudaStream_t st = (cudaStream_t)stream;
  // With one, many rows are streamed.
  RowsArgs ra;
  memset(&ra, 0, sizeof ra);
  int rnw = 0;
  const bool many = many_rows(ctx, kRowsStats, a.P.V, cells) && ((uintptr_t)draft_stats_lo & 15u) == 0;
  if (const size_t rdyn = many ? plan_rows(ctx, a.P, kRowsStats, &ra, &rnw) : 0) {
    ra.P = a.P;
    ra.cond = a.draft;
    ra.tok_of = draft_tok_lo;
    ra.stats_out = draft_stats_lo;
    ra.tok_hi_out = draft_tok_hi;
    ra.q_hi_out = q_tok_hi;
    ra.dev_status = a.dev_status;
    ra.n_units = cells;
    if (launch_rows<kRowsStats>(ctx, ra, rnw, rdyn, st)) {
      if (!MULO_LAUNCH_LEFT(K_UPSAMPLE_FAILED, general_smem(a.P, false), st, a)) return MULO_ERR_CUDA;
      return launched(ctx, 2);
    }
  }
  if (a.P.top_k == 0 && cells > 4 * ctx->sm_count && (a.P.bf16 || a.P.V <= 8192)) {
    if (!launch_general(ctx, K_UPSAMPLE(false), (unsigned)cells, 0, st, a)) return MULO_ERR_CUDA;
    return launched(ctx, 1);
  }
  if (!MULO_LAUNCH_GENERAL(K_UPSAMPLE, cells, general_smem(a.P, false), st, a)) return MULO_ERR_CUDA;
  return launched(ctx, 1);
}

mulo_status mulo_island_schedule(mulo_ctx* ctx, const mulo_params* p, const int32_t* labels, int32_t window,
                                 int32_t* step, int32_t* n_steps, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!labels || !step || !n_steps || window < 1) return MULO_ERR_INVALID_ARG;
  if ((size_t)p->H * p->W > (size_t)kIslandMaxCells) return MULO_ERR_UNSUPPORTED;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  ScheduleArgs a;
  a.H = p->H; a.W = p->W; a.window = window > p->W ? p->W : window;
  a.labels = labels; a.step = step; a.n_steps = n_steps;
  const auto kernel = p->W <= 32 ? k_island_schedule<1> : p->W <= 64 ? k_island_schedule<2> : k_island_schedule<4>;
  const size_t smem = schedule_smem(p->H, p->W);
  if (ctas_per_sm(ctx, kernel, kScheduleThreads, smem) < 1) return MULO_ERR_UNSUPPORTED;
  if (!launch_after(kernel, (unsigned)p->B, kScheduleThreads, smem, (cudaStream_t)stream, a)) return MULO_ERR_CUDA;
  return launched(ctx, 1);
}

mulo_status mulo_redraw_plan(mulo_ctx* ctx, const mulo_params* p, const int32_t* step, int32_t max_step,
                             int32_t* pos_list, int32_t* step_offsets, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!step || !pos_list || !step_offsets || max_step < 1) return MULO_ERR_INVALID_ARG;
  if ((size_t)max_step > (size_t)p->H * p->W) return MULO_ERR_INVALID_ARG;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const int n = p->B * p->H * p->W;
  int32_t* cursor = step_offsets + max_step + 2;
  if (cudaMemsetAsync(step_offsets, 0, sizeof(int32_t) * 2 * ((size_t)max_step + 2), st) != cudaSuccess) return MULO_ERR_CUDA;
  if (n == 0) return MULO_OK;
  const int blocks = (n + 255) / 256 < 4 * ctx->sm_count ? (n + 255) / 256 : 4 * ctx->sm_count;
  k_redraw_count<<<blocks, 256, 0, st>>>(step, n, max_step, cursor);
  if (!launch_after(k_redraw_scan, 1u, kScanThreads, 0, st, max_step, step_offsets, cursor) ||
      !launch_after(k_redraw_fill, (unsigned)blocks, 256, 0, st, step, n, max_step, cursor, pos_list))
    return MULO_ERR_CUDA;
  return launched(ctx, 3);
}

mulo_status mulo_redraw_step(mulo_ctx* ctx, const mulo_params* p, int32_t s_index, int32_t max_step,
                             const int32_t* pos_list, const int32_t* step_offsets, const void* tgt_cond,
                             const void* tgt_uncond, int32_t* out_tok, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!pos_list || !step_offsets || !tgt_cond || !out_tok || !aligned16(tgt_cond) || !aligned16(tgt_uncond))
    return MULO_ERR_INVALID_ARG;
  if (s_index < 1 || s_index > max_step) return MULO_ERR_INVALID_ARG;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  RedrawArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.cond = (const char*)tgt_cond;
  a.uncond = (const char*)tgt_uncond;
  a.pos_list = pos_list;
  a.offsets = step_offsets;
  a.out_tok = out_tok;
  a.s = s_index;
  const int np = a.P.V <= 4 * kRedrawIds ? 1 : a.P.V <= 8 * kRedrawIds ? 2 : 4, ctas = (a.P.V + np * kRedrawIds - 1) / (np * kRedrawIds);
  // Eight ids per thread as long as four CTAs hold the row: a row's chain is the shorter the fewer ids a thread has.  64 x 64, 4 images,
  // V = 16384, window 16, an ordinary kernel (1.3 us) between any two steps: 12.9 us a step with four CTAs, 15.6 with two, 19.6 with
  // one; V = 8192: 11.9 with two, 13.6 with one; V = 32768: 17.1 with four, 22.2 with two.
  // The step's positions are counted on the device: a fixed number of clusters strides over them, 128 CTAs' worth, and as many as a
  // schedule of window 8 has positions at a time (W / 8 per image) if that is more.  No more: what is left of the chip draws the
  // next steps' rows meanwhile.  64 x 64, 4 images, V = 16384, window 16 (15 positions): 4.7 us a step with 32 clusters of four, 7.5 with 64 (as
  // a graph; the host's calls take 4.9).
  // A step of more positions than clusters (small windows; the first steps of sparse islands; any plan of the caller's) is shared out
  // to single CTAs, each with a whole row in shared memory.  us a step, clusters only / so / the resident kernel with 296 CTAs that
  // this one replaced: window 4 (64 positions) 14.7 / 12.4 / 9.0, window 1 (up to 256) 39 / 19 / 13, sparse islands at 2 % rejections
  // (202 positions at first, 40 on average) 13 / 8.5 / 9.9, 4096 positions of one image at once 1050 / 312 / 227; V = 4096, window 1: 24 / 6.3 /
  // 9.5.  Where two whole rows do not fit an SM (V > 24576) the clusters stride: room for a single row per SM would leave none
  // for the next steps.
  const int room = ctx->sm_count * (np == 4 ? 1 : 2) / ctas;
  const long long likely = (long long)p->B * (p->W > 8 ? p->W / 8 : 1), base = 128 / ctas, wanted = likely > base ? likely : base;
  const int clusters = wanted < room ? (int)wanted : room;
  size_t dyn = (size_t)ctas * kRedrawWords * sizeof(uint32_t);
  a.single = ctas > 1 && np < 4 && 2 * (resident_bytes(a.P.V) + sizeof(RedrawSmem) + sizeof(ResScratch) + 1024) <= (size_t)ctx->smem_optin;
  if (a.single) dyn = resident_bytes(a.P.V) > dyn ? resident_bytes(a.P.V) : dyn;
  auto kern = a.P.bf16 ? (np == 1 ? k_redraw_step<true, 1> : np == 2 ? k_redraw_step<true, 2> : k_redraw_step<true, 4>)
                       : (np == 1 ? k_redraw_step<false, 1> : np == 2 ? k_redraw_step<false, 2> : k_redraw_step<false, 4>);
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3((unsigned)(clusters * ctas));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)ctas;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (clusters < 1 || ctas_per_sm(ctx, kern, kThreads, cfg.dynamicSmemBytes) < 1) return MULO_ERR_CUDA;
  if (cudaLaunchKernelEx(&cfg, kern, a) != cudaSuccess) {
    cudaGetLastError();
    return MULO_ERR_CUDA;
  }
  return launched(ctx, 1);
}

mulo_status mulo_sample_draft(mulo_ctx* ctx, const mulo_params* p, const void* draft_logits_lo,
                              int32_t* draft_tok_lo, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!draft_logits_lo || !draft_tok_lo || !aligned16(draft_logits_lo)) return MULO_ERR_INVALID_ARG;
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  RowKernelArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.draft = (const char*)draft_logits_lo;
  a.out_tok = draft_tok_lo;
  a.dev_status = (uint32_t*)ctx->ws;
  // fast paths: without a top-k cut one kernel does it; with one, a workspace large enough for the list of cells
  // that the kernel may leave to the general routines
  FlatArgs fa;
  memset(&fa, 0, sizeof fa);
  bool fres = false;
  const size_t fdyn = ctx->force_dense ? 0 : plan_flat(ctx, a.P, true, &fa, &fres);
  if (fdyn) {
    fa.cond = a.draft;
    fa.sample_out = draft_tok_lo;
    fa.dev_status = a.dev_status;
    fa.n_units = p->B * a.P.h * a.P.w;
    if (launch_flat(ctx, fa, true, fres, fdyn, st)) return launched(ctx, 1);
  }
  // With one, few rows go to the chunked kernel, whose eight warps bring a row through sooner: up to four per SM for 4096 ids
  // (64, 576, 1024 cells with k = V / 8: 24, 25, 35 us there, 28, 28, 31 us with two warps per row), three for 8192, two for more
  // (16384 ids, 256, 400, 576 cells: 31, 38, 59 us, 39, 42, 43 us); above 16384 ids only short lists, k up to V / 25 (32768 ids,
  // 64 cells, k = V / 8: 50 us there, 15 us).
  Workspace w;
  const bool listed = !ctx->force_dense && check_ws(ctx, p, &w) == MULO_OK;   // (there is room for the list)
  StreamArgs sa;
  memset(&sa, 0, sizeof sa);
  const int V = a.P.V, per_sm = V <= 4096 ? 4 : V <= 8192 ? 3 : 2;
  const bool few = p->B * a.P.h * a.P.w <= per_sm * ctx->sm_count && (V <= 16384 || a.P.top_k <= V / 25);
  size_t sdyn = listed && few ? plan_stream(ctx, a.P, &sa) : 0;
  RowsArgs ra;
  memset(&ra, 0, sizeof ra);
  int rnw = 0;
  const size_t rdyn = listed && !sdyn ? plan_rows(ctx, a.P, kRowsSample, &ra, &rnw) : 0;
  if (rdyn) {
    ra.P = a.P;
    ra.cond = a.draft;
    ra.sample_out = draft_tok_lo;
    ra.dev_status = w.status;
    ra.fail_list = w.fail_list;
    ra.n_units = p->B * a.P.h * a.P.w;
    if (cudaMemsetAsync(w.status + kFailCount, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
    if (launch_rows<kRowsSample>(ctx, ra, rnw, rdyn, st)) {
      if (!MULO_LAUNCH_LEFT(K_SAMPLE_FAILED, general_smem(a.P, false), st, a, w.fail_list, w.status + kFailCount)) return MULO_ERR_CUDA;
      return launched(ctx, 2);
    }
  }
  if (listed && !sdyn) sdyn = plan_stream(ctx, a.P, &sa);
  if (sdyn) {
    sa.P = a.P;
    sa.draft = a.draft;
    sa.sample_out = draft_tok_lo;
    sa.dev_status = w.status;
    sa.fail_list = w.fail_list;
    sa.n_parents = p->B * a.P.h * a.P.w;
    if (cudaMemsetAsync(w.status + kFailCount, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
    const bool fast = a.P.bf16 ? launch_stream_t<true, false, true>(ctx, sa, sdyn, st)
                               : launch_stream_t<false, false, true>(ctx, sa, sdyn, st);
    if (fast) {
      if (!MULO_LAUNCH_LEFT(K_SAMPLE_FAILED, general_smem(a.P, false), st, a, w.fail_list, w.status + kFailCount)) return MULO_ERR_CUDA;
      return launched(ctx, 2);
    }
  }
  if (!MULO_LAUNCH_GENERAL(K_SAMPLE, p->B * a.P.h * a.P.w, general_smem(a.P, false), st, a)) return MULO_ERR_CUDA;
  return launched(ctx, 1);
}

mulo_status mulo_downsample(mulo_ctx* ctx, const mulo_params* p, const int32_t* tok_hi, int32_t* tok_lo,
                            void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!tok_hi || !tok_lo) return MULO_ERR_INVALID_ARG;
  if (p->r > 16) return MULO_ERR_UNSUPPORTED;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  const int h = p->H / p->r, w = p->W / p->r, cells = p->B * h * w;
  if (!launch_after(k_downsample, (unsigned)((cells + 255) / 256), 256, 0, (cudaStream_t)stream, tok_hi, tok_lo, cells, h, w, p->W, p->r))
    return MULO_ERR_CUDA;
  return launched(ctx, 1);
}

mulo_status mulo_verify(mulo_ctx* ctx, const mulo_params* p, const void* tgt_cond, const void* tgt_uncond,
                        const void* draft_logits_lo, const float* draft_stats_lo,
                        const int32_t* draft_tok_hi, const uint16_t* nn, float* p_tok, float* q_tok,
                        float* accept_prob, uint32_t* reject_bits, int32_t* n_reject,
                        int32_t* first_reject, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!tgt_cond || !draft_logits_lo || !draft_stats_lo || !draft_tok_hi || !p_tok || !q_tok || !accept_prob ||
      !reject_bits || !n_reject || !first_reject)
    return MULO_ERR_INVALID_ARG;
  if (p->pool_k > 1 && !nn) return MULO_ERR_INVALID_ARG;
  if (!aligned16(tgt_cond) || !aligned16(tgt_uncond) || !aligned16(draft_logits_lo)) return MULO_ERR_INVALID_ARG;
  Workspace w;
  if ((s = check_ws(ctx, p, &w)) != MULO_OK) return s;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  RowKernelArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.cond = (const char*)tgt_cond;
  a.uncond = (const char*)tgt_uncond;
  a.draft = (const char*)draft_logits_lo;
  a.stats_in = draft_stats_lo;
  a.draft_tok_hi = draft_tok_hi;
  a.nn = nn;
  a.p_tok = p_tok; a.q_tok = q_tok; a.accept_prob = accept_prob;
  a.flags = w.flags;
  a.dev_status = w.status;
  const size_t dyn = general_smem(a.P, true);
  cudaStream_t st = (cudaStream_t)stream;
  // Many rows with a cut and without pooling are streamed.
  bool fast = false;
  RowsArgs ra;
  memset(&ra, 0, sizeof ra);
  int rnw = 0;
  const long long rows = (long long)p->B * p->H * p->W;
  const bool many = a.P.pool_k <= 1 && many_rows(ctx, kRowsVerify, a.P.V, rows);
  if (const size_t rdyn = many ? plan_rows(ctx, a.P, kRowsVerify, &ra, &rnw) : 0) {
    ra.P = a.P;
    ra.cond = a.cond; ra.uncond = a.uncond; ra.draft = a.draft;
    ra.tok_of = draft_tok_hi;
    ra.stats_in = draft_stats_lo;
    ra.p_tok = p_tok; ra.q_tok = q_tok; ra.accept_prob = accept_prob;
    ra.flags = w.flags;
    ra.dev_status = w.status;
    ra.fail_list = w.fail_list;
    ra.n_units = (int)rows;
    if (cudaMemsetAsync(w.status + kFailCount, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
    fast = launch_rows<kRowsVerify>(ctx, ra, rnw, rdyn, st);
    if (fast && !MULO_LAUNCH_LEFT(K_VERIFY_LEFT, dyn, st, a, w.fail_list, w.status + kFailCount)) return MULO_ERR_CUDA;
  }
  if (!fast && !MULO_LAUNCH_GENERAL(K_VERIFY, rows, dyn, st, a)) return MULO_ERR_UNSUPPORTED;
  MaskArgs m;
  memset(&m, 0, sizeof m);
  m.H = p->H; m.W = p->W; m.r = p->r; m.radius = p->radius; m.clip = a.P.clip; m.resample_mode = p->resample_mode;
  m.flags = w.flags;
  m.reject_bits = reject_bits; m.n_reject = n_reject; m.first_reject = first_reject;
  if (!launch_after(k_mask<0>, (unsigned)p->B, kMaskThreads, mask_smem(p), st, m)) return MULO_ERR_CUDA;
  return launched(ctx, fast ? 3 : 2);
}

mulo_status mulo_local_reject_expand(mulo_ctx* ctx, const mulo_params* p, const uint32_t* reject_bits,
                                     const int32_t* first_reject, uint32_t* expand_bits,
                                     int32_t* n_expand, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!reject_bits || !first_reject || !expand_bits || !n_expand) return MULO_ERR_INVALID_ARG;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  MaskArgs m;
  memset(&m, 0, sizeof m);
  m.H = p->H; m.W = p->W; m.r = p->r; m.radius = p->radius; m.clip = p->clip_before_first != 0;
  m.resample_mode = p->resample_mode;
  m.reject_in = reject_bits; m.first_in = first_reject;
  m.expand_bits = expand_bits; m.n_expand = n_expand;
  k_mask<1><<<p->B, kMaskThreads, mask_smem(p), (cudaStream_t)stream>>>(m);
  return launched(ctx, 1);
}

mulo_status mulo_islands(mulo_ctx* ctx, const mulo_params* p, const uint32_t* expand_bits, int32_t* labels,
                         int32_t* n_islands, int32_t max_islands, int32_t* island_rows,
                         int32_t* island_size, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!expand_bits || !labels || !n_islands || max_islands < 0) return MULO_ERR_INVALID_ARG;
  if ((size_t)p->H * p->W > (size_t)kIslandMaxCells) return MULO_ERR_UNSUPPORTED;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  IslandArgs a;
  a.H = p->H; a.W = p->W; a.max_islands = max_islands;
  a.bits = expand_bits; a.labels = labels; a.n_islands = n_islands;
  a.rows = max_islands > 0 ? island_rows : nullptr;
  a.size = max_islands > 0 ? island_size : nullptr;
  const size_t smem = ((size_t)2 * p->H * p->W + (size_t)p->H * ((p->W + 31) / 32)) * sizeof(int);
  if (ctas_per_sm(ctx, k_islands, kIslandThreads, smem) < 1) return MULO_ERR_UNSUPPORTED;
  if (!launch_after(k_islands, (unsigned)p->B, kIslandThreads, smem, (cudaStream_t)stream, a)) return MULO_ERR_CUDA;
  return launched(ctx, 1);
}

mulo_status mulo_resample(mulo_ctx* ctx, const mulo_params* p, const void* tgt_cond, const void* tgt_uncond,
                          const void* draft_logits_lo, const float* draft_stats_lo,
                          const int32_t* draft_tok_hi, const uint16_t* nn, const uint32_t* reject_bits,
                          const uint32_t* expand_bits, int32_t* out_tok, void* stream) {
  if (!ctx) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!tgt_cond || !draft_logits_lo || !draft_stats_lo || !draft_tok_hi || !reject_bits || !expand_bits || !out_tok)
    return MULO_ERR_INVALID_ARG;
  if (p->pool_k > 1 && !nn) return MULO_ERR_INVALID_ARG;
  if (!aligned16(tgt_cond) || !aligned16(tgt_uncond) || !aligned16(draft_logits_lo)) return MULO_ERR_INVALID_ARG;
  if (!ctx->ws) return MULO_ERR_WORKSPACE;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  RowKernelArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.cond = (const char*)tgt_cond;
  a.uncond = (const char*)tgt_uncond;
  a.draft = (const char*)draft_logits_lo;
  a.stats_in = draft_stats_lo;
  a.draft_tok_hi = draft_tok_hi;
  a.nn = nn;
  a.reject_bits = reject_bits;
  a.expand_bits = expand_bits;
  a.out_tok = out_tok;
  a.dev_status = (uint32_t*)ctx->ws;
  const cudaStream_t st = (cudaStream_t)stream;
  const size_t dyn = general_smem(a.P, true);
  const long long rows = (long long)p->B * p->H * p->W;
  // Many rows with a cut and without pooling are streamed.  (Whether a rejection is isolated depends on its neighbours, which the
  // general kernel looks up.)
  RowsArgs ra;
  memset(&ra, 0, sizeof ra);
  int rnw = 0;
  const bool many = a.P.pool_k <= 1 && many_rows(ctx, kRowsResample, a.P.V, rows) && (size_t)p->H * p->W <= (size_t)kPickIndex &&
                    p->resample_mode != MULO_RESAMPLE_ISOLATED_RESIDUAL;
  if (const size_t rdyn = many ? plan_rows(ctx, a.P, kRowsResample, &ra, &rnw) : 0) {
    ra.P = a.P;
    ra.cond = a.cond; ra.uncond = a.uncond; ra.draft = a.draft;
    ra.tok_of = draft_tok_hi;
    ra.stats_in = draft_stats_lo;
    ra.reject_bits = reject_bits;
    ra.expand_bits = expand_bits;
    ra.sample_out = out_tok;
    ra.dev_status = a.dev_status;
    ra.n_units = (int)rows;   // (at most)
    if (launch_rows<kRowsResample>(ctx, ra, rnw, rdyn, st)) {
      if (!MULO_LAUNCH_LEFT(K_RESAMPLE_LEFT, dyn, st, a)) return MULO_ERR_CUDA;
      return launched(ctx, 2);
    }
  }
  if (!MULO_LAUNCH_GENERAL(K_RESAMPLE, rows, dyn, st, a)) return MULO_ERR_UNSUPPORTED;
  return launched(ctx, 1);
}

mulo_status mulo_round(mulo_ctx* ctx, const mulo_params* p, const void* tgt_cond, const void* tgt_uncond,
                       const void* draft_logits_lo, const int32_t* draft_tok_lo, const uint16_t* nn,
                       int32_t* out_tok, uint32_t* reject_bits, uint32_t* expand_bits, float* p_tok,
                       float* q_tok, float* accept_prob, int32_t* n_reject, int32_t* n_expand,
                       int32_t* first_reject, void* stream) {
  mulo_status s = check_round_args(ctx, p, tgt_cond, tgt_uncond, draft_logits_lo, draft_tok_lo, nn, out_tok,
                                   reject_bits, expand_bits);
  if (s != MULO_OK) return s;
  Workspace w;
  if ((s = check_ws(ctx, p, &w)) != MULO_OK) return s;
  if (p->B == 0) return MULO_OK;
  RowKernelArgs a;
  memset(&a, 0, sizeof a);
  a.P = to_dev(p);
  a.cond = (const char*)tgt_cond;
  a.uncond = (const char*)tgt_uncond;
  a.draft = (const char*)draft_logits_lo;
  a.draft_tok_lo = draft_tok_lo;
  a.nn = nn;
  a.p_tok = p_tok; a.q_tok = q_tok; a.accept_prob = accept_prob;
  a.flags = w.flags; a.cand_res = w.cand_res; a.cand_tgt = w.cand_tgt;
  a.dev_status = w.status;
  const size_t dyn = general_smem(a.P, true);
  cudaStream_t st = (cudaStream_t)stream;
  const bool timed = ctx->ev_used + 2 <= ctx->ev.size();
  if (timed) cudaEventRecord(ctx->ev[ctx->ev_used], st);
  bool fast = false;
  int fast_launches = 2;   // a fast kernel and the one that redoes the rows it left
  // Eq. 5 with every redraw from the target distribution never looks at q: no kernel reports it
  // (the kernels of rows without a cut do not even read the draft logits), the output is zero-filled
  if (!round_needs_q(a.P) && q_tok) {
    if (cudaMemsetAsync(q_tok, 0, sizeof(float) * (size_t)p->B * p->H * p->W, st) != cudaSuccess) return MULO_ERR_CUDA;
    a.q_tok = nullptr;
    q_tok = nullptr;
  }
  FullArgs ua;
  memset(&ua, 0, sizeof ua);
  const size_t udyn = ctx->force_dense ? 0 : plan_full(ctx, a.P, tgt_uncond != nullptr, &ua);
  if (udyn) {
    ua.P = a.P;
    ua.cond = a.cond; ua.uncond = a.uncond; ua.draft = a.draft; ua.draft_tok_lo = draft_tok_lo;
    ua.nn = a.nn;
    ua.p_tok = p_tok; ua.q_tok = q_tok; ua.accept_prob = accept_prob;
    ua.flags = w.flags; ua.cand_tgt = w.cand_tgt;
    ua.dev_status = w.status;
    ua.n_units = p->B * p->H * p->W;
    fast = launch_full(ctx, ua, udyn, st);
    if (fast) fast_launches = 1;
  }
  FlatArgs fa;
  memset(&fa, 0, sizeof fa);
  bool fres = false;
  const size_t fdyn = (ctx->force_dense || fast) ? 0 : plan_flat(ctx, a.P, false, &fa, &fres);
  if (fdyn) {
    fa.cond = a.cond; fa.uncond = a.uncond; fa.draft = a.draft; fa.draft_tok_lo = draft_tok_lo;
    fa.nn = a.nn;
    fa.p_tok = p_tok; fa.q_tok = q_tok; fa.accept_prob = accept_prob;
    fa.flags = w.flags; fa.cand_res = w.cand_res; fa.cand_tgt = w.cand_tgt;
    fa.dev_status = w.status;
    fa.n_units = p->B * p->H * p->W;
    fast = launch_flat(ctx, fa, false, fres, fdyn, st);
    if (fast) fast_launches = 1;
  }
  RowsArgs ra;
  memset(&ra, 0, sizeof ra);
  int rnw = 0;
  const size_t rdyn = (ctx->force_dense || fast) ? 0 : plan_rows(ctx, a.P, kRowsRound, &ra, &rnw);
  if (rdyn) {
    ra.P = a.P;
    ra.cond = a.cond; ra.uncond = a.uncond; ra.draft = a.draft; ra.draft_tok_lo = draft_tok_lo;
    ra.nn = a.nn;
    ra.p_tok = p_tok; ra.q_tok = q_tok; ra.accept_prob = accept_prob;
    ra.flags = w.flags; ra.cand_res = w.cand_res; ra.cand_tgt = w.cand_tgt;
    ra.dev_status = w.status;
    ra.fail_list = w.fail_list;
    ra.n_units = p->B * p->H * p->W;
    if (cudaMemsetAsync(w.status + kFailCount, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
    fast = launch_rows<kRowsRound>(ctx, ra, rnw, rdyn, st);
    if (fast && !MULO_LAUNCH_LEFT(K_ROUND_FAILED, dyn, st, a, w.fail_list, w.status + kFailCount)) return MULO_ERR_CUDA;
  }
  StreamArgs sa;
  memset(&sa, 0, sizeof sa);
  const size_t sdyn = (ctx->force_dense || fast) ? 0 : plan_stream(ctx, a.P, &sa);
  if (sdyn) {
    sa.P = a.P;
    sa.cond = a.cond; sa.uncond = a.uncond; sa.draft = a.draft; sa.draft_tok_lo = draft_tok_lo;
    sa.nn = a.nn;
    sa.p_tok = p_tok; sa.q_tok = q_tok; sa.accept_prob = accept_prob;
    sa.flags = w.flags; sa.cand_res = w.cand_res; sa.cand_tgt = w.cand_tgt;
    sa.dev_status = w.status;
    sa.fail_list = w.fail_list;
    sa.n_parents = p->B * a.P.h * a.P.w;
    if (cudaMemsetAsync(w.status + kFailCount, 0, sizeof(uint32_t), st) != cudaSuccess) return MULO_ERR_CUDA;
    fast = launch_stream(ctx, sa, sdyn, st);
    // the rows the streaming kernel gave up on (usually a handful, often none)
    if (fast && !MULO_LAUNCH_LEFT(K_ROUND_FAILED, dyn, st, a, w.fail_list, w.status + kFailCount)) return MULO_ERR_CUDA;
  }
  if (!fast && !MULO_LAUNCH_GENERAL(K_ROUND, p->B * a.P.h * a.P.w, dyn, st, a)) return MULO_ERR_UNSUPPORTED;
  if (timed) {
    cudaEventRecord(ctx->ev[ctx->ev_used + 1], st);
    ctx->ev_used += 2;
  }
  MaskArgs m;
  memset(&m, 0, sizeof m);
  m.H = p->H; m.W = p->W; m.r = p->r; m.radius = p->radius; m.clip = a.P.clip; m.resample_mode = p->resample_mode;
  m.flags = w.flags;
  m.reject_bits = reject_bits; m.expand_bits = expand_bits;
  m.n_reject = n_reject; m.first_reject = first_reject; m.n_expand = n_expand;
  m.cand_res = w.cand_res; m.cand_tgt = w.cand_tgt;
  m.draft_tok_lo = draft_tok_lo; m.out_tok = out_tok;
  if (!launch_after(k_mask<2>, (unsigned)p->B, kMaskThreads, mask_smem(p), st, m)) return MULO_ERR_CUDA;
  return launched(ctx, fast ? 1 + fast_launches : 2);
}

mulo_status mulo_round_kernel(const mulo_ctx* ctx, const mulo_params* p, int has_uncond, int* kernel) {
  if (!ctx || !kernel) return MULO_ERR_INVALID_ARG;
  const mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  const DevParams d = to_dev(p);
  RowsArgs ra;
  StreamArgs sa;
  int nw;
  memset(&ra, 0, sizeof ra);
  memset(&sa, 0, sizeof sa);
  *kernel = MULO_KERNEL_GENERAL;
  if (ctx->force_dense) return MULO_OK;
  FullArgs ua;
  FlatArgs fa;
  memset(&ua, 0, sizeof ua);
  memset(&fa, 0, sizeof fa);
  bool fres;
  if (plan_full(ctx, d, has_uncond != 0, &ua) || plan_flat(ctx, d, false, &fa, &fres)) *kernel = MULO_KERNEL_FULL;
  else if (plan_rows(ctx, d, kRowsRound, &ra, &nw)) *kernel = d.pool_k > 1 ? MULO_KERNEL_STREAM : MULO_KERNEL_LANE;
  else if (plan_stream(ctx, d, &sa)) *kernel = MULO_KERNEL_STREAM;
  return MULO_OK;
}

// ---- host-buffer variant -------------------------------------------------------------

struct HostArena {
  size_t ws, cond, uncond, draft, tok_lo, nn, out_tok, rbits, ebits, ptok, qtok, aprob, nrej, nexp, first, total;
};

static HostArena carve_arena(const mulo_params* p, int has_uncond) {
  const size_t n = (size_t)p->B * p->H * p->W, nlo = n / ((size_t)p->r * p->r);
  const size_t esz = p->logit_dtype == MULO_BF16 ? 2 : 4;
  const size_t nwords = (size_t)p->B * p->H * ((p->W + 31) / 32);
  HostArena a;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes ? bytes : 1, 256); return o; };
  a.ws = take(carve_ws(nullptr, p).bytes);
  a.cond = take(n * p->V * esz);
  a.uncond = take(has_uncond ? n * p->V * esz : 0);
  a.draft = take(nlo * p->V * esz);
  a.tok_lo = take(nlo * 4);
  a.nn = take(p->pool_k > 1 ? (size_t)p->V * p->pool_k * 2 : 0);
  a.out_tok = take(n * 4);
  a.rbits = take(nwords * 4);
  a.ebits = take(nwords * 4);
  a.ptok = take(n * 4); a.qtok = take(n * 4); a.aprob = take(n * 4);
  a.nrej = take((size_t)p->B * 4); a.nexp = take((size_t)p->B * 4); a.first = take((size_t)p->B * 4);
  a.total = off;
  return a;
}

mulo_status mulo_round_host_arena_bytes(const mulo_params* p, int has_uncond, size_t* bytes) {
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!bytes) return MULO_ERR_INVALID_ARG;
  *bytes = carve_arena(p, has_uncond).total;
  return MULO_OK;
}

mulo_status mulo_round_host(mulo_ctx* ctx, const mulo_params* p, void* arena, size_t arena_bytes,
                            const void* tgt_cond, const void* tgt_uncond, const void* draft_logits_lo,
                            const int32_t* draft_tok_lo, const uint16_t* nn, int32_t* out_tok,
                            uint32_t* reject_bits, uint32_t* expand_bits, float* p_tok, float* q_tok,
                            float* accept_prob, int32_t* n_reject, int32_t* n_expand,
                            int32_t* first_reject, void* stream) {
  if (!ctx || !arena || ((uintptr_t)arena & 255u)) return MULO_ERR_INVALID_ARG;
  mulo_status s = validate(p);
  if (s != MULO_OK) return s;
  if (!tgt_cond || !draft_logits_lo || !draft_tok_lo || !out_tok || !reject_bits || !expand_bits)
    return MULO_ERR_INVALID_ARG;
  if (p->pool_k > 1 && !nn) return MULO_ERR_INVALID_ARG;
  const HostArena A = carve_arena(p, tgt_uncond != nullptr);
  if (A.total > arena_bytes) return MULO_ERR_WORKSPACE;
  if (p->B == 0) return MULO_OK;
  if ((s = on_context_device(ctx)) != MULO_OK) return s;
  char* d = (char*)arena;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t n = (size_t)p->B * p->H * p->W, nlo = n / ((size_t)p->r * p->r);
  const size_t esz = p->logit_dtype == MULO_BF16 ? 2 : 4;
  const size_t nwords = (size_t)p->B * p->H * ((p->W + 31) / 32);
  bool ok = true;
  ok &= cudaMemsetAsync(d + A.ws, 0, kStatusBytes, st) == cudaSuccess;
  ctx->ws = d + A.ws;
  ctx->ws_bytes = carve_ws(nullptr, p).bytes;
  ok &= cudaMemcpyAsync(d + A.draft, draft_logits_lo, nlo * p->V * esz, cudaMemcpyHostToDevice, st) == cudaSuccess;
  ok &= cudaMemcpyAsync(d + A.tok_lo, draft_tok_lo, nlo * 4, cudaMemcpyHostToDevice, st) == cudaSuccess;
  if (p->pool_k > 1)
    ok &= cudaMemcpyAsync(d + A.nn, nn, (size_t)p->V * p->pool_k * 2, cudaMemcpyHostToDevice, st) == cudaSuccess;
  ok &= cudaMemcpyAsync(d + A.cond, tgt_cond, n * p->V * esz, cudaMemcpyHostToDevice, st) == cudaSuccess;
  if (tgt_uncond)
    ok &= cudaMemcpyAsync(d + A.uncond, tgt_uncond, n * p->V * esz, cudaMemcpyHostToDevice, st) == cudaSuccess;
  if (!ok) return MULO_ERR_CUDA;
  s = mulo_round(ctx, p, d + A.cond, tgt_uncond ? d + A.uncond : nullptr, d + A.draft,
                 (const int32_t*)(d + A.tok_lo), p->pool_k > 1 ? (const uint16_t*)(d + A.nn) : nullptr,
                 (int32_t*)(d + A.out_tok), (uint32_t*)(d + A.rbits), (uint32_t*)(d + A.ebits),
                 p_tok ? (float*)(d + A.ptok) : nullptr, q_tok ? (float*)(d + A.qtok) : nullptr,
                 accept_prob ? (float*)(d + A.aprob) : nullptr, (int32_t*)(d + A.nrej),
                 (int32_t*)(d + A.nexp), (int32_t*)(d + A.first), stream);
  if (s != MULO_OK) return s;
  ok &= cudaMemcpyAsync(out_tok, d + A.out_tok, n * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  ok &= cudaMemcpyAsync(reject_bits, d + A.rbits, nwords * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  ok &= cudaMemcpyAsync(expand_bits, d + A.ebits, nwords * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (p_tok) ok &= cudaMemcpyAsync(p_tok, d + A.ptok, n * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (q_tok) ok &= cudaMemcpyAsync(q_tok, d + A.qtok, n * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (accept_prob) ok &= cudaMemcpyAsync(accept_prob, d + A.aprob, n * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (n_reject) ok &= cudaMemcpyAsync(n_reject, d + A.nrej, (size_t)p->B * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (n_expand) ok &= cudaMemcpyAsync(n_expand, d + A.nexp, (size_t)p->B * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  if (first_reject) ok &= cudaMemcpyAsync(first_reject, d + A.first, (size_t)p->B * 4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
  ok &= cudaStreamSynchronize(st) == cudaSuccess;
  return ok ? MULO_OK : MULO_ERR_CUDA;
}

}  // extern "C"

// ---- allocation-free variant of the fused round ------------------------------------------

// Scratch of mulo_round_static: lives in the library image, one copy per device that
// loads it.  In host code this name is only a handle for the runtime's symbol table,
// never a device address; the kernels get the address cudaGetSymbolAddress returns.
static __device__ __align__(256) unsigned char g_static_scratch[MULO_STATIC_SCRATCH_BYTES];

static const int kMaxStaticDevices = 64;
static void* g_static_scratch_addr[kMaxStaticDevices];   // per device, nullptr until looked up
static std::mutex g_static_scratch_mutex;

// Device address of g_static_scratch on `device`: looked up once per device, with that
// device current, then served from the table.
static mulo_status static_scratch_address(int device, void** out) {
  if (device < 0 || device >= kMaxStaticDevices) return MULO_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
  if (!g_static_scratch_addr[device]) {
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return MULO_ERR_CUDA;
    if (prev != device && cudaSetDevice(device) != cudaSuccess) return MULO_ERR_CUDA;
    void* addr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&addr, g_static_scratch);
    if (prev != device) cudaSetDevice(prev);
    if (e != cudaSuccess || !addr) {
      cudaGetLastError();
      return MULO_ERR_CUDA;
    }
    g_static_scratch_addr[device] = addr;
  }
  *out = g_static_scratch_addr[device];
  return MULO_OK;
}

extern "C" mulo_status mulo_round_static(mulo_ctx* ctx, const mulo_params* p, const void* tgt_cond,
                                         const void* tgt_uncond, const void* draft_logits_lo,
                                         const int32_t* draft_tok_lo, const uint16_t* nn, int32_t* out_tok,
                                         uint32_t* reject_bits, uint32_t* expand_bits, float* p_tok,
                                         float* q_tok, float* accept_prob, int32_t* n_reject,
                                         int32_t* n_expand, int32_t* first_reject, uint32_t* device_status,
                                         void* stream) {
  // every refusal comes before the shared array is touched
  mulo_status s = check_round_args(ctx, p, tgt_cond, tgt_uncond, draft_logits_lo, draft_tok_lo, nn, out_tok,
                                   reject_bits, expand_bits);
  if (s != MULO_OK) return s;
  if (carve_ws(nullptr, p).bytes > (size_t)MULO_STATIC_SCRATCH_BYTES) return MULO_ERR_WORKSPACE;
  void* scratch = nullptr;
  if ((s = static_scratch_address(ctx->device, &scratch)) != MULO_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  // The status word is OR-ed into and must start at zero; flags and candidates are written
  // for every position of this call before the mask kernel reads them.
  if (cudaMemsetAsync(scratch, 0, kStatusBytes, st) != cudaSuccess) return MULO_ERR_CUDA;
  void* const saved_ws = ctx->ws;
  const size_t saved_bytes = ctx->ws_bytes;
  ctx->ws = scratch;
  ctx->ws_bytes = MULO_STATIC_SCRATCH_BYTES;
  s = mulo_round(ctx, p, tgt_cond, tgt_uncond, draft_logits_lo, draft_tok_lo, nn, out_tok, reject_bits,
                 expand_bits, p_tok, q_tok, accept_prob, n_reject, n_expand, first_reject, stream);
  ctx->ws = saved_ws;
  ctx->ws_bytes = saved_bytes;
  if (s != MULO_OK) return s;
  if (device_status &&
      cudaMemcpyAsync(device_status, scratch, sizeof(uint32_t), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return MULO_ERR_CUDA;
  return MULO_OK;
}
