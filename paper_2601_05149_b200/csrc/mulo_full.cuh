// Pooled rows without a top-k cut whose redraws all come from the target distribution (the paper's Eq. 5 as printed,
// its default sampling setting), when the vocabulary splits evenly over a CTA's 256 threads and the rows of one position
// fit in shared memory.  The other rows without a cut are mulo_flat.cuh's.
//
// A persistent CTA owns a contiguous range of target rows, parent (low-res) cell by parent cell.  Per parent it brings the
// draft row into shared memory once (plain bulk copies, never multicast) -- unless the decision rule never looks at q
// (Eq. 5), in which case the draft logits are not read at all -- and then, child by child, the target position's
// conditional and unconditional rows.  Every thread owns a contiguous range of W = V / 256 ids of the resident row, so that
// per-thread sums are slices of the ascending-id CDF:
//
//   softmax      one pass: a running maximum and a sum of exponentials against it per thread
//                (the sum is rescaled on the rare occasions the maximum moves), then the block
//                maximum, the threads' sums rescaled to it, and one block scan in double that
//                gives both the partition sum and the CDF slice of every thread.
//   pooling      Eq. 3-4 on the resident row: a few consecutive entries of x~'s neighbour list per thread, asked for
//                before the wait for the row; prefix masses by a block scan; the pooled ids are marked in a V-bit map and
//                their weights leave their owners' sums through fixed-point shared atomics (integer addition: the result
//                does not depend on the order), in two halves of 32 bits.
//   draws        the thread sums are known, the owner of u * total walks its W ids.
//
// The 128-bit shared loads of a warp are spread over the bank groups by starting every thread
// at a different 16-byte piece of its range (sums do not depend on the order; the walk of a
// draw's owner thread is in ascending id).
//
// Bound by instruction issue: 12.7 k warp instructions per position of V = 16384 at 0.58 per scheduler cycle, three CTAs
// per SM.  64 x 64, 16 images, lists of 1000: 1462 us with the list read entry by entry behind the wait for each row, 64-bit
// atomics (a loop each) and the row kept until the draw was done; 1240 us now, 1280 with these rows on mulo_flat.cuh's
// kernel.  The next row asked into L2 meanwhile: 5 % slower.
#pragma once

#include "mulo_flat.cuh"

namespace mulo {

constexpr int kFThreads = 256;
constexpr int kFWarps = kFThreads / 32;
constexpr uint32_t kFPiece = 16384;      // bytes per bulk copy
constexpr float kFix40 = 1099511627776.0f;   // 2^40: fixed-point scale of the pooled weights (each at most 1, at most 256 per thread)

struct FullArgs {
  DevParams P;
  const char* cond;
  const char* uncond;
  const char* draft;
  const int32_t* draft_tok_lo;
  const uint16_t* nn;
  float* p_tok;
  float* q_tok;
  float* accept_prob;
  uint8_t* flags;
  int32_t* cand_tgt;
  uint32_t* dev_status;
  int n_units;   // target rows, parent by parent
  int W;         // ids per thread
  int need_q;    // 0: neither the decision nor any draw uses the draft distribution
};

struct FullSmem {
  uint64_t bar_q, bar_t;
  double wtot[2][kFWarps];   // block scans; consecutive scans alternate
  double bd[kFWarps];        // block sums
  float bf[2][kFWarps];      // block maxima; consecutive reductions alternate
  uint32_t rnd[3];
  double p_tok, q_tok;       // exp(z - max) of x~ at the current position; q(x~) of the parent
  double p_row;              // p(x~)
  double cJ;                 // pooled prefix mass c_J
  int first_bad;
  int tok;
  int abort;
};

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// z of one id of a resident row
template <bool BF16, bool ROW_U>
__device__ __forceinline__ float full_one(const unsigned char* crow, const unsigned char* urow, int x, float s, float invT) {
  float c, u = 0.f;
  if (BF16) {
    c = __uint_as_float((uint32_t) reinterpret_cast<const unsigned short*>(crow)[x] << 16);
    if (ROW_U) u = __uint_as_float((uint32_t) reinterpret_cast<const unsigned short*>(urow)[x] << 16);
  } else {
    c = reinterpret_cast<const float*>(crow)[x];
    if (ROW_U) u = reinterpret_cast<const float*>(urow)[x];
  }
  return mix_logit(c, u, ROW_U, s, invT);
}

template <bool BF16, bool HAS_U>
__global__ void __launch_bounds__(kFThreads, 3) k_round_full(const __grid_constant__ FullArgs a) {
  constexpr int esz = BF16 ? 2 : 4;
  constexpr int N = 16 / esz;   // ids per 16-byte piece
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ FullSmem sm;
  const DevParams& P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  let_next_begin();
  const int u_begin = (int)(((long long)a.n_units * blockIdx.x) / gridDim.x);
  const int u_end = (int)(((long long)a.n_units * (blockIdx.x + 1)) / gridDim.x);
  if (u_end <= u_begin) return;
  const int V = P.V, W = a.W, nch = W / N, rr = P.r * P.r, NN = P.H * P.W;
  const uint32_t row_bytes = (uint32_t)V * esz;
  const bool need_q = a.need_q != 0;
  unsigned char* const qrow = dyn;
  unsigned char* const crow = dyn + (need_q ? row_bytes : 0u);
  unsigned char* const urow = crow + row_bytes;
  uint32_t* const bitmap = reinterpret_cast<uint32_t*>(crow + (HAS_U ? 2u : 1u) * row_bytes);
  uint2* const adj = reinterpret_cast<uint2*>(bitmap + V / 32);   // pooled weight times 2^40: 24 bits below, the rest above
  const uint32_t my_off = (uint32_t)tid * (uint32_t)W * esz;
  const uint32_t q_at = smem_u32(qrow) + my_off, c_at = smem_u32(crow) + my_off, u_at = smem_u32(urow) + my_off;
  const int start = tid % nch;   // this thread's first piece (bank spreading)
  const int id0 = tid * W;
  const float inv_W = 1.0f / (float)W;
  const int nb = P.pool_k - 1, per = (nb + kFThreads - 1) / kFThreads, j0 = tid * per;

  if (tid == 0) {
    mbar_init(&sm.bar_q, 1);
    mbar_init(&sm.bar_t, 1);
    mbar_fence_init();
    sm.abort = 0;
  }
  __syncthreads();
  uint32_t ph_q = 0, ph_t = 0;

  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return;
    if (*(volatile int*)&sm.abort) return;
#pragma unroll 1
    for (uint32_t it = 0; it < kSpinLimit; ++it)
      if (mbar_try_wait(bar, parity)) return;
    atomicOr(a.dev_status, MULO_DEV_TIMEOUT);
    *(volatile int*)&sm.abort = 1;
  };
  // one thread: a row from global memory into a resident buffer
  auto fetch = [&](unsigned char* dst, const char* src, uint64_t* bar) {
    for (uint32_t o = 0; o < row_bytes; o += kFPiece) {
      const uint32_t n = row_bytes - o < kFPiece ? row_bytes - o : kFPiece;
      bulk_load(dst + o, src + o, n, bar);
    }
  };
  auto fetch_target = [&](size_t g) {   // one thread
    fence_async_smem();
    mbar_expect_tx(&sm.bar_t, HAS_U ? 2u * row_bytes : row_bytes);
    fetch(crow, a.cond + g * (size_t)row_bytes, &sm.bar_t);
    if (HAS_U) fetch(urow, a.uncond + g * (size_t)row_bytes, &sm.bar_t);
  };
  // ---- block helpers (every thread gets the result; fixed order)
  int max_call = 0;
  auto block_max_f = [&](float v) -> float {   // one barrier: consecutive calls alternate buffers
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    float* const bf = sm.bf[max_call & 1];
    ++max_call;
    if (lane == 0) bf[warp] = v;
    __syncthreads();
    float t = bf[0];
#pragma unroll
    for (int w = 1; w < kFWarps; ++w) t = fmaxf(t, bf[w]);
    return t;
  };
  int scan_call = 0;
  // inclusive scan over the threads in id order: returns the total; `before` = mass of the threads below
  auto block_scan = [&](double v, double& before, double& incl) -> double {
    double inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double n = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += n;
    }
    double* const wt = sm.wtot[scan_call & 1];
    ++scan_call;
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    double pre = 0.0, total = 0.0;
#pragma unroll
    for (int w = 0; w < kFWarps; ++w) {
      const double x = wt[w];
      if (w == warp) pre = total;
      total += x;
    }
    // (the mass below this thread comes from its neighbour's inclusive sum, not from inc - v,
    // which would cancel the small masses before a large v)
    double exc = __shfl_up_sync(kFull, inc, 1);
    if (lane == 0) exc = 0.0;
    incl = pre + inc;
    before = pre + exc;
    return total;
  };

  // ---- one pass over this thread's part of a resident row: running maximum m and the sum of
  //      2^((z - m) log2 e) against it
  auto softmax_pass_t = [&](auto row_u_tag, auto scale_tag, uint32_t at_c, uint32_t at_u, float s, float& m, float& sum) {
    constexpr bool ROW_U = decltype(row_u_tag)::value;
    constexpr bool SCALE = decltype(scale_tag)::value;
    constexpr int NP = N / 2;   // pairs per piece
    const float2 s2 = make_float2(s, s), t2 = make_float2(P.invT, P.invT), l2 = make_float2(kLog2e, kLog2e);
    m = -1e30f;   // (not -inf: pieces whose ids are all forbidden, at -inf under guidance, would be inf - inf)
    float2 acc = make_float2(0.f, 0.f);
    int ci = start;
#pragma unroll 1
    for (int i = 0; i < nch; ++i) {
      float2 z[NP];
      const uint4 cv = lds128(at_c + (uint32_t)ci * 16u);
      flat_logits<BF16, ROW_U, SCALE>(cv, ROW_U ? lds128(at_u + (uint32_t)ci * 16u) : cv, s2, t2, z);
      if (++ci == nch) ci = 0;
      float cm = fmaxf(z[0].x, z[0].y);
#pragma unroll
      for (int j = 1; j < NP; ++j) cm = fmaxf(cm, fmaxf(z[j].x, z[j].y));
      if (cm > m) {
        const float f = ex2f((m - cm) * kLog2e);   // (0 * 0 on the first piece)
        acc = __fmul2_rn(acc, make_float2(f, f));
        m = cm;
      }
      const float c0 = -m * kLog2e;
      const float2 c2 = make_float2(c0, c0);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const float2 t = __ffma2_rn(z[j], l2, c2);
        acc = __fadd2_rn(acc, make_float2(ex2f(t.x), ex2f(t.y)));
      }
    }
    sum = acc.x + acc.y;
  };
  const bool scale = P.invT != 1.0f;
  auto softmax_pass = [&](auto row_u_tag, uint32_t at_c, uint32_t at_u, float s, float& m, float& sum) {
    if (scale) softmax_pass_t(row_u_tag, std::true_type{}, at_c, at_u, s, m, sum);   // block-uniform
    else softmax_pass_t(row_u_tag, std::false_type{}, at_c, at_u, s, m, sum);
  };

  for (int parent = u_begin / rr; parent * rr < u_end; ++parent) {
    const int c_begin = max(0, u_begin - parent * rr), c_end = min(rr, u_end - parent * rr);
    const int hw = P.h * P.w, b = parent / hw, cell = parent - b * hw, ca = cell / P.w, cc = cell - ca * P.w;
    int di = c_begin / P.r, dj = c_begin - di * P.r;
    int t = (ca * P.r + di) * P.W + cc * P.r + dj;   // the row's place in its image
    // ------------------------------------------------------------ the parent's draft row
    if (tid == 0 && !sm.abort) {
      sm.tok = checked_token(__ldg(a.draft_tok_lo + parent), V, a.dev_status);
      if (need_q) {
        fence_async_smem();
        mbar_expect_tx(&sm.bar_q, row_bytes);
        fetch(qrow, a.draft + (size_t)parent * row_bytes, &sm.bar_q);
      }
      fetch_target((size_t)b * NN + t);
    }
    __syncthreads();
    // A wait of this CTA gave up (block-uniform: raised before the last barrier, and nothing was
    // requested since): nothing more is written for its rows; the copy that did not arrive gets a
    // bounded time to land before the shared memory is given up.
    if (*(volatile int*)&sm.abort) {
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
      return;
    }
    const int tok = sm.tok;
    // This thread's `per` consecutive entries of the neighbour list (at most 8: the list has at most 2047), asked for here,
    // once for all rows under the parent: one after the other behind the wait for each row they cost it 5 k cycles.
    uint32_t ids[4];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const uint16_t* const from = a.nn + (size_t)tok * P.pool_k + 1;
      const uint32_t lo = i < per ? __ldg(from + min(j0 + i, nb - 1)) : 0u, hi = i + 1 < per ? __ldg(from + min(j0 + i + 1, nb - 1)) : 0u;
      ids[i / 2] = lo | hi << 16;
    }
    double q_tok = 0.0;
    if (need_q) {
      wait(&sm.bar_q, ph_q);
      ph_q ^= 1u;
      float mt, st;
      softmax_pass(std::false_type{}, q_at, q_at, 0.f, mt, st);
      const float m_q = block_max_f(mt);
      const double mine = (double)(st * ex2f((mt - m_q) * kLog2e));
      double before, incl;
      const double Zq = block_scan(mine, before, incl);
      if (tid == 0) {
        const float zq = full_one<BF16, false>(qrow, qrow, tok, 0.f, P.invT);
        const double q = row_exp2(((double)zq - (double)m_q) * 1.4426950408889634) / Zq;
        if (q <= 0.0) atomicOr(a.dev_status, MULO_DEV_ZERO_DRAFT_PROB);
        sm.q_tok = q;
      }
      __syncthreads();
      q_tok = sm.q_tok;
    }

    for (int child = c_begin; child < c_end; ++child) {
      const size_t g = (size_t)b * NN + t;
      if (tid == 32) {
        const uint4 rnd = row_philox(make_uint4((uint32_t)t, (uint32_t)b + P.image_offset, P.round, 0u),
                                      make_uint2(P.seed_lo, P.seed_hi));
        sm.rnd[0] = rnd.x;
        sm.rnd[1] = rnd.y;
        sm.rnd[2] = rnd.z;
      }
      wait(&sm.bar_t, ph_t);
      ph_t ^= 1u;
      float mt, st;
      softmax_pass(std::integral_constant<bool, HAS_U>{}, c_at, u_at, P.cfg_scale, mt, st);
      const float M = block_max_f(mt);
      const float c0 = -M * kLog2e;
      const float S_t = st * ex2f((mt - M) * kLog2e);   // this thread's ids, against the row maximum
      const float z_tok = full_one<BF16, HAS_U>(crow, urow, tok, P.cfg_scale, P.invT);
      const float e_tok = ex2f(fmaf(z_tok, kLog2e, c0));
      // exp(z_tok - M) in double by one thread, published by the scan's barrier
      if (tid == 0) sm.p_tok = row_exp2(((double)z_tok - (double)M) * 1.4426950408889634);
      double before, incl;
      const double Z = block_scan((double)S_t, before, incl);

      // ---- Eq. 3-4: the leading run of the neighbour list whose prefix mass stays below delta
      int J = 0;
      double cJ = 0.0;
      {
        for (int x = tid; x < V / 32; x += kFThreads) bitmap[x] = 0u;
        adj[tid] = make_uint2(0u, 0u);
        if (tid == 0) {
          sm.first_bad = nb;
          sm.p_row = sm.p_tok / Z;
        }
        int id[8];
        bool bad_id = false;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          id[i] = (int)(ids[i / 2] >> (16 * (i & 1)) & 0xffffu);
          bad_id |= id[i] >= V;
          id[i] = min(id[i], V - 1);
        }
        if (bad_id) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
        float e[8];
        double mine = 0.0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          e[i] = 0.f;
          if (i < per && j0 + i < nb) {
            e[i] = ex2f(fmaf(full_one<BF16, HAS_U>(crow, urow, id[i], P.cfg_scale, P.invT), kLog2e, c0));
            mine += (double)e[i];
          }
        }
        double bef, inc;
        block_scan(mine, bef, inc);   // (its barrier also publishes first_bad and the cleared map)
        // c_j < delta, in units of the partition sum
        const double limit = P.pool_delta * Z;
        {
          double c = bef;
          int bad = nb;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i < per && j0 + i < nb) {
              c += (double)e[i];
              if (bad == nb && !(c < limit)) bad = j0 + i;
            }
          if (bad < nb) atomicMin(&sm.first_bad, bad);
        }
        __syncthreads();
        J = sm.first_bad;   // the leading run n_1 .. n_J keeps its prefix mass below delta
        if (J - 1 >= j0 && J - 1 < j0 + per) {
          double c = bef;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (j0 + i < J) c += (double)e[i];
          sm.cJ = c / Z;
        }
        // the pooled ids: out of the map of drawable ids, their weights out of their owners' sums
        uint32_t old[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < per && j0 + i < J) old[i] = atomicOr(&bitmap[id[i] >> 5], 1u << (id[i] & 31));
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < per && j0 + i < J && !(old[i] >> (id[i] & 31) & 1u) && id[i] != tok) {   // (a list may name an id twice, or x~ again)
            const unsigned long long f = __float2ull_rz(e[i] * kFix40);
            uint2* const at = &adj[(int)(((float)id[i] + 0.5f) * inv_W)];   // its owner
            atomicAdd(&at->x, (uint32_t)f & 0xffffffu);
            atomicAdd(&at->y, (uint32_t)(f >> 24));
          }
        __syncthreads();
        if (J > 0) cJ = sm.cJ;
      }
      const double p_tok = sm.p_row;
      const double mass = p_tok + cJ;   // pooled mass P of Eq. 3

      // ---- the decision (Eq. 1 / Eq. 5), the same in every thread
      double thr;
      int accepted;
      if (P.accept_mode == MULO_ACCEPT_THRESHOLD) {
        thr = mass;
        accepted = mass >= P.tau;
      } else {
        if (q_tok <= 0.0) thr = mass > 0.0 ? 1.0 : 0.0;
        else thr = fmin(1.0, mass / q_tok);
        accepted = uniform24(sm.rnd[0]) < thr;
      }
      // ---- the draw, from the target weights in units of 2^((z - M) log2 e): the entry's own, nothing for a pooled id,
      // mass * Z for x~
      double S = (double)S_t;
      {
        const uint2 out = adj[tid];
        S -= (double)(((unsigned long long)out.y << 24) + out.x) * (1.0 / (double)kFix40);
      }
      if (tok >= id0 && tok < id0 + W) S += mass * Z - (double)e_tok;
      S = fmax(S, 0.0);
      double bef, inc;
      const double total = block_scan(S, bef, inc);
      const double y = uniform24(sm.rnd[2]) * total;
      // One thread owns u * total; its warp walks that thread's ids together, 32 at a time in ascending order: weights, an
      // inclusive scan in double, the first id whose running sum passes y.  With the weights in registers the row can go:
      // the next one is asked for before the scans.
      const unsigned owner_mask = total > 0.0 ? __ballot_sync(kFull, bef <= y && y < inc) : 0u;
      const int src = owner_mask ? __ffs(owner_mask) - 1 : 0, o_id0 = __shfl_sync(kFull, id0, src);
      float w[8];   // (W <= 256)
      if (owner_mask) {   // warp-uniform
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int x = o_id0 + i * 32 + lane;
          w[i] = 0.f;
          if (i * 32 < W && x < o_id0 + W) {
            if (!((bitmap[x >> 5] >> (x & 31)) & 1u))
              w[i] = ex2f(fmaf(full_one<BF16, HAS_U>(crow, urow, x, P.cfg_scale, P.invT), kLog2e, c0));
            if (x == tok) w[i] = (float)(mass * Z);
          }
        }
      }
      __syncthreads();   // everybody is done with the resident target row
      if (++dj == P.r) {
        dj = 0;
        t += P.W - P.r;
      }
      ++t;
      if (tid == 0 && child + 1 < c_end && !sm.abort) fetch_target((size_t)b * NN + t);
      if (owner_mask) {
        double c = __shfl_sync(kFull, bef, src);
        int pick = -1, last_pos = -1;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i * 32 < W && pick < 0) {
            double run = (double)w[i];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const double n = __shfl_up_sync(kFull, run, o);
              if (lane >= o) run += n;
            }
            const unsigned has = __ballot_sync(kFull, w[i] > 0.f);
            const unsigned hit = __ballot_sync(kFull, w[i] > 0.f && c + run > y);
            if (has) last_pos = o_id0 + i * 32 + 31 - __clz(has);
            if (hit) pick = o_id0 + i * 32 + __ffs(hit) - 1;
            c += __shfl_sync(kFull, run, 31);
          }
        // (rounding left the walk short of y: the last id with weight; none at all cannot be, the thread's sum being
        // positive -- then the thread's first id stands in)
        if (lane == 0) a.cand_tgt[g] = pick >= 0 ? pick : last_pos >= 0 ? last_pos : o_id0;
      }
      if (tid == 32 * (kFWarps - 1)) {
        if (!(total > 0.0)) a.cand_tgt[g] = -1;   // (a row whose largest logit mixes to +inf)
        a.flags[g] = accepted ? 0 : 1;
        if (a.p_tok) a.p_tok[g] = (float)p_tok;
        if (a.q_tok) a.q_tok[g] = (float)q_tok;
        if (a.accept_prob) a.accept_prob[g] = (float)thr;
      }
    }
  }
}

}  // namespace mulo
