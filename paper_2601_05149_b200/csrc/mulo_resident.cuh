// The general path for rows that fit shared memory (V <= 49152): one CTA of 512 threads per row, the row's
// pre-processed logits resident as fp32.
//
// What a row costs here is a chain of passes with block barriers between them, so the passes are few and short: the
// row comes in once (coalesced 128-bit loads; maximum, minimum and sum on the way), the k-th largest value is found by
// ONE histogram of 1024 bins between the mean and the maximum (a second one inside the crossing bin if more than 128
// entries share it) and an exact ranking of the crossing bin's entries, one pass turns logits into exp(z - max) in
// place, and one block scan in double gives the partition sum and every thread's slice of the ascending-id CDF.  A
// draw from the target weights needs nothing more than the walk of the owner's run by its warp.  The routines of
// mulo_device.cuh / mulo_dense.cuh, which read the row nine times (radix select), took 55 us for a row of 16384
// bf16 ids with guidance on one CTA; this takes 7.6 us.
//
// A thread owns a contiguous run of E ids; runs are E + 4 floats apart, so that 128-bit accesses of a quarter warp
// hit different banks.
#pragma once

#include "mulo_rows.cuh"

namespace mulo {

constexpr int kResBins = 1024;
constexpr int kResMembers = 128;

struct ResScratch {
  unsigned hist[kResBins];
  unsigned spill[32];           // where the ids outside the bracket are counted
  double scan[2][kWarps];       // block scans; consecutive ones alternate
  unsigned top[kWarps], low[kWarps];   // keys of block maxima and minima
  float sum[kWarps];
  float sa[kResMembers];
  unsigned n_sa;
  int first_bad;
  int tok[2];                   // draws: residual, target
  double bd[4];
};

__host__ __device__ inline int resident_run(int V) { return 8 * ((V + 8 * kThreads - 1) / (8 * kThreads)); }
__host__ inline size_t resident_bytes(int V) { return (size_t)kThreads * (resident_run(V) + 4) * sizeof(float); }
__host__ inline bool resident_fits(int V) { return V <= 49152; }

// One row in shared memory: logits after load(), weights exp(z - max) (0 below the threshold) after weigh().
struct ResRow {
  float* w;
  int V, E, beg, end;           // this thread's run
  float inv_E;
  __device__ ResRow(float* smem, int V_) : w(smem), V(V_), E(resident_run(V_)), inv_E(1.0f / (float)resident_run(V_)) {
    beg = min(V, (int)threadIdx.x * E);
    end = min(V, beg + E);
  }
  __device__ __forceinline__ float* run() const { return w + threadIdx.x * (E + 4); }
  __device__ __forceinline__ float* place(int x) const {   // (x + 0.5) / E in fp32 truncates to x / E for x < 2^16)
    return w + x + 4 * (int)(((float)x + 0.5f) * inv_E);
  }
  __device__ __forceinline__ float& at(int x) const { return *place(x); }
};

struct ResSums {      // block scan of one value per thread, in id order
  double before, incl, total;
};

__device__ __forceinline__ ResSums res_scan(double v, ResScratch& rs, int& calls) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double n = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += n;
  }
  double* const wt = rs.scan[calls++ & 1];
  if (lane == 31) wt[warp] = inc;
  __syncthreads();
  double t = wt[lane & (kWarps - 1)], ti = t;   // every warp scans the warps' totals
#pragma unroll
  for (int o = 1; o < kWarps; o <<= 1) {
    const double n = __shfl_up_sync(kFull, ti, o, kWarps);
    if ((lane & (kWarps - 1)) >= o) ti += n;
  }
  ResSums r;
  r.total = __shfl_sync(kFull, ti, kWarps - 1);
  const double up = __shfl_sync(kFull, ti, warp > 0 ? warp - 1 : 0), here = __shfl_sync(kFull, ti, warp);
  const double pre = warp > 0 ? up : 0.0;
  double exc = __shfl_up_sync(kFull, inc, 1);
  if (lane == 0) exc = 0.0;
  r.incl = lane == 31 ? here : pre + inc;   // (the next warp's `before`, to the bit)
  r.before = pre + exc;
  return r;
}

// Eight logits of a piece, two per packed instruction.
template <bool BF16>
__device__ __forceinline__ void res_mix(const RowSrc& r, const raw_piece<BF16>& c, const raw_piece<BF16>& u, float (&z)[8]) {
  const float2 s2 = make_float2(r.s, r.s), t2 = make_float2(r.invT, r.invT);
  auto all = [&](auto row_u) {
    constexpr bool U = decltype(row_u)::value;
#pragma unroll
    for (int i = 0; i < (BF16 ? 1 : 2); ++i) {
      float2 q[4];
      q[0] = row_pair<BF16, U, true, 0>(c.w[i], u.w[i], s2, t2);
      q[1] = row_pair<BF16, U, true, 1>(c.w[i], u.w[i], s2, t2);
      if (BF16) {
        q[2] = row_pair<BF16, U, true, 2>(c.w[i], u.w[i], s2, t2);
        q[3] = row_pair<BF16, U, true, 3>(c.w[i], u.w[i], s2, t2);
      }
#pragma unroll
      for (int j = 0; j < (BF16 ? 4 : 2); ++j) {
        z[4 * i + 2 * j] = q[j].x;
        z[4 * i + 2 * j + 1] = q[j].y;
      }
    }
  };
  if (r.uncond) all(std::true_type{});
  else all(std::false_type{});
}

// The row from global memory into shared memory; every thread gets the row's maximum and mean.
__device__ __forceinline__ void res_load(const ResRow& row, const RowSrc& src, ResScratch& rs, float& mx, float& mean) {
  float hi = -INFINITY, sum = 0.f;
#pragma unroll 2
  for (int x = (int)threadIdx.x * 8; x < row.V; x += 8 * kThreads) {
    float v[8];
    if (src.bf16) {
      raw_piece<true> c, u = {};
      ask8<true>(src, x, c, u);
      res_mix<true>(src, c, u, v);
    } else {
      raw_piece<false> c, u = {};
      ask8<false>(src, x, c, u);
      res_mix<false>(src, c, u, v);
    }
    float4* const to = reinterpret_cast<float4*>(row.place(x));
    to[0] = make_float4(v[0], v[1], v[2], v[3]);
    to[1] = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      hi = fmaxf(hi, v[j]);
      sum += v[j];
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  const unsigned key = __reduce_max_sync(kFull, float_key(hi));
  if (lane == 0) {
    rs.top[warp] = key;
    rs.sum[warp] = sum;
  }
  if (threadIdx.x == 0) rs.n_sa = 0;
#pragma unroll
  for (int i = 0; i < kResBins / kThreads; ++i) rs.hist[threadIdx.x + i * kThreads] = 0;
  __syncthreads();
  mx = key_float(__reduce_max_sync(kFull, rs.top[lane & (kWarps - 1)]));
  sum = rs.sum[lane & (kWarps - 1)];
#pragma unroll
  for (int o = kWarps / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  mean = sum / (float)row.V;
}

// What the histogram of a bracket says about rank `want` from the top: the bin that holds it, the entries above that
// bin, the entries in it (-1: the bracket holds fewer).  Every warp finds it, 32 bins per lane, lane 0 the highest.
__device__ __forceinline__ int res_crossing(const ResScratch& rs, unsigned want, unsigned& over, int& in_bin) {
  const int lane = threadIdx.x & 31;
  unsigned mine = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 h = *reinterpret_cast<const uint4*>(&rs.hist[(31 - lane) * 32 + 4 * ((i + lane) & 7)]);
    mine += (h.x + h.y) + (h.z + h.w);
  }
  unsigned inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += t;
  }
  const unsigned hit = __ballot_sync(kFull, inc >= want);
  if (hit == 0) return -1;
  const int src = __ffs(hit) - 1;
  over = __shfl_sync(kFull, inc - mine, src);
  const unsigned h = rs.hist[(31 - src) * 32 + 31 - lane];
  inc = h;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += t;
  }
  const int k = __ffs(__ballot_sync(kFull, over + inc >= want)) - 1;
  in_bin = (int)__shfl_sync(kFull, h, k);
  over += __shfl_sync(kFull, inc - h, k);
  return (31 - src) * 32 + 31 - k;
}

// The value of rank r from the top among the n >= r entries set aside.
__device__ __forceinline__ float res_rank(const ResScratch& rs, int n, unsigned r) {
  float th = 0.f;
  bool found = false;
#pragma unroll 1
  for (int i = threadIdx.x & 31; i < n; i += 32) {
    const float vi = rs.sa[i];
    unsigned more = 0, geq = 0;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const float vj = rs.sa[j];
      more += vj > vi;
      geq += vj >= vi;
    }
    if (more < r && r <= geq) {
      th = vi;
      found = true;
    }
  }
  return __shfl_sync(kFull, th, __ffs(__ballot_sync(kFull, found)) - 1);   // (found: the entries hold the rank)
}

// The top_k-th largest of the row's values, zhi being the largest, by brackets that shrink by a factor of 512 or more per
// round, in steps of the order-preserving integer keys: for rows whose first histogram did not settle it (many entries in
// one bin, fewer than top_k above the mean).  The first bracket goes down to -inf, which finite logits may mix to.  The
// histogram's memory is free (all threads are past a barrier since its last use) and is left so.
__device__ __noinline__ float res_refine(const ResRow& row, int top_k, float zhi, ResScratch& rs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_mine = row.end - row.beg;
  const float* const z = row.run();
  float zlo = -INFINITY;
  int above = 0;   // values larger than zhi
  for (;;) {
    const uint32_t lo = float_key(zlo), hi = float_key(zhi);
    if (lo == hi) return zhi;
    const int shift = max(0, 22 - __clz(hi - lo));
    for (int i = threadIdx.x; i < kResBins; i += kThreads) rs.hist[i] = 0;
    if (threadIdx.x == 0) rs.n_sa = 0;
    __syncthreads();
    for (int i = 0; i < n_mine; ++i) {
      const uint32_t k = float_key(z[i]);
      if (k >= lo && k <= hi) atomicAdd(&rs.hist[(k - lo) >> shift], 1u);
    }
    __syncthreads();
    unsigned over = 0;
    int in_bin = 0;
    const unsigned want = (unsigned)(top_k - above);
    const int bin = res_crossing(rs, want, over, in_bin);
    if (bin < 0) {   // (uniform; fewer than top_k values are numbers at all: nothing is cut)
      __syncthreads();
      return -INFINITY;
    }
    uint32_t vhi = 0u, vlo = ~0u;
    for (int i = 0; i < n_mine; ++i) {
      const uint32_t k = float_key(z[i]);
      if (k >= lo && k <= hi && (int)((k - lo) >> shift) == bin) {
        if (in_bin <= kResMembers) rs.sa[atomicAdd(&rs.n_sa, 1u)] = z[i];
        vhi = max(vhi, k);
        vlo = min(vlo, k);
      }
    }
    vhi = __reduce_max_sync(kFull, vhi);
    vlo = __reduce_min_sync(kFull, vlo);
    if (lane == 0) {
      rs.top[warp] = vhi;
      rs.low[warp] = vlo;
    }
    __syncthreads();
    if (in_bin <= kResMembers) return res_rank(rs, in_bin, want - over);
    zhi = key_float(__reduce_max_sync(kFull, rs.top[lane & (kWarps - 1)]));
    zlo = key_float(__reduce_min_sync(kFull, rs.low[lane & (kWarps - 1)]));
    above += (int)over;
    __syncthreads();
  }
}

// The top_k-th largest value of the resident row (1 <= top_k < V): a histogram between the mean and the maximum, the
// crossing bin's entries ranked exactly.  The map z -> bin is monotone, so a bin's entries are consecutive in rank
// whatever the rounding (z - mean and the product round monotonically; adding 1.5 * 2^23 leaves the rounded integer in
// the low bits; an entry that rounds up into the first bin from below it is simply one of its entries).
__device__ __forceinline__ float res_select(const ResRow& row, int top_k, float mx, float mean, ResScratch& rs) {
  const int lane = threadIdx.x & 31;
  // (Finite logits may sum to -inf, or mix to it under guidance: two ids at the lowest value of the type do.  Then there
  // is no mean, and no first histogram; sc is 0 where mx - mean is infinite.)
  const float sc = (float)(kResBins - 1) / (mx - mean);
  if (!(mean < mx) || !(sc > 0.f && sc < 1e30f)) {   // (uniform)
    __syncthreads();
    return res_refine(row, top_k, mx, rs);
  }
  auto bits_of = [&](float v) -> int { return __float_as_int(fmaf(__fsub_rn(v, mean), sc, kRMagic)); };
  auto eight = [&](int i, float (&v)[8]) {   // eight of this thread's logits
    const float4 a = *reinterpret_cast<const float4*>(row.run() + i), b = *reinterpret_cast<const float4*>(row.run() + i + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  };
  const uint32_t hist = smem_u32(rs.hist), spill = smem_u32(rs.spill) + (uint32_t)lane * 4u;
  // No branch: what lies below the first bin counts in a word of its lane.  Both ends are tested (as unsigned): no value,
  // whatever its bits, may form an address beyond the bins.
  auto count = [&](float v) {
    const uint32_t b = (uint32_t)bits_of(v) - __float_as_uint(kRMagic);
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(b < (uint32_t)kResBins ? hist + 4u * b : spill) : "memory");
  };
  const int n_mine = row.end - row.beg;
#pragma unroll 1
  for (int i = 0; i < n_mine; i += 8) {
    float v[8];
    eight(i, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) count(v[j]);
  }
  __syncthreads();
  unsigned over = 0;
  int in_bin = 0;
  const int bin = res_crossing(rs, (unsigned)top_k, over, in_bin);
  if (bin < 0 || in_bin > kResMembers) {   // (uniform)
    __syncthreads();
    return res_refine(row, top_k, mx, rs);
  }
  const int want_bits = bin + __float_as_int(kRMagic);
  auto aside = [&](float v) { rs.sa[atomicAdd(&rs.n_sa, 1u)] = v; };
#pragma unroll 1
  for (int i = 0; i < n_mine; i += 8) {
    float v[8];
    eight(i, v);
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) m |= bits_of(v[j]) == want_bits ? 1u << j : 0u;
#pragma unroll 1
    for (; m; m &= m - 1u) aside(row.run()[i + __ffs(m) - 1]);
  }
  __syncthreads();
  return res_rank(rs, in_bin, (unsigned)top_k - over);
}

// Logits -> weights in place; returns the scan of the threads' sums (total = partition sum).  With a threshold most
// entries are zero: a thread marks those it keeps and exponentiates only them.  Every weight goes into a double by itself:
// partial sums in fp32, even of eight, show in Z (relative error of Z_q, 512 draft rows of 264 to 49152 ids: at most 3.3e-8 so,
// 1.8e-7 with them).
__device__ __forceinline__ ResSums res_weigh(const ResRow& row, float theta, float m, ResScratch& rs, int& calls) {
  float* const z = row.run();
  const int n = row.end - row.beg;
  double acc = 0.0;
  if (theta > -INFINITY) {   // uniform
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32) {
      uint32_t keep = 0;
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        if (i0 + i < n) {
          float4 a = *reinterpret_cast<float4*>(z + i0 + i);
          if (a.x >= theta) keep |= 1u << i;
          else a.x = 0.f;
          if (a.y >= theta) keep |= 2u << i;
          else a.y = 0.f;
          if (a.z >= theta) keep |= 4u << i;
          else a.z = 0.f;
          if (a.w >= theta) keep |= 8u << i;
          else a.w = 0.f;
          *reinterpret_cast<float4*>(z + i0 + i) = a;
        }
#pragma unroll 1
      for (; keep; keep &= keep - 1u) {
        float* const p = z + i0 + __ffs(keep) - 1;
        const float e = expf(__fsub_rn(*p, m));
        *p = e;
        acc += (double)e;
      }
    }
  } else {
#pragma unroll 1
    for (int i = 0; i < n; i += 8) {
      float4 a = *reinterpret_cast<float4*>(z + i), b = *reinterpret_cast<float4*>(z + i + 4);
      a = make_float4(expf(__fsub_rn(a.x, m)), expf(__fsub_rn(a.y, m)), expf(__fsub_rn(a.z, m)), expf(__fsub_rn(a.w, m)));
      b = make_float4(expf(__fsub_rn(b.x, m)), expf(__fsub_rn(b.y, m)), expf(__fsub_rn(b.z, m)), expf(__fsub_rn(b.w, m)));
      *reinterpret_cast<float4*>(z + i) = a;
      *reinterpret_cast<float4*>(z + i + 4) = b;
      acc += (((double)a.x + (double)a.y) + ((double)a.z + (double)a.w)) + (((double)b.x + (double)b.y) + ((double)b.z + (double)b.w));
    }
  }
  return res_scan(acc, rs, calls);
}

// The draw of u over per-thread sums `s` of weight(x): the owner's warp walks the owner's run, 32 ids at a time, and
// one lane writes the token to *out (shared memory).  No barrier.
template <class Weight>
__device__ inline void res_pick(const ResRow& row, const ResSums& s, double u, Weight weight, int* out) {
  const int lane = threadIdx.x & 31;
  const double y = u * s.total;
  const unsigned own = __ballot_sync(kFull, s.before <= y && y < s.incl);
  if (!own) return;   // warp-uniform
  const int src = __ffs(own) - 1;
  const int x_beg = __shfl_sync(kFull, row.beg, src), x_end = __shfl_sync(kFull, row.end, src);
  double c = __shfl_sync(kFull, s.before, src);
  int pick = -1, last = -1;
  for (int x0 = x_beg; x0 < x_end && pick < 0; x0 += 32) {
    const int x = x0 + lane;
    const double w = x < x_end ? weight(x) : 0.0;
    double run = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double n = __shfl_up_sync(kFull, run, o);
      if (lane >= o) run += n;
    }
    const unsigned has = __ballot_sync(kFull, w > 0.0), hit = __ballot_sync(kFull, w > 0.0 && c + run > y);
    if (has) last = x0 + 31 - __clz(has);
    if (hit) pick = x0 + __ffs(hit) - 1;
    c += __shfl_sync(kFull, run, 31);
  }
  if (lane == 0) *out = pick >= 0 ? pick : last >= 0 ? last : x_beg;   // (rounding: the last id with weight)
}

// Statistics of a row (threshold, maximum, partition sum); the row's weights stay in shared memory.
__device__ inline ResSums res_row_stats(const ResRow& row, const RowSrc& src, int top_k, ResScratch& rs, int& calls,
                                        int tok, float& z_tok, RowStats& st) {
  float mx, mean;
  res_load(row, src, rs, mx, mean);
  z_tok = tok >= 0 ? row.at(tok) : 0.f;   // (before the logits become weights)
  st.m = mx;
  st.theta = -INFINITY;
  if (top_k > 0 && top_k < row.V) st.theta = res_select(row, top_k, mx, mean, rs);
  else __syncthreads();                   // everybody has z_tok
  const ResSums s = res_weigh(row, st.theta, mx, rs, calls);
  st.Z = s.total;
  return s;
}

// Everything for one target position on resident rows; arguments as dense_position's, whose results it gives.
template <class WantDraws>
__device__ inline void res_position(const DevParams& P, const ResRow& row, const RowSrc& tr, const RowSrc& qr,
                                    const RowStats& sq, int tok, const uint16_t* nn, uint32_t image, uint32_t position,
                                    bool decide, int given_accept, WantDraws want, ResScratch& rs, int& calls,
                                    uint32_t* dev_status, PositionOut& out) {
  float zq_tok = 0.f;
  if (threadIdx.x == 0) zq_tok = load1(qr, tok);   // asked for now, used after the row's statistics
  RowStats sp;
  float z_tok;
  ResSums sums = res_row_stats(row, tr, P.top_k, rs, calls, tok, z_tok, sp);
  const float invZp = (float)(1.0 / sp.Z), invZq = (float)(1.0 / sq.Z);
  if (threadIdx.x == 0) {
    const double p = (z_tok >= sp.theta) ? exp((double)z_tok - (double)sp.m) / sp.Z : 0.0;
    const double q = (zq_tok >= sq.theta) ? exp((double)zq_tok - (double)sq.m) / sq.Z : 0.0;
    rs.bd[0] = p;
    rs.bd[1] = q;
    rs.first_bad = P.pool_k - 1;
    if (q <= 0.0) atomicOr(dev_status, MULO_DEV_ZERO_DRAFT_PROB);
  }
  __syncthreads();
  const double p_tok = rs.bd[0], q_tok = rs.bd[1];
  double mass = p_tok;
  bool moved = false;   // the resident weights were changed (pooling)
  if (P.pool_k > 1) {
    // Eq. 3-4: the leading run of the neighbour list whose prefix mass stays below delta; four entries per thread
    // (the list has at most 2047), one block scan
    const uint16_t* const list = nn + (size_t)tok * P.pool_k;
    const int nb = P.pool_k - 1, per = (nb + kThreads - 1) / kThreads, j0 = (int)threadIdx.x * per;
    double pj[4], mine = 0.0;
    int id[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      pj[i] = 0.0;
      id[i] = -1;
      if (i < per && j0 + i < nb) {
        id[i] = list[j0 + i + 1];
        if (id[i] >= P.V) {
          atomicOr(dev_status, MULO_DEV_BAD_TOKEN);
          id[i] = P.V - 1;
        }
        pj[i] = (double)row.at(id[i]) / sp.Z;
        mine += pj[i];
      }
    }
    const ResSums c = res_scan(mine, rs, calls);
    {
      double run = c.before;
      int bad = nb;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (id[i] >= 0) {
          run += pj[i];
          if (bad == nb && !(run < P.pool_delta)) bad = j0 + i;
        }
      if (bad < nb) atomicMin(&rs.first_bad, bad);
    }
    __syncthreads();
    const int J = rs.first_bad;
    if (J > 0 && (J - 1) / per == (int)threadIdx.x) {
      double run = c.before;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (id[i] >= 0 && j0 + i < J) run += pj[i];
      rs.bd[2] = run;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (id[i] >= 0 && j0 + i < J) row.at(id[i]) = 0.f;   // the pooled ids leave the row
    moved = J > 0;
    __syncthreads();
    if (moved) mass = p_tok + rs.bd[2];
  }

  // acceptance (Eq. 1 / Eq. 5)
  const uint4 rnd = philox4x32_10(make_uint4(position, image, P.round, 0u), make_uint2(P.seed_lo, P.seed_hi));
  double thr;
  int accepted;
  if (P.accept_mode == MULO_ACCEPT_THRESHOLD) {
    thr = mass;
    accepted = mass >= P.tau;
  } else {
    if (q_tok <= 0.0) thr = mass > 0.0 ? 1.0 : 0.0;
    else thr = fmin(1.0, mass / q_tok);
    accepted = uniform24(rnd.x) < thr;
  }
  if (!decide) accepted = given_accept;

  // draws: weights max(0, p' - lambda q) with x~'s own taken in double
  const int draws = want(accepted);
  if (threadIdx.x < 2) rs.tok[threadIdx.x] = -1;
  const bool own_tok = tok >= row.beg && tok < row.end;
  auto target = [&](int x) -> double { return x == tok ? mass * sp.Z : (double)row.at(x); };
  bool have_target = !moved;   // `sums` are those of the target weights
  auto target_draw = [&](double u, int* to) {
    if (!have_target) {
      const float* const w = row.run();
      double acc = 0.0;
      for (int i = 0; i < row.end - row.beg; i += 4) {
        const float4 a = *reinterpret_cast<const float4*>(w + i);
        acc += ((double)a.x + (double)a.y) + ((double)a.z + (double)a.w);
      }
      if (own_tok) acc += mass * sp.Z - (double)row.at(tok);
      sums = res_scan(fmax(acc, 0.0), rs, calls);
      have_target = true;
    } else {
      __syncthreads();   // rs.tok
    }
    if (sums.total > 0.0) res_pick(row, sums, u, target, to);
  };
  if (draws & kDrawResidual) {
    auto residual = [&](int x) -> double {
      if (x == tok) return fmax(0.0, mass - q_tok);
      const float q = prob_f(load1(qr, x), sq.theta, sq.m, invZq);
      return (double)fmaxf(__fsub_rn(__fmul_rn(row.at(x), invZp), q), 0.f);
    };
    const float* const w = row.run();
    double acc = 0.0;
#pragma unroll 1
    for (int x = row.beg; x < row.end; x += 8) {
      float zq[8];
      load8(qr, x, zq);
      const float4 a = *reinterpret_cast<const float4*>(w + x - row.beg), b = *reinterpret_cast<const float4*>(w + x - row.beg + 4);
      const float e[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float q = prob_f(zq[j], sq.theta, sq.m, invZq);
        acc += x + j == tok ? 0.0 : (double)fmaxf(__fsub_rn(__fmul_rn(e[j], invZp), q), 0.f);
      }
    }
    if (own_tok) acc += fmax(0.0, mass - q_tok);
    const ResSums r = res_scan(acc, rs, calls);
    if (r.total > 0.0) res_pick(row, r, uniform24(rnd.y), residual, &rs.tok[0]);
    else target_draw(uniform24(rnd.y), &rs.tok[0]);   // a residual without mass: the lambda = 0 weights, same uniform
  }
  if (draws & kDrawTarget) target_draw(uniform24(rnd.z), &rs.tok[1]);
  __syncthreads();
  out.p_tok = (float)p_tok;
  out.q_tok = (float)q_tok;
  out.accept_prob = (float)thr;
  out.accepted = accepted;
  out.tok_residual = rs.tok[0];
  out.tok_target = rs.tok[1];
}

}  // namespace mulo
