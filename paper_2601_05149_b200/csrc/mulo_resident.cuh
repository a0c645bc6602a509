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
// bf16 ids with guidance on one CTA; this takes REDRAW_US us.
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
  double scan[2][kWarps];       // block scans; consecutive ones alternate
  float red[2][kWarps][3];      // block maxima, minima, sums
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
  __device__ ResRow(float* smem, int V_) : w(smem), V(V_), E(resident_run(V_)) {
    beg = min(V, (int)threadIdx.x * E);
    end = min(V, beg + E);
  }
  __device__ __forceinline__ float* run() const { return w + threadIdx.x * (E + 4); }
  __device__ __forceinline__ float& at(int x) const {
    const int o = x / E;
    return w[o * (E + 4) + x - o * E];
  }
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

// The row from global memory into shared memory; every thread gets the row's maximum, minimum and mean.
__device__ inline void res_load(const ResRow& row, const RowSrc& src, ResScratch& rs, float& mx, float& mn, float& mean) {
  float hi = -INFINITY, lo = INFINITY, sum = 0.f;
#pragma unroll 2
  for (int x = (int)threadIdx.x * 8; x < row.V; x += 8 * kThreads) {
    float z[8];
    load8<true>(src, x, z);
    const int o = x / row.E;
    float4* const to = reinterpret_cast<float4*>(row.w + o * (row.E + 4) + x - o * row.E);
    to[0] = make_float4(z[0], z[1], z[2], z[3]);
    to[1] = make_float4(z[4], z[5], z[6], z[7]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      hi = fmaxf(hi, z[j]);
      lo = fminf(lo, z[j]);
      sum += z[j];
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
    lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
    sum += __shfl_xor_sync(kFull, sum, o);
  }
  if (lane == 0) {
    rs.red[0][warp][0] = hi;
    rs.red[0][warp][1] = lo;
    rs.red[0][warp][2] = sum;
  }
  if (threadIdx.x == 0) rs.n_sa = 0;
#pragma unroll
  for (int i = 0; i < kResBins / kThreads; ++i) rs.hist[threadIdx.x + i * kThreads] = 0;
  __syncthreads();
  hi = rs.red[0][lane & (kWarps - 1)][0];
  lo = rs.red[0][lane & (kWarps - 1)][1];
  sum = rs.red[0][lane & (kWarps - 1)][2];
#pragma unroll
  for (int o = kWarps / 2; o > 0; o >>= 1) {
    hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
    lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
    sum += __shfl_xor_sync(kFull, sum, o);
  }
  mx = hi;
  mn = lo;
  mean = sum / (float)row.V;
}

// The top_k-th largest value of the resident row (1 <= top_k < V).  The map z -> bin is monotone, so the crossing
// bin's entries are consecutive in rank whatever the rounding.
__device__ inline float res_select(const ResRow& row, int top_k, float mx, float mn, float mean, ResScratch& rs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float zlo = mean > mn && mean < mx ? mean : mn, zhi = mx;
  int above = 0;   // entries above zhi
  for (;;) {
    if (!(zlo < zhi)) {   // one value left (uniform)
      __syncthreads();
      return zhi;
    }
    const float sc = (float)(kResBins - 1) / (zhi - zlo);
    auto bin_of = [&](float v) -> int { return min((int)__fmul_rn(__fsub_rn(v, zlo), sc), kResBins - 1); };
    const float* const z = row.run();
#pragma unroll 1
    for (int i = 0; i < row.end - row.beg; i += 4) {
      const float4 q = *reinterpret_cast<const float4*>(z + i);
      const float v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v[j] >= zlo && v[j] <= zhi) atomicAdd(&rs.hist[bin_of(v[j])], 1u);
    }
    __syncthreads();
    // the crossing bin, from the top: every warp finds it (32 bins per lane, lane 0 the highest)
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
    const unsigned want = (unsigned)(top_k - above);   // rank from the top within [zlo, zhi]
    const unsigned hit = __ballot_sync(kFull, inc >= want);
    if (hit == 0) {   // (fewer than top_k entries reach the mean)
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kResBins / kThreads; ++i) rs.hist[threadIdx.x + i * kThreads] = 0;
      __syncthreads();
      zlo = mn;
      continue;
    }
    const int src = __ffs(hit) - 1;
    unsigned over = __shfl_sync(kFull, inc - mine, src);
    const unsigned h = rs.hist[(31 - src) * 32 + 31 - lane];
    inc = h;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += t;
    }
    const int k = __ffs(__ballot_sync(kFull, over + inc >= want)) - 1;
    const int bin = (31 - src) * 32 + 31 - k;
    const int in_bin = (int)__shfl_sync(kFull, h, k);
    over += __shfl_sync(kFull, inc - h, k);
    // its entries: set aside if few, else their range for the next histogram
    float vhi = -INFINITY, vlo = INFINITY;
#pragma unroll 1
    for (int i = 0; i < row.end - row.beg; i += 4) {
      const float4 q = *reinterpret_cast<const float4*>(z + i);
      const float v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (v[j] >= zlo && v[j] <= zhi && bin_of(v[j]) == bin) {
          if (in_bin <= kResMembers) rs.sa[atomicAdd(&rs.n_sa, 1u)] = v[j];
          vhi = fmaxf(vhi, v[j]);
          vlo = fminf(vlo, v[j]);
        }
    }
    if (in_bin <= kResMembers) {
      __syncthreads();
      const unsigned r = want - over;   // rank from the top within the bin
      float th = 0.f;
      bool found = false;
      for (int i = lane; i < in_bin; i += 32) {
        const float vi = rs.sa[i];
        unsigned more = 0, geq = 0;
        for (int j = 0; j < in_bin; ++j) {
          const float vj = rs.sa[j];
          more += vj > vi;
          geq += vj >= vi;
        }
        if (more < r && r <= geq) {
          th = vi;
          found = true;
        }
      }
      return __shfl_sync(kFull, th, __ffs(__ballot_sync(kFull, found)) - 1);   // (found: the bin holds the rank)
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      vhi = fmaxf(vhi, __shfl_xor_sync(kFull, vhi, o));
      vlo = fminf(vlo, __shfl_xor_sync(kFull, vlo, o));
    }
    if (lane == 0) {
      rs.red[1][warp][0] = vhi;
      rs.red[1][warp][1] = vlo;
    }
    __syncthreads();   // (also: everybody is done with the histogram)
#pragma unroll
    for (int i = 0; i < kResBins / kThreads; ++i) rs.hist[threadIdx.x + i * kThreads] = 0;
    vhi = rs.red[1][lane & (kWarps - 1)][0];
    vlo = rs.red[1][lane & (kWarps - 1)][1];
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) {
      vhi = fmaxf(vhi, __shfl_xor_sync(kFull, vhi, o));
      vlo = fminf(vlo, __shfl_xor_sync(kFull, vlo, o));
    }
    zhi = vhi;
    zlo = vlo;
    above += (int)over;
    __syncthreads();
  }
}

// Logits -> weights in place; returns the scan of the threads' sums (total = partition sum).
__device__ inline ResSums res_weigh(const ResRow& row, float theta, float m, ResScratch& rs, int& calls) {
  float* const z = row.run();
  double acc = 0.0;
#pragma unroll 1
  for (int i = 0; i < row.end - row.beg; i += 8) {
    float4 a = *reinterpret_cast<float4*>(z + i), b = *reinterpret_cast<float4*>(z + i + 4);
    auto weigh = [&](float v) -> float {
      const float e = expf(__fsub_rn(v, m));
      return v >= theta ? e : 0.f;
    };
    a = make_float4(weigh(a.x), weigh(a.y), weigh(a.z), weigh(a.w));
    b = make_float4(weigh(b.x), weigh(b.y), weigh(b.z), weigh(b.w));
    *reinterpret_cast<float4*>(z + i) = a;
    *reinterpret_cast<float4*>(z + i + 4) = b;
    acc += (double)(((a.x + a.y) + (a.z + a.w)) + ((b.x + b.y) + (b.z + b.w)));
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
  float mx, mn, mean;
  res_load(row, src, rs, mx, mn, mean);
  z_tok = tok >= 0 ? row.at(tok) : 0.f;   // (before the logits become weights)
  st.m = mx;
  st.theta = -INFINITY;
  if (top_k > 0 && top_k < row.V) st.theta = res_select(row, top_k, mx, mn, mean, rs);
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
        acc += (double)((a.x + a.y) + (a.z + a.w));
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
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float q = prob_f(zq[j], sq.theta, sq.m, invZq);
        s += x + j == tok ? 0.f : fmaxf(__fsub_rn(__fmul_rn(e[j], invZp), q), 0.f);
      }
      acc += (double)s;
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
