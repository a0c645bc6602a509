// One sequential step of the redraw of R_X (Sec. 3.4, Algorithm 1 Step 6): every position of the step's slice of the list
// draws its token from the target distribution of the given logits.
//
// Steps follow one another by the thousand with a handful of positions each, so a step is bound by the latency of ONE row.
// A row's ids stay in the registers of a cluster of up to four CTAs of 512 threads, eight ids per thread up to V = 16384:
//
//   load       128-bit loads, mixed at once
//   select     a histogram of 4096 bins over the upper bits of the values as they are (the sign, sixteen binary orders of
//              magnitude, seven bits of the mantissa), so nothing about the row needs to be known before; one block scan finds
//              the bin that holds the k-th largest.  A bin of more than 128 entries is split again, by key ranges.  CTAs of a
//              cluster write their 16-bit counts into one another's shared memory and go on by themselves.
//   weigh      exp(z - max) of what lies above the bin, summed in double per warp; the bin's entries are ranked (shared out
//              over the warps); every warp has the warps' weights scanned in id order, and the one that owns u * total walks
//              its ids.
//
// The launch may begin while the kernels before it in the stream still run (programmatic dependent launch).  The first row of
// a cluster is drawn BEFORE it waits for them, from the list and the logits as they are at that moment; after the wait both are
// read again, and the token counts only if every logit mixes to the same value as before and the list names the same
// position -- otherwise the row is drawn again from what is there now.  So a step costs its successor a re-read instead of
// the whole chain.  Before the wait anything may be rewritten at any moment: ONE thread of the cluster reads the list and tells
// the others what it found, and every later verdict is one for the whole cluster, so no barrier is ever met by a part of it.
// Where another kernel runs between two steps nothing overlaps, and drawing ahead only costs (the agreement before the row, the
// re-read after it: 2.5 us).  64 x 64, 4 images, V = 16384, window 16: 4.7 us a step back to back, 13.3 with a copy of 1.3 us between any
// two; without drawing ahead 9.9 and 10.5.
//
// A step with more positions than clusters is bound by their number instead: after the wait every CTA takes whole rows for itself, by
// the resident routines, two CTAs to an SM.
#pragma once

#include "mulo_resident.cuh"

namespace mulo {

constexpr int kRedrawBins = 4096;        // two 16-bit counts to a word: a CTA has at most 16384 ids of a row
constexpr int kRedrawWords = kRedrawBins / 2;
constexpr int kRedrawMembers = 128;      // entries of the crossing bin that are ranked
constexpr int kRedrawMaxCtas = 4;        // CTAs per row
constexpr int kRedrawIds = 8 * kThreads; // ids of a CTA per piece

struct RedrawArgs {
  DevParams P;
  int single;              // a step of more positions than clusters: every CTA draws rows of its own
  const char* cond;
  const char* uncond;
  const int32_t* pos_list;
  const int32_t* offsets;
  int32_t* out_tok;
  int s;
};

struct RedrawSmem {
  double w_sum[kRedrawMaxCtas * kWarps];      // weight above the crossing bin, per warp of the cluster
  double m_sum[kRedrawMaxCtas * kWarps];      // ... of the crossing bin's kept entries
  uint2 member[kRedrawMembers];               // value, warp
  uint32_t w_max[kRedrawMaxCtas * kWarps];
  uint32_t tot[kWarps];
  uint32_t same[kRedrawMaxCtas];
  uint2 ahead;                                // the list's start and the row to draw before the wait, as one thread found them
  int bin, in_bin;
  unsigned over, n_member;
  float theta;
};

// a 4-byte load that is neither taken from the read-only cache nor moved
__device__ __forceinline__ int ld_fresh(const int32_t* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ---- a peer's shared memory, and the cluster's barrier
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_peer(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, uint2 v) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, uint4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The first histogram: eight bits of exponent held to [2^-5, 2^11) and seven of the mantissa; values from +0 up in bins 0 to
// 2047, from -0 down in 4095 to 2048.
constexpr int kRedrawLow = (127 - 5) << 7;
__device__ __forceinline__ int redraw_bin(float z) {
  const uint32_t bits = __float_as_uint(z);
  const int b = min(max((int)(bits >> 16 & 0x7fffu) - kRedrawLow, 0), kRedrawBins / 2 - 1);
  return b ^ ((int32_t)bits >> 31 & (kRedrawBins - 1));
}
// The first and last key of a bin.
__device__ __forceinline__ void redraw_range(int bin, uint32_t& lo, uint32_t& hi) {
  const bool neg = bin >= kRedrawBins / 2;
  const int b = neg ? kRedrawBins - 1 - bin : bin;
  const uint32_t m0 = b == 0 ? 0u : (uint32_t)(b + kRedrawLow) << 16;
  const uint32_t m1 = b == kRedrawBins / 2 - 1 ? 0x7fffffffu : ((uint32_t)(b + 1 + kRedrawLow) << 16) - 1u;
  lo = neg ? 0x7fffffffu - m1 : 0x80000000u + m0;
  hi = neg ? 0x7fffffffu - m0 : 0x80000000u + m1;
}

// NP: pieces of eight ids per thread.  A cluster of `ctas` CTAs holds ctas * NP * 4096 >= V ids; a warp's are consecutive.
template <bool BF16, int NP>
__global__ void __launch_bounds__(kThreads, NP == 4 ? 1 : 2) k_redraw_step(const __grid_constant__ RedrawArgs a) {
  extern __shared__ __align__(128) unsigned char dyn[];   // [ctas][kRedrawWords]: every CTA's counts, one's own at its rank; or a whole row
  __shared__ RedrawSmem sm;
  __shared__ typename std::conditional<NP < 4, ResScratch, int>::type rs;   // (rows drawn by one CTA)
  const DevParams& P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t rank, ctas;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(ctas));
  let_next_begin();
  const int cluster = (int)(blockIdx.x / ctas), clusters = (int)(gridDim.x / ctas);
  const uint32_t N = (uint32_t)P.H * (uint32_t)P.W, total = (uint32_t)P.B * N;   // (positions fit 31 bits)
  const uint32_t bytes = (uint32_t)P.V * (BF16 ? 2u : 4u);
  uint32_t* const copies = reinterpret_cast<uint32_t*>(dyn);
  uint32_t* const hist = copies + rank * kRedrawWords;
  const bool cut = P.top_k > 0;
  const int my_warp = (int)rank * kWarps + warp, n_warps = (int)ctas * kWarps;
  const int x0 = my_warp * (NP * 256) + lane * 8;        // piece j: eight ids from x0 + 256 j on
  auto meet = [&]() {                                    // all threads of the cluster
    if (ctas == 1) __syncthreads();
    else cluster_meet();
  };

  // what the step will find, if the list stays as it is
  uint2 found = make_uint2(0u, total);
  if (tid == 0) {
    const int beg = ld_fresh(a.offsets + a.s), end = ld_fresh(a.offsets + a.s + 1);
    const bool many = a.single && (long long)end - beg > clusters;
    const long long at = (long long)beg + cluster + (many ? (int)rank * clusters : 0);
    if (beg >= 0 && at < end && at < (long long)total && (many || rank == 0)) {
      const uint32_t row = (uint32_t)ld_fresh(a.pos_list + at);
      if (!many) {
        found = make_uint2((uint32_t)beg, row);
      } else if (row < total) {   // (a hint, nothing else: no row is drawn ahead)
        prefetch_l2(a.cond + (size_t)row * bytes, bytes);
        if (a.uncond) prefetch_l2(a.uncond + (size_t)row * bytes, bytes);
      }
    }
    sm.ahead = found;
  }
  auto clear = [&]() {
    reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < n_warps) sm.m_sum[tid] = 0.0;
    if (tid == 0) sm.n_member = 0;
  };
  static_assert(kRedrawWords == 4 * kThreads && kRedrawMaxCtas * kWarps <= kThreads, "one 16-byte word per thread");
  clear();
  RowSrc src;
  src.s = P.cfg_scale;
  src.invT = P.invT;
  // A row's ids of this thread, piece by piece (F of them are asked for before any is used).  -0 and, under a cut, what is no
  // number (it counts as below every other) leave here.
  constexpr int F = BF16 || NP < 4 ? NP : NP / 2;
  auto load = [&](uint32_t row, auto take) {
    src.cond = a.cond + (size_t)row * bytes;
    src.uncond = a.uncond ? a.uncond + (size_t)row * bytes : nullptr;
#pragma unroll
    for (int f = 0; f < NP; f += F) {
      raw_piece<BF16> c[F], u[F] = {};
#pragma unroll
      for (int j = 0; j < F; ++j)
        if (x0 + 256 * (f + j) < P.V) ask8<BF16>(src, x0 + 256 * (f + j), c[j], u[j]);
#pragma unroll
      for (int j = 0; j < F; ++j) {
        float v[8];
        if (x0 + 256 * (f + j) < P.V) {
          res_mix<BF16>(src, c[j], u[j], v);
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = __fadd_rn(cut ? fmaxf(v[k], -INFINITY) : v[k], 0.f);
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = -INFINITY;
        }
        take(f + j, v);
      }
    }
  };
  auto uniform_of = [&](uint32_t at) -> double {
    const uint32_t b = at / N, t = at - b * N;
    return uniform24(philox4x32_10(make_uint4(t, b + P.image_offset, P.round, 1u + (uint32_t)a.s), make_uint2(P.seed_lo, P.seed_hi)).x);
  };
  meet();   // (the peers run, everybody's memory is cleared)
  if (ctas > 1) {
    if (rank == 0 && tid == 0)
      for (uint32_t q = 1; q < ctas; ++q) st_peer(peer_addr(smem_u32(&sm.ahead), q), found);
    meet();
  }
  const uint32_t beg0 = sm.ahead.x;
  uint32_t g = sm.ahead.y;
  bool waited = g >= total;
  int i = 0, end = 0;
  bool single = false;
  auto look = [&]() {   // after the wait: the same in every CTA
    wait_for_previous();
    i = ld_fresh(a.offsets + a.s);
    end = ld_fresh(a.offsets + a.s + 1);
    single = a.single && end - i > clusters;
  };
  if (waited) {
    look();
    i += cluster;
  }
  bool used = false;   // the shared memory, by a row before
#pragma unroll 1
  for (;;) {   // (what decides here is the same in every CTA of the cluster)
    if (waited) {
      if (single || i >= end) break;
      g = (uint32_t)ld_fresh(a.pos_list + i);
      if (g >= total) {
        i += clusters;
        continue;
      }
    }
    if (used) {
      meet();
      clear();
      meet();
    }
    used = true;
    // ---- the ids; the row's maximum; counts
    float z[NP][8];
    float mx = -INFINITY;
    load(g, [&](int j, const float (&v)[8]) {
#pragma unroll
      for (int k = 0; k < 8; ++k) z[j][k] = v[k];
    });
#pragma unroll
    for (int j = 0; j < NP; ++j) {
#pragma unroll
      for (int k = 0; k < 8; ++k) mx = fmaxf(mx, z[j][k]);
      if (cut && x0 + 256 * j < P.V) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int b = redraw_bin(z[j][k]);
          atomicAdd(&hist[b >> 1], 1u << ((b & 1) * 16));
        }
      }
    }
    const unsigned mk = __reduce_max_sync(kFull, float_key(mx));
    if (ctas == 1) {
      if (lane == 0) sm.w_max[warp] = mk;
    } else if (lane < (int)ctas) {
      st_peer(peer_addr(smem_u32(&sm.w_max[my_warp]), lane), mk);
    }
    // counts to the peers, and the cluster's barrier
    auto exchange = [&]() {
      if (cut && ctas > 1) {
        __syncthreads();
        const uint4 v = reinterpret_cast<const uint4*>(hist)[tid];
        const uint32_t at = smem_u32(hist) + (uint32_t)tid * 16u;
#pragma unroll 1
        for (uint32_t q = 0; q < ctas; ++q)
          if (q != rank) st_peer(peer_addr(at, q), v);
      }
      meet();
    };
    exchange();
    unsigned mk_all = 0;
    for (int w = lane; w < n_warps; w += 32) mk_all = max(mk_all, sm.w_max[w]);
    const float m = key_float(__reduce_max_sync(kFull, mk_all));

    // ---- the bin that holds the k-th largest: values from lo to hi, `above` ids beyond it, n_in in it
    float lo = -INFINITY, hi = -INFINITY;
    int n_in = 0;
    unsigned above = 0;
    if (cut) {
      // rank `want` from the top; a thread has the eight bins from 8 `block` on, thread 0 the highest
      auto crossing = [&](unsigned want, int block) {
        unsigned n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
        for (uint32_t q = 0; q < ctas; ++q) {
          const uint4 v = reinterpret_cast<const uint4*>(copies + q * kRedrawWords)[block];
          n[0] += v.x & 0xffffu; n[1] += v.x >> 16;
          n[2] += v.y & 0xffffu; n[3] += v.y >> 16;
          n[4] += v.z & 0xffffu; n[5] += v.z >> 16;
          n[6] += v.w & 0xffffu; n[7] += v.w >> 16;
        }
        const unsigned own = ((n[0] + n[1]) + (n[2] + n[3])) + ((n[4] + n[5]) + (n[6] + n[7]));
        unsigned inc = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned t = __shfl_up_sync(kFull, inc, o);
          if (lane >= o) inc += t;
        }
        if (lane == 31) sm.tot[warp] = inc;
        __syncthreads();
        unsigned run = __reduce_add_sync(kFull, lane < warp ? sm.tot[lane & (kWarps - 1)] : 0u) + inc - own;
        if (run < want && want <= run + own) {
#pragma unroll
          for (int k = 7; k >= 0; --k) {
            if (run < want && want <= run + n[k]) {
              sm.bin = block * 8 + k;
              sm.over = run;
              sm.in_bin = (int)n[k];
            }
            run += n[k];
          }
        }
        __syncthreads();
      };
      crossing((unsigned)P.top_k, (kThreads / 2 - 1 - tid) & (kThreads - 1));
      int bin = sm.bin;   // (always found: every id is counted)
      uint32_t klo, khi;
      redraw_range(bin, klo, khi);
      n_in = sm.in_bin;
      above = sm.over;
      // (Entries of a bin are weighed in any order, so its sums in double have to be exact: 128 weights of 24 bits that lie within
      // a factor of e^15 of one another.  The bins at the ends of the first histogram have no such bound, nor have ranges of
      // keys far out.)
      auto wide = [&]() { return !(key_float(khi) - key_float(klo) <= 15.0f); };
#pragma unroll 1
      while ((n_in > kRedrawMembers || wide()) && klo != khi) {   // a crowded or wide bin is split again
        meet();   // (everybody has read the counts)
        reinterpret_cast<uint4*>(hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        const int shift = max(0, 20 - __clz(khi - klo));
#pragma unroll
        for (int j = 0; j < NP; ++j)
          if (x0 + 256 * j < P.V) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint32_t key = float_key(z[j][k]);
              if (key >= klo && key <= khi) {
                const int b = (int)((key - klo) >> shift);
                atomicAdd(&hist[b >> 1], 1u << ((b & 1) * 16));
              }
            }
          }
        exchange();
        crossing((unsigned)P.top_k - above, kThreads - 1 - tid);
        bin = sm.bin;
        klo += (uint32_t)bin << shift;
        khi = min(khi, klo + ((1u << shift) - 1u));
        n_in = sm.in_bin;
        above += sm.over;
      }
      // as values (none of the row's is -0; the bins at the ends hold keys that are no numbers)
      lo = klo < float_key(-INFINITY) ? -INFINITY : key_float(klo);
      hi = khi > float_key(INFINITY) ? INFINITY : khi == 0x7fffffffu ? key_float(khi - 1u) : key_float(khi);
      if (n_in <= kRedrawMembers) {
        // the bin's entries to every CTA, one CTA's behind the other's
        int at0 = 0;
#pragma unroll 1
        for (uint32_t q = 0; q < rank; ++q) at0 += (int)(copies[q * kRedrawWords + (bin >> 1)] >> ((bin & 1) * 16) & 0xffffu);
#pragma unroll
        for (int j = 0; j < NP; ++j)
          if (x0 + 256 * j < P.V) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (z[j][k] >= lo && z[j][k] <= hi) {
                const int at = (at0 + (int)atomicAdd(&sm.n_member, 1u)) & (kRedrawMembers - 1);
                const uint2 e = make_uint2(__float_as_uint(z[j][k]), (uint32_t)my_warp);
                if (ctas == 1) {
                  sm.member[at] = e;
                } else {
#pragma unroll 1
                  for (uint32_t q = 0; q < ctas; ++q) st_peer(peer_addr(smem_u32(&sm.member[at]), q), e);
                }
              }
          }
      } else {
        n_in = 0;   // all of them the same value: the threshold, and all are kept
        // (below +0 comes the largest negative value, not -0; below -inf comes no number)
        hi = klo <= float_key(-INFINITY) ? -INFINITY : key_float(klo == 0x80000000u ? klo - 2u : klo - 1u);
      }
    }
    // ---- weights of what lies above the bin (every weight goes into a double by itself)
    auto weight = [&](float v) -> float { return expf(__fsub_rn(v, m)); };
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j)
      if (x0 + 256 * j < P.V) {
        float w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = !cut || z[j][k] > hi ? weight(z[j][k]) : 0.f;
        acc += (((double)w[0] + (double)w[1]) + ((double)w[2] + (double)w[3])) +
               (((double)w[4] + (double)w[5]) + ((double)w[6] + (double)w[7]));
      }
    acc = warp_sum(acc);
    if (ctas == 1) {
      if (lane == 0) sm.w_sum[warp] = acc;
    } else if (lane < (int)ctas) {
      st_peer(peer_addr(smem_u32(&sm.w_sum[my_warp]), lane), acc);
    }
    meet();
    // ---- the threshold among the bin's entries; what is kept of them, per warp of the cluster
    float theta = INFINITY;
    if (n_in > 0) {
      float v[kRedrawMembers / 32];
#pragma unroll
      for (int q = 0; q < kRedrawMembers / 32; ++q) v[q] = lane + 32 * q < n_in ? __uint_as_float(sm.member[lane + 32 * q].x) : NAN;
      const int want = P.top_k - (int)above;
#pragma unroll 1
      for (int j = warp; j < n_in; j += kWarps) {
        const float vj = __uint_as_float(sm.member[j].x);
        int more = 0, geq = 0;
#pragma unroll
        for (int q = 0; q < kRedrawMembers / 32; ++q)
          if (32 * q < n_in) {
            more += __popc(__ballot_sync(kFull, v[q] > vj));
            geq += __popc(__ballot_sync(kFull, v[q] >= vj));
          }
        if (more < want && want <= geq && lane == 0) sm.theta = vj;   // (equal entries say the same)
      }
      __syncthreads();
      theta = sm.theta;
      if (tid < n_in) {
        const uint2 e = sm.member[tid];
        // (exact in double, whatever the order, and so the same in every CTA: see above)
        if (__uint_as_float(e.x) >= theta) atomicAdd(&sm.m_sum[e.y & (kRedrawMaxCtas * kWarps - 1)], (double)weight(__uint_as_float(e.x)));
      }
      __syncthreads();
    }
    // ---- the warp that owns u * total: every warp has the same sums, `per` warps to a lane
    constexpr int kPer = kRedrawMaxCtas * kWarps / 32;
    const int per = (n_warps + 31) >> 5;
    double t[kPer], lane_sum = 0.0;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int wi = lane * per + e;
      t[e] = e < per && wi < n_warps ? sm.w_sum[wi] + sm.m_sum[wi] : 0.0;
      lane_sum += t[e];
    }
    double inc = lane_sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double n = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += n;
    }
    double exc = __shfl_up_sync(kFull, inc, 1);
    if (lane == 0) exc = 0.0;
    const double sum = __shfl_sync(kFull, inc, 31);
    int owner = 0, tok = -1;   // (no mass, a row whose largest logit mixes to +inf: -1)
    if (sum > 0.0) {
      const double y = uniform_of(g) * sum;
      const unsigned hit_l = __ballot_sync(kFull, lane_sum > 0.0 && inc > y), has_l = __ballot_sync(kFull, lane_sum > 0.0);
      const int from = hit_l ? __ffs(hit_l) - 1 : 31 - __clz(has_l);
      double run = exc, below = exc;
      int e_own = 0;
      bool past = false;
#pragma unroll
      for (int e = 0; e < kPer; ++e) {   // the first element past y, else the last one with weight
        if (t[e] > 0.0 && !past) {
          e_own = e;
          below = run;
          past = run + t[e] > y;
        }
        run += t[e];
      }
      owner = __shfl_sync(kFull, lane * per + e_own, from);
      double done = __shfl_sync(kFull, below, from);
      if (owner == my_warp) {
        // ---- its ids, piece by piece: the lane, then the id
        int last = -1;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          float w[8];
          double s = 0.0;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            w[k] = x0 + 256 * j < P.V && (!cut || z[j][k] > hi || z[j][k] >= theta) ? weight(z[j][k]) : 0.f;
            s += (double)w[k];
          }
          double si = s;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double n = __shfl_up_sync(kFull, si, o);
            if (lane >= o) si += n;
          }
          double cum = __shfl_up_sync(kFull, si, 1);
          cum = done + (lane == 0 ? 0.0 : cum);
          const unsigned hit = __ballot_sync(kFull, s > 0.0 && done + si > y), has = __ballot_sync(kFull, s > 0.0);
          int k_first = -1, k_last = -1;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            cum += (double)w[k];
            if (w[k] > 0.f) {
              k_last = k;
              if (k_first < 0 && cum > y) k_first = k;
            }
          }
          const int x_first = x0 + 256 * j + (k_first >= 0 ? k_first : k_last), x_last = x0 + 256 * j + k_last;
          if (tok < 0 && hit) tok = __shfl_sync(kFull, x_first, __ffs(hit) - 1);
          if (has) last = __shfl_sync(kFull, x_last, 31 - __clz(has));
          done += __shfl_sync(kFull, si, 31);
        }
        if (tok < 0) tok = last;   // (rounding: the last id with weight)
      }
    }
    const bool mine = owner == my_warp && lane == 0;
    if (waited) {
      if (mine) a.out_tok[g] = tok;
      i += clusters;
      continue;
    }
    // ---- drawn ahead: does it hold?
    look();
    waited = true;
    const int now = ld_fresh(a.pos_list + beg0 + cluster);
    bool same = i == (int)beg0 && i + cluster < end && (uint32_t)now == g && !single;
    load(g, [&](int j, const float (&v)[8]) {
#pragma unroll
      for (int k = 0; k < 8; ++k) same = same && __float_as_uint(v[k]) == __float_as_uint(z[j][k]);
    });
    bool holds = __syncthreads_and(same);
    if (ctas > 1) {
      if (tid < (int)ctas) st_peer(peer_addr(smem_u32(&sm.same[rank]), tid), (uint32_t)holds);
      meet();
      for (uint32_t q = 0; q < ctas; ++q) holds = holds && sm.same[q] != 0;
    }
    i += cluster;
    if (holds) {
      if (mine) a.out_tok[g] = tok;
      i += clusters;
    }
  }
  if constexpr (NP < 4) {
    if (single) {   // (nothing is under way between the cluster's CTAs any more)
      const ResRow row(reinterpret_cast<float*>(dyn), P.V);
#pragma unroll 1
      for (i += (int)rank * clusters; i < end; i += (int)gridDim.x) {   // (i: the list's start, and this cluster's number)
        g = (uint32_t)ld_fresh(a.pos_list + i);
        if (g >= total) continue;
        src.cond = a.cond + (size_t)g * bytes;
        src.uncond = a.uncond ? a.uncond + (size_t)g * bytes : nullptr;
        src.V = P.V;
        src.bf16 = BF16;
        int calls = 0;
        float unused;
        RowStats st;
        const ResSums sums = res_row_stats(row, src, P.top_k, rs, calls, -1, unused, st);
        if (sums.total > 0.0) res_pick(row, sums, uniform_of(g), [&](int x) -> double { return (double)row.at(x); }, a.out_tok + g);
        else if (tid == 0) a.out_tok[g] = -1;
        __syncthreads();
      }
    }
  }
}

}  // namespace mulo
