// The fast path for rows with a top-k cut: NW warps per row.
//
// A CTA owns a contiguous range of target rows (in parent order).  Per parent it streams the draft row and then
// the target rows under it, each ONCE.  The ids are split into 4 NW contiguous parts, one for every group of eight
// lanes.
//
//   stream     128-byte pieces of each group's part (16 bytes per lane) through registers, four in flight per lane
//              (two when sampling), the next row asked into L2 by a bulk prefetch.  Per id: unpack, CFG mix (packed
//              fp32, one IEEE rounding per step), compare with a predicted pivot and a predicated append to the
//              thread's PRIVATE list plus a bit in its survivor mask (one word per four pieces).  The loads run
//              on into the next row, so a row's first pieces are in registers when its turn comes.
//   lists      threads t and t + 32 (of an even and the next odd warp) share a column of R rows, growing towards
//              each other.
//   first pass over the list: exp against a predicted maximum.  Entries above the selection window are done
//              with here (their exp replaces the logit in the list); those in the window go into a 256-bin
//              histogram and a bit mask.
//   selection  the bin that holds the k-th largest; the window's entries once more: above the bin -> exp, below
//              -> 0, in the bin -> set aside and ranked exactly; then each thread turns its own ones into weights (a bit
//              mask says which).  From here on the list holds the row's weights, zeros below the threshold included.
//   draws      sums of p (target) or of max(0, p - q) (residual; the sum of p minus that of min(p, q) over the ids
//              that both rows kept, found by intersecting the masks) per thread and group.  The group that owns
//              u * total is searched by the whole CTA, a mask word or so per eight threads; the owner's warp takes
//              it from there (piece, lane, id) while the others go on with the next row.
//   pooling    (POOL, Eq. 3-4) between selection and decision: the neighbour list of x~ is walked in tiles, eight
//              entries per thread, their weights found in the lists by popcount on the survivor masks (most neighbours are not
//              kept at all, which their mask bit says); prefix masses by block scan; the pooled ids' weights change their sign,
//              which counts as nothing from then on, and leave their owners' sums (64-bit fixed point, so the order does not
//              matter).  x~ carries its pooled weight outside the lists.
//
// Three block barriers per draft row, four per target row.  Pivot, histogram scale and exp reference are predicted from the CTA's previous
// rows of the same kind; a row without prediction takes them from the mean and spread of its first pieces.  A
// row whose prediction misses (too few candidates, a full column, rank beyond the histogram, maximum far from the
// reference) is streamed again with corrected values; one that still fails, or has too many ties at the
// threshold, goes to a list that a second launch works off with the general routines, so results never depend
// on the prediction.
#pragma once

#include <type_traits>

#include "mulo_stream.cuh"

namespace mulo {

constexpr int kRPieceBytes = 128;        // of a group: 16 bytes per lane
constexpr int kRBins = 256;
constexpr int kRSetAside = 128;          // entries of the crossing bin that are ranked exactly
constexpr int kRTries = 6;               // times a row is streamed before it is given up
constexpr int kRSlack = 12;              // list rows kept free between the two lists of a column: a piece's entries and the closing ones
constexpr float kRMagic = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kNearRefGap = 8.0f;      // a row whose maximum lies further from the predicted exp reference is streamed again
                                         // against its own maximum (large exponents cost relative accuracy)

// What the kernel is run for: a whole round; the drafter's draws; or one stage of a round.  Two stages want sums of a row and
// nothing drawn: the target rows' probabilities of x~ and its acceptance, the draft rows' statistics.  kRowsResample draws for the
// positions of R_X, with the draft rows' statistics given: a draft row is only streamed, its entries above the given threshold are
// its list.  The stages are no less exact than the general routines whose place they take: weights by sums_exp, added in double,
// the maximum's own in double where the sum is handed on, a draw's sums and its search in double.  (The exp reference is a whole
// number: subtracting it loses no bits of the logits near the maximum.)
constexpr int kRowsRound = 0, kRowsSample = 1, kRowsVerify = 2, kRowsStats = 3, kRowsResample = 4;
// What is left to the general routines is marked in the stage's own output, so that calls on other streams share nothing but
// status bits: in the place of a threshold a NaN that no logit gives, in the place of a token what no draw gives.
constexpr uint32_t kStatsLeft = 0xffa5c3e1u;
constexpr int32_t kPickLeft = INT32_MIN;
// A position of R_X: its index in its image, whether it is drawn from the residual, whether any position of its parent is (the
// draft row is not read otherwise).
constexpr uint32_t kPickIndex = (1u << 30) - 1u, kPickResidual = 1u << 31, kPickDraft = 1u << 30;

// running prediction for one kind of row (draft / target), per CTA
struct RowPredictor {
  int have;
  int age;                    // rows learnt from since the prediction was last lost
  float theta, rho, mx;       // running k-th largest, density below it, row maximum
  float pivot, inv_w, ref;    // what the next row starts from (valid while have != 0)
  float shift, step;          // bootstrap adaptation, as in the general streaming kernel
  int dir;
};

struct RowsArgs {
  DevParams P;
  const char* cond;
  const char* uncond;
  const char* draft;
  const int32_t* draft_tok_lo;
  const uint16_t* nn;       // POOL
  float* p_tok;
  float* q_tok;
  float* accept_prob;
  uint8_t* flags;
  int32_t* cand_res;
  int32_t* cand_tgt;
  int32_t* sample_out;      // kRowsSample: the drafter's token per cell
  const int32_t* tok_of;    // kRowsVerify, kRowsStats, kRowsResample: x~ of each row
  const float* stats_in;    // kRowsVerify, kRowsResample: the draft rows' statistics
  const uint32_t* reject_bits;   // kRowsResample
  const uint32_t* expand_bits;
  float* stats_out;         // kRowsStats
  int32_t* tok_hi_out;
  float* q_hi_out;
  uint32_t* dev_status;
  int32_t* fail_list;
  int n_units;              // rows: target rows, parent by parent (kRowsSample, kRowsStats: low-res cells; kRowsVerify: in raster order)
  uint32_t row_bytes;
  int ppg;                  // pieces of a group's part of a row
  int n_words;              // mask words per thread: ceil(ppg / 4)
  int R;                    // rows of a list column (shared by two threads)
  uint32_t o_dlist, o_tmask, o_dmask;   // dynamic shared memory: the lists first, then these
  int margin;
  float a_theta, a_boot, a_max;
};

template <int NW, bool POOL = false>
struct RowsSmem {
  alignas(16) unsigned hist[kRBins + 4];   // (+ one bin that rounding may reach)
  unsigned spill[32];                      // where the entries outside the window are counted
  alignas(16) float closer[4][32];         // -inf: what a thread past its list's end reads
  alignas(16) float sa_z[kRSetAside];      // (before the set-aside: where such a thread writes)
  RowPredictor pred[2];                   // draft rows / target rows
  double w_all[NW];                        // exp sums of each warp without the crossing bin
  double w_draw[2][NW * 4];                // weights of a draw, per group; consecutive draws alternate
  uint32_t fx[2][NW * 4];                  // ... and of the parts of the owning group
  double e_tok;
  float z_tok;
  alignas(8) uint32_t rnd[2][16][3];       // (kRowsResample: `fx` in double) uniforms of sixteen of the parent's children, by parity of the parent
  unsigned n_sa;
  int wn[NW];
  unsigned wmax[NW];
  float red[NW][3];
  unsigned char cnt[NW * 32];
  unsigned char over[NW];
  // POOL
  unsigned long long adj[POOL ? NW * 32 : 1];   // weight that left a thread's entries, times 2^40
  double pool_sum[2][POOL ? NW : 1], pool_cj;
  int pool_bad[POOL ? NW : 1];
};

// Dynamic shared memory of a CTA (bytes); the parts' offsets go into `s`.
inline uint32_t rows_layout(RowsArgs& s, int nw, bool bf16, int kind) {
  const uint32_t cols = (uint32_t)s.R * (uint32_t)(nw / 2);
  uint32_t off = cols * 128u;   // the target row's lists
  auto take = [&](uint32_t bytes) {
    const uint32_t o = off;
    off += bytes;
    return o;
  };
  const bool draws = kind == kRowsRound || kind == kRowsResample;
  s.o_dlist = take(draws ? cols * (bf16 ? 64u : 128u) : 0u);
  s.o_tmask = take(draws || kind == kRowsSample ? (uint32_t)s.n_words * nw * 128u : 0u);
  s.o_dmask = draws ? take((uint32_t)s.n_words * nw * 128u) : s.o_tmask;
  return off;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float lds_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// 2^t by the special-function unit (relative error about 2^-22)
__device__ __forceinline__ float ex2f(float t) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(t));
  return r;
}

template <int J>
__device__ __forceinline__ uint32_t word_of(const uint4& v) {
  return J == 0 ? v.x : J == 1 ? v.y : J == 2 ? v.z : v.w;
}

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// a logit of the draft list (bf16 or fp32)
template <bool BF16>
__device__ __forceinline__ void dlist_put(uint32_t addr, float z) {
  if (BF16) asm volatile("{\n\t.reg .b16 h;\n\tcvt.rn.bf16.f32 h, %1;\n\tst.shared.b16 [%0], h;\n\t}" ::"r"(addr), "f"(z) : "memory");
  else sts_f32(addr, z);
}
template <bool BF16>
__device__ __forceinline__ float dlist_get(uint32_t addr) {
  if (!BF16) return lds_f32(addr);
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return __uint_as_float((uint32_t)v << 16);
}
__device__ __forceinline__ uint4 ldg_stream(const char* p) {   // 16 bytes, read once: not kept in L1
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ void prefetch_l2(const char* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Appends z to the thread's list if z >= pivot (cursor step: one list row of 128 bytes, up or down) and
// marks its bit (MARK).
template <bool MARK, int BIT>
__device__ __forceinline__ void row_put(float z, float pivot, uint32_t& cur, uint32_t step, uint32_t& m) {
  if constexpr (!MARK)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ge.f32 p, %1, %2;\n\t"
        "@p st.shared.f32 [%0], %1;\n\t"
        "@p add.u32 %0, %0, %3;\n\t}"
        : "+r"(cur)
        : "f"(z), "f"(pivot), "r"(step)
        : "memory");
  else asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ge.f32 p, %2, %3;\n\t"
      "@p st.shared.f32 [%0], %2;\n\t"
      "@p add.u32 %0, %0, %4;\n\t"
      "@p or.b32 %1, %1, %5;\n\t}"
      : "+r"(cur), "+r"(m)
      : "f"(z), "f"(pivot), "r"(step), "n"(1u << BIT)
      : "memory");
}

// The pre-processed logits of a piece (8 bf16 / 4 fp32 ids), two per packed instruction: d = c - u;
// v = fma(s, d, u); z = v * invT, each half one IEEE rounding.
template <bool BF16, bool ROW_U, bool SCALE, int J>
__device__ __forceinline__ float2 row_pair(const uint4& c, const uint4& u, float2 s2, float2 t2) {
  float2 v, un;
  if (BF16) {
    const uint32_t cw = word_of<J>(c);
    v = make_float2(bf16_lo(cw), bf16_hi(cw));
    if (ROW_U) {
      const uint32_t uw = word_of<J>(u);
      un = make_float2(bf16_lo(uw), bf16_hi(uw));
    }
  } else {
    v = make_float2(__uint_as_float(word_of<(2 * J) & 3>(c)), __uint_as_float(word_of<(2 * J + 1) & 3>(c)));
    if (ROW_U)
      un = make_float2(__uint_as_float(word_of<(2 * J) & 3>(u)), __uint_as_float(word_of<(2 * J + 1) & 3>(u)));
  }
  if (ROW_U) v = __ffma2_rn(s2, __ffma2_rn(un, make_float2(-1.f, -1.f), v), un);   // fma(u, -1, c) rounds as c - u
  if (SCALE) v = __fmul2_rn(v, t2);
  return v;
}
template <bool BF16, bool ROW_U, bool SCALE, bool MARK, int BIT0>
__device__ __forceinline__ void row_piece(const uint4& c, const uint4& u, float2 s2, float2 t2, float pivot,
                                          uint32_t& cur, uint32_t step, uint32_t& m) {
  float2 z = row_pair<BF16, ROW_U, SCALE, 0>(c, u, s2, t2);
  row_put<MARK, BIT0>(z.x, pivot, cur, step, m);
  row_put<MARK, BIT0 + 1>(z.y, pivot, cur, step, m);
  z = row_pair<BF16, ROW_U, SCALE, 1>(c, u, s2, t2);
  row_put<MARK, BIT0 + 2>(z.x, pivot, cur, step, m);
  row_put<MARK, BIT0 + 3>(z.y, pivot, cur, step, m);
  if (BF16) {
    z = row_pair<BF16, ROW_U, SCALE, 2>(c, u, s2, t2);
    row_put<MARK, (BIT0 + 4) & 31>(z.x, pivot, cur, step, m);
    row_put<MARK, (BIT0 + 5) & 31>(z.y, pivot, cur, step, m);
    z = row_pair<BF16, ROW_U, SCALE, 3>(c, u, s2, t2);
    row_put<MARK, (BIT0 + 6) & 31>(z.x, pivot, cur, step, m);
    row_put<MARK, (BIT0 + 7) & 31>(z.y, pivot, cur, step, m);
  }
}

// 2^x in double, out of line: three call sites, a few hundred instructions each otherwise
__device__ __noinline__ double row_exp2(double x) { return exp2(x); }

__device__ __noinline__ double row_exp(double x) { return exp(x); }

// e^d for d from -80 (below: that of -80) to 80, within 7.5e-8 (0.91 units in the last place), 2.65e-8 rms, by 4 M values per range:
// d = n ln 2 + f with ln 2 in two parts (Cody and Waite), and on |f| <= ln 2 / 2 a polynomial 1 + f + f^2 q(f), q of degree four
// fitted to (e^f - 1 - f) / f^2 (largest error in e^f 5.2e-9; the rest are the roundings of f and of the last two steps).
__device__ __forceinline__ float sums_exp(float d) {
  d = fmaxf(d, -80.0f);
  const float t = fmaf(d, kLog2e, kRMagic), n = t - kRMagic;   // n to nearest
  float f = fmaf(n, -0.693145751953125f, d);                   // (n times these sixteen bits of ln 2 is exact)
  f = fmaf(n, -1.4286068203094e-6f, f);
  float q = fmaf(1.3950488064e-3f, f, 8.3688879386e-3f);
  q = fmaf(q, f, 4.1666205972e-2f);
  q = fmaf(q, f, 1.6666518152e-1f);
  q = fmaf(q, f, 0.5f);
  q = fmaf(q, f, 1.0f);
  q = fmaf(q, f, 1.0f);
  return __fmul_rn(q, __int_as_float((__float_as_int(t) + 127) << 23));
}
// What the weight of the row's maximum in a sum of these lacks: with one id far above the rest that is the sum's whole error.
__device__ __forceinline__ double sums_exp_rest(float d) { return exp((double)d) - (double)sums_exp(d); }

// x~'s own weight, in double, beside weights 2^(z * kLog2e + c0), c0 = -ref * kLog2e in fp32.  That constant is off by 1.3e-8
// (relative), which acts on z - ref: it averages out in sums near the maximum, a single weight far below it shows it whole
// and is corrected.  (p(x~) against 64 bits, relative error, mean and largest of 1024 positions, V = 16384: 6.0e-8 and 1.8e-7 at
// top-k 2048 with the weights' constant, 2.5e-8 and 1.5e-7 so; without a cut 5.8e-8 and 2.2e-7, 2.5e-8 and 1.5e-7 so.)
constexpr double kLog2eRest = 1.4426950408889634 - (double)kLog2e;
__device__ __noinline__ double token_weight(float z, float ref, float c0) {   // (out of line: hundreds of instructions)
  return exp2((double)z * (double)kLog2e + (double)c0 + (double)(z - ref) * kLog2eRest);
}

// Philox4x32-10 as a rolled loop (one thread per row runs it; the unrolled form is ten times the code)
__device__ __noinline__ uint4 row_philox(uint4 c, uint2 k) {
#pragma unroll 1
  for (int i = 0; i < 10; ++i) {
    const uint32_t a = 0xD2511F53u, b = 0xCD9E8D57u;
    const uint32_t h0 = __umulhi(a, c.x), l0 = a * c.x;
    const uint32_t h1 = __umulhi(b, c.z), l1 = b * c.z;
    c = make_uint4(h1 ^ c.y ^ k.x, l1, h0 ^ c.w ^ k.y, l0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// The optional probability outputs of a position (one thread; out of line: double divisions).
__device__ __noinline__ void row_write_probs(float* p_tok, float* q_tok_out, float* accept_prob, size_t g, double e_tok,
                                              double mass, double q_tok, double Z, bool threshold_rule) {
  const double p = e_tok / Z;
  if (p_tok) p_tok[g] = (float)p;
  if (q_tok_out) q_tok_out[g] = (float)q_tok;
  if (accept_prob) {
    const double P = mass / Z;
    double thr;
    if (threshold_rule) thr = P;
    else if (q_tok <= 0.0) thr = P > 0.0 ? 1.0 : 0.0;
    else thr = fmin(1.0, P / q_tok);
    accept_prob[g] = (float)thr;
  }
}

// The predictor of one kind of row after a row (ok: theta found exactly).  One thread; out of line.
__device__ __noinline__ void row_learn(RowPredictor* prp, bool ok, int reason, float theta, float pivot, int n,
                                        int n_ge, float mx, int margin, float a_theta, float a_boot) {
  RowPredictor pr = *prp;
  if (!ok) {
    pr.have = 0;
    pr.age = 0;
    const int dir = reason == 2 ? -1 : (reason == 1 || reason == 3) ? 1 : 0;
    if (dir != 0) {
      const float unit = 0.5f * (a_theta - a_boot);
      if (pr.dir == 0) pr.step = unit;
      else if (pr.dir == dir) pr.step = fminf(2.0f * pr.step, 64.0f * unit);
      else pr.step = fmaxf(0.5f * pr.step, 0.25f * unit);
      pr.shift += (float)dir * pr.step;
      pr.dir = dir;
    }
  } else {
    pr.dir = 0;
    const int below = n - n_ge;   // candidates in [pivot, theta)
    // running means: a plain average over the first four rows, weight 1/4 for the newest after that
    const float w_new = pr.have ? fmaxf(0.25f, 1.0f / (float)(pr.age + 1)) : 1.0f;
    float rho = pr.rho;
    bool rho_ok = pr.have != 0;
    if (theta > pivot && below >= 16) {
      const float r_new = (float)below / (theta - pivot);
      rho = pr.have ? pr.rho + w_new * (r_new - pr.rho) : r_new;
      rho_ok = true;
    }
    if (!rho_ok) {
      pr.have = 0;
      pr.age = 0;
    } else {
      pr.theta = pr.have ? pr.theta + w_new * (theta - pr.theta) : theta;
      pr.mx = pr.have ? pr.mx + w_new * (mx - pr.mx) : mx;
      pr.rho = rho;
      pr.have = 1;
      if (pr.age < 8) ++pr.age;
      // a prediction that rests on a single row carries that row's noise in the threshold and in
      // the density: the row after it aims for a wider margin
      const float d = (pr.age < 2 ? 1.4f : 1.0f) * (float)margin / rho;
      pr.pivot = pr.theta - d;
      pr.inv_w = (float)kRBins / (2.0f * d);   // the histogram spans twice the distance pivot -> threshold
      pr.ref = pr.mx;
    }
  }
  *prp = pr;
}

// One logit as it is in memory, and its value.
template <bool BF16>
__device__ __forceinline__ uint32_t raw_logit(const char* row, int x) {
  if constexpr (BF16) return __ldg(reinterpret_cast<const unsigned short*>(row) + x);
  else return __ldg(reinterpret_cast<const uint32_t*>(row) + x);
}
template <bool BF16>
__device__ __forceinline__ float wide_logit(uint32_t raw) {
  return __uint_as_float(BF16 ? raw << 16 : raw);
}

// Double division, out of line.
__device__ __noinline__ double rows_div(double a, double b) { return a / b; }

// Eight entries of a neighbour list from `first` (a multiple of eight; entry 0 is x~ itself) on, packed; past the list's
// end the last ones again.
__device__ __forceinline__ uint4 pool_ids(const uint16_t* row, int pool_k, int first) {
  if ((pool_k & 7) == 0 && ((uintptr_t)row & 15) == 0) return __ldg(reinterpret_cast<const uint4*>(row + min(first, pool_k - 8)));
  uint32_t v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __ldg(row + min(first + i, pool_k - 1));
  return make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
}
// Puts V - 1 in the place of what is no id; returns whether there was one (entry 0, x~ itself, does not count).
__device__ __forceinline__ bool pool_clamp(uint4& v, bool from0, int V) {
  const uint32_t top = (uint32_t)(V - 1) * 0x10001u;
  const uint4 c = make_uint4(__vminu2(v.x, top), __vminu2(v.y, top), __vminu2(v.z, top), __vminu2(v.w, top));
  const uint32_t diff = ((c.x ^ v.x) & (from0 ? 0xffff0000u : 0xffffffffu)) | (c.y ^ v.y) | (c.z ^ v.z) | (c.w ^ v.w);
  v = c;
  return diff != 0u;
}
// One of them.
__device__ __forceinline__ int pool_id(const uint4& v, int i) {
  const uint32_t w = i < 2 ? v.x : i < 4 ? v.y : i < 6 ? v.z : v.w;
  return (int)(w >> (16 * (i & 1)) & 0xffffu);
}
// Asks a neighbour list into L2 (one thread; the whole 16 bytes in it).
__device__ __forceinline__ void pool_prefetch(const uint16_t* row, int pool_k) {
  const uintptr_t from = ((uintptr_t)row + 15) & ~(uintptr_t)15, to = (uintptr_t)(row + pool_k) & ~(uintptr_t)15;
  if (to > from) prefetch_l2(reinterpret_cast<const char*>(from), (uint32_t)(to - from));
}

// Warps per SM the kernel is compiled for: 16 (128 registers, four pieces in flight; eight CTAs of two warps are also
// what the lists of V = 16384, top-k 2000 leave room for), 24 for the draft rows' kernels, which keep no draft list, 20 for the
// target rows' sums.
__host__ __device__ constexpr int rows_warps(int kind) { return kind == kRowsRound || kind == kRowsResample ? 16 : kind == kRowsVerify ? 20 : 24; }

// The end of a row of the stages (out of line: double divisions and exponentials).  One thread; e_tok: weight of x~ in the row's
// units, 0 below its threshold.
__device__ __noinline__ void rows_verified(const RowsArgs* a, uint32_t g, double e_tok, double Z, float m, float ref, float zq,
                                           float theta_q, float m_q, double Zq) {
  const DevParams& P = a->P;
  Z += sums_exp_rest(__fsub_rn(m, ref));
  const uint32_t N = (uint32_t)P.H * (uint32_t)P.W, b = g / N, t = g - b * N;
  const double p = e_tok / Z, q = zq >= theta_q ? exp((double)zq - (double)m_q) / Zq : 0.0;
  if (q <= 0.0) atomicOr(a->dev_status, MULO_DEV_ZERO_DRAFT_PROB);
  double thr;
  bool accepted;
  if (P.accept_mode == MULO_ACCEPT_THRESHOLD) {
    thr = p;
    accepted = p >= P.tau;
  } else {
    thr = q <= 0.0 ? (p > 0.0 ? 1.0 : 0.0) : fmin(1.0, p / q);
    accepted = uniform24(row_philox(make_uint4(t, b + P.image_offset, P.round, 0u), make_uint2(P.seed_lo, P.seed_hi)).x) < thr;
  }
  a->flags[g] = accepted ? 0 : 1;
  a->p_tok[g] = (float)p;
  a->q_tok[g] = (float)q;
  a->accept_prob[g] = (float)thr;
}
__device__ __noinline__ void rows_stats(const RowsArgs* a, uint32_t cell, float z_tok, float theta, float m, float ref, double Z) {
  const DevParams& P = a->P;
  Z = (Z + sums_exp_rest(__fsub_rn(m, ref))) * exp((double)ref - (double)m);
  const float hi = (float)Z, lo = (float)(Z - (double)hi);
  reinterpret_cast<float4*>(a->stats_out)[cell] = make_float4(theta, m, hi, lo);
  const float q = z_tok >= theta ? (float)(exp((double)z_tok - (double)m) / ((double)hi + (double)lo)) : 0.f;
  const uint32_t hw = (uint32_t)P.h * (uint32_t)P.w, b = cell / hw, ca = (cell - b * hw) / P.w, cc = cell - b * hw - ca * P.w;
  const int32_t tok = a->tok_of[cell];
  for (int di = 0; di < P.r; ++di)
    for (int dj = 0; dj < P.r; ++dj) {
      const size_t t = ((size_t)b * P.H + (size_t)ca * P.r + di) * P.W + (size_t)cc * P.r + dj;
      a->tok_hi_out[t] = tok;
      a->q_hi_out[t] = q;
    }
}

// PLAIN: T = 1 and every piece a thread's whole 16 bytes (V splits evenly), so no scaling and no bounds checks.
template <bool BF16, bool HAS_U, int KIND, bool POOL, bool PLAIN, int NW>
__global__ void __launch_bounds__(NW * 32, rows_warps(KIND) / NW) k_round_rows(const __grid_constant__ RowsArgs a) {
  constexpr bool LISTED = KIND == kRowsResample;
  constexpr bool ONE_KIND = KIND != kRowsRound && !LISTED;       // of row: either target or draft rows, and no parents
  constexpr bool SUMS = KIND == kRowsVerify || KIND == kRowsStats;   // nothing is drawn
  constexpr int NT = NW * 32;
  constexpr int IDS = BF16 ? 8 : 4;              // ids per lane per piece
  constexpr int kRDepth = KIND == kRowsSample || KIND == kRowsStats ? 2 : 4;   // pieces in flight per lane
  constexpr bool EXACT = SUMS || LISTED;         // weights by sums_exp, sums in double
  using Sum = typename std::conditional<EXACT, double, float>::type;
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ RowsSmem<NW, POOL> sm;
  const DevParams& P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  let_next_begin();
  const int rr = ONE_KIND ? 1 : P.r * P.r;
  int n_units = a.n_units;
  // LISTED: the unit in work and the one after it are found by going down the positions parent by parent (`found`: how far), 32 at a time.
  uint32_t found = 0;
  int left = 0;
  const uint32_t N = (uint32_t)P.H * (uint32_t)P.W, n_at = (uint32_t)P.B * N;
  const int Ww = (P.W + 31) >> 5;
  struct Place {
    int b, i, j, parent;
  };
  auto place_of = [&](uint32_t x) -> Place {
    Place p;
    p.parent = (int)(x / (uint32_t)rr);
    const int c = (int)(x - (uint32_t)p.parent * (uint32_t)rr), hw = P.h * P.w;
    p.b = p.parent / hw;
    const int rem = p.parent - p.b * hw, ca = rem / P.w, di = c / P.r;
    p.i = ca * P.r + di;
    p.j = (rem - ca * P.w) * P.r + c - di * P.r;
    return p;
  };
  auto bit_of = [&](const uint32_t* bits, const Place& p) -> bool {
    return bits[((size_t)p.b * P.H + p.i) * Ww + (p.j >> 5)] >> (p.j & 31) & 1u;
  };
  // Blocks of 32 parents of a row (r words of r rows of the mask): how many positions of R_X, the first position, the one past the last.
  const int nb = (P.w + 31) >> 5, n_blocks = P.B * P.h * nb;
  const uint32_t row_units = (uint32_t)P.w * (uint32_t)rr;
  auto count_block = [&](int q) -> int {
    const int row = q / nb, w0 = (q - row * nb) * P.r, w1 = min(w0 + P.r, Ww);
    int n = 0;
    for (int i = 0; i < P.r; ++i)
      for (int w = w0; w < w1; ++w) {
        uint32_t v = a.expand_bits[((size_t)row * P.r + i) * Ww + w];
        if (w == Ww - 1 && (P.W & 31)) v &= (1u << (P.W & 31)) - 1u;   // (bits past the row's end do not count)
        n += __popc(v);
      }
    return n;
  };
  auto block_start = [&](int q) -> uint32_t {
    const int row = q / nb;
    return (uint32_t)row * row_units + (uint32_t)(q - row * nb) * 32u * (uint32_t)rr;
  };
  auto block_end = [&](int q) -> uint32_t {
    const int row = q / nb;
    return (uint32_t)row * row_units + (uint32_t)min(P.w, (q - row * nb + 1) * 32) * (uint32_t)rr;
  };
  // the first position of R_X from x on, which lies in block `q_at` or at its end, that has `skip` others of the block before it (every
  // warp for itself; there is one)
  int q_at = 0;
  uint32_t e_at = 0;
  auto find_pick = [&](uint32_t x, int skip) -> uint32_t {
#pragma unroll 1
    for (;;) {
#pragma unroll 1
      for (; x < e_at; x += 32) {
        const uint32_t mine = x + (uint32_t)lane;
        uint32_t hit = __ballot_sync(kFull, mine < e_at && bit_of(a.expand_bits, place_of(min(mine, e_at - 1u))));
        const int n = __popc(hit);
        if (skip < n) {
          for (; skip > 0; --skip) hit &= hit - 1u;
          return x + (uint32_t)__ffs(hit) - 1u;
        }
        skip -= n;
      }
      unsigned some = 0;   // the next block that is not empty, 32 at a time
#pragma unroll 1
      for (++q_at; q_at < n_blocks; q_at += 32) {
        some = __ballot_sync(kFull, q_at + lane < n_blocks && count_block(min(q_at + lane, n_blocks - 1)) > 0);
        if (some) break;
      }
      if (!some) return n_at - 1u;
      q_at += __ffs(some) - 1;
      x = block_start(q_at);
      e_at = block_end(q_at);
    }
  };
  if constexpr (LISTED) {
    // x~ where nothing is drawn; of what is drawn, what the general routines report of a position
    for (uint32_t x = blockIdx.x * NT + tid; x < n_at; x += gridDim.x * NT) {
      const int raw = a.tok_of[x], b = (int)(x / N), t = (int)(x - (uint32_t)b * N), i = t / P.W, j = t - i * P.W;
      if (!bit_of(a.expand_bits, Place{b, i, j, 0})) {
        a.sample_out[x] = raw;
      } else {
        const int tok = min(max(raw, 0), P.V - 1);
        if (tok != raw) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
        const size_t cell = ((size_t)b * P.h + i / P.r) * P.w + j / P.r;
        const float zq = mix_logit(wide_logit<BF16>(raw_logit<BF16>(a.draft + cell * a.row_bytes, tok)), 0.f, false, 0.f, P.invT);
        const float* const st = a.stats_in + cell * 4;
        if (!(zq >= st[0]) || row_exp((double)zq - (double)st[1]) / ((double)st[2] + (double)st[3]) <= 0.0) atomicOr(a.dev_status, MULO_DEV_ZERO_DRAFT_PROB);
      }
    }
    // how many positions R_X has, and which is this CTA's first: a run of blocks per thread
    const int per = (n_blocks + NT - 1) / NT, q0 = min(n_blocks, tid * per), q1 = min(n_blocks, q0 + per);
    int mine = 0;
    for (int q = q0; q < q1; ++q) mine += count_block(q);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) sm.wn[warp] = inc;
    __syncthreads();
    n_units = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      if (w < warp) inc += sm.wn[w];
      n_units += sm.wn[w];
    }
    const int first = (int)(((long long)n_units * blockIdx.x) / gridDim.x);
    if (first >= inc - mine && first < inc) {   // (one thread, unless there is nothing to do)
      int q = q0, skip = first - (inc - mine);
      for (int n = count_block(q); skip >= n; n = count_block(++q)) skip -= n;
      sm.n_sa = (unsigned)q;
      sm.wmax[0] = (unsigned)skip;
    }
    __syncthreads();
  }
  int unit = (int)(((long long)n_units * blockIdx.x) / gridDim.x);
  const int u_end = (int)(((long long)n_units * (blockIdx.x + 1)) / gridDim.x);
  if (unit >= u_end) return;
  if constexpr (LISTED) {
    q_at = (int)sm.n_sa;
    e_at = block_end(q_at);
    found = find_pick(block_start(q_at), (int)sm.wmax[0]);
    __syncthreads();
  }
  const uint32_t row_bytes = a.row_bytes;
  const int n_words = a.n_words, R = a.R;
  const float inv_ppg = 1.0f / (float)a.ppg;

  // ---- this thread's places in shared memory.  Lists grow upwards (even warps) or downwards (odd warps).
  const bool up = (warp & 1) == 0;
  const uint32_t my = smem_u32(dyn);
  const uint32_t first_row = (uint32_t)(warp >> 1) * (uint32_t)R + (up ? 0u : (uint32_t)(R - 1));
  const uint32_t step = up ? 128u : 0u - 128u;
  uint32_t col = (uint32_t)lane;                   // this thread's column (see `rot` below)
  uint32_t tl = my + first_row * 128u + col * 4u;
  const uint32_t low4 = up ? 0u : 0u - 384u;       // from an entry to the lowest address of the four from it on
  // the draft row's kept logits (bf16 if they came as such: exact, half the memory)
  constexpr uint32_t DROW = BF16 ? 64u : 128u;
  const uint32_t dstep = up ? DROW : 0u - DROW;
  uint32_t dl = my + a.o_dlist + first_row * DROW + col * (DROW / 32u);
  const uint32_t tm = my + a.o_tmask + (uint32_t)tid * 4u, dm = my + a.o_dmask + (uint32_t)tid * 4u;
  const uint32_t hbase = smem_u32(sm.hist) - (__float_as_uint(kRMagic) << 2);
  const uint32_t closer = smem_u32(sm.closer) + (uint32_t)lane * 4u, dump = smem_u32(sm.sa_z) + (uint32_t)lane * 4u;
  const uint32_t dl_dump = smem_u32(sm.sa_z) + (uint32_t)lane * (DROW / 32u), spill = smem_u32(sm.spill) + (uint32_t)lane * 4u;

#pragma unroll 1
  for (int i = tid; i < kRBins + 4; i += NT) sm.hist[i] = 0;
#pragma unroll 1
  for (int i = tid; i < 128; i += NT) (&sm.closer[0][0])[i] = -INFINITY;
  if (tid < 2) {
    RowPredictor& pr = sm.pred[tid];
    pr.have = 0;
    pr.age = 0;
    pr.theta = 0.f; pr.rho = 1.f; pr.mx = 0.f;
    pr.pivot = 0.f; pr.inv_w = 0.f; pr.ref = 0.f;
    pr.shift = 0.f; pr.step = 0.f; pr.dir = 0;
    sm.n_sa = 0;
  }
  __syncthreads();

  // ---- where the current row is.  parent = low-res cell (b, ca, cc); child (di, dj) of a target row.
  int parent, b, ca, cc, di = 0, dj = 0;
  {
    parent = unit / rr;
    const int child = unit - parent * rr, hw = P.h * P.w;
    b = parent / hw;
    const int rem = parent - b * hw;
    ca = rem / P.w;
    cc = rem - ca * P.w;
    if (!ONE_KIND) {
      di = child / P.r;
      dj = child - di * P.r;
    }
  }
  // LISTED: the position in work (b: its image) and the one after it
  uint32_t pick = 0, pick_next = 0;
  int b_next = 0, parent_next = 0;
  auto look_at = [&](uint32_t x, uint32_t& p, int& image, int& par) {
    const Place pl = place_of(x);
    const int mode = P.resample_mode;
    bool some = mode == MULO_RESAMPLE_RESIDUAL_ALL;
    if (mode == MULO_RESAMPLE_MIXED) {
#pragma unroll 1
      for (int c0 = 0; c0 < rr; c0 += 32) {
        const Place c = place_of((uint32_t)pl.parent * (uint32_t)rr + (uint32_t)min(c0 + lane, rr - 1));
        some = some || __any_sync(kFull, bit_of(a.expand_bits, c) && bit_of(a.reject_bits, c));
      }
    }
    const bool resid = mode == MULO_RESAMPLE_RESIDUAL_ALL || (mode == MULO_RESAMPLE_MIXED && bit_of(a.reject_bits, pl));
    p = (uint32_t)(pl.i * P.W + pl.j) | (resid ? kPickResidual : 0u) | (some ? kPickDraft : 0u);
    image = pl.b;
    par = pl.parent;
  };
  auto next_pick = [&]() {   // (there is one)
    found = find_pick(found + 1u, 0);
    look_at(found, pick_next, b_next, parent_next);
  };
  if constexpr (LISTED) {
    look_at(found, pick, b, parent);
    left = u_end - unit - 1;
  }
  auto target_index = [&]() -> uint32_t {
    if constexpr (LISTED) return (uint32_t)b * N + (pick & kPickIndex);
    return ((uint32_t)b * P.H + (uint32_t)(ca * P.r + di)) * P.W + (uint32_t)(cc * P.r + dj);
  };
  auto next_parent = [&]() {
    ++parent;
    di = dj = 0;
    if (++cc == P.w) {
      cc = 0;
      if (++ca == P.h) {
        ca = 0;
        ++b;
      }
    }
  };

  // ---- this thread's part of a row: np pieces from part_off on
  const uint32_t part_off = (uint32_t)((tid >> 3) * a.ppg) * kRPieceBytes + (uint32_t)(lane & 7) * 16u;
  const int np = part_off < row_bytes ? min(a.ppg, (int)((row_bytes - part_off + kRPieceBytes - 1) / kRPieceBytes)) : 0;
  uint4 c[kRDepth], u[kRDepth];   // the pieces in flight
  const uint4 none = make_uint4(~0u, ~0u, ~0u, ~0u);   // NaN in either type: never appended
#pragma unroll
  for (int j = 0; j < kRDepth; ++j) c[j] = u[j] = none;
  auto prologue = [&](const char* rc, const char* ru) {
#pragma unroll
    for (int j = 0; j < kRDepth; ++j) {
      c[j] = j < np ? ldg_stream(rc + j * kRPieceBytes) : none;
      if (HAS_U) u[j] = j < np && ru ? ldg_stream(ru + j * kRPieceBytes) : none;
    }
  };
  const float2 s2 = make_float2(P.cfg_scale, P.cfg_scale), t2 = make_float2(P.invT, P.invT);

  // ---- one row through the registers into the list; the loads run on into the row (nc, nu).  Returns
  //      the list's end.  (All row pointers are this thread's: part_off is in them.)
  auto stream_t = [&](auto row_u_tag, const char* rc, const char* ru, const char* nc, const char* nu, float pivot,
                      uint32_t cur, uint32_t lim, uint32_t mask_at) -> uint32_t {
    constexpr bool ROW_U = decltype(row_u_tag)::value;
#pragma unroll 1
    for (int w = 0; w < n_words; ++w) {
      const bool last = w + 1 == n_words;
      // the pieces to ask for: kRDepth ahead; those of the next word may be the next row's first
      const char* const fc = last ? nc : rc + 4 * kRPieceBytes;
      const char* const fu = !HAS_U ? nullptr : last ? nu : ROW_U ? ru + 4 * kRPieceBytes : nullptr;
      const bool do_u = HAS_U && fu != nullptr;
      const int f0 = last ? 0 : 4 * w + 4;
      uint32_t m = 0;
#define MULO_PIECE(J)                                                                                      \
  {                                                                                                        \
    constexpr int S = J % kRDepth, A = (J + kRDepth) & 3;                                                  \
    constexpr bool SAME = J + kRDepth < 4;                                                                 \
    cur = up ? min(cur, lim) : max(cur, lim);                                                              \
    row_piece<BF16, ROW_U, !PLAIN, !SUMS, J * IDS>(c[S], u[S], s2, t2, pivot, cur, step, m);                      \
    const char* const pc = SAME ? rc : fc;                                                                 \
    const char* const pu = SAME ? ru : fu;                                                                 \
    const bool want_u = SAME ? ROW_U : do_u;                                                               \
    if (PLAIN) {                                                                                           \
      c[S] = ldg_stream(pc + A * kRPieceBytes);                                                            \
      if (HAS_U && want_u) u[S] = ldg_stream(pu + A * kRPieceBytes);                                       \
    } else {                                                                                               \
      const bool in = (SAME ? 4 * w : f0) + A < np;                                                        \
      c[S] = in ? ldg_stream(pc + A * kRPieceBytes) : none;                                                \
      if (HAS_U) u[S] = in && want_u ? ldg_stream(pu + A * kRPieceBytes) : none;                           \
    }                                                                                                      \
  }
      MULO_PIECE(0) MULO_PIECE(1) MULO_PIECE(2) MULO_PIECE(3)
#undef MULO_PIECE
      if constexpr (!SUMS) sts_u32(mask_at + (uint32_t)(w * NT) * 4u, m);
      rc += 4 * kRPieceBytes;
      if (HAS_U && ROW_U) ru += 4 * kRPieceBytes;
    }
    return cur;
  };

  // ---- pivot, histogram scale and exp reference of a row whose first pieces are in registers
  auto boot_pivot = [&](bool row_u, float shift, float& pivot, float& inv_w, float& ref, float& per) {
    float s1 = 0.f, sq = 0.f, cnt = 0.f;
    auto add = [&](float z) {
      if (z == z) {
        s1 += z;
        sq += z * z;
        cnt += 1.f;
      }
    };
#pragma unroll
    for (int j = 0; j < kRDepth; ++j) {
      const uint32_t cw[4] = {c[j].x, c[j].y, c[j].z, c[j].w}, uw[4] = {u[j].x, u[j].y, u[j].z, u[j].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (BF16) {
          add(mix_logit(bf16_lo(cw[k]), bf16_lo(uw[k]), row_u, P.cfg_scale, P.invT));
          add(mix_logit(bf16_hi(cw[k]), bf16_hi(uw[k]), row_u, P.cfg_scale, P.invT));
        } else {
          add(mix_logit(__uint_as_float(cw[k]), __uint_as_float(uw[k]), row_u, P.cfg_scale, P.invT));
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_xor_sync(kFull, s1, o);
      sq += __shfl_xor_sync(kFull, sq, o);
      cnt += __shfl_xor_sync(kFull, cnt, o);
    }
    if (lane == 0) {
      sm.red[warp][0] = s1;
      sm.red[warp][1] = sq;
      sm.red[warp][2] = cnt;
    }
    __syncthreads();
    s1 = sq = cnt = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      s1 += sm.red[w][0];
      sq += sm.red[w][1];
      cnt += sm.red[w][2];
    }
    __syncthreads();
    const float mean = s1 / cnt;
    const float sd = sqrtf(fmaxf(sq / cnt - mean * mean, 1e-20f));
    const float d = fmaxf((a.a_theta - a.a_boot) * sd, 1e-20f);
    pivot = mean + (a.a_boot + shift) * sd;
    inv_w = (float)kRBins / (3.0f * d);   // (a predicted row's histogram spans 2 d)
    ref = mean + a.a_max * sd;
    per = d / (1.75f * (float)a.margin);  // distance per candidate near the pivot
  };

  bool is_q = LISTED ? (pick & kPickDraft) != 0u : !ONE_KIND;   // the row in work is a draft row
  uint32_t g = !LISTED || is_q ? (uint32_t)parent : target_index();   // ... and its index in its tensor
  if (LISTED && left > 0) next_pick();

  // ---- first pass over the list (see the top of the file); returns the exp sum of the entries above the window.
  //      A draft row (Q) puts its logits into the draft list instead of their exps into its own.  Written with
  //      predicated PTX: left to the compiler, every entry becomes two branches.
  //      (c0: the exp reference as the weights take it, see below)
  auto weight_of = [&](float z, float c0) -> float { return EXACT ? sums_exp(__fsub_rn(z, c0)) : ex2f(fmaf(z, kLog2e, c0)); };
  auto pass_one = [&](auto q_tag, int n, float inv_w, float hoff, float c0, uint32_t& low_a, uint32_t& low_b) -> Sum {
    constexpr bool Q = decltype(q_tag)::value;
    const int n_max = __reduce_max_sync(kFull, n);
    float mx = -INFINITY;
    Sum s0 = 0, s1 = 0;
    low_a = low_b = 0;
    const uint32_t end = tl + (uint32_t)n * step;
#pragma unroll
    for (int k = 0; k < 3; ++k) sts_f32(end + (uint32_t)k * step, -INFINITY);
    const float hm = hoff + kRMagic;
    const float T = 1.0f / P.invT;   // (fl(v * invT) * T rounds back to the bf16 value v)
    uint32_t ad = tl + low4, dd = dl + (up ? 0u : 0u - 3u * DROW);
#pragma unroll 1
    for (int i = 0; i < n_max; i += 4, ad += 4 * step, dd += 4 * dstep) {
      const bool in = i < n;
      const uint32_t from = in ? ad : closer;
      [[maybe_unused]] const uint32_t to = !Q && in ? ad : dump;
      float z[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) z[k] = lds_f32(from + k * 128);
      uint32_t l4 = 0;
// (entries outside the window count in a word of their own lane: a predicated reduction becomes a branch)
#define MULO_ENTRY(K, S)                                                                       \
  if constexpr (!(LISTED && Q)) {   /* (nothing is selected there, and the sum is given) */    \
    float e = weight_of(z[K], c0);                                                             \
    const uint32_t bin = __float_as_uint(fmaf(z[K], inv_w, hm));                               \
    const uint32_t at = hbase + (bin << 2);                                                    \
    if constexpr (LISTED) {                                                                    \
      asm volatile(                                                                            \
          "{\n\t.reg .pred p;\n\t.reg .u32 t, w;\n\t"                                            \
          "sub.u32 t, %2, %3;\n\t"                                                             \
          "setp.le.u32 p, t, %4;\n\t"                                                          \
          "selp.u32 w, %5, %7, p;\n\t"                                                         \
          "red.shared.add.u32 [w], 1;\n\t"                                                     \
          "@p or.b32 %0, %0, %6;\n\t"                                                          \
          "@!p st.shared.f32 [%8 + %9], %1;\n\t"                                               \
          "@p mov.f32 %1, 0f00000000;\n\t}"                                                    \
          : "+r"(l4), "+f"(e)                                                                  \
          : "r"(bin), "n"(0x4B400000), "n"(kRBins), "r"(at), "n"(1 << K), "r"(spill), "r"(to), "n"(K * 128) \
          : "memory");                                                                         \
      S += (double)e;                                                                          \
    } else if constexpr (SUMS) {                                                               \
      asm volatile(                                                                            \
          "{\n\t.reg .pred p;\n\t.reg .u32 t, w;\n\t"                                            \
          "sub.u32 t, %2, %3;\n\t"                                                             \
          "setp.le.u32 p, t, %4;\n\t"                                                          \
          "selp.u32 w, %5, %7, p;\n\t"                                                         \
          "red.shared.add.u32 [w], 1;\n\t"                                                     \
          "@p or.b32 %0, %0, %6;\n\t"                                                          \
          "@p mov.f32 %1, 0f00000000;\n\t}"                                                    \
          : "+r"(l4), "+f"(e)                                                                  \
          : "r"(bin), "n"(0x4B400000), "n"(kRBins), "r"(at), "n"(1 << K), "r"(spill)           \
          : "memory");                                                                         \
      S += (double)e;                                                                          \
    } else asm volatile(                                                                       \
        "{\n\t.reg .pred p;\n\t.reg .u32 t, w;\n\t"                                            \
        "sub.u32 t, %2, %3;\n\t"                                                               \
        "setp.le.u32 p, t, %4;\n\t"                                                            \
        "selp.u32 w, %5, %10, p;\n\t"                                                          \
        "red.shared.add.u32 [w], 1;\n\t"                                                       \
        "@p or.b32 %0, %0, %6;\n\t"                                                            \
        "@!p add.f32 %1, %1, %7;\n\t"                                                          \
        "@!p st.shared.f32 [%8 + %9], %7;\n\t}"                                                \
        : "+r"(l4), "+f"(reinterpret_cast<float&>(S))                                          \
        : "r"(bin), "n"(0x4B400000), "n"(kRBins), "r"(at), "n"(1 << K), "f"(e), "r"(to), "n"(K * 128), "r"(spill) \
        : "memory");                                                                           \
  }
      MULO_ENTRY(0, s0) MULO_ENTRY(1, s1) MULO_ENTRY(2, s0) MULO_ENTRY(3, s1)
#undef MULO_ENTRY
      if (Q) {   // (rows past the end of the list take -inf, or go where nobody reads)
        const uint32_t dt = in ? dd : dl_dump;
#pragma unroll
        for (int k = 0; k < 4; ++k) dlist_put<BF16>(dt + k * DROW, BF16 && !PLAIN ? __fmul_rn(z[k], T) : z[k]);
      }
      mx = fmaxf(mx, fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])));
      if (i < 32) low_a |= l4 << i;   // (uniform)
      else low_b |= l4 << (i & 31);
    }
    const unsigned mk = __reduce_max_sync(kFull, float_key(mx));
    const int nw = __reduce_add_sync(kFull, n);
    sm.cnt[tid] = (unsigned char)n;
    if (lane == 0) {
      sm.wn[warp] = nw;
      sm.wmax[warp] = mk;
    }
    return s0 + s1;
  };

  // ---- the window's entries once more (after the crossing bin is known): the exp of those above it and 0 for those
  //      below replace the logit (draft row: those below leave the draft list); returns the exp sum of those above.  Of the
  //      masks, the entries in the crossing bin are left, which keep their logits.
  const uint32_t flip = up ? 0u : 3u;      // (a mask's bits run along memory)
  auto window = [&](uint32_t& low_a, uint32_t& low_b, float inv_w, float hoff, float c0, int bstar) -> Sum {
    const float hm = hoff + kRMagic;
    const uint32_t bm = __float_as_uint(kRMagic) + (uint32_t)bstar;
    Sum s = 0;
    uint32_t first = 0;
    auto one = [&](uint32_t bit, float& z) -> bool {   // does the entry lie in the crossing bin?
      const uint32_t i = first + ((uint32_t)__popc(bit - 1u) ^ flip);
      const uint32_t at = tl + i * step;
      z = lds_f32(bit ? at : closer);
      const uint32_t bin = __float_as_uint(fmaf(z, inv_w, hm));   // (-inf: as unsigned above every bin; its exp is 0, e^-80 where sums_exp gives it)
      float e = weight_of(z, c0);
      e = bin > bm ? e : 0.f;
      s += (Sum)e;
      if (SUMS) {
      } else if (is_q) {
        if (bin < bm) dlist_put<BF16>(dl + i * dstep, -INFINITY);
      } else {
        const uint32_t there = bin == bm ? 0u : bit;
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(at), "f"(e), "r"(there) : "memory");
      }
      return bin == bm;
    };
    auto aside = [&](float z) { sm.sa_z[atomicAdd(&sm.n_sa, 1u) & (unsigned)(kRSetAside - 1)] = z; };
    uint32_t left_a = 0;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int trips = __reduce_max_sync(kFull, __popc(low_a));
      uint32_t left = 0;
#pragma unroll 1
      for (int t = 0; t < trips; t += 2) {
        const uint32_t b0 = low_a & (0u - low_a);
        low_a ^= b0;
        const uint32_t b1 = low_a & (0u - low_a);
        low_a ^= b1;
        float z0, z1;
        const bool h0 = one(b0, z0), h1 = one(b1, z1);
        if (h0 || h1) {
          if (h0) aside(z0);
          if (h1) aside(z1);
          left |= (h0 ? b0 : 0u) | (h1 ? b1 : 0u);
        }
      }
      if (h == 0) left_a = left;
      low_a = low_b;
      low_b = left;
      first = 32;
    }
    low_a = left_a;
    return s;
  };

  auto count_failure = [&](int reason) {   // one thread
    if (reason < 1 || reason > 4) return;
    const int slot = reason == 1 ? kCntListFull : reason == 2 ? kCntTooFew : reason == 3 ? kCntAboveRange : kCntCrowdedBin;
    atomicAdd(a.dev_status + slot, 1u);
  };
  auto defer = [&](uint32_t g) {           // one thread: position (cell) g goes to the general routines
    if constexpr (KIND == kRowsStats || LISTED) {
      if (LISTED) a.sample_out[g] = kPickLeft;
      else reinterpret_cast<uint32_t*>(a.stats_out)[(size_t)g * 4] = kStatsLeft;
      atomicAdd(a.dev_status + kCntRows, 1u);
      atomicOr(a.dev_status, MULO_DEV_DENSE_FALLBACK);
      return;
    }
    const unsigned at = atomicAdd(a.dev_status + kFailCount, 1u);
    a.fail_list[at] = (int32_t)g;
    atomicAdd(a.dev_status + kCntRows, 1u);
    atomicOr(a.dev_status, MULO_DEV_DENSE_FALLBACK);
  };

  auto row_c = [&](bool q, uint32_t g) -> const char* { return (q ? a.draft : a.cond) + (size_t)g * row_bytes; };
  auto row_u = [&](bool q, uint32_t g) -> const char* { return HAS_U && !q ? a.uncond + (size_t)g * row_bytes : nullptr; };
  auto part = [&](const char* row) -> const char* { return row ? row + part_off : nullptr; };
  auto prefetch = [&](const char* rc, const char* ru) {   // one thread
    prefetch_l2(rc, row_bytes);
    if (HAS_U && ru) prefetch_l2(ru, row_bytes);
  };

  // A column can be too full for its two threads although both have few enough entries: when a row is streamed
  // again for that, the odd warps' threads move to other columns (lane ^ rot).
  uint32_t rot = 0, rot_q = 0;            // of the row in work / of the parent's draft row
  int tries = 0, tok = 0, child = 0;      // child: which row under the parent
  int partner_n = 0;                      // entries of the previous target row in the list this thread's list grows towards
  int partner_q = 0;                      // ... and of the draft row's list
  float c0_q = 0.f;                       // of the parent's draft row
  Sum Zq = 1;
  double q_tok = 0.0;
  int tok_next = KIND == kRowsSample || LISTED ? 0 : __ldg((SUMS ? a.tok_of : a.draft_tok_lo) + parent);
  float pivot = 0.f, inv_w = 0.f, ref = 0.f, per = 0.f, lo = 0.f, hi = 0.f;   // of the row in work
  prologue(part(row_c(is_q, g)), part(row_u(is_q, g)));
  if (tid == 0) prefetch(row_c(is_q, g), row_u(is_q, g));

#pragma unroll 1
  for (;;) {
    const char* const rc = row_c(is_q, g);
    const char* const ru = row_u(is_q, g);
    // ---- the row after this one
    bool nq = false, more = true;
    uint32_t ng = 0;
    if (ONE_KIND) {
      more = unit + 1 < u_end;
      ng = more ? g + 1 : g;
    } else if (is_q) {
      ng = target_index();
    } else if (unit + 1 >= u_end) {
      more = false;
      ng = g;
    } else if (LISTED) {
      nq = parent_next != parent && (pick_next & kPickDraft) != 0u;
      ng = nq ? (uint32_t)parent_next : (uint32_t)b_next * N + (pick_next & kPickIndex);
    } else {
      if (dj + 1 < P.r || di + 1 < P.r) {
        if (++dj == P.r) {
          dj = 0;
          ++di;
        }
        ng = target_index();
      } else {
        nq = true;
        ng = (uint32_t)parent + 1u;
        tok_next = __ldg(a.draft_tok_lo + ng);
      }
    }
    const char* const nc = row_c(nq, ng);            // (no row left: this one's first pieces again)
    const char* const nu = more ? row_u(nq, ng) : nullptr;
    // the logit of x~ in this row: asked for now, used after the first pass
    uint32_t raw_c = 0u, raw_u = 0u;   // (as they are: a conversion here would wait for them)
    if constexpr (SUMS) {
      if (tries == 0) {
        tok = tok_next;
        if (tok < 0 || tok >= P.V) {
          if (tid == 0) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
          tok = min(max(tok, 0), P.V - 1);
        }
        tok_next = __ldg(a.tok_of + ng);
      }
      if (warp == NW - 1) {
        raw_c = raw_logit<BF16>(rc, tok);
        if (HAS_U) raw_u = raw_logit<BF16>(ru, tok);
      }
    } else if (KIND == kRowsRound) {
      if (is_q) {
        tok = tok_next;
        if (tok < 0 || tok >= P.V) {
          if (tid == 0) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
          tok = min(max(tok, 0), P.V - 1);
        }
        if (POOL && tid == 0) pool_prefetch(a.nn + (size_t)tok * P.pool_k, P.pool_k);
      }
      if (warp == NW - 1) {
        raw_c = raw_logit<BF16>(rc, tok);
        if (HAS_U && !is_q) raw_u = raw_logit<BF16>(ru, tok);
      }
    }

    RowPredictor& pr = sm.pred[is_q ? 0 : 1];
    float theta_q = 0.f;
    if (LISTED && is_q) {   // the threshold is given: what lies above it, and no selection
      const float* const st = a.stats_in + (size_t)g * 4;
      theta_q = pivot = __ldg(st);
      ref = __ldg(st + 1);
      inv_w = 1.0f;
    } else if (tries == 0) {   // (a row streamed again keeps its corrected values)
      lo = -INFINITY;
      hi = INFINITY;
      if (pr.have) {
        pivot = pr.pivot;
        inv_w = pr.inv_w;
        ref = pr.ref;
        per = 1.0f / pr.rho;
      } else {
        boot_pivot(HAS_U && !is_q, pr.shift, pivot, inv_w, ref, per);
      }
    }

    if (SUMS || (LISTED && !is_q)) ref = rintf(ref);
    col = (uint32_t)lane ^ (up ? 0u : rot);
    tl = my + first_row * 128u + col * 4u;
    if (is_q) dl = my + a.o_dlist + first_row * DROW + col * (DROW / 32u);
    const uint32_t mask_at = is_q ? dm : tm;
    const uint32_t lim = tl + (uint32_t)(R - kRSlack - (is_q ? max(partner_n, partner_q) : partner_n)) * step;   // a piece appends at most 8 entries
    const uint32_t end = HAS_U && !is_q
                             ? stream_t(std::integral_constant<bool, HAS_U>{}, part(rc), part(ru), part(nc), part(nu), pivot, tl, lim, mask_at)
                             : stream_t(std::false_type{}, part(rc), part(ru), part(nc), part(nu), pivot, tl, lim, mask_at);
    if (more && tid == 0) prefetch(nc, nu);
    const int n_raw = (int)(up ? end - tl : tl - end) >> 7;
    const int n = min(n_raw, 64);
    // (a list that reached its limit was held there: its entries are incomplete; one of more than R - kRSlack
    // entries would leave its neighbour's next row no room at all)
    const bool over = (up ? end >= lim : end <= lim) || n_raw > 64 || n_raw > R - kRSlack;
    const float c0 = EXACT ? ref : -ref * kLog2e, hoff = -pivot * inv_w;
    uint32_t low_a, low_b;
    Sum s_t = is_q ? pass_one(std::integral_constant<bool, !ONE_KIND>{}, n, inv_w, hoff, c0, low_a, low_b)
                     : pass_one(std::false_type{}, n, inv_w, hoff, c0, low_a, low_b);
    {
      const bool any_over = __any_sync(kFull, over);
      if (lane == 0) sm.over[warp] = any_over;
    }
    if (KIND != kRowsSample && !LISTED && warp == NW - 1) {
      // the token's own weight (its z against theta later)
      const float z = mix_logit(wide_logit<BF16>(raw_c), wide_logit<BF16>(raw_u), HAS_U && !is_q, P.cfg_scale, P.invT);
      const double e = SUMS ? row_exp((double)z - (double)ref) : token_weight(z, ref, c0);
      if (lane == 0) {
        sm.e_tok = e;
        sm.z_tok = z;
      }
    }
    // the uniforms of the parent's rows, sixteen at a time: those around the first one with the draft row, the next with every
    // sixteenth row (barrier 3 of the row before lies behind everybody who read the last ones)
    if (KIND == kRowsRound && warp == 0 && lane < min(rr, 16) && (is_q || (rr > 16 && (child & 15) == 0))) {
      const int i = rr > 16 ? ((is_q ? di * P.r + dj : child) & ~15) + lane : lane;
      const int ddi = i / P.r, ddj = i - ddi * P.r;
      const uint32_t t = (uint32_t)(ca * P.r + ddi) * P.W + (uint32_t)(cc * P.r + ddj);
      const uint4 v = row_philox(make_uint4(t, (uint32_t)b + P.image_offset, P.round, 0u), make_uint2(P.seed_lo, P.seed_hi));
      sm.rnd[parent & 1][lane][0] = v.x;
      sm.rnd[parent & 1][lane][1] = v.y;
      sm.rnd[parent & 1][lane][2] = v.z;
    }
    __syncthreads();   // ---- barrier 1
    int n_all = 0, reason = 0;
    unsigned mk = 0;
    bool any_over = false;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      n_all += sm.wn[w];
      mk = max(mk, sm.wmax[w]);
      any_over |= sm.over[w] != 0;
    }
    const float mx = key_float(mk);
    const int pair_n = sm.cnt[(uint32_t)tid ^ 32u ^ rot];
#pragma unroll
    for (int w = 0; w < NW; w += 2)   // (three rows close each of the two lists)
      any_over |= (int)sm.cnt[w * 32 + lane] + (int)sm.cnt[w * 32 + 32 + (lane ^ (int)rot)] + 6 > R;
    if (__any_sync(kFull, any_over)) reason = 1;
    else if (LISTED && is_q) reason = 0;
    else if (n_all < P.top_k) reason = 2;
    else if (!(fabsf(mx - ref) <= kNearRefGap)) reason = 5;
    unsigned cum = 0, in_bin = 0;
    int bstar = 0;
    const int rank = n_all - P.top_k + 1;   // 1-based rank from the bottom of the k-th largest
    const bool select = reason == 0 && !(LISTED && is_q);
    if (select) {
      // ---- the bin that holds the k-th largest: which eight bins, then which of them
      const uint4 h0 = *reinterpret_cast<const uint4*>(sm.hist + lane * 8);
      const uint4 h1 = *reinterpret_cast<const uint4*>(sm.hist + lane * 8 + 4);
      const unsigned own = ((h0.x + h0.y) + (h0.z + h0.w)) + ((h1.x + h1.y) + (h1.z + h1.w));
      unsigned inc = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += t;
      }
      const unsigned owners = __ballot_sync(kFull, inc >= (unsigned)rank);
      if (owners == 0) {
        reason = 3;
      } else {
        const int src = __ffs(owners) - 1;
        cum = __shfl_sync(kFull, inc - own, src);
        const unsigned h = sm.hist[src * 8 + (lane & 7)];
        inc = h;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          const unsigned t = __shfl_up_sync(kFull, inc, o, 8);
          if ((lane & 7) >= o) inc += t;
        }
        const int k = __ffs(__ballot_sync(kFull, cum + inc >= (unsigned)rank)) - 1;
        bstar = src * 8 + k;
        in_bin = __shfl_sync(kFull, h, k);
        cum += __shfl_sync(kFull, inc - h, k);
        if (in_bin > (unsigned)kRSetAside) reason = 4;
      }
    }
    float theta = 0.f;
    int n_ge = 0;
    double Z = 0.0;
    if (select && reason == 0) {
      s_t += window(low_a, low_b, inv_w, hoff, c0, bstar);
      const double w = warp_sum((double)s_t);
      if (lane == 0) sm.w_all[warp] = w;
    }
    __syncthreads();   // ---- barrier 2
#pragma unroll 1
    for (int i = tid; i < kRBins + 4; i += NT) sm.hist[i] = 0;
    if (select && reason == 0) {
      // ---- the crossing bin's entries: exact rank, and their weights
      const int want = rank - (int)cum, mcount = (int)in_bin;
      float vmin = INFINITY, vmax = -INFINITY;
#pragma unroll 1
      for (int i = lane; i < mcount; i += 32) {
        const float v = sm.sa_z[i];
        vmin = fminf(vmin, v);
        vmax = fmaxf(vmax, v);
      }
      const unsigned kmin = __reduce_min_sync(kFull, float_key(vmin)), kmax = __reduce_max_sync(kFull, float_key(vmax));
      int less_at = 0;
      theta = key_float(kmin);
      if (kmin != kmax) {   // several values in the bin: rank them
        float th = 0.f;
        bool found = false;
#pragma unroll 1
        for (int i = lane; i < mcount; i += 32) {
          const float vi = sm.sa_z[i];
          int less = 0, leq = 0;
#pragma unroll 1
          for (int k = 0; k < mcount; ++k) {
            const float vk = sm.sa_z[k];
            less += vk < vi;
            leq += vk <= vi;
          }
          if (less < want && want <= leq) {
            th = vi;
            less_at = less;
            found = true;
          }
        }
        const unsigned fm = __ballot_sync(kFull, found);
        const int fs = fm ? __ffs(fm) - 1 : 0;   // (always found: the bin holds the rank)
        theta = __shfl_sync(kFull, th, fs);
        less_at = __shfl_sync(kFull, less_at, fs);
      }
      n_ge = n_all - (int)cum - less_at;
      // (values of one bin share their exponent: sums of them in double are exact, whatever the order)
      double all = (double)mcount * (double)weight_of(theta, c0);
      if (kmin != kmax) {
        all = 0.0;
#pragma unroll 1
        for (int i = lane; i < mcount; i += 32) {
          const float v = sm.sa_z[i];
          if (v >= theta) all += (double)weight_of(v, c0);
        }
        all = warp_sum(all);
      }
      if (!SUMS && (kmin != kmax || !is_q)) {   // (a draft row keeps its logits: nothing changes unless some fall below)
        double own = 0.0;
        uint32_t at = tl;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {   // this thread's own
#pragma unroll 1
          for (; low_a; low_a &= low_a - 1u) {
            const uint32_t i = (uint32_t)(__ffs(low_a) - 1) ^ flip;
            const float v = lds_f32(at + i * step);
            const float e = v >= theta ? weight_of(v, c0) : 0.f;
            own += (double)e;
            if (!is_q) sts_f32(at + i * step, e);
            else if (!(v >= theta)) dlist_put<BF16>(dl + (i + 32 * h) * dstep, -INFINITY);
          }
          low_a = low_b;
          at += 32 * step;
        }
        s_t = (Sum)((double)s_t + own);
      }
      Z = all;
#pragma unroll
      for (int w = 0; w < NW; ++w) Z += sm.w_all[w];
    }
    if (LISTED && is_q) {
      theta = theta_q;
      const float* const st = a.stats_in + (size_t)g * 4;
      Z = (double)__ldg(st + 2) + (double)__ldg(st + 3);
    }
    const bool ok = reason == 0 && Z > 0.0 && Z < 1e300;
    const bool again = !ok && reason != 0 && reason != 4 && tries + 1 < kRTries;
    if (tid == 32 && !again && !(LISTED && is_q))
      row_learn(&pr, ok, reason, theta, pivot, n_all, n_ge, mx, a.margin, a.a_theta, a.a_boot);

    if (!ok) {   // CTA-uniform
      __syncthreads();   // ---- barrier 3
      if (tid == 0) sm.n_sa = 0;
      partner_n = 0;     // (nothing of the target rows before is read any more)
      if (is_q) partner_q = 0;
      if (again) {
        // once more: with the maximum just found, with other columns, or with the pivot moved by the candidates it
        // was off by (the values that were too high and too low bracket it)
        ++tries;
        const bool first_full = reason == 1 && rot == 0 && n_all <= P.top_k + 2 * a.margin;
        if (reason == 1) rot = (uint32_t)(11 * tries) & 31u;
        if (reason == 5) {
          ref = mx;
        } else if (!first_full) {
          const float aim = (float)P.top_k + (reason == 1 ? 0.4f : 0.7f) * (float)a.margin;
          float next = pivot + ((float)n_all - aim) * per;
          if (reason == 2) hi = pivot;
          if (reason == 3) lo = pivot;
          if (!(next > lo && next < hi))
            next = lo > -INFINITY && hi < INFINITY ? 0.5f * (lo + hi) : pivot + (reason == 2 ? -1.f : 1.f) * (float)a.margin * per;
          if (reason != 1) per *= 1.5f;   // (should the density be off, the next correction is larger)
          pivot = next;
        }
        prologue(part(rc), part(ru));
        if (KIND == kRowsRound && !is_q && more && !nq) {   // (the position was advanced to the next row above)
          if (--dj < 0) {
            dj = P.r - 1;
            --di;
          }
        }
        continue;
      }
      tries = 0;
      rot = 0;
      if (tid == 0) count_failure(reason);
      if (!is_q) {
        if (tid == 0) defer(g);
      } else {
        // the draft row is lost: its parent's rows go with it (those of this CTA)
        if constexpr (LISTED) {
          for (;;) {
            if (tid == 0) defer(target_index());
            if (++unit >= u_end) break;
            const int before = parent;
            b = b_next;
            pick = pick_next;
            parent = parent_next;
            if (--left > 0) next_pick();
            if (parent != before) break;
          }
          if (unit >= u_end) break;
          is_q = (pick & kPickDraft) != 0u;
          g = is_q ? (uint32_t)parent : target_index();
          prologue(part(row_c(is_q, g)), part(row_u(is_q, g)));
          continue;
        } else {
#pragma unroll 1
        while (true) {
          if (tid == 0) defer(target_index());
          ++unit;
          if (dj + 1 < P.r || di + 1 < P.r) {
            if (++dj == P.r) {
              dj = 0;
              ++di;
            }
            if (unit >= u_end) break;
          } else {
            break;
          }
        }
        if (unit >= u_end) break;
        next_parent();
        g = (uint32_t)parent;
        tok_next = __ldg(a.draft_tok_lo + parent);
        prologue(part(row_c(true, g)), nullptr);
        continue;
        }
      }
    } else if (!ONE_KIND && is_q) {
      tries = 0;
      // ---- a draft row ends here
      c0_q = c0;
      Zq = (Sum)Z;
      if (!LISTED) {
        q_tok = sm.z_tok >= theta ? rows_div(sm.e_tok, Z) : 0.0;
        if (q_tok <= 0.0 && tid == 0) atomicOr(a.dev_status, MULO_DEV_ZERO_DRAFT_PROB);
      }
      __syncthreads();   // ---- barrier 3
      if (tid == 0) sm.n_sa = 0;
      partner_n = 0;
      partner_q = pair_n;
      rot_q = rot;
    } else if constexpr (SUMS) {
      tries = 0;
      if (tid == (NW - 1) * 32) {   // (who wrote x~'s weight)
        if constexpr (KIND == kRowsVerify) {
          const uint32_t N = (uint32_t)P.H * (uint32_t)P.W, image = g / N, t = g - image * N, i = t / P.W, j = t - i * P.W;
          const uint32_t cell = (image * P.h + i / P.r) * P.w + j / P.r;
          const float zq = mix_logit(wide_logit<BF16>(raw_logit<BF16>(a.draft + (size_t)cell * row_bytes, tok)), 0.f, false, 0.f, P.invT);
          const float* const st = a.stats_in + (size_t)cell * 4;
          rows_verified(&a, g, sm.z_tok >= theta ? sm.e_tok : 0.0, Z, mx, ref, zq, st[0], st[1], (double)st[2] + (double)st[3]);
        } else {
          rows_stats(&a, g, sm.z_tok, theta, mx, ref, Z);
        }
      }
      __syncthreads();   // ---- barrier 3
      if (tid == 0) sm.n_sa = 0;
      partner_n = 0;
    } else {
      tries = 0;
      const double e_tok = KIND == kRowsRound && sm.z_tok >= theta ? sm.e_tok : 0.0;
      double mass = e_tok;   // x~'s weight with what is pooled onto it
      // where an id of the row is: the thread, its mask word, the bit in it
      struct Spot {
        int thread, word;
        uint32_t bit;
      };
      auto spot_of = [&](int x) -> Spot {
        const int pc = (x * (BF16 ? 2 : 4)) >> 7, grp = (int)(((float)pc + 0.5f) * inv_ppg), in_grp = pc - grp * a.ppg;
        return {grp * 8 + ((x / IDS) & 7), in_grp >> 2, 1u << ((in_grp & 3) * IDS + x % IDS)};
      };
      const Spot tok_spot = POOL ? spot_of(tok) : Spot{-1, 0, 0u};
      if constexpr (POOL) {
        // where N ids' weights are in the lists, and whose (<< 20); 0: not kept
        auto find = [&](auto n_tag, const int* x, uint32_t* at) {
          constexpr int N = decltype(n_tag)::value;
          Spot sp[N];
          uint32_t tm_at[N], last[N];
#pragma unroll
          for (int i = 0; i < N; ++i) {
            sp[i] = spot_of(max(x[i], 0));
            const bool o_up = ((sp[i].thread >> 5) & 1) == 0;
            tm_at[i] = my + a.o_tmask + (uint32_t)sp[i].thread * 4u;
            at[i] = my + ((uint32_t)(sp[i].thread >> 6) * (uint32_t)R + (o_up ? 0u : (uint32_t)(R - 1))) * 128u +
                    (((uint32_t)sp[i].thread & 31u) ^ (o_up ? 0u : rot)) * 4u;
            last[i] = x[i] >= 0 ? lds_u32(tm_at[i] + (uint32_t)(sp[i].word * NT) * 4u) & sp[i].bit : 0u;
          }
          bool any = false;
#pragma unroll
          for (int i = 0; i < N; ++i) any = any || last[i];
          if (__any_sync(kFull, any)) {
#pragma unroll 1
            for (int w = 0; w < n_words; ++w) {
#pragma unroll
              for (int i = 0; i < N; ++i) {   // entries of the words before the id's, of its own those below it
                const uint32_t m = lds_u32(tm_at[i] + (uint32_t)(w * NT) * 4u);
                const int n = __popc(w < sp[i].word ? m : w == sp[i].word ? m & (sp[i].bit - 1u) : 0u);
                at[i] += (uint32_t)(sp[i].thread & 32 ? -n : n) * 128u;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < N; ++i) at[i] = last[i] ? at[i] | (uint32_t)sp[i].thread << 20 : 0u;
        };
        // takes a weight out of its owner's list and sum (a list may name an id twice, or x~ itself)
        auto remove = [&](float w, uint32_t at) {
          uint32_t old;
          asm volatile("atom.shared.exch.b32 %0, [%1], %2;" : "=r"(old) : "r"(at & 0xfffffu), "r"(__float_as_uint(-w)) : "memory");
          if (__uint_as_float(old) > 0.f) atomicAdd(&sm.adj[at >> 20], __float2ull_rz(w * 1099511627776.0f));
        };
        const uint16_t* const list = a.nn + (size_t)tok * P.pool_k;   // (x~ first)
        const int nb = P.pool_k;
        const double limit = P.pool_delta * Z;
        double carry = 0.0;
        sm.adj[tid] = 0ull;
        if (tid == 0) sm.pool_cj = 0.0;
        __syncthreads();   // (every thread's entries are weights)
        int tile = 0;
#pragma unroll 1
        for (int base = 0; base < nb; base += NT * 8, ++tile) {
          const int j0 = base + tid * 8;
          float e[8];
          int id[8];
          uint32_t at[8];
          double sum = 0.0;
          {
            uint4 ids = pool_ids(list, nb, j0);
            if (pool_clamp(ids, j0 == 0, P.V)) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
#pragma unroll
            for (int i = 0; i < 8; ++i) id[i] = j0 + i < 1 || j0 + i >= nb ? -1 : pool_id(ids, i);
          }
          find(std::integral_constant<int, 4>{}, id, at);
          find(std::integral_constant<int, 4>{}, id + 4, at + 4);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            e[i] = at[i] ? fabsf(lds_f32(at[i] & 0xfffffu)) : 0.f;
            sum += (double)e[i];
          }
          double inc = sum;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += t;
          }
          // (the mass below a thread comes from its neighbour's inclusive sum: inc - sum would cancel small masses)
          double run = __shfl_up_sync(kFull, inc, 1);
          if (lane == 0) run = 0.0;
          if (lane == 31) sm.pool_sum[tile & 1][warp] = inc;
          __syncthreads();
          double total = carry;
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            if (w == warp) run += total;
            total += sm.pool_sum[tile & 1][w];
          }
          carry = total;
          int bad = nb;
          double c = run;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (id[i] >= 0) {
              c += (double)e[i];
              if (bad == nb && !(c < limit)) bad = j0 + i;
            }
          bad = __reduce_min_sync(kFull, bad);
          if (lane == 0) sm.pool_bad[warp] = bad;
          __syncthreads();
          bool in[8];
          int J = nb;   // the leading run n_1 .. n_J keeps its prefix mass below delta
#pragma unroll
          for (int w = 0; w < NW; ++w) J = min(J, sm.pool_bad[w]);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            in[i] = id[i] >= 0 && j0 + i < J;
            if (in[i]) {
              run += (double)e[i];
              if (j0 + i == J - 1 || (j0 + i == base + NT * 8 - 1)) sm.pool_cj = run;
            }
            if (in[i] && e[i] > 0.f) remove(e[i], at[i]);
          }
          if (J < nb) break;   // (uniform)
          __syncthreads();     // (the last tile's prefix mass before the next one's)
        }
        if (warp == NW - 1 && e_tok > 0.0) {   // x~ is drawn with its pooled weight, outside the lists
          uint32_t at;
          find(std::integral_constant<int, 1>{}, &tok, &at);
          if (lane == 0 && at) remove(fabsf(lds_f32(at & 0xfffffu)), at);
        }
        __syncthreads();
        mass = e_tok + sm.pool_cj;
        s_t = (float)fmax((double)s_t - (double)sm.adj[tid] * (1.0 / 1099511627776.0), 0.0);
      }
      // ---- the decision (Eq. 1 / Eq. 5) and what has to be drawn, the same in every warp
      int pending = kDrawTarget;
      double u_res = 0.0, u_tgt;
      if (ONE_KIND) {
        const uint32_t cell = g - (uint32_t)b * (uint32_t)(P.h * P.w);
        const uint4 v = row_philox(make_uint4(cell, (uint32_t)b + P.image_offset, P.round, 1u), make_uint2(P.seed_lo, P.seed_hi));
        u_tgt = uniform24(v.x);
      } else if (LISTED) {
        const uint4 v = row_philox(make_uint4(pick & kPickIndex, (uint32_t)b + P.image_offset, P.round, 0u), make_uint2(P.seed_lo, P.seed_hi));
        u_res = uniform24(v.y);
        u_tgt = uniform24(v.z);
        pending = (pick & kPickResidual) != 0u ? kDrawResidual : kDrawTarget;
      } else {
        const uint32_t* const rnd = sm.rnd[parent & 1][child & 15];
        int accepted;
        if (P.accept_mode == MULO_ACCEPT_THRESHOLD) accepted = mass >= P.tau * Z;
        else if (q_tok <= 0.0) accepted = mass > 0.0;
        else accepted = uniform24(rnd[0]) * q_tok * Z < mass;
        u_res = uniform24(rnd[1]);
        u_tgt = uniform24(rnd[2]);
        if (tid == 0) {
          a.flags[g] = accepted ? 0 : 1;
          if (a.p_tok || a.q_tok || a.accept_prob)
            row_write_probs(a.p_tok, a.q_tok, a.accept_prob, g, e_tok, mass, q_tok, Z,
                             P.accept_mode == MULO_ACCEPT_THRESHOLD);
        }
        pending = draws_for(P.resample_mode, accepted);
      }
      // weights in units of e = exp(z - ref): p -> e, q -> ratio * e_q
      const float ratio = LISTED ? (float)(Z / (double)Zq) : __fdividef((float)Z, (float)Zq);
      auto q_weight = [&](uint32_t at) -> float {
        float zq = dlist_get<BF16>(at);
        if (BF16 && !PLAIN) zq = __fmul_rn(zq, P.invT);
        return __fmul_rn(weight_of(zq, c0_q), ratio);
      };
      partner_n = pair_n;   // (this row's entries may still be searched when the next row is streamed)
      // weights of the owning group's parts: in fixed point, 2^31 = its weight, or (LISTED) as they are
      using Fx = typename std::conditional<LISTED, double, uint32_t>::type;
      const Fx past = LISTED ? (Fx)INFINITY : (Fx)~0u;
      auto fx_of = [&](Sum v, float to_fx) -> Fx {
        if constexpr (LISTED) return v;
        else return __float2uint_rn(__fmul_rn(v, to_fx));
      };
      static_assert(!LISTED || sizeof sm.rnd[0] >= NW * 4 * sizeof(double), "a double per set of eight threads");
      bool no_mass = false;
      int dcall = 0;
#pragma unroll 1
      do {
        const bool is_res = (pending & kDrawResidual) != 0;
        const bool resid = !ONE_KIND && is_res && !no_mass;
        Sum v_t = s_t;
        if (resid) {
          // sum of max(0, p - q) = p - min(p, q); min is not zero only where both rows kept the id
          uint32_t tp = tl, dp = dl;
          Sum mins = 0;
#pragma unroll 1
          for (int w = 0; w < n_words; ++w) {
            const uint32_t m = lds_u32(tm + (uint32_t)(w * NT) * 4u), d = lds_u32(dm + (uint32_t)(w * NT) * 4u);
            uint32_t im = m & d;
            const int trips = __reduce_max_sync(kFull, __popc(im));
            auto both = [&]() -> float {   // the next entry of the intersection
              const uint32_t bit = im & (0u - im), below = bit - 1u;
              im ^= bit;
              const float e = lds_f32(tp + (uint32_t)__popc(m & below) * step);
              const float q = q_weight(dp + (uint32_t)__popc(d & below) * dstep);
              return bit ? fminf(POOL ? fmaxf(e, 0.f) : e, q) : 0.f;
            };
#pragma unroll 1
            for (int i = 0; i < trips; i += 4) {   // four at a time: their chains overlap
              const float v0 = both(), v1 = both(), v2 = both(), v3 = both();
              mins += ((Sum)v0 + (Sum)v1) + ((Sum)v2 + (Sum)v3);
            }
            tp += (uint32_t)__popc(m) * step;
            dp += (uint32_t)__popc(d) * dstep;
          }
          v_t = s_t > mins ? s_t - mins : (Sum)0;
        }
        constexpr int NG = NW * 4;   // groups, and sets of eight threads in the search
        const double w_tok = !POOL ? 0.0 : resid ? fmax(mass - q_tok * Z, 0.0) : mass;   // x~'s weight outside the lists
        double w_grp = (double)v_t;
        if (POOL && tid == tok_spot.thread) w_grp += w_tok;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) w_grp += __shfl_xor_sync(kFull, w_grp, o);
        double* const ws = sm.w_draw[dcall & 1];
        Fx* const fxs = LISTED ? reinterpret_cast<Fx*>(sm.rnd[dcall & 1]) : reinterpret_cast<Fx*>(sm.fx[dcall & 1]);
        ++dcall;
        if ((lane & 7) == 0) ws[tid >> 3] = w_grp;
        __syncthreads();   // ---- barrier 3
        if (tid == 0) sm.n_sa = 0;
        // the group that owns u * total (the same in every warp)
        w_grp = ws[lane & (NG - 1)];
        double inc_d = w_grp;
#pragma unroll
        for (int o = 1; o < NG; o <<= 1) {
          const double t = __shfl_up_sync(kFull, inc_d, o, NG);
          if ((lane & (NG - 1)) >= o) inc_d += t;
        }
        const double total = __shfl_sync(kFull, inc_d, NG - 1);
        if (!(total > 0.0)) {
          if (resid) {
            no_mass = true;   // the same draw again, from the target weights
            continue;
          }
        } else {
          const double yt = (is_res ? u_res : u_tgt) * total;
          double exc_d = __shfl_up_sync(kFull, inc_d, 1, NG);
          if ((lane & (NG - 1)) == 0) exc_d = 0.0;
          const unsigned hit_g = __ballot_sync(kFull, lane < NG && inc_d > yt), has_g = __ballot_sync(kFull, lane < NG && w_grp > 0.0);
          const int og = hit_g ? __ffs(hit_g) - 1 : 31 - __clz(has_g);
          const float to_fx = __fdividef(2147483648.0f, (float)__shfl_sync(kFull, w_grp, og));
          const double yg = yt - __shfl_sync(kFull, exc_d, og);
          Fx y = past;
          if (hit_g) {
            if constexpr (LISTED) y = yg;
            else y = __double2uint_rz(yg * (double)to_fx);
          }
          const uint32_t tok_fx = POOL ? __double2uint_rn(fmin(w_tok * (double)to_fx, 4294967294.0)) : 0u;
          // the thread of the group whose entries this thread looks at, and where they are
          const int own = og * 8 + (lane & 7);
          const bool o_up = ((own >> 5) & 1) == 0;
          const uint32_t o_row = (uint32_t)(own >> 6) * (uint32_t)R + (o_up ? 0u : (uint32_t)(R - 1));
          const uint32_t o_step = o_up ? 128u : 0u - 128u, o_dstep = o_up ? DROW : 0u - DROW;
          const uint32_t o_tm = my + a.o_tmask + (uint32_t)own * 4u, o_dm = my + a.o_dmask + (uint32_t)own * 4u;
          const uint32_t o_tl = my + o_row * 128u + (((uint32_t)own & 31u) ^ (o_up ? 0u : rot)) * 4u;
          const uint32_t o_dl = my + a.o_dlist + o_row * DROW + (((uint32_t)own & 31u) ^ (o_up ? 0u : rot_q)) * (DROW / 32u);
          uint32_t m = 0, d = 0, ta = 0, da = 0;   // masks of the word in work and where its entries start
          auto weight = [&](uint32_t bit, uint32_t at) -> float {
            float e = fmaxf(lds_f32(bit ? at : closer), 0.f);   // (the closer's -inf)
            if (resid) {
              const float qv = q_weight(da + (uint32_t)__popc(d & (bit - 1u)) * o_dstep);
              e = (d & bit) ? fmaxf(__fsub_rn(e, qv), 0.f) : e;
            }
            return e;
          };
          auto entries = [&](uint32_t mm, uint32_t at) -> Fx {   // sum of the entries at the bits mm
            Sum sum = 0;
#pragma unroll 1
            while (mm) {
              const uint32_t b0 = mm & (0u - mm);
              mm ^= b0;
              const uint32_t b1 = mm & (0u - mm);
              mm ^= b1;
              const uint32_t b2 = mm & (0u - mm);
              mm ^= b2;
              const float v0 = weight(b0, at), v1 = weight(b1, at + o_step), v2 = weight(b2, at + 2 * o_step);
              sum += ((Sum)v0 + (Sum)v1) + (Sum)v2;
              at += 3 * o_step;
            }
            return fx_of(sum, to_fx);
          };
          auto go_to = [&](int w) {   // the state of word w
            ta = o_tl;
            da = o_dl;
#pragma unroll 1
            for (int k = 0; k < w; ++k) {
              ta += (uint32_t)__popc(lds_u32(o_tm + (uint32_t)(k * NT) * 4u)) * o_step;
              if (resid) da += (uint32_t)__popc(lds_u32(o_dm + (uint32_t)(k * NT) * 4u)) * o_dstep;
            }
          };
          auto load_word = [&](int w) {
            m = lds_u32(o_tm + (uint32_t)(w * NT) * 4u);
            d = resid ? lds_u32(o_dm + (uint32_t)(w * NT) * 4u) : 0u;
          };
          auto next_word = [&]() {
            ta += (uint32_t)__popc(m) * o_step;
            da += (uint32_t)__popc(d) * o_dstep;
          };
          const int wps = (n_words + NG - 1) / NG;   // words per set of eight threads
          {
            const int w0 = min((tid >> 3) * wps, n_words), w1 = min(w0 + wps, n_words);
            Fx v = 0;
            go_to(w0);
#pragma unroll 1
            for (int w = w0; w < w1; ++w) {
              load_word(w);
              v += entries(m, ta);
              if (POOL && own == tok_spot.thread && w == tok_spot.word) v += tok_fx;
              next_word();
            }
            __syncwarp();
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
            if ((lane & 7) == 0) fxs[tid >> 3] = v;
          }
          __syncthreads();   // ---- barrier 4
          if (warp == (og >> 2)) {
            Fx v = fxs[lane & (NG - 1)], inc = v;
#pragma unroll
            for (int o = 1; o < NG; o <<= 1) {
              const Fx t = __shfl_up_sync(kFull, inc, o, NG);
              if ((lane & (NG - 1)) >= o) inc += t;
            }
            unsigned hit = __ballot_sync(kFull, lane < NG && v > 0 && inc > y), has = __ballot_sync(kFull, lane < NG && v > 0);
            int src = hit ? __ffs(hit) - 1 : has ? 31 - __clz(has) : 0;
            y = hit ? y - __shfl_sync(kFull, inc - v, src) : past;
            // the set's words one by one: eight lanes to a piece
            const uint32_t piece_bits = ((1u << IDS) - 1u) << ((lane >> 3) * IDS), under = (1u << ((lane >> 3) * IDS)) - 1u;
            const int w0 = src * wps, w1 = min(w0 + wps, n_words);
            int w = w0, last_w = w0;
            bool seek = false;   // rounding left the sums short: the last word with weight
            go_to(w0);
#pragma unroll 1
            for (;;) {
              load_word(w);
              v = entries(m & piece_bits, ta + (uint32_t)__popc(m & under) * o_step);
              if (POOL && own == tok_spot.thread && w == tok_spot.word && (tok_spot.bit & piece_bits)) v += tok_fx;
              __syncwarp();
              Fx t;
              if constexpr (LISTED) t = warp_sum(v);
              else t = __reduce_add_sync(kFull, v);
              if (t > 0) last_w = w;
              if (seek ? w == last_w : y < t && (!LISTED || t > 0)) break;   // (in double y may be a rounding below 0)
              if (y != past) y -= t;
              next_word();
              if (++w == w1) {
                seek = true;
                y = past;
                w = last_w;
                go_to(w);
              }
            }
            inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const Fx t = __shfl_up_sync(kFull, inc, o);
              if (lane >= o) inc += t;
            }
            hit = __ballot_sync(kFull, v > 0 && inc > y);
            has = __ballot_sync(kFull, v > 0);
            src = hit ? __ffs(hit) - 1 : has ? 31 - __clz(has) : 0;
            y = hit ? y - __shfl_sync(kFull, inc - v, src) : past;
            // ... and the ids of the lane found: lane i takes id i
            m = __shfl_sync(kFull, m, src);
            d = __shfl_sync(kFull, d, src);
            ta = __shfl_sync(kFull, ta, src);
            da = __shfl_sync(kFull, da, src);
            const uint32_t bit = lane < IDS ? m & (1u << ((src >> 3) * IDS + lane)) : 0u;
            float wt = weight(bit, ta + (uint32_t)__popc(m & (bit - 1u)) * o_step);
            if (POOL && og * 8 + (src & 7) == tok_spot.thread && w == tok_spot.word && lane < IDS &&
                tok_spot.bit == 1u << ((src >> 3) * IDS + lane))
              wt += (float)w_tok;
            inc = fx_of((Sum)wt, to_fx);
#pragma unroll
            for (int o = 1; o < IDS; o <<= 1) {
              const Fx t = __shfl_up_sync(kFull, inc, o);
              if (lane >= o) inc += t;
            }
            hit = __ballot_sync(kFull, wt > 0.f && inc > y);
            has = __ballot_sync(kFull, wt > 0.f);
            // (no id with weight: a sum that was rounding noise of a difference -- to the general routines)
            const int chosen = hit ? __ffs(hit) - 1 : has ? 31 - __clz(has) : -1;
            int32_t* const out = ONE_KIND || LISTED ? a.sample_out + g : (is_res ? a.cand_res : a.cand_tgt) + g;
            if (lane == chosen) *out = (((og * a.ppg + w * 4 + (src >> 3)) << 3) + (src & 7)) * IDS + chosen;
            if (chosen < 0 && lane == 0) defer(g);
          }
        }
        pending &= ~(is_res ? kDrawResidual : kDrawTarget);
        no_mass = false;
      } while (pending);
    }

    if (rot != 0 || (nq && rot_q != 0)) {   // (the next row's columns pair up differently: nobody may still be at this one's)
      __syncthreads();
      rot = 0;
      partner_n = 0;
      if (nq) partner_q = 0;
    }
    // ---- on to the next row (its first pieces are in registers)
    if (!is_q) ++unit;
    if (!more) break;
    if (KIND == kRowsRound) {
      if (is_q) child = di * P.r + dj;
      else ++child;
    }
    if constexpr (LISTED) {
      if (!is_q) {
        b = b_next;
        pick = pick_next;
        parent = parent_next;
        if (--left > 0) next_pick();
      }
    } else {
      if (KIND == kRowsSample || nq) next_parent();
    }
    is_q = nq;
    g = ng;
  }
}

}  // namespace mulo
