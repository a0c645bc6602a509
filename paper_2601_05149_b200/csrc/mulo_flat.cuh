// The fast path for rows WITHOUT a top-k cut (the paper's default sampling setting): NW warps per row.
//
// Without a cut there is nothing to select: every entry of a row is exponentiated once, on its way through registers,
// and nothing of it is kept but sums.  A CTA owns a contiguous range of target rows (in parent order); per parent the
// draft row comes first, unless the decision rule and the resample mode never look at q (Eq. 5 with redraws from the
// target distribution), in which case the draft logits are not read at all.  The ids are split into 4 NW contiguous
// parts, one for every group of eight lanes, as in mulo_rows.cuh.
//
//   stream     128-byte pieces of each group's part, four in flight per lane, running on into the next row: CFG mix, exp
//              against a predicted maximum (the previous row's of the kind; a row whose maximum lies far from it is
//              streamed again), sums in fp32 per word of four pieces, in double above.  One block barrier, and the
//              partition sum and every group's slice of the ascending-id CDF are known.
//   draws      the group that owns u * total; in its warp the word that owns what is left, its 256 ids once more from the
//              row (L2, one 16-byte load per lane), the id.  The other warps are on their way with the next row.
//
// RES: where a row is needed again -- pooling, residual redraws -- its weights (fp32) stay in shared memory, 4 V bytes, and
// eight warps share a row (pooled rows with target redraws only: where mulo_full.cuh's kernel cannot take them).
//
//   pooling    (POOL, Eq. 3-4) eight entries of x~'s neighbour list per thread, their weights straight from shared memory;
//              prefix masses by a block scan; what is pooled is set to zero there, x~'s own weight too (it is drawn apart).
//              Then the draw's pass below adds up what is left.
//   residual   one pass over the weights and the draft row (L2): sums of max(0, p' - q).
//   draws      the owning group's weights, 16 ids per lane, then the owning lane's ids, one per lane.
//
// Bound: without RES by the loads (16384 rows of V = 16384 bf16 with guidance, no pooling: 207 us, 5.2 TB/s); with it by
// instruction issue and by the barriers of a row at two CTAs per SM (the same rows with residual redraws: 416 us; with lists
// of 1000 too: 388 us, 12.7 k warp instructions per row and its quarter of a draft row).  The kernel before this one copied
// the raw rows to shared memory, 64 to 96 KB per position, with nothing of the next row in flight: 273, 724 and 566 us.
// Draft draws without a cut went to the general routines: 195 us for 4096 rows, now 35.
// Measured and not kept: pooled logits gathered from L2 instead of shared memory (470 us: half of the time the row is out of
// L2), three CTAs per SM at 80 registers (spills, which share what shared memory leaves of L1: 384 to 411 us).
#pragma once

#include "mulo_rows.cuh"

namespace mulo {

// Warps per row.  Two without RES: what each warp of a row repeats counts least (four 217 us, eight 254 us where two take
// 207; at 256 and 1024 rows they are within 10 % of each other).  Eight with it: two CTAs of 64 KB are what an SM holds, and
// a neighbour list of 2048 is eight entries per thread.
constexpr int kFlatWarps = 2, kFlatResWarps = 8;
constexpr int kFlatMaxRatio = 8;   // the uniforms of r * r children are kept

struct FlatArgs {
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
  int32_t* cand_res;
  int32_t* cand_tgt;
  int32_t* sample_out;      // SAMPLE: the drafter's token per cell
  uint32_t* dev_status;
  int n_units;              // target rows, parent by parent (SAMPLE: low-res cells)
  uint32_t row_bytes;
  int ppg;                  // pieces of a group's part of a row
  int n_words;              // words of four pieces per thread
  int need_q;               // 0: neither the decision nor any draw uses the draft distribution
};

template <int NW>
struct FlatSmem {
  double w_grp[2][NW * 4];                 // weights of the groups; consecutive uses alternate
  unsigned wmax[2][NW];
  double e_tok[2];                         // x~'s own weight
  uint32_t rnd[2][kFlatMaxRatio * kFlatMaxRatio][3];   // uniforms of the parent's children, by parity of the parent
  double pool_sum[NW], pool_cj[NW];
};

// Dynamic shared memory of a CTA (bytes): the row's weights, or a sum per word and thread.
inline uint32_t flat_smem(const FlatArgs& s, int nw, bool res) {
  return res ? (uint32_t)((s.P.V + 31) & ~31) * 4u : (uint32_t)s.n_words * nw * 128u;
}

// Inclusive and exclusive sums over every W lanes of a warp.  (Inlined: the row waits for it, and a rolled copy took 10 % off
// the whole kernel's rate.)
struct FlatScan {
  double inc, exc;
};
// v += the value O lanes below, where there is one among W (the shuffle's own predicate)
template <int O, int W>
__device__ __forceinline__ void flat_scan_step(double& v) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 lo, hi;\n\t.reg .f64 t;\n\t"
      "mov.b64 {lo, hi}, %0;\n\t"
      "shfl.sync.up.b32 lo, lo, %1, %2, 0xffffffff;\n\t"
      "shfl.sync.up.b32 hi|p, hi, %1, %2, 0xffffffff;\n\t"
      "mov.b64 t, {lo, hi};\n\t"
      "@p add.f64 %0, %0, t;\n\t}"
      : "+d"(v)
      : "n"(O), "n"((32 - W) << 8));
}
template <int W>
__device__ __forceinline__ FlatScan flat_scan(double v) {
  if constexpr (W > 1) flat_scan_step<1, W>(v);
  if constexpr (W > 2) flat_scan_step<2, W>(v);
  if constexpr (W > 4) flat_scan_step<4, W>(v);
  if constexpr (W > 8) flat_scan_step<8, W>(v);
  if constexpr (W > 16) flat_scan_step<16, W>(v);
  // (not inc - v: that would cancel small values)
  const double e = __shfl_up_sync(kFull, v, 1);
  return {v, (threadIdx.x & (W - 1)) == 0 ? 0.0 : e};
}

struct FlatGroups {
  double w, inc, exc, total;   // of group (lane % NG): its weight, inclusive and exclusive sums; the total
};

// the logits of one lane's 16 bytes
template <bool BF16, bool ROW_U, bool SCALE>
__device__ __forceinline__ void flat_logits(const uint4& c, const uint4& u, float2 s2, float2 t2, float2 (&z)[BF16 ? 4 : 2]) {
  z[0] = row_pair<BF16, ROW_U, SCALE, 0>(c, u, s2, t2);
  z[1] = row_pair<BF16, ROW_U, SCALE, 1>(c, u, s2, t2);
  if constexpr (BF16) {
    z[2] = row_pair<BF16, ROW_U, SCALE, 2>(c, u, s2, t2);
    z[3] = row_pair<BF16, ROW_U, SCALE, 3>(c, u, s2, t2);
  }
}

// EVEN: every word four whole pieces (V splits evenly), so no bounds checks; they cost up to 45 us of 145 (4608 rows of 8192
// fp32 ids with guidance, T = 0.9, no pooling).  SCALE: T is not 1.
template <bool BF16, bool HAS_U, bool SAMPLE, bool POOL, bool RES, bool EVEN, bool SCALE>
__global__ void __launch_bounds__((RES ? kFlatResWarps : kFlatWarps) * 32, (SAMPLE ? 24 : 16) / (RES ? kFlatResWarps : kFlatWarps))
    k_round_flat(const __grid_constant__ FlatArgs a) {
  constexpr int NW = RES ? kFlatResWarps : kFlatWarps;
  constexpr int NT = NW * 32, NG = NW * 4;
  constexpr int IDS = BF16 ? 8 : 4;              // ids per lane per piece
  constexpr int DEPTH = 4;                       // pieces in flight per lane
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ FlatSmem<NW> sm;
  const DevParams& P = a.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  let_next_begin();
  int unit = (int)(((long long)a.n_units * blockIdx.x) / gridDim.x);
  const int u_end = (int)(((long long)a.n_units * (blockIdx.x + 1)) / gridDim.x);
  if (unit >= u_end) return;
  const int rr = SAMPLE ? 1 : P.r * P.r;
  const bool need_q = !SAMPLE && a.need_q != 0;
  const uint32_t row_bytes = a.row_bytes;
  const int n_words = a.n_words;
  const float inv_ppg = 1.0f / (float)a.ppg;
  float* const wsum = reinterpret_cast<float*>(dyn);   // [n_words][NT]
  // RES: place of an id's weight: 16-byte chunks, the upper four of eight lanes' first chunks moved to the other banks
  auto e_at = [&](int x) -> float* { return reinterpret_cast<float*>(dyn + ((x << 2) ^ ((x >> 1) & 16))); };

  // ---- where the current row is.  parent = low-res cell (b, ca, cc); child (di, dj) of a target row.
  int parent, b, ca, cc, di = 0, dj = 0;
  {
    parent = unit / rr;
    const int child = unit - parent * rr, hw = P.h * P.w;
    b = parent / hw;
    const int rem = parent - b * hw;
    ca = rem / P.w;
    cc = rem - ca * P.w;
    if (!SAMPLE) {
      di = child / P.r;
      dj = child - di * P.r;
    }
  }
  auto target_index = [&]() -> uint32_t {
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
  const uint32_t part_off = (uint32_t)((tid >> 3) * a.ppg) * kRPieceBytes + (uint32_t)(lane & 7) * 16u;
  const int np = part_off < row_bytes ? min(a.ppg, (int)((row_bytes - part_off + kRPieceBytes - 1) / kRPieceBytes)) : 0;
  uint4 c[DEPTH], u[DEPTH];   // the pieces in flight
  const uint4 zero = make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int j = 0; j < DEPTH; ++j) c[j] = u[j] = zero;
  auto prologue = [&](const char* rc, const char* ru) {
#pragma unroll
    for (int j = 0; j < DEPTH; ++j)
      if (j < np) {
        c[j] = ldg_stream(rc + j * kRPieceBytes);
        if (HAS_U && ru) u[j] = ldg_stream(ru + j * kRPieceBytes);
      }
  };
  const float2 s2 = make_float2(P.cfg_scale, P.cfg_scale), t2 = make_float2(P.invT, P.invT), l2 = make_float2(kLog2e, kLog2e);
  // ---- one row through the registers; the loads run on into the row (nc, nu).  (All row pointers are this thread's.)
  //      Word sums of exp(z - ref) to shared memory; returns their sum, and the maximum in mx.
  auto stream = [&](auto row_u_tag, const char* rc, const char* ru, const char* nc, const char* nu, float c0, bool keep, float& mx) -> double {
    constexpr bool ROW_U = decltype(row_u_tag)::value;
    const float2 c2 = make_float2(c0, c0);
    double sum = 0.0;
    mx = -INFINITY;
    int x0 = (int)part_off / (BF16 ? 2 : 4);
#pragma unroll 1
    for (int w = 0; w < n_words; ++w) {
      const bool last = w + 1 == n_words;
      const char* const fc = last ? nc : rc + 4 * kRPieceBytes;
      const char* const fu = !HAS_U ? nullptr : last ? nu : ROW_U ? ru + 4 * kRPieceBytes : nullptr;
      const bool do_u = HAS_U && fu != nullptr;
      const int f0 = last ? 0 : 4 * w + 4;
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (EVEN || 4 * w + j < np) {
          float2 z[IDS / 2];
          flat_logits<BF16, ROW_U, SCALE>(c[j], u[j], s2, t2, z);
#pragma unroll
          for (int k = 0; k < IDS / 2; ++k) {
            mx = fmaxf(mx, fmaxf(z[k].x, z[k].y));
            const float2 t = __ffma2_rn(z[k], l2, c2);
            z[k] = make_float2(ex2f(t.x), ex2f(t.y));
            acc = __fadd2_rn(acc, z[k]);
          }
          if (RES && keep) {
            *reinterpret_cast<float4*>(e_at(x0 + j * (8 * IDS))) = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
            if constexpr (BF16)
              *reinterpret_cast<float4*>(e_at(x0 + j * (8 * IDS) + 4)) = make_float4(z[2].x, z[2].y, z[3].x, z[3].y);
          }
        }
        if (EVEN || f0 + j < np) {
          c[j] = ldg_stream(fc + j * kRPieceBytes);
          if (do_u) u[j] = ldg_stream(fu + j * kRPieceBytes);
        }
      }
      const float s = acc.x + acc.y;
      if (!RES) wsum[w * NT + tid] = s;
      sum += (double)s;
      x0 += 32 * IDS;
      rc += 4 * kRPieceBytes;
      if (HAS_U && ROW_U) ru += 4 * kRPieceBytes;
    }
    return sum;
  };

  // ---- group sums of a value per thread, scanned in id order (every warp has them; one block barrier)
  int call = 0;   // consecutive calls alternate between two buffers
  auto scan_groups = [&](double v) -> FlatGroups {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
    double* const ws = sm.w_grp[call & 1];
    if ((lane & 7) == 0) ws[tid >> 3] = v;
    __syncthreads();
    ++call;
    FlatGroups s;
    s.w = fmax(ws[lane & (NG - 1)], 0.0);
    const FlatScan sc = flat_scan<NG>(s.w);
    s.inc = sc.inc;
    s.exc = sc.exc;
    s.total = __shfl_sync(kFull, s.inc, NG - 1);
    return s;
  };

  auto block_sum = [&](double v) -> double {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    double* const ws = sm.w_grp[call & 1];
    if (lane == 0) ws[warp] = v;
    __syncthreads();
    ++call;
    double sum = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) sum += ws[w];
    return sum;
  };

  auto row_c = [&](bool q, uint32_t g) -> const char* { return (q ? a.draft : a.cond) + (size_t)g * row_bytes; };
  auto row_u = [&](bool q, uint32_t g) -> const char* { return HAS_U && !q ? a.uncond + (size_t)g * row_bytes : nullptr; };
  auto part = [&](const char* row) -> const char* { return row ? row + part_off : nullptr; };
  auto prefetch = [&](const char* rc, const char* ru) {   // one thread
    prefetch_l2(rc, row_bytes);
    if (HAS_U && ru) prefetch_l2(ru, row_bytes);
  };

  bool is_q = need_q;                     // the row in work is a draft row
  uint32_t g = is_q || SAMPLE ? (uint32_t)parent : target_index();   // ... and its index in its tensor
  bool again = false, first = true;       // the row is streamed again / the first under its parent
  int tok = 0;
  float ref_q = 0.f, ref_t = 0.f;         // the last row's maximum, by kind
  bool have_q = false, have_t = false;
  float c0_q = 0.f, Zq = 1.f;             // of the parent's draft row
  double q_tok = 0.0;
  int tok_next = SAMPLE ? 0 : __ldg(a.draft_tok_lo + parent);
  prologue(part(row_c(is_q, g)), part(row_u(is_q, g)));

#pragma unroll 1
  for (;;) {
    const char* const rc = row_c(is_q, g);
    const char* const ru = row_u(is_q, g);
    // ---- the row after this one (place of the next child in ndi, ndj)
    bool nq = false, np_new = false, more = true;
    uint32_t ng = g;
    int ndi = di, ndj = dj;
    if (SAMPLE) {
      more = unit + 1 < u_end;
      ng = more ? g + 1 : g;
      np_new = true;
    } else if (is_q) {
      ng = target_index();
    } else if (unit + 1 >= u_end) {
      more = false;
    } else if (dj + 1 < P.r || di + 1 < P.r) {
      if (++ndj == P.r) {
        ndj = 0;
        ++ndi;
      }
      ng = ((uint32_t)b * P.H + (uint32_t)(ca * P.r + ndi)) * P.W + (uint32_t)(cc * P.r + ndj);
    } else {
      np_new = true;
      nq = need_q;
      if (need_q) {
        ng = (uint32_t)parent + 1u;
      } else {
        const bool wrap = cc + 1 == P.w, wrap2 = wrap && ca + 1 == P.h;
        ng = ((uint32_t)(b + (wrap2 ? 1 : 0)) * P.H + (uint32_t)((wrap2 ? 0 : ca + (wrap ? 1 : 0)) * P.r)) * P.W +
             (uint32_t)((wrap ? 0 : cc + 1) * P.r);
      }
    }
    const char* const nc = row_c(nq, ng);            // (no row left: this one's first pieces again)
    const char* const nu = more ? row_u(nq, ng) : nullptr;
    if (RES && more && tid == 0) prefetch(nc, nu);   // (without RES as many rows as there are CTAs do not fit into L2: 207 -> 251 us)
    // the logit of x~ in this row: asked for now, used after the row
    uint32_t raw_c = 0u, raw_u = 0u;   // (as they are: a conversion here would wait for them)
    if (!SAMPLE) {
      if (first) {
        tok = tok_next;
        if (tok < 0 || tok >= P.V) {
          if (tid == 0) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
          tok = min(max(tok, 0), P.V - 1);
        }
        tok_next = __ldg(a.draft_tok_lo + min(parent + 1, P.B * P.h * P.w - 1));
        if (POOL && tid == 0) pool_prefetch(a.nn + (size_t)tok * P.pool_k, P.pool_k);
      }
      if (warp == NW - 1) {
        raw_c = raw_logit<BF16>(rc, tok);
        if (HAS_U && !is_q) raw_u = raw_logit<BF16>(ru, tok);
      }
    }
    // ---- the exp reference
    float ref = is_q ? ref_q : ref_t;
    if (!again && !(is_q ? have_q : have_t)) {   // the maximum of the first pieces
      float m = -INFINITY;
#pragma unroll
      for (int j = 0; j < DEPTH; ++j)
        if (j < np) {
          float2 z[IDS / 2];
          if (HAS_U && !is_q) flat_logits<BF16, HAS_U, SCALE>(c[j], u[j], s2, t2, z);
          else flat_logits<BF16, false, SCALE>(c[j], u[j], s2, t2, z);
#pragma unroll
          for (int k = 0; k < IDS / 2; ++k) m = fmaxf(m, fmaxf(z[k].x, z[k].y));
        }
      const unsigned mk = __reduce_max_sync(kFull, float_key(m));
      if (lane == 0) sm.wmax[call & 1][warp] = mk;
      __syncthreads();
      unsigned all = 0;
#pragma unroll
      for (int w = 0; w < NW; ++w) all = max(all, sm.wmax[call & 1][w]);
      ref = key_float(all);
      __syncthreads();
    }
    const float c0 = -ref * kLog2e;
    float mx;
    const uint16_t* const list = POOL ? a.nn + (size_t)tok * P.pool_k : nullptr;   // the neighbours of x~ (itself first)
    const int nb = P.pool_k;
    uint4 ids = zero;
    if (POOL && !is_q && warp * 256 < nb) ids = pool_ids(list, nb, tid * 8);
    double s_t;
    if (HAS_U && !is_q) s_t = stream(std::integral_constant<bool, HAS_U>{}, part(rc), part(ru), part(nc), part(nu), c0, !is_q, mx);
    else s_t = stream(std::false_type{}, part(rc), part(ru), part(nc), part(nu), c0, !is_q, mx);
    {
      const unsigned mk = __reduce_max_sync(kFull, float_key(mx));
      if (lane == 0) sm.wmax[call & 1][warp] = mk;
    }
    if (!SAMPLE && warp == NW - 1) {
      // the token's own weight
      const float z = mix_logit(wide_logit<BF16>(raw_c), wide_logit<BF16>(raw_u), HAS_U && !is_q, P.cfg_scale, P.invT);
      const double e = token_weight(z, ref, c0);
      if (lane == 0) sm.e_tok[call & 1] = e;
    }
    if (warp == 0 && first) {   // the uniforms of the parent's rows (the cell's)
#pragma unroll 1
      for (int i = lane; i < rr; i += 32) {
        const int ddi = SAMPLE ? 0 : i / P.r, ddj = i - ddi * P.r;
        const uint32_t t = SAMPLE ? (uint32_t)ca * P.w + (uint32_t)cc : (uint32_t)(ca * P.r + ddi) * P.W + (uint32_t)(cc * P.r + ddj);
        const uint4 v = row_philox(make_uint4(t, (uint32_t)b + P.image_offset, P.round, SAMPLE ? 1u : 0u),
                                    make_uint2(P.seed_lo, P.seed_hi));
        sm.rnd[parent & 1][i][0] = v.x;
        sm.rnd[parent & 1][i][1] = v.y;
        sm.rnd[parent & 1][i][2] = v.z;
      }
    }
    first = false;
    const int buf = call & 1;
    // ---- the row's block barrier.  (With pooling the draws make their own sums; of the row, only the total is needed.)
    FlatGroups gs;
    if constexpr (POOL) {
      gs.total = block_sum(s_t);
      gs.w = gs.inc = gs.exc = 0.0;
    } else {
      gs = scan_groups(s_t);
    }
    unsigned mk = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) mk = max(mk, sm.wmax[buf][w]);
    mx = key_float(mk);
    if (!(fabsf(mx - ref) <= kNearRefGap) && !again) {   // CTA-uniform
      again = true;
      (is_q ? ref_q : ref_t) = mx;
      prologue(part(rc), part(ru));
      continue;
    }
    again = false;
    const double Z = gs.total > 0.0 ? gs.total : (double)NAN;   // (no number, and no probability, where the largest logit is +inf)
    if (is_q) {
      ref_q = mx;
      have_q = true;
      c0_q = c0;
      Zq = (float)Z;
      q_tok = rows_div(sm.e_tok[buf], Z);
      if (q_tok <= 0.0 && tid == 0) atomicOr(a.dev_status, MULO_DEV_ZERO_DRAFT_PROB);
    } else {
      ref_t = mx;
      have_t = true;
      const double e_tok = SAMPLE ? 0.0 : sm.e_tok[buf];
      double mass = e_tok;   // x~'s weight with what is pooled onto it
      // the thread that x~'s weight belongs to
      const int tok_owner = [&] {
        const int pc = (tok * (BF16 ? 2 : 4)) >> 7;
        return POOL ? (int)(((float)pc + 0.5f) * inv_ppg) * 8 + ((tok / IDS) & 7) : -1;
      }();
      if constexpr (POOL) {
        static_assert(!POOL || (RES && NT * 8 >= 2048), "a neighbour list is at most this long");
        const double limit = P.pool_delta * Z;
        const int j0 = tid * 8;
        const bool bad_id = pool_clamp(ids, tid == 0, P.V);
        if (tid == 0) ids.x = (ids.x & 0xffff0000u) | (uint32_t)tok;   // (entry 0 is x~ itself)
        const bool mine = warp * 256 < nb;   // (warp-uniform)
        float e[8];
        double sum = 0.0, run = 0.0, cj = 0.0;
        if (mine) {
          if (bad_id) atomicOr(a.dev_status, MULO_DEV_BAD_TOKEN);
#pragma unroll
          for (int i = 0; i < 8; ++i) e[i] = *e_at(pool_id(ids, i));
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if (j0 + i >= nb || j0 + i == 0) e[i] = 0.f;
            sum += (double)e[i];
          }
          const FlatScan sc = flat_scan<32>(sum);
          run = sc.exc;
          if (lane == 31) sm.pool_sum[warp] = sc.inc;
        }
        __syncthreads();
        if (mine) {
          double below = 0.0;
#pragma unroll
          for (int w = 0; w < NW; ++w) below += w < warp ? sm.pool_sum[w] : 0.0;
          run += below;
          // the leading run of neighbours whose prefix mass is below delta (prefix masses do not fall, so each thread
          // can tell for its own entries); its mass is the largest of them
          int n_in = 0;
          if (run + sum < limit) {
            n_in = 8;
            cj = run + sum;
          } else if (run < limit) {
            bool go = true;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              go = go && run + (double)e[i] < limit;
              if (go) {
                run += (double)e[i];
                n_in = i + 1;
              }
            }
            cj = run;
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i < n_in) *e_at(pool_id(ids, i)) = 0.f;   // (past the list's end: the last one again, which the run has reached)
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) cj = fmax(cj, __shfl_xor_sync(kFull, cj, o));
        }
        if (lane == 0) sm.pool_cj[warp] = cj;
        if (tid == NT - 1) *e_at(tok) = 0.f;   // x~ is drawn with its pooled weight
        __syncthreads();
        cj = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) cj = fmax(cj, sm.pool_cj[w]);
        mass = e_tok + cj;
      }
      // ---- the decision (Eq. 1 / Eq. 5) and what has to be drawn, the same in every warp
      int pending = kDrawTarget, accepted = 0, owner = 0;
      double u_res = 0.0, u_tgt;
      if (SAMPLE) {
        u_tgt = uniform24(sm.rnd[parent & 1][0][0]);
      } else {
        const uint32_t* const rnd = sm.rnd[parent & 1][di * P.r + dj];
        if (P.accept_mode == MULO_ACCEPT_THRESHOLD) accepted = mass >= P.tau * Z;
        else if (q_tok <= 0.0) accepted = mass > 0.0;
        else accepted = !(uniform24(rnd[0]) * q_tok * Z >= mass);
        u_res = uniform24(rnd[1]);
        u_tgt = uniform24(rnd[2]);
        pending = draws_for(P.resample_mode, accepted);
      }
      // weights in units of e = exp(z - ref): p -> e, q -> ratio * e_q
      const float ratio = __fdividef((float)Z, Zq);
      const char* const qrow = SAMPLE ? nullptr : a.draft + (size_t)parent * row_bytes;
      // the weights of one lane's ids from x on: those of the row, or max(0, p - q) with the draft's 16 bytes
      auto weights = [&](auto resid_tag, const uint4& qv, int x, float* w) {
        *reinterpret_cast<float4*>(w) = *reinterpret_cast<const float4*>(e_at(x));
        if constexpr (BF16) *reinterpret_cast<float4*>(w + 4) = *reinterpret_cast<const float4*>(e_at(x + 4));
        if constexpr (decltype(resid_tag)::value) {
          float2 z[IDS / 2];
          flat_logits<BF16, false, SCALE>(qv, qv, s2, t2, z);
          const float2 cq = make_float2(c0_q, c0_q);
#pragma unroll
          for (int k = 0; k < IDS / 2; ++k) {
            const float2 t = __ffma2_rn(z[k], l2, cq);
            w[2 * k] = fmaxf(__fsub_rn(w[2 * k], __fmul_rn(ex2f(t.x), ratio)), 0.f);
            w[2 * k + 1] = fmaxf(__fsub_rn(w[2 * k + 1], __fmul_rn(ex2f(t.y), ratio)), 0.f);
          }
        }
      };
      bool no_mass = false;
#pragma unroll 1
      do {
        const bool is_res = (pending & kDrawResidual) != 0;
        const bool resid = RES && is_res && !no_mass;
        const double w_tok = !POOL ? 0.0 : resid ? fmax(mass - q_tok * Z, 0.0) : mass;   // x~'s weight outside the sums
        FlatGroups ds = gs;
        // sums of the draw's weights per thread and word; returns this thread's
        auto pass = [&](auto resid_tag) -> double {
          constexpr bool RESID = decltype(resid_tag)::value;
          double sum = 0.0;
          const char* pq = RESID ? qrow + part_off : nullptr;
          int x = (int)part_off / (BF16 ? 2 : 4);
#pragma unroll 1
          for (int w = 0; w < n_words; ++w) {
            float2 s0 = make_float2(0.f, 0.f), s1 = s0;
            uint4 qv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              qv[j] = zero;
              if (RESID && (EVEN || 4 * w + j < np)) qv[j] = ldg_stream(pq + j * kRPieceBytes);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (EVEN || 4 * w + j < np) {
                alignas(16) float v[IDS];
                weights(resid_tag, qv[j], x + j * (8 * IDS), v);
#pragma unroll
                for (int k = 0; k < IDS; k += 4) {
                  s0 = __fadd2_rn(s0, make_float2(v[k], v[k + 1]));
                  s1 = __fadd2_rn(s1, make_float2(v[k + 2], v[k + 3]));
                }
              }
            sum += (double)((s0.x + s1.x) + (s0.y + s1.y));
            if (RESID) pq += 4 * kRPieceBytes;
            x += 32 * IDS;
          }
          if (POOL && tid == tok_owner) sum += w_tok;
          return sum;
        };
        if constexpr (RES) {
          if (resid) ds = scan_groups(pass(std::true_type{}));
          else if constexpr (POOL) ds = scan_groups(pass(std::false_type{}));
        }
        if (!(ds.total > 0.0)) {
          if (resid) {
            no_mass = true;   // the same draw again, from the target weights
            continue;
          }
          if (tid == 0) (SAMPLE ? a.sample_out : is_res ? a.cand_res : a.cand_tgt)[g] = -1;
        } else {
          const double yt = (is_res ? u_res : u_tgt) * ds.total;
          const unsigned hit_g = __ballot_sync(kFull, lane < NG && ds.inc > yt), has_g = __ballot_sync(kFull, lane < NG && ds.w > 0.0);
          const int og = hit_g ? __ffs(hit_g) - 1 : 31 - __clz(has_g);
          owner = og >> 2;
          if (warp == owner) {
            double y = hit_g ? yt - __shfl_sync(kFull, ds.exc, og) : 1e300;
            __syncwarp();
            int pick;
            if constexpr (RES) {
              // ---- the group's ids, 16 to a lane, until the lane is found that owns y; then its ids, one to a lane
              const int g_ids = a.ppg * (kRPieceBytes / (BF16 ? 2 : 4)), g0 = og * g_ids, g1 = min(g0 + g_ids, P.V);
              auto weight16 = [&](int x, float (&v)[16]) {
#pragma unroll
                for (int k = 0; k < 16; k += IDS) {
                  if (x + k < g1) {
                    if (resid) weights(std::true_type{}, ldg_stream(qrow + (size_t)(x + k) * (BF16 ? 2 : 4)), x + k, v + k);
                    else weights(std::false_type{}, zero, x + k, v + k);
                  } else {
#pragma unroll
                    for (int i = 0; i < IDS; ++i) v[k + i] = 0.f;
                  }
                }
                if (POOL) {
#pragma unroll
                  for (int k = 0; k < 16; ++k)
                    if (x + k == tok) v[k] = (float)w_tok;
                }
              };
              alignas(16) float v[16];
              double done = 0.0, y16 = 1e300;
              int x16 = -1, src = 0;
#pragma unroll 1
              for (int x0 = g0; x0 < g1; x0 += 512) {
                weight16(x0 + lane * 16, v);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < 16; k += 4) s += (v[k] + v[k + 1]) + (v[k + 2] + v[k + 3]);
                const FlatScan sc = flat_scan<32>((double)s);
                const unsigned hit = __ballot_sync(kFull, s > 0.f && done + sc.inc > y), has = __ballot_sync(kFull, s > 0.f);
                if (hit || has) {   // (rounding may leave the sums short of y: the last with weight stands in)
                  src = hit ? __ffs(hit) - 1 : 31 - __clz(has);
                  x16 = x0 + src * 16;
                  if (hit) {
                    y16 = y - (done + __shfl_sync(kFull, sc.exc, src));
                    break;
                  }
                }
                done += __shfl_sync(kFull, sc.inc, 31);
              }
              x16 = max(x16, g0);
              float w1 = 0.f;
              const int x = x16 + (lane & 15);
              if (x < g1) {
                w1 = *e_at(x);
                if (resid) {
                  const uint32_t rq = raw_logit<BF16>(qrow, x);
                  const float zq = mix_logit(wide_logit<BF16>(rq), 0.f, false, 0.f, P.invT);
                  w1 = fmaxf(__fsub_rn(w1, __fmul_rn(ex2f(fmaf(zq, kLog2e, c0_q)), ratio)), 0.f);
                }
                if (POOL && x == tok) w1 = (float)w_tok;
              }
              const FlatScan sc = flat_scan<16>((double)w1);
              const unsigned hit = __ballot_sync(kFull, w1 > 0.f && sc.inc > y16) & 0xffffu, has = __ballot_sync(kFull, w1 > 0.f) & 0xffffu;
              pick = x16 + (hit ? __ffs(hit) - 1 : has ? 31 - __clz(has) : 0);
              if (lane == 0) {
                int32_t* const out = (is_res ? a.cand_res : a.cand_tgt) + g;
                *out = pick;
              }
            } else {
            // ---- the word: lane l adds up word l of the group's eight threads
            int word = 0;
            {
              double done = 0.0;
              int last_w = 0;
              double last_exc = 0.0;
              bool found = false;
#pragma unroll 1
              for (int w0 = 0; w0 < n_words && !found; w0 += 32) {
                const int w = w0 + lane;
                double t = 0.0;
                if (w < n_words) {
                  const float4 p0 = *reinterpret_cast<const float4*>(wsum + w * NT + og * 8);
                  const float4 p1 = *reinterpret_cast<const float4*>(wsum + w * NT + og * 8 + 4);
                  t = (((double)p0.x + (double)p0.y) + ((double)p0.z + (double)p0.w)) +
                      (((double)p1.x + (double)p1.y) + ((double)p1.z + (double)p1.w));
                }
                const FlatScan sc = flat_scan<32>(t);
                const double inc = sc.inc, exc = sc.exc;
                const unsigned hit = __ballot_sync(kFull, t > 0.0 && done + inc > y), has = __ballot_sync(kFull, t > 0.0);
                if (hit || has) {
                  const int src = hit ? __ffs(hit) - 1 : 31 - __clz(has);
                  last_w = w0 + src;
                  last_exc = done + __shfl_sync(kFull, exc, src);
                  found = hit != 0;
                }
                done += __shfl_sync(kFull, inc, 31);
              }
              word = last_w;
              y = found ? y - last_exc : 1e300;   // (rounding left the sums short: the last word with weight)
            }
            // ---- its ids once more from the row: eight lanes to a piece
            const int pg = word * 4 + (lane >> 3);
            const uint32_t at = (uint32_t)(og * a.ppg + pg) * kRPieceBytes + (uint32_t)(lane & 7) * 16u;
            alignas(16) float v[IDS];
#pragma unroll
            for (int k = 0; k < IDS; ++k) v[k] = 0.f;
            const int x0 = (int)(at / (BF16 ? 2u : 4u));
            if (pg < a.ppg && at < row_bytes) {
              float2 z[IDS / 2];
              const uint4 cv = ldg_stream(rc + at), uv = HAS_U ? ldg_stream(ru + at) : zero;
              flat_logits<BF16, HAS_U, SCALE>(cv, uv, s2, t2, z);
#pragma unroll
              for (int k = 0; k < IDS; ++k) v[k] = ex2f(fmaf(k & 1 ? z[k / 2].y : z[k / 2].x, kLog2e, c0));
            }
            __syncwarp();
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < IDS; ++k) t += (double)v[k];
            const FlatScan sc = flat_scan<32>(t);
            const double inc = sc.inc, exc = sc.exc;
            const unsigned hit = __ballot_sync(kFull, t > 0.0 && inc > y), has = __ballot_sync(kFull, t > 0.0);
            const int src = hit ? __ffs(hit) - 1 : has ? 31 - __clz(has) : 0;
            if (!hit) y = 1e300;
            if (lane == src) {
              pick = -1;
              double cum = exc;
#pragma unroll
              for (int k = 0; k < IDS; ++k) {
                if (v[k] > 0.f && !(pick >= 0 && cum > y)) pick = k;   // (the first past y, else the last with weight)
                cum += (double)v[k];
              }
              int32_t* const out = SAMPLE ? a.sample_out + g : (is_res ? a.cand_res : a.cand_tgt) + g;
              *out = x0 + max(pick, 0);
            }
            }
          }
        }
        pending &= ~(is_res ? kDrawResidual : kDrawTarget);
        no_mass = false;
      } while (pending);
      if (!SAMPLE && tid == ((owner + 1) & (NW - 1)) * 32) {   // (the owner is the last one on its way already)
        a.flags[g] = accepted ? 0 : 1;
        if (a.p_tok || a.q_tok || a.accept_prob)
          row_write_probs(a.p_tok, a.q_tok, a.accept_prob, g, e_tok, mass, q_tok, Z, P.accept_mode == MULO_ACCEPT_THRESHOLD);
      }
    }

    // ---- on to the next row (its first pieces are in registers)
    if (!is_q) ++unit;
    if (!more) break;
    if (!is_q) {
      di = ndi;
      dj = ndj;
    }
    if (np_new) {
      next_parent();
      first = true;
    }
    is_q = nq;
    g = ng;
  }
}

}  // namespace mulo
