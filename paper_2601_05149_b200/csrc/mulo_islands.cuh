// Rejection islands (Sec. 3.4, Eq. 8): {I_m} = CC_8(R_X), the 8-connected components of the
// set of positions to redraw, one CTA per image.
//
// The grid of one image (at most kIslandMaxCells positions) lives in shared memory as a
// forest: parent[t] is an earlier raster index of the same island, a root points at itself.
// Horizontal links cost nothing: every position starts out pointing at the first position of
// its run of consecutive R_X bits in the row, found with bit operations on the mask words.
// Only the first position of a run then works: it joins its run with every run of the row
// above that reaches into columns [first - 1, last + 1].  Joining hangs the later root under
// the earlier one with atomicMin, so the root of an island is its first raster position;
// numbering the roots in raster order (a block-wide count) numbers the islands by their
// first position.
#pragma once
#include <climits>
#include <cstdint>

#include "mulo_device.cuh"

namespace mulo {

constexpr int kIslandThreads = 1024;
constexpr int kIslandMaxCells = 16384;

struct IslandArgs {
  int H, W, max_islands;
  const uint32_t* bits;   // [B, H, ceil(W/32)]
  int32_t* labels;        // [B, H, W]
  int32_t* n_islands;     // [B]
  int32_t* rows;          // [B, max_islands, 2] or null
  int32_t* size;          // [B, max_islands] or null
};

// Root of x.  Parents only ever decrease and a root points at itself, so the walk ends.
__device__ __forceinline__ int island_root(const volatile int* parent, int x) {
  int p = parent[x];
  while (p != x) {
    x = p;
    p = parent[x];
  }
  return x;
}

// Joins the islands of a and b.  If another thread re-parents the later root between the
// look-up and the atomicMin, the link it made is kept by carrying on from that parent.
__device__ __forceinline__ void island_join(int* parent, int a, int b) {
  for (;;) {
    a = island_root(parent, a);
    b = island_root(parent, b);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    const int old = atomicMin(&parent[a], b);
    if (old == a) return;
    a = old;
  }
}

__global__ void __launch_bounds__(kIslandThreads) k_islands(IslandArgs a) {
  extern __shared__ int island_smem[];
  const int H = a.H, W = a.W, N = H * W, Ww = (W + 31) / 32, nw = H * Ww;
  int* const parent = island_smem;                                        // [N]
  int* const number = island_smem + N;                                    // [N], roots only
  uint32_t* const word = reinterpret_cast<uint32_t*>(island_smem + 2 * N);   // [nw]
  __shared__ int s_warp[kIslandThreads / 32];
  __shared__ int s_carry;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  let_next_begin();
  wait_for_previous();
  for (int w = tid; w < nw; w += kIslandThreads) {
    uint32_t v = a.bits[(size_t)b * nw + w];
    if (w % Ww == Ww - 1 && (W & 31)) v &= (1u << (W & 31)) - 1u;   // bits past the row's end do not count
    word[w] = v;
  }
  if (tid == 0) s_carry = 0;
  __syncthreads();
  // t = i * W + j without an integer division (t < 2^14: the float quotient is off by one at most)
  const float inv_w = 1.0f / (float)W;
  auto split = [&](int t, int& i, int& j) {
    i = (int)((float)t * inv_w);
    j = t - i * W;
    if (j < 0) {
      --i;
      j += W;
    } else if (j >= W) {
      ++i;
      j -= W;
    }
  };
  auto in_rx = [&](int i, int j) -> bool {
    return i >= 0 && j >= 0 && j < W && ((word[i * Ww + (j >> 5)] >> (j & 31)) & 1u);
  };
  // first column of the run of R_X bits that holds (i, j); (i, j) itself is in R_X
  auto run_first = [&](int i, int j) -> int {
    int w = j >> 5;
    uint32_t gaps = ~word[i * Ww + w] & ((1u << (j & 31)) - 1u);   // zeros below j in its word
    while (gaps == 0u && w > 0) {
      --w;
      gaps = ~word[i * Ww + w];
    }
    return gaps ? (w << 5) + 32 - __clz(gaps) : 0;
  };
  // last column of the run that starts at (i, j)
  auto run_last = [&](int i, int j) -> int {
    int w = j >> 5;
    uint32_t gaps = ~word[i * Ww + w] & ~((2u << (j & 31)) - 1u);   // zeros above j in its word
    while (gaps == 0u && w + 1 < Ww) {
      ++w;
      gaps = ~word[i * Ww + w];
    }
    return gaps ? (w << 5) + __ffs(gaps) - 2 : W - 1;
  };
  for (int t = tid; t < N; t += kIslandThreads) {
    int i, j;
    split(t, i, j);
    parent[t] = in_rx(i, j) ? i * W + run_first(i, j) : -1;
  }
  __syncthreads();

  for (int t = tid; t < N; t += kIslandThreads) {
    int i, j;
    split(t, i, j);
    if (i == 0 || !in_rx(i, j) || in_rx(i, j - 1)) continue;   // only the first position of a run works
    const int last = run_last(i, j);
    // runs of the row above inside columns [lo, hi]: one join per run, at its first bit there
    const int lo = j > 0 ? j - 1 : 0, hi = last + 1 < W ? last + 1 : W - 1;
    for (int w = lo >> 5; w <= hi >> 5; ++w) {
      uint32_t up = word[(i - 1) * Ww + w];
      uint32_t below = w > (lo >> 5) ? word[(i - 1) * Ww + w - 1] >> 31 : 0u;   // bit left of this word
      if (w == lo >> 5) up &= ~((1u << (lo & 31)) - 1u);
      if (w == hi >> 5 && (hi & 31) != 31) up &= (2u << (hi & 31)) - 1u;
      uint32_t firsts = up & ~((up << 1) | below);   // first bit, inside the window, of each run
      while (firsts) {
        const int x = (w << 5) + __ffs(firsts) - 1;
        firsts &= firsts - 1u;
        island_join(parent, t, (i - 1) * W + x);
      }
    }
  }
  __syncthreads();
  // first positions of runs point straight at their root (a reader that meets a half-updated
  // chain still walks to the same root); then everybody else, one hop behind
  for (int t = tid; t < N; t += kIslandThreads) {
    int i, j;
    split(t, i, j);
    if (parent[t] >= 0 && !in_rx(i, j - 1)) parent[t] = island_root(parent, t);
  }
  __syncthreads();
  for (int t = tid; t < N; t += kIslandThreads) {
    int i, j;
    split(t, i, j);
    const int q = parent[t];
    if (q >= 0 && in_rx(i, j - 1)) parent[t] = parent[q];
  }
  __syncthreads();

  // number the roots in raster order
  for (int base = 0; base < N; base += kIslandThreads) {
    const int t = base + tid;
    const bool is_root = t < N && parent[t] == t;
    const unsigned roots = __ballot_sync(0xffffffffu, is_root);
    if (lane == 0) s_warp[warp] = __popc(roots);
    __syncthreads();
    // every warp scans the 32 warp counts
    static_assert(kIslandThreads == 1024, "one count per lane");
    const int mine = s_warp[lane];
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const int before = s_carry + __shfl_sync(0xffffffffu, inc - mine, warp);
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    if (is_root) number[t] = before + __popc(roots & ((1u << lane) - 1u)) + 1;
    __syncthreads();
    if (tid == 0) s_carry += total;
  }
  __syncthreads();
  const int M = s_carry;
  if (tid == 0) a.n_islands[b] = M;

  const int cap = a.max_islands;
  int32_t* const rows = a.rows ? a.rows + (size_t)b * cap * 2 : nullptr;
  int32_t* const size = a.size ? a.size + (size_t)b * cap : nullptr;
  for (int m = tid; m < cap; m += kIslandThreads) {
    if (rows) {
      rows[2 * m] = m < M ? H : -1;
      rows[2 * m + 1] = -1;
    }
    if (size) size[m] = 0;
  }
  __syncthreads();
  for (int t = tid; t < N; t += kIslandThreads) {
    const int root = parent[t];
    const int m = root >= 0 ? number[root] : 0;
    a.labels[(size_t)b * N + t] = m;
    int i, j;
    split(t, i, j);
    if (m > 0 && m <= cap && !in_rx(i, j - 1)) {   // one contribution per run of the row
      if (rows) {
        atomicMin(&rows[2 * (m - 1)], i);
        atomicMax(&rows[2 * (m - 1) + 1], i);
      }
      if (size) atomicAdd(&size[m - 1], run_last(i, j) - j + 1);
    }
  }
}

// Island schedule (Sec. 3.4: islands redrawn concurrently, a ZipAR-style row window inside an island):
// the sequential step at which each position of R_X is decoded,
//   step(t) = 1 + max(step of the island's earlier positions in the row,
//                     step of the island's positions in the row above up to column col(t) + window - 1).
// Steps grow along an island's positions in a row, so of the row above only the last position inside the window
// counts, and along the island's positions of the row the recurrence s_k = max(s_{k-1} + 1, d_k) is a prefix maximum of
// d_k - k.  One CTA per image.  All threads first find where every position comes when its row is sorted by island, then by
// column (its slot), and the slot in the row above that it depends on -- with bit operations on the rows' masks; nothing of
// that needs a step.  ONE warp then goes down the rows: what the row above demands, one scan over the slots (a term that grows
// from island to island keeps them apart, however their runs interleave), and the steps are there; a row's slots are asked
// for one row ahead.  What bounds the kernel is this chain of H rows.
// (64 x 64, 32 images: 43.1 k of 61 k cycles with the slots' keys formed in the chain, 36 us in all, 44 with a second pass over an
// island's runs; 25 to 30 us with everything at hand that does not depend on a step.)
struct ScheduleArgs {
  int H, W, window;
  const int32_t* labels;   // [B, H, W]
  int32_t* step;           // [B, H, W]
  int32_t* n_steps;        // [B]
};

constexpr int kScheduleThreads = 1024;
constexpr int kScheduleSlack = 128;    // slots past the last row's, which the chain's lanes may touch
constexpr int kIslandTerm = 1 << 15;   // more than two steps, or columns, of one image can differ by

__host__ inline size_t schedule_smem(int H, int W) {
  const size_t N = (size_t)H * W, nw = (size_t)H * ((W + 31) / 32);
  return (N + kScheduleSlack) * 12 + 2 * nw * 4;   // (at most 225,536 bytes: 4000 x 4)
}

// M: slots per lane in the chain of rows; rows of more than 32 M columns take several turns.
template <int M>
__global__ void __launch_bounds__(kScheduleThreads) k_island_schedule(ScheduleArgs a) {
  extern __shared__ __align__(16) unsigned char sched_smem[];
  const int H = a.H, W = a.W, N = H * W, Ww = (W + 31) / 32, nw = H * Ww, b = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int S = N + kScheduleSlack;
  int* const lab = reinterpret_cast<int*>(sched_smem);
  uint16_t* const steps = reinterpret_cast<uint16_t*>(sched_smem) + 1;      // by slot, once the labels are not needed any more
  // by slot: what the step loses to become the key of the scan, its number among its island's in the row less a term that grows
  // with the island's first slot; 1 + the slot of the row above that it depends on, counted through the rows (0: none, steps[-1])
  int* const less = lab + S;
  uint32_t* const pos = reinterpret_cast<uint32_t*>(less + S);              // bit: the position is in R_X
  uint32_t* const first = pos + nw;                                         // bit: ... and starts a run
  uint16_t* const above = reinterpret_cast<uint16_t*>(first + nw);
  uint16_t* const slot = above + S;                                         // by column
  __shared__ int s_max;
  if (tid == 0) s_max = 0;
  let_next_begin();
  wait_for_previous();
  const int32_t* const labels = a.labels + (size_t)b * N;
  for (int t = tid; t < N; t += kScheduleThreads) {
    lab[t] = labels[t];
    above[t] = 0;
    less[t] = 0;
  }
  for (int t = N + tid; t < S; t += kScheduleThreads) {
    above[t] = 0;
    less[t] = 0;
  }
  __syncthreads();
  for (int w = warp; w < nw; w += kScheduleThreads / 32) {   // the rows' masks
    const int i = w / Ww, j = (w % Ww) * 32 + lane;
    const int m = j < W ? lab[i * W + j] : 0, left = j > 0 && j < W ? lab[i * W + j - 1] : 0;
    const unsigned in = __ballot_sync(0xffffffffu, m > 0), fs = __ballot_sync(0xffffffffu, m > 0 && m != left);
    if (lane == 0) {
      pos[w] = in;
      first[w] = fs;
    }
  }
  __syncthreads();
  // slots: the row's runs, cut at the masks' words, one after the other
  for (int w = warp; w < nw; w += kScheduleThreads / 32) {
    if (pos[w] == 0u) continue;
    const int i = w / Ww, j = (w % Ww) * 32 + lane;
    const int m = pos[w] >> lane & 1u ? lab[i * W + j] : 0;
    int below = 0, before = 0;   // positions of islands with a lower label; the island's own to the left
    for (int v = 0; v < Ww; ++v) {
      const uint32_t in = pos[i * Ww + v], stops = first[i * Ww + v] | ~in;
      for (uint32_t starts = (first[i * Ww + v] | 1u) & in; starts; starts &= starts - 1u) {
        const int at = __ffs(starts) - 1;
        const uint32_t stop = stops & ~((2u << at) - 1u);
        const int len = (stop ? __ffs(stop) - 1 : 32) - at, x = v * 32 + at, other = lab[i * W + x];
        if (other < m) below += len;
        if (other == m) before += min(max(j - x, 0), len);
      }
    }
    if (m > 0) {
      slot[i * W + j] = (uint16_t)(below + before);
      less[i * W + below + before] = before - below * kIslandTerm;
    }
  }
  __syncthreads();
  // the last set bit of a row's mask at or before column x, -1: none
  auto last_at = [&](const uint32_t* row, int x) -> int {
    if (x < 0) return -1;
    int w = x >> 5;
    uint32_t v = row[w] & (0xffffffffu >> (31 - (x & 31)));
    while (v == 0u && w > 0) v = row[--w];
    return v ? (w << 5) + 31 - __clz(v) : -1;
  };
  for (int w = warp; w < nw; w += kScheduleThreads / 32) {
    const int i = w / Ww, j = (w % Ww) * 32 + lane;
    if (!(pos[w] >> lane & 1u)) continue;
    const int m = lab[i * W + j], at = slot[i * W + j];
    int u = 0;
    if (i > 0) {   // the island's last position of the row above inside the window: run by run
      int x = last_at(pos + (i - 1) * Ww, min(W - 1, j + a.window - 1));
      while (x >= 0 && lab[(i - 1) * W + x] != m) x = last_at(pos + (i - 1) * Ww, last_at(first + (i - 1) * Ww, x) - 1);
      if (x >= 0) u = 1 + (i - 1) * W + slot[(i - 1) * W + x];
    }
    above[i * W + at] = (uint16_t)u;
  }
  __syncthreads();
  if (warp == 0) {
    if (lane == 0) steps[-1] = 0;
    __syncwarp();
    // A lane has M slots in a row.  Lanes past the row's end work on the next row's entries, or on slots that are not used: what they
    // find comes after everything of this row in the scan, and is overwritten when its row's turn comes.
    const int turns = (W + 32 * M - 1) / (32 * M);
    int u[M], l[M];
    auto ask = [&](int at) {
#pragma unroll
      for (int k = 0; k < M; ++k) {
        u[k] = above[at + k];
        l[k] = less[at + k];
      }
    };
    ask(lane * M);
    for (int i = 0, row = lane * M; i < H; ++i, row += W) {
      int carry = INT_MIN;
      for (int c = 0, at = row; c < turns; ++c, at += 32 * M) {
        int v[M], back[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
          back[k] = l[k];
          v[k] = (int)steps[u[k] - 1] + 1 - l[k];
        }
        const bool on = c + 1 < turns;
        if (on ? at + 32 * M < S - M : i + 1 < H) ask(on ? at + 32 * M : row + W);
#pragma unroll
        for (int k = 1; k < M; ++k) v[k] = max(v[k], v[k - 1]);
        int inc = v[M - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) inc = max(inc, __shfl_up_sync(0xffffffffu, inc, o));   // (the first lanes get their own)
        const int left = __shfl_up_sync(0xffffffffu, inc, 1);
        const int exc = max(lane == 0 ? INT_MIN : left, carry);
        if (turns > 1) carry = max(carry, __shfl_sync(0xffffffffu, inc, 31));
        if (turns == 1 || at < S - M) {
#pragma unroll
          for (int k = 0; k < M; ++k) steps[at + k] = (uint16_t)(max(v[k], exc) + back[k]);
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  int mine = 0;
  for (int w = warp; w < nw; w += kScheduleThreads / 32) {
    const int i = w / Ww, j = (w % Ww) * 32 + lane;
    if (j >= W) continue;
    const int s = pos[w] >> lane & 1u ? (int)steps[i * W + slot[i * W + j]] : 0;
    a.step[(size_t)b * N + i * W + j] = s;
    mine = max(mine, s);
  }
  mine = __reduce_max_sync(0xffffffffu, mine);
  if (lane == 0) atomicMax(&s_max, mine);
  __syncthreads();
  if (tid == 0) a.n_steps[b] = s_max;
}

}  // namespace mulo
