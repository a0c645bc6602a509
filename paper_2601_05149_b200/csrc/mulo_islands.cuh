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
// counts, and along a run of neighbours the recurrence s_k = max(s_{k-1} + 1, d_k) is a prefix maximum of d_k - k.
// One CTA per image.  All threads first find, for every position, what it depends on -- its run, the position of the
// row above, for a run the island's previous run in the row -- with bit operations on the rows' masks; nothing of that
// needs a step.  ONE warp then goes down the rows with shuffles instead of block barriers; the runs of a row share one
// scan (a term that grows from run to run keeps them apart).  In rows where an island has several runs, a run adds to
// the next one's steps: lane r takes run r and the chains are followed by doubling.  What bounds the kernel is this
// chain of H rows (three barriers and two searches per row made them 2.5 us each at 64 columns).
struct ScheduleArgs {
  int H, W, window;
  const int32_t* labels;   // [B, H, W]
  int32_t* step;           // [B, H, W]
  int32_t* n_steps;        // [B]
};

constexpr int kScheduleThreads = 1024;
constexpr int kRunTerm = 1 << 15;   // more than two steps, or columns, of one image can differ by

// Linked: the type of a row's number of runs -- int where it fits (16-bit loads in the chain of rows cost 5 %).
template <class Linked>
__host__ inline size_t schedule_smem(int H, int W) {
  const size_t N = (size_t)H * W, nw = (size_t)H * ((W + 31) / 32);
  return N * 12 + 2 * nw * 4 + (size_t)H * sizeof(Linked);   // (in 16 bits at most 232,000 bytes: 4000 x 4; an SM has 232,448)
}

template <class Linked>
__global__ void __launch_bounds__(kScheduleThreads) k_island_schedule(ScheduleArgs a) {
  extern __shared__ __align__(16) unsigned char sched_smem[];
  const int H = a.H, W = a.W, N = H * W, Ww = (W + 31) / 32, nw = H * Ww, b = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  int* const lab = reinterpret_cast<int*>(sched_smem);                      // labels, then steps
  uint32_t* const pos = reinterpret_cast<uint32_t*>(lab + N);               // bit: the position is in R_X
  uint32_t* const first = pos + nw;                                         // bit: ... and starts a run
  // by position: number of its run in the row (-1 outside R_X) << 16 | column of the row above (0xffff: none)
  int* const place = reinterpret_cast<int*>(first + nw);
  // by run of the row: the island's previous run in the row (-1: none) << 16 | last column
  int* const table = place + N;
  Linked* const linked = reinterpret_cast<Linked*>(table + N);              // runs of a row where one has a predecessor, else 0
  __shared__ int s_max, s_many;
  if (tid == 0) s_max = s_many = 0;
  const int32_t* const labels = a.labels + (size_t)b * N;
  for (int t = tid; t < N; t += kScheduleThreads) lab[t] = labels[t];
  for (int i = tid; i < H; i += kScheduleThreads) linked[i] = 0;
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
  // the last set bit of a row's mask at or before column x, -1: none
  auto last_at = [&](const uint32_t* row, int x) -> int {
    if (x < 0) return -1;
    int w = x >> 5;
    uint32_t v = row[w] & (0xffffffffu >> (31 - (x & 31)));
    while (v == 0u && w > 0) v = row[--w];
    return v ? (w << 5) + 31 - __clz(v) : -1;
  };
  // the last position of label m in row i at or before column x: run by run
  auto last_of = [&](int i, int x, int m) -> int {
    for (;;) {
      x = last_at(pos + i * Ww, x);
      if (x < 0 || lab[i * W + x] == m) return x;
      x = last_at(first + i * Ww, x) - 1;
    }
  };
  // the number, within the row, of the run that holds column x
  auto run_of = [&](int i, int x) -> int {
    int n = -1;
    for (int w = 0; w < x >> 5; ++w) n += __popc(first[i * Ww + w]);
    return n + __popc(first[i * Ww + (x >> 5)] & (0xffffffffu >> (31 - (x & 31))));
  };
  for (int w = warp; w < nw; w += kScheduleThreads / 32) {
    const int i = w / Ww, j = (w % Ww) * 32 + lane;
    if (j >= W) continue;
    const int t = i * W + j, m = lab[t];
    int r = -1, u = -1;
    if (m > 0) {
      r = run_of(i, j);
      if (i > 0) u = last_of(i - 1, min(W - 1, j + a.window - 1), m);
      if (j + 1 == W || lab[t + 1] != m) {   // the run's last position enters it in the row's table
        const int l = last_of(i, last_at(first + i * Ww, j) - 1, m);
        table[i * W + r] = (l >= 0 ? run_of(i, l) : -1) << 16 | j;
        const int nr = run_of(i, W - 1) + 1;
        if (l >= 0) linked[i] = (Linked)nr;
        if (nr > 32) s_many = 1;
      }
    }
    place[t] = r << 16 | (u & 0xffff);
  }
  __syncthreads();
  if (warp == 0) {
    // the key of a position: what the row above demands, less its column, plus its run's term
    auto key = [&](int pl, int j, const int* above) -> int {
      const int u = pl & 0xffff, r = pl >> 16;
      const int d = u != 0xffff ? above[u] + 1 : 1;
      return r >= 0 ? d - j + r * kRunTerm : INT_MIN;
    };
    // Chains of runs: run r hands on max(c + len, its last step); maps of this kind composed by doubling (lane r: run r).
    // Returns the step before the run's first one that its predecessor demands (0: none); beg: that first column.
    auto follow = [&](int i, int nr, const int* row, int& beg) -> int {
      int top = 0, len = 0, p = -1;
      beg = 0;
      if (lane < nr) {
        const int e = table[i * W + lane];
        p = e >> 16;
        top = row[e & 0xffff];
        beg = last_at(first + i * Ww, e & 0xffff);
        len = (e & 0xffff) - beg + 1;
      }
      const int p0 = p;
      while (__any_sync(0xffffffffu, p >= 0)) {
        const int q = max(p, 0);
        const int t2 = __shfl_sync(0xffffffffu, top, q), l2 = __shfl_sync(0xffffffffu, len, q), p2 = __shfl_sync(0xffffffffu, p, q);
        if (p >= 0) {
          top = max(top, t2 + len);
          len += l2;
          p = p2;
        }
      }
      const int c = __shfl_sync(0xffffffffu, top, max(p0, 0));
      return p0 >= 0 ? c : 0;
    };
    int* row = lab;
    if (Ww <= 2 && !s_many) {   // a row is two values per lane, which stay in registers
      const int j0 = lane, j1 = min(32 + lane, W - 1);
      const bool in0 = j0 < W, in1 = 32 + lane < W;
      for (int i = 0; i < H; ++i, row += W) {
        const int nr = linked[i], p0 = in0 ? place[i * W + j0] : -1, p1 = in1 ? place[i * W + j1] : -1;
        int v0 = key(p0, j0, row - W), v1 = key(p1, j1, row - W);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          v0 = max(v0, __shfl_up_sync(0xffffffffu, v0, o));   // (the first lanes get their own value)
          v1 = max(v1, __shfl_up_sync(0xffffffffu, v1, o));
        }
        v1 = max(v1, __shfl_sync(0xffffffffu, v0, 31));
        const int r0 = p0 >> 16, r1 = p1 >> 16;
        int s0 = r0 >= 0 ? v0 + j0 - r0 * kRunTerm : 0, s1 = r1 >= 0 ? v1 + j1 - r1 * kRunTerm : 0;
        if (in0) row[j0] = s0;
        if (in1) row[j1] = s1;
        __syncwarp();
        if (nr > 0) {
          int beg;
          const int c = follow(i, nr, row, beg);
          const int c0 = __shfl_sync(0xffffffffu, c, r0 & 31), c1 = __shfl_sync(0xffffffffu, c, r1 & 31);
          const int b0 = __shfl_sync(0xffffffffu, beg, r0 & 31), b1 = __shfl_sync(0xffffffffu, beg, r1 & 31);
          if (r0 >= 0 && c0 > 0) row[j0] = max(s0, c0 + 1 + j0 - b0);
          if (r1 >= 0 && c1 > 0) row[j1] = max(s1, c1 + 1 + j1 - b1);
          __syncwarp();
        }
      }
    } else {
      for (int i = 0; i < H; ++i, row += W) {
        int carry = INT_MIN;
        for (int w = 0; w < Ww; ++w) {
          const int j = (w << 5) + lane, pl = j < W ? place[i * W + j] : -1, r = pl >> 16;
          int v = key(pl, j, row - W);
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) v = max(v, __shfl_up_sync(0xffffffffu, v, o));
          v = max(v, carry);
          carry = __shfl_sync(0xffffffffu, v, 31);
          if (j < W) row[j] = r >= 0 ? v + j - r * kRunTerm : 0;
        }
        __syncwarp();
        const int nr = linked[i];
        if (nr == 0) continue;
        int c = 0, beg = 0;
        if (nr <= 32) {
          c = follow(i, nr, row, beg);
        } else {   // run by run
          if (lane == 0)
            for (int r = 0; r < nr; ++r) {
              const int e = table[i * W + r] & 0xffff, p = table[i * W + r] >> 16;
              if (p >= 0) row[e] = max(row[e], row[table[i * W + p] & 0xffff] + e - last_at(first + i * Ww, e) + 1);
            }
          __syncwarp();
        }
        for (int w = 0; w < Ww; ++w) {
          const int j = (w << 5) + lane, r = j < W ? place[i * W + j] >> 16 : -1;
          int cr = 0, br = 0;
          if (nr <= 32) {
            cr = __shfl_sync(0xffffffffu, c, r & 31);
            br = __shfl_sync(0xffffffffu, beg, r & 31);
          } else if (r >= 0 && (table[i * W + r] >> 16) >= 0) {
            cr = row[table[i * W + (table[i * W + r] >> 16)] & 0xffff];
            br = last_at(first + i * Ww, j);
          }
          if (r >= 0 && cr > 0) row[j] = max(row[j], cr + 1 + j - br);
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  int mine = 0;
  for (int t = tid; t < N; t += kScheduleThreads) {
    const int s = lab[t];
    a.step[(size_t)b * N + t] = s;
    mine = max(mine, s);
  }
  mine = __reduce_max_sync(0xffffffffu, mine);
  if (lane == 0) atomicMax(&s_max, mine);
  __syncthreads();
  if (tid == 0) a.n_steps[b] = s_max;
}

}  // namespace mulo
