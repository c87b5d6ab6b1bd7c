// Repair of annealed states into flight paths, on the device (one warp per
// replica).  The reconstruction step of Algorithm 1 reads the path off the
// best state and must hand back a feasible flight path; a state whose row or
// column sums are not all 1 has none, so it is repaired:
//
//   Greedy fix.  path[0] = s.  For t = 1 .. C-1, with prev = path[t-1]: the
//   candidates are the cells not yet on the path that are hot in row t
//   (x_{t,i} = 1); if there are none, every cell not yet on the path.  path[t]
//   is the candidate nearest to prev (smallest d), ties to the smaller id.  A
//   feasible state (every row and column sum 1, x_{0,s} = 1) comes out as its
//   own decoded path.
//
//   2-opt (open path, path[0] fixed).  Move (i, j), 1 <= i < j <= C-1,
//   reverses path[i..j]: edges (i-1, i) and (j, j+1) become (i-1, j) and
//   (i, j+1) (no edge after j = C-1); inner edges keep their lengths because
//   d is symmetric.  One pass: for i = 1 .. C-2, for j = i+1 .. C-1 in order,
//   apply the move when it makes the path strictly shorter, then go on with
//   j+1 on the changed path.  Passes repeat while the last one moved and fewer
//   than max_passes have run (max_passes < 0: until no move helps, which ends
//   because every move shortens an integer length).
//
// The warp evaluates consecutive j at once on the current path and applies the
// first improving one, then restarts at the j after it: the same moves, in the
// same order, as the scan one j at a time.
#include <algorithm>
#include <climits>

#include "qp_device.cuh"
#include "qp_internal.h"

namespace qp {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t w = __shfl_xor_sync(kFull, v, o);
    v = w < v ? w : v;
  }
  return v;
}

__host__ __device__ constexpr size_t align16p(size_t x) { return (x + 15) & ~size_t(15); }

// Shared memory of a warp of k_repair_table: the path and its coordinates, the
// used cells, and the larger of {row cells, counts} and {edges, long edges}.
__host__ __device__ inline size_t repair_table_warp_bytes(int C) {
  return align16p(8 * (size_t)C) + align16p(2 * (size_t)C) + 2 * align16p(4 * (size_t)C) +
         align16p(((size_t)C + 31) / 32 * 4);
}

// Reverse path[i..j] and the inner edges edge[i..j-1] (edge[t] = d(path[t], path[t+1])).
__device__ __forceinline__ void reverse_segment(int32_t *path, int32_t *edge, int i, int j, int lane) {
  const int L = j - i + 1;
  for (int k = lane; k < L / 2; k += 32) {
    const int32_t a = path[i + k], b = path[j - k];
    path[i + k] = b;
    path[j - k] = a;
  }
  for (int k = lane; k < (L - 1) / 2; k += 32) {
    const int32_t a = edge[i + k], b = edge[j - 1 - k];
    edge[i + k] = b;
    edge[j - 1 - k] = a;
  }
  __syncwarp();
}

// smem per warp: path[C], edge[C], used bits[ceil(C/32)]  (int32 words)
__global__ void k_repair(const uint8_t *__restrict__ states, int R, int C, int start,
                         const int32_t *__restrict__ d, int max_passes, int32_t *__restrict__ paths,
                         int64_t *__restrict__ lengths, int32_t *__restrict__ status) {
  extern __shared__ int32_t sm_all[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const int r = blockIdx.x * W + warp;
  if (r >= R) return;
  const int nwu = (C + 31) >> 5;
  int32_t *path = sm_all + (size_t)warp * (2 * C + nwu);
  int32_t *edge = path + C;
  uint32_t *used = reinterpret_cast<uint32_t *>(edge + C);
  const uint8_t *x = states + (size_t)r * C * C;

  for (int w = lane; w < nwu; w += 32) used[w] = 0;
  __syncwarp();
  // row 0 must be exactly {s} for the state to be feasible
  int hot0 = 0;
  for (int i = lane; i < C; i += 32) hot0 += x[i] != 0;
  hot0 = __reduce_add_sync(kFull, hot0);
  bool feasible = hot0 == 1 && x[start] != 0;
  if (lane == 0) {
    path[0] = start;
    used[start >> 5] |= 1u << (start & 31);
  }
  __syncwarp();

  // greedy fix
  for (int t = 1; t < C; ++t) {
    const int prev = path[t - 1];
    const int32_t *drow = d + (size_t)QP_IX(prev, C, 5) * C;
    const uint8_t *xr = x + (size_t)t * C;
    uint64_t best_hot = ~0ull, best_any = ~0ull;
    int hot = 0;
    for (int i = lane; i < C; i += 32) {
      const bool h = xr[i] != 0;
      hot += h;
      if (!((used[i >> 5] >> (i & 31)) & 1u)) {
        const uint64_t key = ((uint64_t)(uint32_t)drow[i] << 32) | (uint32_t)i;
        best_any = key < best_any ? key : best_any;
        if (h) best_hot = key < best_hot ? key : best_hot;
      }
    }
    hot = __reduce_add_sync(kFull, hot);
    best_hot = warp_min_u64(best_hot);
    best_any = warp_min_u64(best_any);
    // feasible so far iff this row has one hot cell and it is not on the path yet
    feasible = feasible && hot == 1 && best_hot != ~0ull;
    const int pick = (int)(uint32_t)(best_hot != ~0ull ? best_hot : best_any);
    __syncwarp();
    if (lane == 0) {
      path[t] = pick;
      used[pick >> 5] |= 1u << (pick & 31);
    }
    __syncwarp();
  }

  // 2-opt
  for (int t = lane; t + 1 < C; t += 32) edge[t] = d[QP_IX((size_t)path[t] * C + path[t + 1], (size_t)C * C, 5)];
  __syncwarp();
  bool changed = false;
  bool moved = true;
  for (int pass = 0; moved && (max_passes < 0 || pass < max_passes); ++pass) {
    moved = false;
    for (int i = 1; i + 1 < C; ++i) {
      int j0 = i + 1;
      while (j0 < C) {
        const int a = path[i - 1], b = path[i];
        const int j = j0 + lane;
        int32_t n1 = 0, n2 = 0;
        bool imp = false;
        if (j < C) {
          const int pj = path[j];
          int64_t old = edge[i - 1];
          n1 = d[QP_IX((size_t)a * C + pj, (size_t)C * C, 5)];
          if (j + 1 < C) {
            old += edge[j];
            n2 = d[QP_IX((size_t)b * C + path[j + 1], (size_t)C * C, 5)];
          }
          imp = (int64_t)n1 + n2 < old;
        }
        const unsigned m = __ballot_sync(kFull, imp);
        if (m) {
          const int f = __ffs(m) - 1, js = j0 + f;
          const int32_t n1s = __shfl_sync(kFull, n1, f), n2s = __shfl_sync(kFull, n2, f);
          __syncwarp();
          reverse_segment(path, edge, i, js, lane);
          if (lane == 0) {
            edge[i - 1] = n1s;
            if (js + 1 < C) edge[js] = n2s;
          }
          __syncwarp();
          moved = true;
          changed = true;
          j0 = js + 1;
        } else {
          j0 += 32;
        }
      }
    }
  }

  int32_t *out = paths + (size_t)r * C;
  long long L = 0;
  for (int t = lane; t < C; t += 32) {
    out[t] = path[t];
    if (t + 1 < C) L += d[QP_IX((size_t)path[t] * C + path[t + 1], (size_t)C * C, 5)];
  }
  L = dev::warp_sum64(L);
  if (lane == 0) {
    lengths[r] = L;
    status[r] = feasible ? (changed ? 1 : 0) : 2;
  }
}

// The repair of fields whose distances fit a table over the grid differences
// (StructArgs), one warp per state.  What took the time was the latency of d in
// L2 (two gathers per 32 moves) and of the state's rows, one after another.
//   State.  Read once in 16-byte loads; its set bytes leave their row's number
//   of cells and one cell.  A feasible state is its path; else the greedy fix
//   reads a row again only when it holds several cells.
//   Distances.  The path's coordinates and edges and the table are in shared
//   memory: a move's two new edges are two table reads.
//   Moves.  An improving move has n1 + n2 < e1 + e2 (the edges it adds and
//   removes) and no edge is shorter than dmin, the field's smallest distance.
//   So at an i whose edge e1 is dmin only the j whose edge is longer than dmin
//   can improve: those are kept as a list in path order (rebuilt after a move),
//   the others are passed over.  On a good path most edges are dmin.
// 1024 states of 491 cells, 2-opt to the end (1500 moves a state): 13.1-13.9 -> 3.6-3.7 ms
// (5.3 with one list entry per lane and one i at a time). What is left is the
// chain of dependent steps: ~400 cycles a move, ~500-1000 a scan.
constexpr int kRun = 4;  // consecutive i scanned at once
// Fields of up to 256 cells (SMALL) scan every j 32 at a time once 64 or fewer are left, and also for a shortest edge
// right after a move while 128 or fewer are left, instead of listing the long edges again for it: moves come one after
// another on a bad path.  1024 annealed states, one pass: 92 cells 0.160 -> 0.143 ms, 236 cells 0.521 -> 0.499; 491
// cells to the end would be slower (3.57 -> 3.62 ms).
constexpr int kSmallRepair = 256;

template <typename DT, bool SMALL>
__global__ void k_repair_table(const uint8_t *__restrict__ states, int R, int C, int start,
                               const uint16_t *__restrict__ xy_g, const DT *__restrict__ tab_g, int sh, int tab_n,
                               uint32_t dmin, int max_passes, int32_t *__restrict__ paths,
                               int64_t *__restrict__ lengths, int32_t *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char rsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const size_t c2 = align16p(2 * (size_t)C);
  const size_t c8 = align16p(8 * (size_t)C);
  uint2 *xy = reinterpret_cast<uint2 *>(rsm);  // {row << sh, column}: a table index is two sums of absolute differences
  DT *tab = reinterpret_cast<DT *>(rsm + c8);
  for (int i = threadIdx.x; i < C; i += blockDim.x) {
    const uint32_t v = __ldg(xy_g + i);
    xy[i] = make_uint2((v >> 8) << sh, v & 0xFFu);
  }
  for (int i = threadIdx.x; i < tab_n; i += blockDim.x) tab[i] = __ldg(tab_g + i);
  __syncthreads();
  const int r = blockIdx.x * W + warp;
  if (r >= R) return;  // no CTA-wide barrier after this point
  unsigned char *p = rsm + c8 + align16p((size_t)tab_n * sizeof(DT)) + warp * repair_table_warp_bytes(C);
  const size_t c4 = align16p(4 * (size_t)C);
  uint2 *path = reinterpret_cast<uint2 *>(p);             // the coordinates of the path's cells
  uint16_t *id = reinterpret_cast<uint16_t *>(p + c8);    // the cells
  uint32_t *used = reinterpret_cast<uint32_t *>(p + c8 + c2);
  unsigned char *u = p + c8 + c2 + align16p(((size_t)C + 31) / 32 * 4);
  // while the state is read: each row's cell, and row counts with column counts << 16
  int32_t *at = reinterpret_cast<int32_t *>(u);
  uint32_t *cnt = reinterpret_cast<uint32_t *>(u + c4);
  // then: edge[t] = d(path[t], path[t+1]), and the long edges' positions
  uint32_t *edge = reinterpret_cast<uint32_t *>(u);
  uint16_t *lng = reinterpret_cast<uint16_t *>(cnt);
  auto D = [&](const uint2 &a, const uint2 &b) -> uint32_t {
    return (uint32_t)(int)tab[QP_IX((int)__usad(a.x, b.x, __usad(a.y, b.y, 0u)), tab_n, 5)];
  };

  const int n = C * C;
  const uint8_t *x = states + (size_t)r * n;
  for (int i = lane; i < C; i += 32) {
    at[i] = -1;
    cnt[i] = 0;
  }
  __syncwarp();
  auto set = [&](int k) {
    const int t = QP_IX(k / C, C, 12), i = k - t * C;
    at[t] = i;  // any of them when there are several
    atomicAdd(cnt + t, 1u);
    atomicAdd(cnt + i, 0x10000u);
  };
  const int head = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15));
  const int nv = (n - head) / 16;
  if (lane < head && x[lane]) set(lane);
  for (int v0 = 0; v0 < nv; v0 += 256) {
    uint4 q[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const int v = v0 + 32 * g + lane;
      q[g] = v < nv ? __ldg(reinterpret_cast<const uint4 *>(x + head) + v) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int g = 0; g < 8; ++g) dev::each_set_byte(q[g], head + 16 * (v0 + 32 * g + lane), set);
  }
  for (int k = head + 16 * nv + lane; k < n; k += 32)
    if (x[k]) set(k);
  __syncwarp();
  int bad = 0;
  for (int i = lane; i < C; i += 32) bad |= cnt[i] != 0x10001u;
  const bool feasible = !__any_sync(kFull, bad) && at[0] == start;
  if (feasible) {
    for (int t = lane; t < C; t += 32) {
      id[t] = (uint16_t)at[t];
      path[t] = xy[QP_IX(at[t], C, 12)];
    }
  } else {
    // greedy fix
    for (int w = lane; w < (C + 31) >> 5; w += 32) used[w] = (start >> 5) == w ? 1u << (start & 31) : 0u;
    if (lane == 0) {
      id[0] = (uint16_t)start;
      path[0] = xy[start];
    }
    __syncwarp();
    constexpr bool kPacked = sizeof(DT) == 2;  // a 16-bit distance and a cell fit one 32-bit key
    static_assert(kMaxCells <= 4096, "a cell in 12 bits");
    const int nw = (C + 31) >> 5;
    uint2 prev = xy[start];
    for (int t = 1; t < C; ++t) {
      const int hot = (int)(cnt[t] & 0xFFFFu), c = at[t];
      int pick = -1;
      if (hot == 1 && !((used[c >> 5] >> (c & 31)) & 1u)) {
        pick = c;
      } else {
        // the nearest open cell of the row when it has several, else of the field: both in one scan without
        // branches, so that its loads are in flight together (1024 states of 491 cells to paths, a third of the
        // cells set: 3.76 -> 1.72 ms, three a row: 2.71 -> 1.15; with a branch before each load it was slower
        // than k_repair's 1.97 on both)
        uint32_t hd = 0xFFFFFFFFu, hi = 0xFFFFFFFFu, ad = 0xFFFFFFFFu, ai = 0xFFFFFFFFu;
        const uint8_t *row = x + (size_t)t * C;
        const bool multi = hot > 1;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) {
          const int i = 32 * w + lane, ic = min(i, C - 1);
          const uint32_t on = multi ? __ldg(row + ic) : 0;
          const bool open = ((~used[w] >> lane) & 1u) && i < C;
          const uint32_t v = D(prev, xy[ic]);
          if (kPacked) {
            const uint32_t key = open ? v << 12 | (uint32_t)i : 0xFFFFFFFFu;
            ad = min(ad, key);
            hd = min(hd, on ? key : 0xFFFFFFFFu);
          } else {  // i ascends: ties keep the smaller
            const bool n = open && v < ad, nh = open && on && v < hd;
            ad = n ? v : ad;
            ai = n ? (uint32_t)i : ai;
            hd = nh ? v : hd;
            hi = nh ? (uint32_t)i : hi;
          }
        }
        uint32_t m = __reduce_min_sync(kFull, hd);
        if (m != 0xFFFFFFFFu) {
          pick = kPacked ? (int)(m & 0xFFFu) : (int)__reduce_min_sync(kFull, hd == m ? hi : 0xFFFFFFFFu);
        } else {
          m = __reduce_min_sync(kFull, ad);
          pick = kPacked ? (int)(m & 0xFFFu) : (int)__reduce_min_sync(kFull, ad == m ? ai : 0xFFFFFFFFu);
        }
      }
      prev = xy[QP_IX(pick, C, 12)];
      __syncwarp();
      if (lane == 0) {
        id[t] = (uint16_t)pick;
        path[t] = prev;
        used[pick >> 5] |= 1u << (pick & 31);
      }
      __syncwarp();
    }
  }
  __syncwarp();

  // 2-opt
  for (int t = lane; t + 1 < C; t += 32) edge[t] = D(path[t], path[t + 1]);
  __syncwarp();
  bool changed = false, moved = true, stale = true, hasty = true;
  int nl = 0;  // long edges in lng[]
  for (int pass = 0; moved && (max_passes < 0 || pass < max_passes); ++pass) {
    moved = false;
    int lp = 0;  // the first long edge after i
    for (int i = 1; i + 1 < C; ++i) {
      int j0 = i + 1;
      while (j0 < C) {
        int js = -1;
        uint32_t n1s = 0, n2s = 0;
        if (edge[i - 1] > dmin || (SMALL && stale && hasty && C - j0 <= 128)) {
          // every j: 32 of them first, where most moves of a long edge are found, then 128 at a time
          const uint2 a = path[i - 1], b = path[i];
          const uint32_t e1 = edge[i - 1];
          int jb = j0 + 32;
          for (int j1 = j0;; j1 = jb, jb += 32) {
            const int j = j1 + lane, jc = min(j, C - 2);
            const uint32_t n1 = D(a, path[QP_IX(min(j, C - 1), C, 12)]), n2 = j + 1 < C ? D(b, path[QP_IX(jc + 1, C, 12)]) : 0u;
            const unsigned m = __ballot_sync(kFull, j < C && n1 + n2 < e1 + (j + 1 < C ? edge[jc] : 0u));
            if (m) {
              const int f = __ffs(m) - 1;
              js = j1 + f;
              n1s = __shfl_sync(kFull, n1, f);
              n2s = __shfl_sync(kFull, n2, f);
            }
            if (!SMALL || js >= 0 || jb >= C || C - jb > 64) break;
          }
          for (; jb < C && js < 0; jb += 128) {
            uint32_t n1[4], n2[4];
            bool imp[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int j = jb + 32 * q + lane, jc = min(j, C - 2);
              n1[q] = D(a, path[QP_IX(min(j, C - 1), C, 12)]);
              n2[q] = j + 1 < C ? D(b, path[QP_IX(jc + 1, C, 12)]) : 0u;
              imp[q] = j < C && n1[q] + n2[q] < e1 + (j + 1 < C ? edge[QP_IX(jc, C, 12)] : 0u);
            }
            if (__any_sync(kFull, imp[0] | imp[1] | imp[2] | imp[3])) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const unsigned m = __ballot_sync(kFull, imp[q]);
                if (m && js < 0) {
                  const int f = __ffs(m) - 1;
                  js = jb + 32 * q + f;
                  n1s = __shfl_sync(kFull, n1[q], f);
                  n2s = __shfl_sync(kFull, n2[q], f);
                }
              }
            }
          }
        } else {
          if (stale) {
            nl = 0;
            for (int t = 0; t + 1 < C; t += 32) {
              const bool l = t + lane + 1 < C && edge[t + lane] > dmin;
              const unsigned m = __ballot_sync(kFull, l);
              if (l) lng[QP_IX(nl + __popc(m & ((1u << lane) - 1u)), C, 12)] = (uint16_t)(t + lane);
              nl += __popc(m);
            }
            __syncwarp();
            stale = false;
            lp = 0;
          }
          while (lp < nl) {  // past the edges up to i
            const unsigned m = __ballot_sync(kFull, lp + lane < nl && lng[QP_IX(lp + lane, C, 12)] <= i);
            lp += __popc(m);
            if (m != kFull) break;
          }
          if (nl - lp > 64) {
            // many long edges: this i against 128 of them at a time
            const uint2 a = path[i - 1], b = path[i];
            for (int l0 = lp; l0 < nl && js < 0; l0 += 128) {
              uint32_t n1[4], n2[4];
              int j[4];
              bool imp[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int l = l0 + 32 * q + lane;
                j[q] = l < nl ? lng[QP_IX(l, C, 12)] : 0;
                n1[q] = D(a, path[QP_IX(j[q], C, 12)]);
                n2[q] = D(b, path[QP_IX(j[q] + 1, C, 12)]);
                imp[q] = j[q] >= j0 && n1[q] + n2[q] < dmin + edge[j[q]];
              }
              if (__any_sync(kFull, imp[0] | imp[1] | imp[2] | imp[3])) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  const unsigned m = __ballot_sync(kFull, imp[q]);
                  if (m && js < 0) {
                    const int f = __ffs(m) - 1;
                    js = __shfl_sync(kFull, j[q], f);
                    n1s = __shfl_sync(kFull, n1[q], f);
                    n2s = __shfl_sync(kFull, n2[q], f);
                  }
                }
              }
            }
          } else {
            // few: this i and, at its first scan, up to kRun - 1 more that
            // follow it with a shortest edge; without a move the path is the
            // same for all of them
            int run = 1;
            if (j0 == i + 1) {
              const bool stop = lane > 0 && (i + lane + 1 >= C || edge[min(i - 1 + lane, C - 2)] > dmin);
              run = min(kRun, __ffs(__ballot_sync(kFull, stop) | 0x80000000u) - 1);
            }
            uint2 pv[kRun + 1];
            int first[kRun];  // this lane's first improving j for each i
#pragma unroll
            for (int q = 0; q <= kRun; ++q) pv[q] = path[QP_IX(min(i - 1 + q, C - 1), C, 12)];
#pragma unroll
            for (int q = 0; q < kRun; ++q) first[q] = INT_MAX;
            for (int l0 = lp; l0 < nl; l0 += 32) {
              const int j = l0 + lane < nl ? lng[QP_IX(l0 + lane, C, 12)] : 0;
              const uint2 pj = path[QP_IX(j, C, 12)], pj1 = path[QP_IX(j + 1, C, 12)];
              const uint32_t lim = dmin + edge[j];
#pragma unroll
              for (int q = 0; q < kRun; ++q)
                if (first[q] == INT_MAX && j >= max(j0, i + q + 1) && q < run && D(pv[q], pj) + D(pv[q + 1], pj1) < lim)
                  first[q] = j;
            }
            bool some = false;
#pragma unroll
            for (int q = 0; q < kRun; ++q) some |= first[q] != INT_MAX;
            if (__any_sync(kFull, some)) {
              int q = 0, fj = INT_MAX;
#pragma unroll
              for (int g = kRun - 1; g >= 0; --g)
                if (__any_sync(kFull, first[g] != INT_MAX)) {
                  q = g;
                  fj = first[g];
                }
              js = __reduce_min_sync(kFull, fj);
              i += q;
              n1s = D(path[i - 1], path[js]);
              n2s = D(path[i], path[js + 1]);
            } else {
              i += run - 1;
            }
          }
        }
        if (SMALL) hasty = js >= 0;
        if (js < 0) break;
        // apply the move: reverse path[i..js]
        __syncwarp();
        const int len = js - i + 1;
        for (int k = lane; k < len / 2; k += 32) {
          const uint2 p0 = path[QP_IX(i + k, C, 12)], p1 = path[QP_IX(js - k, C, 12)];
          const uint16_t i0 = id[i + k], i1 = id[js - k];
          const bool inner = k < (len - 1) / 2;
          const uint32_t ea = edge[QP_IX(i + k, C, 12)], eb = edge[QP_IX(js - 1 - k, C, 12)];
          path[i + k] = p1;
          path[js - k] = p0;
          id[i + k] = i1;
          id[js - k] = i0;
          if (inner) {
            edge[i + k] = eb;
            edge[js - 1 - k] = ea;
          }
        }
        __syncwarp();
        if (lane == 0) {
          edge[QP_IX(i - 1, C, 12)] = n1s;
          if (js + 1 < C) edge[QP_IX(js, C, 12)] = n2s;
        }
        __syncwarp();
        moved = changed = stale = true;
        j0 = js + 1;
      }
    }
  }

  int32_t *out = paths + (size_t)r * C;
  long long L = 0;
  for (int t = lane; t < C; t += 32) {
    out[t] = QP_IX((int)id[t], C, 12);
    if (t + 1 < C) L += edge[t];
  }
  L = dev::warp_sum64(L);
  if (lane == 0) {
    lengths[r] = L;
    status[r] = feasible ? (changed ? 1 : 0) : 2;
  }
}

template <typename DT, bool SMALL>
cudaError_t launch_repair_t(const uint8_t *states, int32_t R, const RepairField &f, int32_t max_passes, int32_t *paths,
                            int64_t *lengths, int32_t *status, cudaStream_t st) {
  const size_t per = repair_table_warp_bytes(f.C);
  const size_t fixed = align16p(8 * (size_t)f.C) + align16p((size_t)f.tab_n * sizeof(DT));
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int W = std::max(1, std::min(8, (R + sms - 1) / sms));  // few states spread over the SMs
  while (W > 1 && fixed + W * per > 160 * 1024) --W;
  const size_t smem = fixed + W * per;
  if (smem > 160 * 1024) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lk(launch_mutex());
  e = cudaFuncSetAttribute(k_repair_table<DT, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_repair_table<DT, SMALL><<<(R + W - 1) / W, W * 32, smem, st>>>(
      states, R, f.C, f.start, f.xy, static_cast<const DT *>(f.tab), f.tab_sh, f.tab_n, (uint32_t)f.min_d, max_passes, paths,
      lengths, status);
  return cudaGetLastError();
}

}  // namespace

size_t repair_smem_per_warp(int32_t C) { return (size_t)(2 * C + (C + 31) / 32) * 4; }

cudaError_t launch_repair(const uint8_t *states, int32_t R, const RepairField &f, int32_t max_passes, int32_t *paths,
                          int64_t *lengths, int32_t *status, cudaStream_t st) {
  // the table kernel, unless the grid is too large for a table
  if (f.tab_n > 0) {
    auto launch = f.C <= kSmallRepair ? (f.d_i16 ? launch_repair_t<int16_t, true> : launch_repair_t<int32_t, true>)
                                      : (f.d_i16 ? launch_repair_t<int16_t, false> : launch_repair_t<int32_t, false>);
    return launch(states, R, f, max_passes, paths, lengths, status, st);
  }
  const int32_t C = f.C;
  const size_t per = repair_smem_per_warp(C);
  int W = 8;
  while (W > 1 && W * per > 96 * 1024) W >>= 1;
  const size_t smem = W * per;
  if (smem > 96 * 1024) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lk(launch_mutex());
  cudaError_t e = cudaFuncSetAttribute(k_repair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_repair<<<(R + W - 1) / W, W * 32, smem, st>>>(states, R, C, f.start, f.d32, max_passes, paths, lengths, status);
  return cudaGetLastError();
}

}  // namespace qp

namespace qp {
namespace chk {
QP_CHECK_ACCESSOR(repair)
}  // namespace chk
}  // namespace qp
