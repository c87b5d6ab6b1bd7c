// Event-driven structured sweep (sm_103a): the same sequential chain as the
// row kernels, with the proposals that cannot be accepted passed over in
// groups by bounds that hold for the current state.
//
// With r the sum of row t and c the sum of column i (both including x_{t,i})
// and f = sum of d over the cells of rows t-1 and t+1, Eq. 6 gives
//   x = 0:  dE = B f + 2A (r + c - 1),      x = 1:  dE = 2A (3 - r - c) - B f.
// So a cell proposed into a row and a column that hold one between them at
// least twice (r + c >= 2) costs dE >= 2A.  Such a proposal is accepted only
// if its draw u is below thr[2A], and never when the table ends at or before
// 2A: a test that does not look at the state.  What is left in a row with
// r >= 1 are few columns: the row's own cells (x = 1), the empty columns
// (c = 0) and the columns whose draw passed the test ("survivors").  At
// T = 1000 that is 1 in 170 draws on a 10x10 field and 1 in 400,000 on a
// 24x24 one; sweeps whose table ends at 2A have none and draw nothing.
// A row without cells (r = 0) has no such bound: all its columns are evaluated.
//
// One warp anneals one replica.  A sweep goes through windows of 32 rows:
//   draws   (only when len > 2A) every Philox block of the window, one per
//           lane and step, each word compared with thr[2A]; the rows that have
//           a survivor are kept as a mask.
//   check   lane j looks at row t0 + j as the state stands: rows that do not
//           hold exactly one cell, that have a survivor, or whose cell or an
//           empty column would be accepted are events.  The first event row
//           is found by one ballot; every row before it is final.
//   event   the row evaluated exactly, 128 columns at a time (a lane takes the
//           four columns of one Philox block), the first accepted proposal
//           applied and the rest re-evaluated, in proposal order.  Of a row of
//           several blocks those that hold none of its cells, no empty column
//           and no survivor are passed over (491 cells: 100.9 -> 91.4 ms).
// After an event the check resumes at the next row.  A sweep most of whose
// rows are events goes from row to row without draws and checks of its own.
// Every decision is the sequential chain's: the same words of the generator
// against the same tables.
//
// What bounds it: the latency of one chain, that is its count of dependent
// instructions (92 cells, T = 1000: 369 warp instructions a row at 3.2 cycles
// each with one warp on the SM, memory idle), and in hot sweeps of large fields
// the Philox multiplies (88 cycles of a scheduler per warp-wide block, whatever
// the occupancy; 43 of the 83.2 ms below).  Against the row kernels, which
// evaluate every column of every row (one GB300): 92 cells, 1024 chains x 5000
// sweeps: 166 -> 32.8 ms (161 -> 63 us a sweep at T = 1000, 1.2 flips a row);
// 491 cells, 4096 chains x 1000 sweeps: 899 -> 83.2 ms; 893 cells, 512 chains x
// 40 sweeps (the general kernel): 272 -> 22.0 ms.  It is also the faster one far
// above the temperatures of a useful schedule (T = 1e6, a third of the cells
// set: 1.5 to 2.2 times), so every structured launch uses it.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "qp_device.cuh"
#include "qp_internal.h"

namespace qp {
namespace {

using namespace dev;

constexpr int kZCheck = 4;    // most empty columns the check looks at; above, rows are processed one by one
constexpr int kRowCells = 3;  // cells of a row kept in its record
// What rows a kernel is compiled for: of one block of columns (C <= kNarrow), of
// several, or both.  A single field's launch knows, and each kernel holds only its
// own row loops (92 cells, 5000 sweeps: 33.3 -> 32.8 ms; instruction fetch is a
// fifteenth of a chain's time).  The batch, whose SMs run fields of both kinds at
// once, takes one body for both: with two bodies 13.5 -> 21.8 ms (256 fields).
enum { kOneBlock, kWide, kAny };
constexpr int kNarrow = 125;  // most cells of a row that is one block of 128 columns, whatever t C mod 4
constexpr int kPad = 8;       // entries before and after the arrays read by four columns at a time

__host__ __device__ constexpr size_t align16e(size_t x) { return (x + 15) & ~size_t(15); }

// A row's record: its number of cells and, when there are at most three, the
// cells themselves (c0 = C in an empty row); of a row with more, one of its
// cells (c0), and the row's bits hold them all.  The bits of other rows are
// not kept.
struct Row {
  int n, c0, c1, c2;
};
__device__ __forceinline__ Row unpack_row(uint2 q) {
  return Row{(int)(q.x & 0xFFFFu), (int)(q.x >> 16), (int)(q.y & 0xFFFFu), (int)(q.y >> 16)};
}
__device__ __forceinline__ uint2 pack_row(int n, int c0, int c1, int c2) {
  return make_uint2((uint32_t)n | ((uint32_t)c0 << 16), (uint32_t)c1 | ((uint32_t)c2 << 16));
}

// d_{h,i}: from the matrix in global memory (DM = 0) or in shared memory
// (DM = 1), with a row of zeros after it and readable entries around it, or from the field's table over (|row difference|, |column
// difference|) in shared memory (DM = 2: 24x24 cells take 1.5 KB instead of
// the matrix's 482 KB).
template <typename DT, int DM>
struct Dist {
  const DT *m;
  int Cp, C;
  const uint16_t *xy;  // row << 8 | column of every cell
  int sh, tab_n;
  __device__ __forceinline__ int lookup(uint32_t a, uint32_t b) const {
    const uint32_t ad = __vabsdiffu4(a, b);
    return QP_VALUE((int)m[QP_IX((int)(((ad >> 8) << sh) + (ad & 0xFFu)), tab_n, 2)], 7);
  }
  // A cell as hx keeps it (its coordinates when they are all a distance needs,
  // which spares the gather of them), and the distance of two of those.
  __device__ __forceinline__ uint32_t code(int h) const { return DM == 2 ? (uint32_t)xy[QP_IX(h, C, 2)] : (uint32_t)h; }
  __device__ __forceinline__ int near(uint32_t a, uint32_t b) const {
    if (DM == 2) return lookup(a, b);
    const int k = QP_IX((int)a * Cp + (int)b, (C + 1) * Cp, 2);
    return DM == 1 ? (int)m[k] : (int)__ldg(m + k);
  }
  // h = C (an empty row's record): 0
  __device__ __forceinline__ int operator()(int h, int i) const {
    if (DM == 2) return h < C ? lookup(xy[QP_IX(h, C, 2)], xy[QP_IX(i, C, 2)]) : 0;
    const int k = QP_IX(h * Cp + i, (C + 1) * Cp, 2);
    return DM == 1 ? (int)m[k] : (int)__ldg(m + k);
  }
  // f[j] += d_{h,i+j}, -4 < i <= C; columns outside the field give anything.
  // xi: the columns' coordinates (DM = 2).
  __device__ __forceinline__ void add4(int h, int i, const uint32_t (&xi)[4], int (&f)[4]) const {
    if (DM == 2) {
      if (h >= C) return;
      const uint32_t a = xy[QP_IX(h, C, 2)];
#pragma unroll
      for (int j = 0; j < 4; ++j) f[j] += lookup(a, xi[j]);
    } else {
      const DT *p = m + QP_IX(h, C + 1, 2) * Cp + QP_RANGE(i, -3, C + 1, 2);
#pragma unroll
      for (int j = 0; j < 4; ++j) f[j] += QP_VALUE(DM == 1 ? (int)p[j] : (int)__ldg(p + j), 7);
    }
  }
};

// SB: the spins' bitsets are in shared memory (up to 256 cells, 8 KB a
// replica); else in global memory (L2, flipped by atomics, read past L1).
template <bool SB>
__device__ __forceinline__ uint32_t bits_word(const uint32_t *p) {
  if (SB) return *p;
  return __ldcg(p);
}

// Sum of d over the cells of row u (whose record is q), for this lane's column i.
template <typename DT, int DM, bool SB>
__device__ __forceinline__ int row_sum_d(const Row &q, int u, const uint32_t *bits, int Cw, int C,
                                         const Dist<DT, DM> &D, int i) {
  int f = 0;
  if (q.n <= kRowCells) {
    if (q.n > 0) f = D(q.c0, i);
    if (q.n > 1) f += D(q.c1, i);
    if (q.n > 2) f += D(q.c2, i);
  } else {
    for (int w = 0; w < Cw; ++w) {
      uint32_t wd = bits_word<SB>(bits + QP_IX(u * Cw + w, C * Cw, 3));
      while (wd) {
        f += D((w << 5) + __ffs(wd) - 1, i);
        wd &= wd - 1;
      }
    }
  }
  return f;
}

// Sums of d over the cells of row t (their number n; more than three, so the
// bits hold them), of the cells but `skip`, for this lane's columns i .. i + 3
// (-4 < i; a multiple of 4 below Cp when ALIGNED): by the whole warp, from the
// matrix in global memory, eight cells' rows in flight at a time.
template <typename DT, bool SB, bool ALIGNED>
__device__ __forceinline__ void add_cells(const DT *d, int Cp, int C, const uint32_t *bits, int Cw, int t, int n, int skip,
                                          int i, int lane, int (&f)[4]) {
  uint32_t word = 0, left = 0, wd = 0;
  int w0 = -32, w = 0;
  auto next = [&]() {  // the next cell, C (the row of zeros) after the last
    while (wd == 0) {
      if (left == 0) {
        w0 += 32;
        if (w0 >= Cw) return C;
        word = w0 + lane < Cw ? bits_word<SB>(bits + QP_IX(t * Cw + w0 + lane, C * Cw, 3)) : 0u;
        if ((skip >> 5) == w0 + lane) word &= ~(1u << (skip & 31));
        left = __ballot_sync(kFull, word != 0);
        continue;
      }
      w = w0 + __ffs(left) - 1;
      left &= left - 1;
      wd = __shfl_sync(kFull, word, w - w0);
    }
    const int h = (w << 5) + __ffs(wd) - 1;
    wd &= wd - 1;
    return h;
  };
  for (int k = 0; k < n; k += 8) {
    const DT *p[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) p[g] = d + (size_t)QP_IX(next(), C + 1, 2) * Cp + i;
    DT v[8][4];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      if (!ALIGNED) {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[g][j] = __ldg(p[g] + j);
      } else if (sizeof(DT) == 2) {
        *reinterpret_cast<int2 *>(v[g]) = __ldg(reinterpret_cast<const int2 *>(p[g]));
      } else {
        *reinterpret_cast<int4 *>(v[g]) = __ldg(reinterpret_cast<const int4 *>(p[g]));
      }
    }
#pragma unroll
    for (int g = 0; g < 8; ++g)
#pragma unroll
      for (int j = 0; j < 4; ++j) f[j] += (int)v[g][j];
  }
}

// This lane's part of the sum of d over the pairs of a cell of row t and one of
// row t + 1, by the whole warp.  (A lane per row, cell by cell, the energy of a state
// with half its cells set was the larger part of a short anneal from it: 230 cells,
// 256 chains, one sweep 31.0 -> 20.7 ms.)
template <typename DT, bool SB>
__device__ __forceinline__ long long pair_distance(const DT *d, int Cp, int C, const uint32_t *bits, int Cw, const uint2 *rec,
                                                int t, int lane) {
  const Row q = unpack_row(rec[t]), p = unpack_row(rec[t + 1]);
  long long sum = 0;
  for (int b = 0; b < Cp; b += 128) {
    const int i = b + 4 * lane, i0 = min(i, Cp - 4);
    int f[4] = {0, 0, 0, 0};
    if (p.n <= kRowCells) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f[j] = (int)__ldg(d + (size_t)p.c0 * Cp + i0 + j);
        if (p.n > 1) f[j] += (int)__ldg(d + (size_t)p.c1 * Cp + i0 + j);
        if (p.n > 2) f[j] += (int)__ldg(d + (size_t)p.c2 * Cp + i0 + j);
      }
    } else {
      add_cells<DT, SB, true>(d, Cp, C, bits, Cw, t + 1, p.n, -1, i0, lane, f);
    }
    uint32_t x = 0;  // row t's cells among the four
    if (q.n > kRowCells) {
      x = bits_word<SB>(bits + QP_IX(t * Cw + (min(i0, C - 1) >> 5), C * Cw, 3)) >> (i0 & 31);
    } else {
      if ((unsigned)(q.c0 - i0) < 4u) x |= 1u << (q.c0 - i0);
      if (q.n > 1 && (unsigned)(q.c1 - i0) < 4u) x |= 1u << (q.c1 - i0);
      if (q.n > 2 && (unsigned)(q.c2 - i0) < 4u) x |= 1u << (q.c2 - i0);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i < Cp && i0 + j < C && ((x >> j) & 1u)) sum += f[j];
  }
  return sum;
}

// The same for every two rows whose numbers of cells multiply to more than `most`.
template <typename DT, bool SB>
__device__ __noinline__ long long pairs_distance(const DT *d, int Cp, int C, const uint32_t *bits, int Cw, const uint2 *rec,
                                                 int most, int lane) {
  long long sum = 0;
  for (int t = 0; t + 1 < C; ++t)
    if ((int)(rec[t].x & 0xFFFFu) * (int)(rec[t + 1].x & 0xFFFFu) > most)
      sum += pair_distance<DT, SB>(d, Cp, C, bits, Cw, rec, t, lane);
  return sum;
}

// Row t's record from its bits (r cells); of a row with more than three, one
// of its cells.
template <bool SB>
__device__ __forceinline__ uint2 record_from_bits(const uint32_t *bits, int Cw, int C, int t, int r, int lane) {
  int c[3] = {C, 0, 0}, k = 0;
  const int want = r <= kRowCells ? r : 1;
  for (int w0 = 0; w0 < Cw && k < want; w0 += 32) {
    const uint32_t word = w0 + lane < Cw ? bits_word<SB>(bits + QP_IX(t * Cw + w0 + lane, C * Cw, 3)) : 0u;
    for (uint32_t b = __ballot_sync(kFull, word != 0); b && k < want; b &= b - 1) {
      const int w = __ffs(b) - 1;
      for (uint32_t wd = __shfl_sync(kFull, word, w); wd && k < want; wd &= wd - 1) {
        const int i = ((w0 + w) << 5) + __ffs(wd) - 1;
        if (k == 0) c[0] = i;
        else if (k == 1) c[1] = i;
        else c[2] = i;
        ++k;
      }
    }
  }
  return pack_row(r, c[0], c[1], c[2]);
}

// The sweeps of one replica.  rec: C + 1 row records (the last stays empty),
// hx: what D.near needs of the cell of a row that holds one, cc:
// column sums with kPad entries on both sides, bits: C x Cw words.
template <typename DT, int DM, bool SB, int ROWS, typename KEY>
__device__ __forceinline__ void events_replica(const StructArgs &a, int rep, uint2 *rec, uint16_t *hx, uint16_t *cc,
                                               uint32_t *bits, const Dist<DT, DM> &D, int lane, const KEY &key) {
  const int C = a.C, s0 = a.start, B = a.B, twoA = 2 * a.A;
  const int Cw = (C + 31) >> 5;
  const int n = C * C;
  const uint32_t rg = (uint32_t)(a.rep_offset + rep);
  const uint32_t magic = (uint32_t)((0x100000000ull + (uint32_t)C - 1) / (uint32_t)C);  // x / C = umulhi(x, magic), x < 2^18

  // ---- initial state: given or all zero; row 0 and column s clamped (x_{0,s} = 1)
  for (int i = lane; i < C + 2 * kPad; i += 32) cc[i - kPad] = 0;
  if (a.init)
    for (int e = lane; e < C * Cw; e += 32) bits[e] = 0;
  for (int t = lane; t <= C; t += 32) rec[t] = a.init ? make_uint2(0, 0) : pack_row(0, C, 0, 0);
  __syncwarp();
  if (lane == 0) {
    rec[0] = pack_row(1, s0, 0, 0);
    cc[s0] = 1;
  }
  __syncwarp();
  if (a.init) {
    // the bytes that are set, found 16 at a time
    const uint8_t *x = a.init + (size_t)rep * n;
    auto set = [&](int k) {
      const int t = QP_IX(k / C, C, 9), i = k - t * C;
      if (t == 0 || i == s0) return;
      atomicOr(bits + QP_IX(t * Cw + (i >> 5), C * Cw, 3), 1u << (i & 31));
      const int at = (int)(atomicAdd(&rec[t].x, 1u) & 0xFFFFu);
      if (at == 0) atomicOr(&rec[t].x, (uint32_t)i << 16);
      else if (at < kRowCells) atomicOr(&rec[t].y, (uint32_t)i << (at == 1 ? 0 : 16));
      uint32_t *cw = reinterpret_cast<uint32_t *>(cc - kPad) + ((i + kPad) >> 1);
      atomicAdd(cw, (i & 1) ? 0x10000u : 1u);
    };
    const int head = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15));
    const int nv = (n - head) / 16;
    if (lane < head && x[lane]) set(lane);
    for (int v0 = 0; v0 < nv; v0 += 128) {
      uint4 q[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int v = v0 + 32 * g + lane;
        q[g] = v < nv ? __ldg(reinterpret_cast<const uint4 *>(x + head) + v) : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        if ((q[g].x | q[g].y | q[g].z | q[g].w) == 0) continue;
        const int k0 = head + 16 * (v0 + 32 * g + lane);
        for (int b = 0; b < 16; ++b)
          if ((word_of(q[g], b >> 2) >> (8 * (b & 3))) & 0xFFu) set(k0 + b);
      }
    }
    for (int k = head + 16 * nv + lane; k < n; k += 32)
      if (x[k]) set(k);
    __syncwarp();
    for (int t = lane; t <= C; t += 32)
      if ((rec[t].x & 0xFFFFu) == 0) rec[t] = pack_row(0, C, 0, 0);
    __syncwarp();
  }
  // ---- energy (Eqs. 3-6), violation count, empty columns
  long long E;
  int viol, nz;
  {
    long long hd = 0, pen = 0;
    int v = 0, z = 0;
    // Rows t and t + 1 of many cells: their pairs by the whole warp (pair_distance), which for fewer takes longer.  Only
    // where the bits are in shared memory: the others' sweeps lose 1% to it (893 cells 22.0 -> 22.2 ms).
    const int most = (C + 127) / 128 * ((C + 127) / 128) * 144;
    bool many = false;
    for (int t = lane; t < C; t += 32) {
      const Row q = unpack_row(rec[t]);
      pen += (long long)(1 - q.n) * (1 - q.n);
      v += q.n != 1;
      if (a.init && t + 1 < C && q.n > 0) {
        const Row p = unpack_row(rec[t + 1]);
        if (ROWS == kWide && SB && q.n * p.n > most) {
          many = true;
        } else if (q.n <= kRowCells) {
          hd += row_sum_d<DT, DM, SB>(p, t + 1, bits, Cw, C, D, q.c0);
          if (q.n > 1) hd += row_sum_d<DT, DM, SB>(p, t + 1, bits, Cw, C, D, q.c1);
          if (q.n > 2) hd += row_sum_d<DT, DM, SB>(p, t + 1, bits, Cw, C, D, q.c2);
        } else {
          for (int w = 0; w < Cw; ++w) {
            uint32_t wd = bits_word<SB>(bits + t * Cw + w);
            while (wd) {
              hd += row_sum_d<DT, DM, SB>(p, t + 1, bits, Cw, C, D, (w << 5) + __ffs(wd) - 1);
              wd &= wd - 1;
            }
          }
        }
      }
    }
    if (ROWS == kWide && SB && __any_sync(kFull, many))
      hd += pairs_distance<DT, SB>(static_cast<const DT *>(a.d), a.Cp, C, bits, Cw, rec, most, lane);
    for (int i = lane; i < C; i += 32) {
      const int c = cc[i];
      pen += (long long)(1 - c) * (1 - c);
      v += c != 1;
      z += c == 0;
    }
    for (int t = lane; t < C; t += 32) {
      const int h = (int)(rec[t].x >> 16);
      hx[t] = (uint16_t)D.code(min(h, C - 1));
    }
    __syncwarp();
    E = (long long)B * warp_sum64(hd) + (long long)a.A * warp_sum64(pen);
    viol = __reduce_add_sync(kFull, v);
    nz = __reduce_add_sync(kFull, z);
  }
  long long best = LLONG_MAX, acc = 0;
  int zreg = 0;          // lane q < nz: an empty column (when zok)
  bool zok = false;
  int rows_flipped = 2 * viol;  // rows the last sweep changed; at first, a guess from the state
  // the lane's valid columns (in the field, not s) of a row's first chunk, by t C mod 4: bit 4 (tC mod 4) + j
  uint32_t vfirst = 0;
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const int i = 4 * lane - (e >> 2) + (e & 3);
    vfirst |= (uint32_t)(i >= 0 && i < C && i != s0) << e;
  }

  // ---- sweeps.  Lane l holds the table's place and length, T ln 2 and thr[2A]
  // of sweep s0 + l, loaded 32 sweeps at a time (a cold sweep is shorter than
  // one load).
  const int lev = a.level ? __ldg(a.level + rep) : -1;
  long long off_l = 0;
  int len_l = 0;
  float cT_l = 0.0f, Tl_l = 0.0f;
  uint32_t q2_l = 0;  // thr[2A], 0 when the table ends before it
  bool settled = false;
  int settled_len = 0;
  for (int s = a.sweep_begin; s < a.sweep_end; ++s) {
    const int sl = (s - a.sweep_begin) & 31;
    if (sl == 0) {
      const int ts = lev >= 0 ? lev : min(s + lane, a.sweep_end - 1);
      off_l = __ldg(reinterpret_cast<const long long *>(a.thr_off) + ts);
      len_l = __ldg(a.thr_len + ts);
      cT_l = __ldg(a.thr_c + ts);
      Tl_l = 1.0f / cT_l;
      q2_l = len_l > twoA ? __ldg(a.thr + off_l + twoA) : 0u;
    }
    const uint32_t *thr = a.thr + __shfl_sync(kFull, off_l, sl);
    const int len = __shfl_sync(kFull, len_l, sl);
    const float cT = __shfl_sync(kFull, cT_l, sl), Tl = __shfl_sync(kFull, Tl_l, sl);
    const uint32_t Q2 = __shfl_sync(kFull, q2_l, sl);
    if (settled && len <= settled_len) continue;
    const bool hot = Q2 != 0;
    const float margin = Tl * (1.0f / 512.0f);  // of the estimate below
    const float top0 = fmaf(32.0f, Tl, margin);
    const int band = (int)(2.0f * margin) + 2;
    bool hit = hot;  // a proposal with dE < len was met

    // The draws of the lane's four columns of row t, block m (first: in the
    // row's first 128 columns), and the largest
    // dE each can accept: u < floor(2^32 exp(-dE/T)) iff dE <= T ln(2^32 /
    // (u + 1)), here with a margin above the estimate's error (100 times it), so
    // that a dE above the bound is rejected for certain, and one more than
    // `band` below it accepted; between them the table decides.
    auto draws = [&](int tC, uint32_t m, uint32_t (&u)[4], int (&top)[4], auto first) {
      const uint4 u4 = philox4x32_10(make_uint4(m, (uint32_t)s, rg, kRngTag), key);
      u[0] = u4.x; u[1] = u4.y; u[2] = u4.z; u[3] = u4.w;
      uint32_t v = vfirst >> (4 * (tC & 3));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float lg;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(__uint2float_rn(u[j]) + 1.0f));
        const int i = (int)(4 * m) - tC + j;
        const bool valid = decltype(first)::value ? (v >> j) & 1u : (unsigned)i < (unsigned)C && i != s0;
        top[j] = valid ? (int)fmaf(-lg, Tl, top0) : INT_MIN;
      }
    };

    // The row in hand: its number of cells r, the cells (l0, l1, l2) unless lost (see Row).
    int r = 0, l0 = 0, l1 = 0, l2 = 0, flips = 0, flips0 = 0;
    bool lost = false;
    auto start_row = [&](const Row &p) {
      r = p.n;
      l0 = p.c0;
      l1 = p.c1;
      l2 = p.c2;
      lost = p.n > kRowCells;
      flips0 = flips;
    };
    // Row t is done (n cells before): its record, stored when it changed.
    auto finish_row = [&](int t, int n) -> uint2 {
      uint2 q = pack_row(r, r > 0 ? l0 : C, l1, l2);
      if (flips != flips0) {
        ++rows_flipped;
        if (ROWS != kWide) zok = false;
        viol += (r != 1) - (n != 1);
        __syncwarp();
        if (lost) q = record_from_bits<SB>(bits, Cw, C, t, r, lane);
        if (lane == 0) {
          rec[QP_RANGE(t, 1, C, 9)] = q;
          if (r == 1) hx[QP_RANGE(t, 1, C, 9)] = (uint16_t)D.code((int)(q.x >> 16));
        }
        __syncwarp();
      }
      return q;
    };

    // dE of the lane's four columns i0 .. i0 + 3 (-4 < i0) of row t, whose
    // records are p1 and, around it, p0 and p2, at the row's sum r; how it moves
    // when the row gains a cell (step), and the columns' place, x and sums
    // (code: j | x << 2 | c << 3).
    auto evaluate = [&](int t, const Row &p0, const Row &p1, const Row &p2, int i0, int (&dE)[4], int (&step)[4],
                        int (&code)[4]) {
      const int ic = min(i0, C);
      int f[4] = {0, 0, 0, 0}, c[4];
      uint32_t xi[4] = {0, 0, 0, 0};
      if (DM == 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j) xi[j] = D.xy[QP_RANGE(ic + j, -kPad, C + kPad, 10)];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) c[j] = cc[QP_RANGE(ic + j, -kPad, C + kPad, 8)];
      D.add4(p0.c0, ic, xi, f);
      D.add4(p2.c0, ic, xi, f);
      bool x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = i0 + j == p1.c0;
      if (p0.n > 1 || p1.n > 1 || p2.n > 1) {  // rows of several cells
        if (p1.n > kRowCells) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int i = i0 + j;
            x[j] = i >= 0 && i < C && ((bits_word<SB>(bits + QP_IX(t * Cw + (i >> 5), C * Cw, 3)) >> (i & 31)) & 1u);
          }
        } else if (p1.n > 1) {
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = x[j] || i0 + j == p1.c1 || (p1.n > 2 && i0 + j == p1.c2);
        }
#pragma unroll 1
        for (int side = -1; side <= 1; side += 2) {
          const Row &p = side < 0 ? p0 : p2;
          if (p.n > kRowCells) {  // the cells from the row's bits, but the one already added
            for (int w0 = 0; w0 < Cw; w0 += 32) {
              uint32_t word = w0 + lane < Cw ? bits_word<SB>(bits + QP_IX((t + side) * Cw + w0 + lane, C * Cw, 3)) : 0u;
              if ((p.c0 >> 5) == w0 + lane) word &= ~(1u << (p.c0 & 31));
              for (uint32_t b = __ballot_sync(kFull, word != 0); b; b &= b - 1) {
                const int w = __ffs(b) - 1;
                for (uint32_t wd = __shfl_sync(kFull, word, w); wd; wd &= wd - 1)
                  D.add4(((w0 + w) << 5) + __ffs(wd) - 1, ic, xi, f);
              }
            }
          } else if (p.n > 1) {
            D.add4(p.c1, ic, xi, f);
            if (p.n > 2) D.add4(p.c2, ic, xi, f);
          }
        }
      }
      // dE of x = 0, and 4A less it for x = 1
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int v = twoA * (c[j] + r - 1) + B * f[j];
        dE[j] = x[j] ? 2 * twoA - v : v;
        step[j] = x[j] ? -twoA : twoA;
        code[j] = c[j] << 3 | (x[j] ? 4 + j : j);
      }
    };

    // The row's proposals of one block, in order: the first that may be accepted
    // is settled, applied to the row and to the state, and the rest looked at again.
    auto resolve = [&](int t, int i0, int (&dE)[4], const int (&step)[4], int (&top)[4], const int (&code)[4],
                       const uint32_t (&u)[4]) {
      while (true) {
        const bool ok0 = dE[0] <= top[0], ok1 = dE[1] <= top[1], ok2 = dE[2] <= top[2], ok3 = dE[3] <= top[3];
        const uint32_t bal = __ballot_sync(kFull, ok0 || ok1 || ok2 || ok3);
        if (bal == 0) break;
        const int L = __ffs(bal) - 1;
        const int dl = ok0 ? dE[0] : (ok1 ? dE[1] : (ok2 ? dE[2] : dE[3]));
        const int tl = ok0 ? top[0] : (ok1 ? top[1] : (ok2 ? top[2] : top[3]));
        const int cl = ok0 ? code[0] : (ok1 ? code[1] : (ok2 ? code[2] : code[3]));
        const int de = __shfl_sync(kFull, dl, L);
        const int pk = __shfl_sync(kFull, cl | (tl - dl <= band ? 1 << 20 : 0), L);
        const int jm = pk & 3;
        const int im = __shfl_sync(kFull, i0, L) + jm;
        if (pk >> 20) {  // within the estimate's band: the table decides
          const uint32_t ul = jm == 0 ? u[0] : (jm == 1 ? u[1] : (jm == 2 ? u[2] : u[3]));
          const uint32_t um = __shfl_sync(kFull, ul, L);
          if (!(de <= 0 || (de < len && um < __ldg(thr + QP_IX(de, len, 1))))) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (lane == L && j == jm) top[j] = INT_MIN;
            continue;
          }
        }
        const int cm = (pk >> 3) & 0x1FFFF, dlt = pk & 4 ? -1 : 1;
        E += de;
        ++flips;
        viol += (cm + dlt != 1) - (cm != 1);
        nz += (cm + dlt == 0) - (cm == 0);
        if (lane == 0) cc[QP_IX(im, C, 8)] = (uint16_t)(cm + dlt);
        if (ROWS == kWide && zok) {  // the list of empty columns follows (491 cells: 91.7 -> 90.6 ms)
          if (cm + dlt == 0) {
            if (lane == nz - 1) zreg = im;
            zok = nz <= kZCheck;
          } else if (cm == 0) {  // the last entry takes the filled column's place
            const int last = __shfl_sync(kFull, zreg, nz);
            if (lane < nz && zreg == im) zreg = last;
          }
        }
        // every proposal up to it is decided; the row's sum moved for the rest
        const int rel = im - i0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          dE[j] += dlt * step[j];
          if (rel >= j) top[j] = INT_MIN;
        }
        if (lost || (dlt > 0 && r >= kRowCells)) {  // a row of more than three cells: its bits
          if (!lost) {
            for (int w = lane; w < Cw; w += 32)
              bits[QP_IX(t * Cw + w, C * Cw, 3)] = ((l0 >> 5) == w ? 1u << (l0 & 31) : 0u) |
                                                   ((l1 >> 5) == w ? 1u << (l1 & 31) : 0u) |
                                                   ((l2 >> 5) == w ? 1u << (l2 & 31) : 0u);
            lost = true;
            __syncwarp();
          }
          if (lane == 0) {
            uint32_t *wp = bits + QP_IX(t * Cw + (im >> 5), C * Cw, 3);
            if (SB) *wp ^= 1u << (im & 31);
            else atomicXor(wp, 1u << (im & 31));
          }
        } else {
          const bool add = dlt > 0, first = l0 == im, second = l1 == im;
          const int n0 = add ? im : (first ? l1 : l0), n1 = add ? l0 : (first || second ? l2 : l1);
          l2 = add ? l1 : l2;
          l1 = n1;
          l0 = n0;
        }
        r += dlt;
      }
    };

    // Row t, exactly.  Blocks of 128 columns in which nothing can be accepted are
    // passed over: with r >= 1 a block needs one of the row's own cells, or (r = 1)
    // an empty column, or a survivor; everything else costs dE >= 2A.  sv: whether
    // the row may hold survivors; a block whose draws all bound dE below 2A has none.
    auto event_row = [&](int t, bool sv) {
      const Row p0 = unpack_row(rec[QP_IX(t - 1, C + 1, 9)]), p1 = unpack_row(rec[QP_IX(t, C + 1, 9)]),
                p2 = unpack_row(rec[QP_IX(t + 1, C + 1, 9)]);
      const int tC = t * C;
      start_row(p1);
      const uint32_t m1 = (uint32_t)(tC + C - 1) >> 2;
      for (uint32_t mb = (uint32_t)tC >> 2; mb <= m1; mb += 32) {
        uint32_t u[4];
        int top[4], dE[4], step[4], code[4];
        const int i0 = (int)(4 * (mb + lane)) - tC;
        bool live = true;
        if (ROWS == kWide && r >= 1 && !lost) {
          const int ib = (int)(4 * mb) - tC;
          live = (unsigned)(l0 - ib) < 128u || (r > 1 && (unsigned)(l1 - ib) < 128u) || (r > 2 && (unsigned)(l2 - ib) < 128u);
          if (!live && r == 1 && nz > 0) {
            bool z = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int i = min(max(i0 + j, 0), C - 1);
              z = z || cc[QP_IX(i, C, 8)] == 0;
            }
            live = __any_sync(kFull, z);
          }
          if (!live && !sv) continue;
        }
        draws(tC, mb + lane, u, top, std::bool_constant<ROWS == kOneBlock>());
        if (ROWS == kWide && !live && !__any_sync(kFull, max(max(top[0], top[1]), max(top[2], top[3])) >= twoA)) continue;
        evaluate(t, p0, p1, p2, i0, dE, step, code);
        resolve(t, i0, dE, step, top, code, u);
        if (ROWS == kOneBlock) break;
      }
      finish_row(t, p1.n);
    };

    // A cold sweep over a permutation (every row and column holds one cell):
    // only removing a row's own cell can cost less than 2A.  32 rows at a time
    // and one vote for the sweep.
    bool quiet = false;
    if (!hot && viol == 0) {
      bool any = false;
#pragma unroll 4
      for (int t = 1 + lane; t < C; t += 32) {
        const uint32_t h = hx[QP_IX(t, C, 9)];
        const int f = D.near(hx[QP_IX(t - 1, C, 9)], h) + (t + 1 < C ? D.near(hx[t + 1], h) : 0);
        any |= twoA - B * f < len;
      }
      quiet = !__any_sync(kFull, any);
    }
    // row by row when half the rows are events anyway: rows changed in the last sweep, rows with survivors
    const float lambda = (float)Q2 * 2.3283064365386963e-10f * (float)C;
    const bool rowwise = (float)rows_flipped + 0.5f * lambda * (float)C > 0.5f * (float)C;
    rows_flipped = 0;
    if (quiet) {
    } else if (ROWS != kWide && rowwise && C <= kNarrow) {  // a row is one block of 128 columns, whatever t C mod 4
      hit = true;
      // the next row's draws and record are fetched beside a row's evaluation, of which they are independent
      uint32_t u[4];
      int top[4];
      draws(C, ((uint32_t)C >> 2) + lane, u, top, std::true_type());
      Row p0 = unpack_row(rec[0]), p1 = unpack_row(rec[1]), p2 = unpack_row(rec[2]);
      for (int t = 1; t < C; ++t) {
        const int tC = t * C;
        uint32_t un[4];
        int topn[4], dE[4], step[4], code[4];
        draws(tC + C, ((uint32_t)(tC + C) >> 2) + lane, un, topn, std::true_type());
        const uint2 q3 = rec[QP_IX(min(t + 2, C), C + 1, 9)];
        start_row(p1);
        const int i0 = 4 * lane - (tC & 3);
        evaluate(t, p0, p1, p2, i0, dE, step, code);
        resolve(t, i0, dE, step, top, code, u);
        p0 = unpack_row(finish_row(t, p1.n));
        p1 = p2;
        p2 = unpack_row(q3);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          u[j] = un[j];
          top[j] = topn[j];
        }
      }
    } else {
      for (int t0 = 1; t0 < C; t0 += 32) {
        const int t1 = min(C, t0 + 32);
        // -- draws of the window: the rows with survivors
        uint32_t smask = 0;
        if (hot && !rowwise) {
          const uint32_t k0 = (uint32_t)(t0 * C), nk = (uint32_t)((t1 - t0) * C);
          const uint32_t mend = (k0 + nk - 1) >> 2;
          auto mark = [&](const uint4 &w4, uint32_t m) {
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t rel = 4 * m + j - k0;
              if (w[j] < Q2 && rel < nk) smask |= 1u << __umulhi(rel, magic);
            }
          };
          for (uint32_t mb = k0 >> 2; mb <= mend; mb += 64) {
            const uint32_t ma = mb + lane, mc = ma + 32;
            const uint4 ua = philox4x32_10(make_uint4(ma, (uint32_t)s, rg, kRngTag), key);
            const uint4 ub = philox4x32_10(make_uint4(mc, (uint32_t)s, rg, kRngTag), key);
            const uint32_t la = min(min(ua.x, ua.y), min(ua.z, ua.w)), lb = min(min(ub.x, ub.y), min(ub.z, ub.w));
            if (min(la, lb) < Q2) {
              mark(ua, ma);
              mark(ub, mc);
            }
          }
          smask = __reduce_or_sync(kFull, smask);
        }
        // -- the window's rows
        bool have_uh = false;
        uint32_t uh = 0;  // the draw of the cell of row t0 + lane
        for (int t = t0; t < t1; ++t) {
          if (!rowwise && nz <= kZCheck) {
            if (!zok) {  // list the empty columns
              int k = 0;
              for (int i0 = 0; i0 < C && k < nz; i0 += 32) {
                uint32_t b = __ballot_sync(kFull, i0 + lane < C && cc[QP_IX(i0 + lane, C, 8)] == 0);
                while (b) {
                  if (lane == k) zreg = i0 + __ffs(b) - 1;
                  b &= b - 1;
                  ++k;
                }
              }
              zok = true;
            }
            // the check: lane = row
            const int tl = t0 + lane;
            const bool in = tl >= t && tl < t1;
            const int tr = min(tl, C - 1);
            const Row p0 = unpack_row(rec[QP_IX(tr - 1, C + 1, 9)]), p1 = unpack_row(rec[QP_IX(tr, C + 1, 9)]),
                      p2 = unpack_row(rec[QP_IX(tr + 1, C + 1, 9)]);
            bool ev = p1.n != 1 || p0.n > 1 || p2.n > 1 || ((smask >> lane) & 1u);
            const int h = p1.c0;
            int dE = len;
            if (in && !ev) dE = twoA * (2 - (int)cc[QP_IX(h, C, 8)]) - B * (D(p0.c0, h) + D(p2.c0, h));
            bool need = dE < len;
            if (__any_sync(kFull, need)) {
              hit = true;
              if (!have_uh) {
                const uint32_t k = (uint32_t)(tr * C + h);
                const uint4 u4 = philox4x32_10(make_uint4(k >> 2, (uint32_t)s, rg, kRngTag), key);
                uh = word_of(u4, k & 3);
                have_uh = true;
              }
              if (need) ev = dE <= 0 || accept_draw(uh, dE, cT, thr, len);
            }
            for (int q = 0; q < nz; ++q) {
              const int z = __shfl_sync(kFull, zreg, q);
              dE = len;
              if (in && !ev) dE = B * (D(p0.c0, z) + D(p2.c0, z));
              need = dE < len;
              if (__any_sync(kFull, need)) {
                hit = true;
                const uint32_t k = (uint32_t)(tr * C + z);
                const uint4 u4 = philox4x32_10(make_uint4(k >> 2, (uint32_t)s, rg, kRngTag), key);
                if (need) ev = dE <= 0 || accept_draw(word_of(u4, k & 3), dE, cT, thr, len);
              }
            }
            const uint32_t bal = __ballot_sync(kFull, in && ev);
            if (bal == 0) break;  // nothing happens in the rest of the window
            t = t0 + __ffs(bal) - 1;
          }
          hit = true;
          event_row(t, hot && (rowwise || ((smask >> (t - t0)) & 1u)));
        }
      }
    }
    acc += flips;
    if (viol == 0 && E < best) best = E;
    settled = a.skip_settled && !hit;
    settled_len = len;
  }

  // ---- outputs: zeros in 16-byte stores, then the cells
  uint8_t *out = a.states_out + (size_t)rep * n;
  const int head = min(n, (int)((16 - (reinterpret_cast<uintptr_t>(out) & 15)) & 15));
  const int nv = (n - head) / 16;
  if (lane < head) out[lane] = 0;
  for (int v = lane; v < nv; v += 32) reinterpret_cast<uint4 *>(out + head)[v] = make_uint4(0, 0, 0, 0);
  for (int e = head + 16 * nv + lane; e < n; e += 32) out[e] = 0;
  __syncwarp();
  for (int t = lane; t < C; t += 32) {
    const Row q = unpack_row(rec[t]);
    uint8_t *o = out + (size_t)t * C;
    if (q.n <= kRowCells) {
      if (q.n > 0) o[QP_IX(q.c0, C, 11)] = 1;
      if (q.n > 1) o[QP_IX(q.c1, C, 11)] = 1;
      if (q.n > 2) o[QP_IX(q.c2, C, 11)] = 1;
    } else {
      for (int w = 0; w < Cw; ++w) {
        uint32_t wd = bits_word<SB>(bits + t * Cw + w);
        while (wd) {
          o[QP_IX((w << 5) + __ffs(wd) - 1, C, 11)] = 1;
          wd &= wd - 1;
        }
      }
    }
  }
  if (lane == 0) {
    a.E_out[rep] = E;
    if (a.best_out) a.best_out[rep] = best;
    if (a.acc_out) a.acc_out[rep] = acc;
  }
}

// Shared memory of one replica.
__host__ __device__ inline size_t events_warp_bytes(int C, bool bits_smem) {
  const int Cw = (C + 31) >> 5;
  return align16e(8 * ((size_t)C + 1)) + align16e(2 * ((size_t)C + 1)) + align16e(2 * ((size_t)C + 2 * kPad)) +
         (bits_smem ? align16e(4 * (size_t)C * Cw) : 0);
}

// Shared memory of the distances: the matrix (DM = 1) or the coordinates and the table (DM = 2).
__host__ __device__ inline size_t events_dist_bytes(int C, int Cp, size_t es, int dm, int tab_n) {
  if (dm == 1) return align16e((((size_t)C + 1) * Cp + 2 * kPad) * es);
  if (dm == 2) return align16e(2 * ((size_t)C + 2 * kPad)) + align16e((size_t)tab_n * es);
  return 0;
}

// A column outside the field is rejected by its bound INT_MIN, so its dE must not
// be INT_MIN too: it stays within the bound that keeps a cell's inside int32.  The
// entries around the matrix are zeros; with the table such a column lies at grid
// difference (0, 0), which the table's owner takes into that bound.
template <typename DT, int DM>
__device__ __forceinline__ Dist<DT, DM> stage_dist(const StructArgs &a, unsigned char *p, int tid, int nthreads) {
  Dist<DT, DM> D{static_cast<const DT *>(a.d), a.Cp, a.C, nullptr, a.tab_sh, a.tab_n};
  if (DM == 1) {
    const int nv = (int)((size_t)a.C * a.Cp * sizeof(DT) / 16);
    const int4 *src = static_cast<const int4 *>(a.d);
    DT *m = reinterpret_cast<DT *>(p) + kPad;
    QP_POISON(p, events_dist_bytes(a.C, a.Cp, sizeof(DT), DM, 0), tid, nthreads);
    for (int v = tid; v < nv; v += nthreads) reinterpret_cast<int4 *>(m)[v] = __ldg(src + v);
    if (tid < kPad) m[tid - kPad] = 0;
    for (int i = tid; i < a.Cp + kPad; i += nthreads) m[a.C * a.Cp + i] = 0;
    D.m = m;
  } else if (DM == 2) {
    uint16_t *xy = reinterpret_cast<uint16_t *>(p) + kPad;
    DT *tab = reinterpret_cast<DT *>(p + align16e(2 * ((size_t)a.C + 2 * kPad)));
    QP_POISON(p, events_dist_bytes(a.C, a.Cp, sizeof(DT), DM, a.tab_n), tid, nthreads);
    for (int i = tid - kPad; i < a.C + kPad; i += nthreads) xy[i] = i >= 0 && i < a.C ? __ldg(a.xy + i) : 0;
    for (int i = tid; i < a.tab_n; i += nthreads) tab[i] = __ldg(static_cast<const DT *>(a.tab) + i);
    D.xy = xy;
    D.m = tab;
  }
  return D;
}

// A warp's arrays of one replica in shared memory (events_warp_bytes(C, SB)).
struct WarpArea {
  uint2 *rec;
  uint16_t *hx, *cc;
  uint32_t *bits;  // with SB
};
__device__ __forceinline__ WarpArea warp_area(unsigned char *p, int C) {
  WarpArea w;
  w.rec = reinterpret_cast<uint2 *>(p);
  p += align16e(8 * ((size_t)C + 1));
  w.hx = reinterpret_cast<uint16_t *>(p);
  p += align16e(2 * ((size_t)C + 1));
  w.cc = reinterpret_cast<uint16_t *>(p) + kPad;
  p += align16e(2 * ((size_t)C + 2 * kPad));
  w.bits = reinterpret_cast<uint32_t *>(p);
  return w;
}

template <typename DT, int DM, bool SB, int ROWS>
__global__ void __launch_bounds__(kMaxWarpsPerCta * 32) k_sweep_events(const StructArgs a, const RoundKeys rk) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  const Dist<DT, DM> D = stage_dist<DT, DM>(a, smem, threadIdx.x, blockDim.x);
  __syncthreads();
  const int rep = blockIdx.x * W + warp;
  if (rep >= a.R) return;  // no CTA-wide barrier after this point
  const WarpArea w = warp_area(smem + events_dist_bytes(a.C, a.Cp, sizeof(DT), DM, a.tab_n) +
                                   warp * events_warp_bytes(a.C, SB), a.C);
  events_replica<DT, DM, SB, ROWS>(a, rep, w.rec, w.hx, w.cc, SB ? w.bits : a.gstate + (size_t)rep * a.nw_pad, D, lane,
                                   rk);
}

// Many fields in one persistent launch: a warp takes (field, replica) units
// from a counter, largest fields first, and reads the field's matrix through
// L1 (consecutive units are replicas of the same field).  No warp waits on
// another.  per: shared memory of a warp, sized for the largest field;
// gbits: one replica's bitsets per warp of the grid (without SB).  256 fields
// of 10-169 cells x 128 replicas x 2000 sweeps: 189 ms (the row kernel's batch:
// 1190), 173 with the matrix staged in shared memory by 8 warps (1054).  At 128
// registers and 16 warps per SM (198 at the time: 96 registers, 20 warps 273; 168, 12 warps 216).
template <bool SB>
__global__ void __launch_bounds__(kMaxWarpsPerCta * 32)
    k_events_batch(const StructArgs *fields, const int2 *units, int n_units, int *counter, size_t per, uint32_t *gbits,
                   int gwords) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  while (true) {
    int u = 0;
    if (lane == 0) u = atomicAdd(counter, 1);
    u = __shfl_sync(kFull, u, 0);
    if (u >= n_units) break;
    const int2 unit = units[u];
    const StructArgs &a = fields[unit.x];
    const Dist<int16_t, 0> D{static_cast<const int16_t *>(a.d), a.Cp, a.C, nullptr, 0, 0};
    const WarpArea w = warp_area(smem + warp * per, a.C);
    uint32_t *bits = SB ? w.bits : gbits + (size_t)(blockIdx.x * W + warp) * gwords;
    events_replica<int16_t, 0, SB, kAny>(a, unit.y, w.rec, w.hx, w.cc, bits, D, lane, PhiloxKey{a.key0, a.key1});
    __syncwarp();
  }
}

// The same with units of W replicas of one field per CTA, whose matrix the CTA
// stages in shared memory.
template <bool SB>
__global__ void __launch_bounds__(kMaxWarpsPerCta * 32)
    k_events_batch_staged(const StructArgs *fields, const int2 *units, int n_units, int *counter, size_t dist,
                          size_t per, uint32_t *gbits, int gwords) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_unit;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  while (true) {
    if (threadIdx.x == 0) s_unit = atomicAdd(counter, 1);
    __syncthreads();
    const int u = s_unit;
    if (u >= n_units) break;  // the same u in every thread
    const int2 unit = units[u];
    const StructArgs &a = fields[unit.x];
    const Dist<int16_t, 1> D = stage_dist<int16_t, 1>(a, smem, threadIdx.x, blockDim.x);
    __syncthreads();
    const int rep = unit.y + warp;
    if (rep < a.R) {
      const WarpArea w = warp_area(smem + dist + warp * per, a.C);
      uint32_t *bits = SB ? w.bits : gbits + (size_t)(blockIdx.x * W + warp) * gwords;
      events_replica<int16_t, 1, SB, kAny>(a, rep, w.rec, w.hx, w.cc, bits, D, lane, PhiloxKey{a.key0, a.key1});
    }
    __syncthreads();  // every warp is done with the matrix and s_unit before the next unit
  }
}

constexpr size_t kSmemLimitEvents = 227 * 1024;
constexpr size_t kBitsSmem = 8 * 1024;       // most bytes of a replica's bitsets kept in shared memory
constexpr size_t kMatrixSmem = 40 * 1024;    // largest distance matrix staged in shared memory
static_assert(4 * kNarrow * ((kNarrow + 31) / 32) <= kBitsSmem, "narrow rows keep their bitsets in shared memory");
static_assert(2 * 181 * 181 > kMatrixSmem && 4 * 181 * ((181 + 31) / 32) <= kBitsSmem, "a staged matrix implies the same");

struct EventsShape {
  int dm;
  bool sb;
  size_t dist, per;
};

EventsShape events_shape(const StructArgs &a, bool d_i16) {
  const size_t es = d_i16 ? 2 : 4;
  const int Cw = (a.C + 31) / 32;
  EventsShape s;
  s.sb = 4 * (size_t)a.C * Cw <= kBitsSmem;
  s.dm = (size_t)a.C * a.Cp * es <= kMatrixSmem ? 1 : (a.tab_n > 0 ? 2 : 0);
  s.dist = events_dist_bytes(a.C, a.Cp, es, s.dm, a.tab_n);
  s.per = events_warp_bytes(a.C, s.sb);
  return s;
}

template <typename DT, int DM, bool SB, int ROWS>
cudaError_t launch_e(const StructArgs &a, const RoundKeys &rk, int W, size_t smem, cudaStream_t st) {
  auto k = k_sweep_events<DT, DM, SB, ROWS>;
  std::lock_guard<std::mutex> lk(launch_mutex());
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k<<<(a.R + W - 1) / W, W * 32, smem, st>>>(a, rk);
  return cudaGetLastError();
}

template <typename DT>
cudaError_t launch_e2(const StructArgs &a, const RoundKeys &rk, const EventsShape &s, int W, size_t smem,
                      cudaStream_t st) {
  if (a.C <= kNarrow)  // the bitsets are in shared memory
    return s.dm == 1   ? launch_e<DT, 1, true, kOneBlock>(a, rk, W, smem, st)
           : s.dm == 2 ? launch_e<DT, 2, true, kOneBlock>(a, rk, W, smem, st)
                       : launch_e<DT, 0, true, kOneBlock>(a, rk, W, smem, st);
  if (s.dm == 1) return launch_e<DT, 1, true, kWide>(a, rk, W, smem, st);  // so here, too
  if (s.dm == 2)
    return s.sb ? launch_e<DT, 2, true, kWide>(a, rk, W, smem, st) : launch_e<DT, 2, false, kWide>(a, rk, W, smem, st);
  return s.sb ? launch_e<DT, 0, true, kWide>(a, rk, W, smem, st) : launch_e<DT, 0, false, kWide>(a, rk, W, smem, st);
}

}  // namespace

size_t events_state_words(int C) {
  const int Cw = (C + 31) / 32;
  const size_t words = ((size_t)C * Cw + 3) / 4 * 4;
  return 4 * (size_t)C * Cw <= kBitsSmem ? 0 : words;
}

cudaError_t launch_events(const StructArgs &a_in, bool d_i16, int W, cudaStream_t st, LaunchInfo *info) {
  StructArgs a = a_in;
  a.nw_pad = (int32_t)events_state_words(a.C);
  const EventsShape s = events_shape(a, d_i16);
  if (!s.sb && a.gstate == nullptr) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // One chain per scheduler first: a chain's latency is its time, so few chains
  // spread over the SMs.  Above 8 per SM 8 share the staged distances, or 4
  // where that leaves fewer chains on the fullest SM, whose time the launch takes
  // (8 -> 4: 491 cells, 4096 chains, 32 -> 28 on it: 90.5 -> 82.7 ms; 1824 chains,
  // 16 -> 12: 46.0 -> 39.0; 92 cells, 4096 chains: 79.2 -> 73.5; where both leave as
  // many 8 stays: 236 cells, 2000 chains, 16 each: 38.5 against 39.8).
  if (W <= 0) {
    auto fullest = [&](int w) { return ((a.R + w - 1) / w + sms - 1) / sms * w; };
    W = a.R <= 8 * sms ? std::max(1, (a.R + sms - 1) / sms) : (fullest(4) < fullest(8) ? 4 : 8);
  }
  while (W > 1 && s.dist + W * s.per > kSmemLimitEvents) --W;
  const size_t smem = s.dist + W * s.per;
  if (smem > kSmemLimitEvents) return cudaErrorInvalidValue;
  if (info) {
    info->warps_per_cta = W;
    info->blocks = (a.R + W - 1) / W;
    info->smem = smem;
    info->variant = s.dm == 1 ? "events,d:smem" : (s.dm == 2 ? "events,d:table" : "events,d:global");
  }
  RoundKeys rk;
  for (int i = 0; i < 10; ++i) {
    rk.k[2 * i] = a.key0 + (uint32_t)i * 0x9E3779B9u;
    rk.k[2 * i + 1] = a.key1 + (uint32_t)i * 0xBB67AE85u;
  }
  return d_i16 ? launch_e2<int16_t>(a, rk, s, W, smem, st) : launch_e2<int32_t>(a, rk, s, W, smem, st);
}

namespace {

// The batched launch's shared memory: bitsets in shared memory when a replica's
// are small and the CTA's fit.
struct BatchShape {
  bool sb;
  size_t dist, per, smem;
};
BatchShape batch_shape(int Cmax, int W, bool staged) {
  BatchShape b;
  b.dist = staged ? events_dist_bytes(Cmax, (Cmax + 7) / 8 * 8, 2, 1, 0) : 0;
  b.sb = 4 * (size_t)Cmax * ((Cmax + 31) / 32) <= kBitsSmem;
  b.per = events_warp_bytes(Cmax, b.sb);
  if (b.sb && b.dist + W * b.per > kSmemLimitEvents) {
    b.sb = false;
    b.per = events_warp_bytes(Cmax, false);
  }
  b.smem = b.dist + W * b.per;
  return b;
}

template <typename K>
cudaError_t prepare_batch(K k, int W, size_t smem, int *blocks_per_sm) {
  std::lock_guard<std::mutex> lk(launch_mutex());
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, W * 32, smem);
}

}  // namespace

// Up to 512 cells, 16 replicas per CTA (8 above 256 cells) whose bitsets and
// one 2-byte entry per row fit 227 KB beside the staged matrix: the entry
// points' limits, which all fit the kernel's own layout too.
bool batch_supported(int Cmax, int W, bool staged) {
  if (Cmax < 2 || Cmax > 512 || W < 1 || W > (Cmax <= 256 ? kMaxWarpsPerCta : 8)) return false;
  const size_t bits = ((size_t)Cmax * ((Cmax + 31) / 32) + 3) / 4 * 16;
  const size_t d = staged ? align16e((size_t)Cmax * ((Cmax + 7) / 8 * 8) * 2) : 0;
  return d + W * (bits + align16e(2 * (size_t)Cmax)) <= kSmemLimitEvents;
}

cudaError_t events_batch_prepare(int Cmax, int W, bool staged, int *blocks_per_sm, size_t *gstate_words) {
  const BatchShape b = batch_shape(Cmax, W, staged);
  *gstate_words = b.sb ? 0 : ((size_t)Cmax * ((Cmax + 31) / 32) + 3) / 4 * 4;
  if (b.smem > kSmemLimitEvents) return cudaErrorInvalidValue;
  if (staged)
    return b.sb ? prepare_batch(k_events_batch_staged<true>, W, b.smem, blocks_per_sm)
                : prepare_batch(k_events_batch_staged<false>, W, b.smem, blocks_per_sm);
  return b.sb ? prepare_batch(k_events_batch<true>, W, b.smem, blocks_per_sm)
              : prepare_batch(k_events_batch<false>, W, b.smem, blocks_per_sm);
}

cudaError_t launch_events_batch(const StructArgs *fields, const int2 *units, int n_units, int *counter, int Cmax, int W,
                                bool staged, int blocks, uint32_t *gstate, cudaStream_t st) {
  const BatchShape b = batch_shape(Cmax, W, staged);
  if (b.smem > kSmemLimitEvents || blocks < 1 || (!b.sb && gstate == nullptr)) return cudaErrorInvalidValue;
  const int gwords = (Cmax * ((Cmax + 31) / 32) + 3) / 4 * 4;
  if (staged) {
    if (b.sb) k_events_batch_staged<true><<<blocks, W * 32, b.smem, st>>>(fields, units, n_units, counter, b.dist, b.per, gstate, gwords);
    else k_events_batch_staged<false><<<blocks, W * 32, b.smem, st>>>(fields, units, n_units, counter, b.dist, b.per, gstate, gwords);
  } else {
    if (b.sb) k_events_batch<true><<<blocks, W * 32, b.smem, st>>>(fields, units, n_units, counter, b.per, gstate, gwords);
    else k_events_batch<false><<<blocks, W * 32, b.smem, st>>>(fields, units, n_units, counter, b.per, gstate, gwords);
  }
  return cudaGetLastError();
}

}  // namespace qp

namespace qp {
namespace chk {
QP_CHECK_ACCESSOR(events)
}  // namespace chk
}  // namespace qp
