// Fused conformal-Hough kernel: map -> rho -> vote -> peaks -> select, one CTA per
// (event, theta tile) work item, the accumulator never leaving shared memory.
//
// Thread organisation (Sec. 3's event / angle-column / hit parallelism, redone for sm_103a):
//   - a work item is one event, or one theta tile of an event when its accumulator
//     does not fit one CTA's shared memory;
//   - every lane of a "worker" warp owns theta columns of the tile for the whole vote.
//     Lane l's cells live in shared-memory bank l only: word ((g * rows + row) * 32 + l),
//     rows = N_rho / 2 packed int16 pairs, so the column-parallel
//     vote is free of bank conflicts whatever rho bins the hits hit; warps sharing
//     columns split the hits and add with red.shared. In mirror pairs a lane owns
//     column j and its mirror N_theta-1-j (th -> pi - th: c -> -c, s -> s), so one pair
//     of products gives both rho values;
//   - for tiled events the neighbour columns of the tile are voted too (halo: mirror pairs by every thread,
//     columns by one extra warp), so the 3x3 peak test is exact on tile edges; the last tile CTA of an
//     event (ticket counter; a run of all tiles in one CTA needs none) merges the tiles' peak lists in tile order
//     and selects. Events of small calls take the tiles of a cluster, which merge without a workspace.
#include <algorithm>
#include <climits>
#include <map>
#include <mutex>
#include <utility>

#include "hough_internal.h"

namespace hgpu {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSelCap = 12;  // peak columns a lane tries alone before its hit goes to a whole warp

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ uint32_t vmax2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__device__ __forceinline__ uint32_t swap16(uint32_t x) { return __funnelshift_l(x, x, 16); }

__device__ __forceinline__ int acc_index(int c, int k, int nrp) {
  return (((c >> 5) * (nrp >> 1) + (k >> 1)) << 5) + (c & 31);
}

__device__ __forceinline__ int acc_get(const uint32_t* acc, int c, int k, int nrp) {
  const uint32_t w = acc[acc_index(c, k, nrp)];
  return (int)((w >> ((k & 1) << 4)) & 0xffffu);
}

// One vote for row k of the column whose row-0 word is at shared address `colbase`.
// No memory clobber: the accumulator is only read after a barrier, and leaving the hit
// loads free to move above the atomics lets consecutive hits overlap.
__device__ __forceinline__ void vote_cell(uint32_t colbase, int k) {
  const uint32_t addr = colbase + (((uint32_t)k >> 1) << 7);
  const uint32_t inc = 1u << (((uint32_t)k & 1u) << 4);
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(inc));
}

// One vote for row k of a halo column: packed int16 pairs stored contiguously.
__device__ __forceinline__ void vote_halo(uint32_t colbase, int k) {
  const uint32_t addr = colbase + (((uint32_t)k >> 1) << 2);
  const uint32_t inc = 1u << (((uint32_t)k & 1u) << 4);
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(inc));
}

// In-place exclusive scan of arr[0, n) by the whole CTA; returns the total.
__device__ int block_exscan(int* arr, int n, int* s_tmp) {
  const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (n + nt - 1) / nt;
  const int lo = min(n, tid * per), hi = min(n, lo + per);
  int sum = 0;
  for (int i = lo; i < hi; ++i) sum += arr[i];
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_tmp[w] = x;
  __syncthreads();
  if (w == 0) {
    int z = (lane < (nt >> 5)) ? s_tmp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, z, o);
      if (lane >= o) z += y;
    }
    s_tmp[lane] = z;
  }
  __syncthreads();
  int excl = x - sum + (w > 0 ? s_tmp[w - 1] : 0);
  const int total = s_tmp[(nt >> 5) - 1];
  for (int i = lo; i < hi; ++i) {
    const int v = arr[i];
    arr[i] = excl;
    excl += v;
  }
  __syncthreads();
  return total;
}

__device__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* s_red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  if (lane == 0) s_red[w] = v;
  __syncthreads();
  unsigned long long t = 0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_red[i];
  __syncthreads();
  return t;  // valid in thread 0
}

// ---- staging hits into shared memory ----

// Maps hits [base, base + cn) and appends those that fit the int32 fast path to hb
// (compacted, order not kept). Valid hits beyond int32 set bit 0 of *s_flags, bad
// hits bit 1.
__device__ void stage_vote32(const int2* __restrict__ xy, long long base, int cn, int2* hb, int* s_nv, int* s_flags,
                             unsigned lsq, uint16_t* idx) {
  const int lane = threadIdx.x & 31;
  // each thread's next hit is loaded one pass ahead, so the loads overlap the mapping
  int2 hn = threadIdx.x < cn ? xy[base + threadIdx.x] : make_int2(0, 0);
  for (int i0 = 0; i0 < cn; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    const int2 h = hn;
    if (i + (int)blockDim.x < cn) hn = xy[base + i + blockDim.x];
    long long u = 0, v = 0;
    int st = 0;
    bool ok = false;
    if (i < cn) {
      st = map_hit(h.x, h.y, u, v);
      ok = (st == 0);
    }
    // fast path: int32 rho, and (mirror-pair layout) rho within one guard bin of the range; the squares of
    // values within kFast32 add up below 2^32
    const int u32 = (int)u, v32 = (int)v;
    const bool f = ok && fits32(u, v) && (unsigned)(u32 * u32) + (unsigned)(v32 * v32) <= lsq;
    const unsigned bal = __ballot_sync(kFull, f);
    if (bal) {
      int slot = 0;
      if (lane == 0) slot = atomicAdd(s_nv, __popc(bal));
      slot = __shfl_sync(kFull, slot, 0);
      // float form for the float bin path: |u|, |v| <= 44061 are exact in float; the mirror-pair
      // layout (idx given) stores hits in pairs (u0, u1, v0, v1) for the vote's f32x2 arithmetic
      if (f) {
        const int at = slot + __popc(bal & lanemask_lt());
        if (idx) {
          float* fp = reinterpret_cast<float*>(hb) + 4 * (at >> 1) + (at & 1);
          fp[0] = (float)u;
          fp[2] = (float)v;
          idx[at] = (uint16_t)i;
        } else {
          hb[at] = make_int2(__float_as_int((float)u), __float_as_int((float)v));
        }
      }
    }
    if (ok && !f) atomicOr(s_flags, 1);
    if (st) atomicOr(s_flags, 2);
  }
}

// Maps hits [base, base + cn) and appends every valid one as int64 to hw (compacted).
__device__ void stage_vote64(const int2* __restrict__ xy, long long base, int cn, longlong2* hw, int* s_nv) {
  const int lane = threadIdx.x & 31;
  for (int i0 = 0; i0 < cn; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    long long u = 0, v = 0;
    bool ok = false;
    if (i < cn) {
      const int2 h = xy[base + i];
      ok = (map_hit(h.x, h.y, u, v) == 0);
    }
    const unsigned bal = __ballot_sync(kFull, ok);
    if (bal) {
      int slot = 0;
      if (lane == 0) slot = atomicAdd(s_nv, __popc(bal));
      slot = __shfl_sync(kFull, slot, 0);
      if (ok) hw[slot + __popc(bal & lanemask_lt())] = make_longlong2(u, v);
    }
  }
}

// Selection staging keeps hit order: hb[i] = (u, v), or (INT_MIN, 0) for a bad hit.
// A valid hit beyond int32 sets *s_wide.
__device__ void stage_sel32(const int2* __restrict__ xy, long long base, int cn, int2* hb, int* s_wide) {
  for (int i = threadIdx.x; i < cn; i += blockDim.x) {
    const int2 h = xy[base + i];
    long long u = 0, v = 0;
    const int st = map_hit(h.x, h.y, u, v);
    if (st) {
      hb[i] = make_int2(INT_MIN, 0);
    } else if (fits32(u, v)) {
      hb[i] = make_int2((int)u, (int)v);
    } else {
      hb[i] = make_int2(INT_MIN, 0);
      *s_wide = 1;
    }
  }
}

__device__ void stage_sel64(const int2* __restrict__ xy, long long base, int cn, longlong2* hw) {
  for (int i = threadIdx.x; i < cn; i += blockDim.x) {
    const int2 h = xy[base + i];
    long long u = 0, v = 0;
    const int st = map_hit(h.x, h.y, u, v);
    hw[i] = st ? make_longlong2(LLONG_MIN, 0) : make_longlong2(u, v);
  }
}

// ---- voting ----

// Which columns a worker lane owns, and where their row-0 words live.
struct VoteLane {
  bool on;          // lane votes
  bool halo;        // columns: lane of the halo warp (tiles > 1)
  int p, P;         // hit partition of this warp, partitions per column set
  int cj, sj;       // trig of the (first) column
  uint32_t col1;    // shared address of column 1, row 0
  uint32_t col2;    // halo column
};

// Bin of the float estimate kf = u A + v B + N_rho/2 of k* = (u c + v s + H) N_rho / 2H, where
// A = c N_rho/2H, B = s N_rho/2H in float. |kf - k*| < N_rho 2^-21 (rounding of A, B and of
// the three float operations, each at most 2^-24 relative of a term below 1.6 N_rho), so
// floor(kf) = floor(k*) unless an integer lies within delta = N_rho 2^-20 of kf. y1 and y2
// round kc - 1/2 + delta and kc - 1/2 - delta to integers (adding 1.5 2^23 leaves no fraction
// bits); they differ exactly when such an integer exists, and then the exact integer path
// decides. Clamping kf to [1/2, N_rho - 1/2] first gives the edge bins for rho outside the
// range, as the integer clamp does.
struct FpBin {
  float khi, dlo, dhi;
};

__device__ __forceinline__ int bin_fp(float kf, const FpBin& K, float uf, float vf, int c, int s, BinMagic m) {
  const float kc = fminf(fmaxf(kf, 0.5f), K.khi);
  const float y1 = __fadd_rn(__fadd_rn(kc, K.dlo), 12582912.0f);
  const float y2 = __fadd_rn(__fadd_rn(kc, K.dhi), 12582912.0f);
  int r = __float_as_int(y1) - 0x4B400000;
  if (__float_as_int(y1) != __float_as_int(y2)) {
    const int u = __float2int_rn(uf), v = __float2int_rn(vf);
    r = rho_bin32(u * c + (v * s + (int)kH), m);
  }
  return r;
}

__device__ __forceinline__ void vote32_fp(const Plan& pl, const VoteLane& L, const int2* hb, int nv) {
  if (!L.on) return;
  const BinMagic m = pl.magic;
  const FpBin K{pl.fp_khi, pl.fp_dlo, pl.fp_dhi};
  const float c0 = pl.fp_c0;
  const int cj = L.cj, sj = L.sj;
  const float A = __fmul_rn((float)cj, pl.fp_scale), B = __fmul_rn((float)sj, pl.fp_scale);
  if (L.halo) {
    const int lane = threadIdx.x & 31;
    for (int i = lane & 15; i < nv; i += 16) {
      const float2 h = reinterpret_cast<const float2*>(hb)[i];
      vote_halo(L.col2, bin_fp(__fmaf_rn(h.x, A, __fmaf_rn(h.y, B, c0)), K, h.x, h.y, cj, sj, m));
    }
    return;
  }
  const float4* hb4 = reinterpret_cast<const float4*>(hb);
  const int np = nv >> 1, P = L.P;
#pragma unroll 4
  for (int q = L.p; q < np; q += P) {
    const float4 h = hb4[q];
    vote_cell(L.col1, bin_fp(__fmaf_rn(h.x, A, __fmaf_rn(h.y, B, c0)), K, h.x, h.y, cj, sj, m));
    vote_cell(L.col1, bin_fp(__fmaf_rn(h.z, A, __fmaf_rn(h.w, B, c0)), K, h.z, h.w, cj, sj, m));
  }
  if ((nv & 1) && L.p == np % P) {
    const float2 h = reinterpret_cast<const float2*>(hb)[nv - 1];
    vote_cell(L.col1, bin_fp(__fmaf_rn(h.x, A, __fmaf_rn(h.y, B, c0)), K, h.x, h.y, cj, sj, m));
  }
}

__device__ __forceinline__ void vote64(const Plan& pl, const VoteLane& L, const longlong2* hw, int nv) {
  if (!L.on) return;
  const BinMagic m = pl.magic;
  const long long cj = L.cj, sj = L.sj;
  if (L.halo) {
    const int lane = threadIdx.x & 31;
    for (int i = lane & 15; i < nv; i += 16) {
      const longlong2 h = hw[i];
      vote_halo(L.col2, rho_bin64(h.x * cj + h.y * sj + kH, m));
    }
    return;
  }
  for (int q = L.p; q < nv; q += L.P) {
    const longlong2 h = hw[q];
    const long long vs = h.y * sj + kH, uc = h.x * cj;
    vote_cell(L.col1, rho_bin64(vs + uc, m));
  }
}

// ---- mirror-pair word layout (even column counts; odd ones where it fits the tiles and threads of their columns) ----
// Word lane w in [0, (N_theta+1)/2) holds column w in its low half and column N_theta-1-w (its
// mirror) in its high half, one word per physical row p = k + 1. With an odd N_theta the last word's column is
// its own mirror (c = 0): the high half then repeats the low one. It serves as the neighbour of the column after it;
// it has no place in the bitmaps, and the fingerprint and the finder's passes leave it out. Rows p = 0 and p = N_rho + 1
// are guard rows: the fast path only takes hits whose rho stays within half a bin of the range,
// so its unclamped bins fall in [-1, N_rho]; the guard rows are folded into rows 0 and
// N_rho - 1 after the vote, which is what clamping would have done.

__device__ __forceinline__ int mp_word(int w, int p, int rows_phys) {
  return (((w >> 5) * rows_phys + p) << 5) + (w & 31);
}

// Cell (c, k) of a mirror-pair tile of wt columns in Wd = (wt + 1) / 2 words; tile-local column c < Wd is word c's low
// half, c >= Wd word wt - 1 - c's high half.
__device__ __forceinline__ int mp_get(const uint32_t* acc, int c, int k, int Wd, int wt, const Plan& pl) {
  const bool hi = c >= Wd;
  const uint32_t x = acc[mp_word(hi ? wt - 1 - c : c, k + 1, pl.rows_phys)];
  return hi ? (int)(x >> 16) : (int)(x & 0xffffu);
}

// Cells of the CTA's accumulator for the iterative finder (one tile): read, and suppress by a
// 16-bit store of zero into the cell's half of its word, which leaves the other half of the word alone.
template <bool MP>
struct FusedCells {
  uint32_t* acc;
  int Wd, NT, nrp, rp;  // words, columns, padded rows (columns), rows with guards (mirror pairs)
  __device__ int get(int j, int k) const {
    if (MP) {
      const bool hi = j >= Wd;
      const uint32_t x = acc[mp_word(hi ? NT - 1 - j : j, k + 1, rp)];
      return hi ? (int)(x >> 16) : (int)(x & 0xffffu);
    }
    return acc_get(acc, j, k, nrp);
  }
  __device__ void clear(int j, int k) {
    if (MP) {
      const bool hi = j >= Wd;
      reinterpret_cast<uint16_t*>(acc)[2 * mp_word(hi ? NT - 1 - j : j, k + 1, rp) + (hi ? 1 : 0)] = 0;
    } else {
      reinterpret_cast<uint16_t*>(acc)[2 * acc_index(j, k, nrp) + (k & 1)] = 0;
    }
  }
};

// The iterative finder's kept set on a whole mirror-pair accumulator: dropped candidates' cells are set to
// zero beside their bits, so a look is a plain maximum over the window's votes (cells that are no candidates
// rank below every candidate). A column of the window a lane, its rows read independently: one
// thread took ~9 k cycles a look at R = 3, its bits and votes one after the other; a group of 8 lanes that
// tests the bits 3.1 k a round of 128 looks. Batched events at 256 x 256 (half the maximum, R = 3; 2,300
// candidates, 490 local maxima, 250 kept), kept set in all, local maxima included: 57 k cycles with rounds on two
// state bits a cell where a thread scans a window at every visit, 64 k with blockers and a thread a look, 46 k
// with groups and bits, 38 k so.
// Ids: j << 16 | k; bitmap word of cell (j, k): j stride + (k >> 5).
struct WholeWindow {
  static constexpr int kVotes = 17;  // at most 227 KB / 2 cells: 17 bits, and 15 of votes
  uint32_t* acc;
  int half, rp, NT, NR, R, stride;
  uint32_t *alive, *surv;
  __device__ int radius() const { return R; }
  __device__ int lg() const { return 2 * R + 1 <= 8 ? 3 : 2 * R + 1 <= 16 ? 4 : 5; }
  __device__ int words() const { return NT * stride; }
  __device__ uint32_t id(int i, int b) const {
    const int j = i / stride;
    return ((uint32_t)j << 16) | (uint32_t)(32 * (i - j * stride) + b);
  }
  __device__ uint32_t bit(uint32_t jk, int& w) const {
    w = (int)(jk >> 16) * stride + (int)((jk & 0xffffu) >> 5);
    return 1u << (jk & 31u);
  }
  template <class Word>
  __device__ void list_bits(Word&& word, uint32_t* list, int room, int* n) const {
    list_cells(NT, NR, stride, word, list, room, n);
  }
  __device__ uint32_t key(uint32_t jk) const {
    const int j = (int)(jk >> 16), k = (int)(jk & 0xffffu);
    return ((uint32_t)*cell(j, k) << kVotes) | (uint32_t)((1 << kVotes) - 1 - (j * NR + k));
  }
  __device__ void cell(uint32_t key, int& j, int& k) const {
    const int c = (1 << kVotes) - 1 - (int)(key & ((1u << kVotes) - 1u));
    j = c / NR;
    k = c - j * NR;
  }
  __device__ uint16_t* cell(int j, int k) const {
    const bool hi = j >= half;
    return reinterpret_cast<uint16_t*>(acc + mp_word(hi ? NT - 1 - j : j, k + 1, rp)) + (hi ? 1 : 0);
  }
  __device__ bool live(uint32_t jk) const { return *cell((int)(jk >> 16), (int)(jk & 0xffffu)) != 0; }
  // Rank within a window in 32 bits: votes (15 bits), then the place of the column in raster order (9 bits; a
  // column from across the wrap, where rho is mirrored, comes after the others at the low end, before them at
  // the high end), then the row (8 bits, from the column's first row).
  __device__ bool look(uint32_t jk, bool on, bool& win, uint32_t& at) const {
    const int lane = threadIdx.x & 31, G = 1 << lg(), sub = lane & (G - 1), W = 2 * R + 1;
    const int j = (int)(jk >> 16), k = (int)(jk & 0xffffu), c0 = max(0, k - R), c1 = min(NR - 1, k + R), n = c1 - c0 + 1;
    uint32_t m = 0u;
    if (on) {
#pragma unroll 1
      for (int a = sub - R; a <= R; a += G) {
        int jj = j + a, r0 = c0, place = 511 - (a + R + W);
        if ((unsigned)jj >= (unsigned)NT) {
          place -= jj < 0 ? W : -W;
          jj += jj < 0 ? NT : -NT;
          r0 = NR - 1 - c1;
        }
        const uint16_t* col = cell(jj, r0);
        uint32_t t = 0u;  // votes << 8 | 255 - row from the first
        if (n == 7) {
#pragma unroll
          for (int i = 0; i < 7; ++i) t = max(t, (uint32_t)col[i << 6] * 256u + (uint32_t)(255 - i));
        } else {
#pragma unroll 4
          for (int i = 0; i < n; ++i) t = max(t, (uint32_t)col[i << 6] * 256u + (uint32_t)(255 - i));
        }
        const uint32_t x = ((t & ~255u) << 9) | (uint32_t)(place << 8) | (t & 255u);
        if (x > m) {
          m = x;
          at = ((uint32_t)jj << 16) | (uint32_t)(r0 + 255 - (int)(t & 255u));
        }
      }
    }
    uint32_t top = m;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) top = max(top, __shfl_xor_sync(kFull, top, o));
    if (G > 8)
      for (int o = 8; o < G; o <<= 1) top = max(top, __shfl_xor_sync(kFull, top, o));
    win = on && m == top;  // ranks are distinct: one lane
    const unsigned self = __ballot_sync(kFull, win && at == jk);
    if (!((self >> (lane & ~(G - 1))) & (0xffffffffu >> (32 - G)))) return false;
#pragma unroll 1
    for (int a = sub - R; a <= R; a += G) {
      int jj = j + a, r0 = c0;
      if ((unsigned)jj >= (unsigned)NT) {
        jj += jj < 0 ? NT : -NT;
        r0 = NR - 1 - c1;
      }
      const int r1 = r0 + n - 1, own = a == 0 ? k : -1;
      uint16_t* col = cell(jj, r0);
#pragma unroll 4
      for (int i = 0; i < n; ++i)
        if (r0 + i != own) col[i << 6] = 0;
#pragma unroll 1
      for (int w = r0 >> 5; w <= (r1 >> 5); ++w) {
        uint32_t x = 0xffffffffu;
        if (w == (r0 >> 5)) x &= 0xffffffffu << (r0 & 31);
        if (w == (r1 >> 5)) x &= 0xffffffffu >> (31 - (r1 & 31));
        if (a == 0 && w == (k >> 5)) x &= ~(1u << (k & 31));
        if (alive[jj * stride + w] & x) atomicAnd(&alive[jj * stride + w], ~x);
      }
    }
    return true;
  }
};

// One pass a peak over a whole accumulator in columns. A function of its own: inlined, a pass took 3.6 k cycles, 3.3 k so
// (459 x 206, 374 peaks; 131 events 1,566 -> 1,462 us).
__device__ __noinline__ int extract_passes_columns(const Plan& pl, hough_peak* dst, int* s) {
  extern __shared__ __align__(16) unsigned char smem[];
  FusedCells<false> cells{reinterpret_cast<uint32_t*>(smem + pl.off_acc), 0, pl.n_theta, pl.nrho_pad, 0};
  return extract_iterative_passes(cells, pl.n_theta, pl.n_rho, kIterSliceRows, pl.threshold, pl.rel_num, pl.rel_den, pl.nms_radius,
                                  pl.max_peaks, reinterpret_cast<uint32_t*>(smem + pl.off_pbits), dst, s);
}

// Maximum of a mirror-pair accumulator's cells (its words lie in one run; guard rows and lanes past the
// last word are zero), to every thread; *s_max must be 0 beforehand.
__device__ int acc_max_mp(const Plan& pl, const uint32_t* acc, int half, int* s_max) {
  const uint4* x4 = reinterpret_cast<const uint4*>(acc);
  const int n4 = ((half + 31) >> 5) * pl.rows_phys * 8;
  uint32_t m = 0u;
  for (int i = threadIdx.x; i < n4; i += blockDim.x) {
    const uint4 x = x4[i];
    m = vmax2(m, vmax2(vmax2(x.x, x.y), vmax2(x.z, x.w)));
  }
  const int top = __reduce_max_sync(kFull, (int)max(m & 0xffffu, m >> 16));
  if ((threadIdx.x & 31) == 0 && top) atomicMax(s_max, top);
  __syncthreads();
  return *s_max;
}

// Shared address of the vote whose float row estimate, shifted by 1 + 2^b + e (2^b > N_rho + 1,
// e = W/2 units of 2^-F, W a power of two), is kfp. In [2^b, 2^(b+1)) a float's low F = 23 - b
// bits are the fraction and the bits above them (127 + b) 2^b + integer part, so
// base2 + ((y >> F) << 7) with base2 = base - ((127 + b) 2^b << 7) is the row's word directly.
// The estimate is within N_rho 2^-21 + 2^-(F+1) <= e of the exact value; when the shifted
// fraction is below W (its bits above log2 W all zero: the exact value within e of an integer)
// the exact integer path (clamped) decides, otherwise the shift by e does not move the integer part.
__device__ __forceinline__ uint32_t mp_addr(float kfp, const Plan& pl, uint32_t base, uint32_t base2, float uf,
                                            float vf, int c, int s) {
  const uint32_t y = (uint32_t)__float_as_int(kfp);
  if ((y & (uint32_t)pl.mp_amask) == 0u) {
    const int u = __float2int_rn(uf), v = __float2int_rn(vf);
    return base + ((uint32_t)(rho_bin32(u * c + (v * s + (int)kH), pl.magic) + 1) << 7);
  }
  return base2 + ((y >> pl.mp_F) << 7);
}

__device__ __forceinline__ void red_u32(uint32_t addr, uint32_t inc) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(inc));
}

// d = a * b + c on pairs of floats (packed f32x2, each lane rounded as one fused multiply-add).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// Hit i of the mirror-pair staging: pairs of hits (u0, u1, v0, v1).
__device__ __forceinline__ float2 staged_hit(const float* f, int i) {
  const float* q = f + 4 * (i >> 1) + (i & 1);
  return make_float2(q[0], q[2]);
}

// d = a + b on pairs of floats, rounded down.
__device__ __forceinline__ float2 add2_rm(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rm.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// Adding 1.5 2^23 rounded down leaves the integer part of a row estimate in the low bits of the
// sum's pattern: row = pattern - mp_zoff.
constexpr float kMagic = 12582912.0f;

// Votes of a staged pair of hits (u0, u1, v0, v1) in one word whose estimates lay in the ambiguous
// window: where the exact row differs from the estimated one that was voted, minus one there and
// plus one at the exact row. (The packed sums are modulo 2^32, so the order of the adds is free.)
__device__ __forceinline__ void pair_fix(const Plan& pl, float4 h, int cj, int sj, uint32_t base) {
  const float A = __fmul_rn((float)cj, pl.fp_scale), B = __fmul_rn((float)sj, pl.fp_scale);
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    const float u = i & 2 ? h.y : h.x, v = i & 2 ? h.w : h.z;
    const float kf = __fmaf_rn(i & 1 ? -u : u, A, __fmaf_rn(v, B, pl.mp_c0));
    const uint32_t y = __float_as_uint(kf);
    if ((y & (uint32_t)pl.mp_amask) != 0u) continue;
    const uint32_t r0 = (y >> pl.mp_F) & (uint32_t)pl.mp_rmask;
    const int ui = __float2int_rn(u), vi = __float2int_rn(v);
    const uint32_t r1 = (uint32_t)rho_bin32(ui * (i & 1 ? -cj : cj) + (vi * sj + (int)kH), pl.magic) + 1u;
    if (r0 != r1) {
      const uint32_t inc = i & 1 ? 0x10000u : 1u;
      red_u32(base + (r0 << 7), 0u - inc);
      red_u32(base + (r1 << 7), inc);
    }
  }
}

// Shared list of vote steps with an estimate in the ambiguous window.
struct AmbList {
  uint32_t* e;  // first pair << 10 | first word
  int* n;       // counts on past cap
  int cap;
};

// Constants of one lane's vote loop (offsets in bytes into the CTA's dynamic shared memory).
template <int W>
struct VoteArgs {
  float A[W], B[W];   // its words' coefficients
  uint32_t bs[W];     // shared address of its words' row "pattern 0"
  float c0;
  uint32_t am;
  int p, P, np;       // pairs p, p + P, ... below np
  int hits;           // staged pairs
  uint32_t tag;       // first word
  int list, n, cap;   // ambiguous steps, their count, room
};

// The vote of a lane's share of the hit pairs into its W words. The loop runs straight through: every
// estimate votes at once, and a step of U pairs x W words with an estimate in the ambiguous window (2e-4
// of the votes at 256 rows) is listed for vote_fix, so that a warp does not run the exact path's ~100
// instructions for one lane. The loop is bound by issue: a vote's estimate, floor, address, add and test
// take 5.5 slots (a packed f32x2 operation takes two), and by the unit that takes the atomics (one warp a
// cycle) and the broadcast loads (an LDS.128 two cycles), which is why a lane's two words share their loads.
// Alone, 2,022 hits at 256 x 256, 1,024 threads: 33.5 k cycles with one word and a branch a pair; straight through
// 28.3 k with one word, 26.8 k with two, 27.6 k with four; 19.4 k with no test, 16.2 k for the atomics alone. A
// test on the distance from the rounded estimate (two more packed operations instead of the masks) took
// 30.4 k. A function of its own, with its arguments in registers: inlined, its registers and schedule
// changed with unrelated code around it (33 k to 40 k cycles an event).
template <int W, int U>
__device__ __noinline__ void vote_loop(const VoteArgs<W> v) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2 AA[W], BB[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    AA[w] = make_float2(v.A[w], v.A[w]);
    BB[w] = make_float2(v.B[w], v.B[w]);
  }
  const float2 CC = make_float2(v.c0, v.c0), MM = make_float2(kMagic, kMagic);
  const uint32_t am = v.am;
  const float4* hb4 = reinterpret_cast<const float4*>(smem + v.hits);
  const int np = v.np, P = v.P;
  auto vote_pair = [&](float4 h) {
    const float2 uu = make_float2(h.x, h.y), nu = make_float2(-h.x, -h.y), vv = make_float2(h.z, h.w);
    bool ok = true;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float2 V = fma2(vv, BB[w], CC);
      const float2 k0 = fma2(uu, AA[w], V), k1 = fma2(nu, AA[w], V);
      const float2 z0 = add2_rm(k0, MM), z1 = add2_rm(k1, MM);
      red_u32(v.bs[w] + (__float_as_uint(z0.x) << 7), 1u);
      red_u32(v.bs[w] + (__float_as_uint(z1.x) << 7), 0x10000u);
      red_u32(v.bs[w] + (__float_as_uint(z0.y) << 7), 1u);
      red_u32(v.bs[w] + (__float_as_uint(z1.y) << 7), 0x10000u);
      ok = ok & ((__float_as_uint(k0.x) & am) != 0u) & ((__float_as_uint(k1.x) & am) != 0u) &
           ((__float_as_uint(k0.y) & am) != 0u) & ((__float_as_uint(k1.y) & am) != 0u);
    }
    return ok;
  };
  auto list = [&](int q) {
    const int at = atomicAdd(reinterpret_cast<int*>(smem + v.n), 1);
    if (at < v.cap) reinterpret_cast<uint32_t*>(smem + v.list)[at] = ((uint32_t)q << 10) | v.tag;
  };
  int q = v.p;
#pragma unroll 1
  for (; q + (U - 1) * P < np; q += U * P) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < U; ++i) ok = vote_pair(hb4[q + i * P]) & ok;
    if (!ok) list(q);
  }
#pragma unroll 1
  for (; q < np; q += P)
    if (!vote_pair(hb4[q])) list(q);
}

// The last hit of an odd count, a word a thread of the first warp of each word group.
__device__ __forceinline__ void vote_last(const Plan& pl, const int16_t* tc, const int16_t* ts, uint32_t acc_s, int aw,
                                          int x, float2 h) {
  const int cj = tc[aw + x], sj = ts[aw + x];
  const float A = __fmul_rn((float)cj, pl.fp_scale), v0 = __fmaf_rn(h.y, __fmul_rn((float)sj, pl.fp_scale), pl.mp_c0);
  const uint32_t base = acc_s + (uint32_t)mp_word(x, 0, pl.rows_phys) * 4u, base2 = base - (uint32_t)pl.mp_k7;
  red_u32(mp_addr(__fmaf_rn(h.x, A, v0), pl, base, base2, h.x, h.y, cj, sj), 1u);
  red_u32(mp_addr(__fmaf_rn(-h.x, A, v0), pl, base, base2, h.x, h.y, -cj, sj), 0x10000u);
}

// All of a chunk's votes into a mirror-pair tile of Wd words (every thread calls it; the votes are
// complete after the next barrier).
template <int W, int U>
__device__ __forceinline__ void vote_words(const Plan& pl, unsigned char* smem, const int16_t* tc, const int16_t* ts,
                                           uint32_t acc_s, int aw, int Wd, int nv, const AmbList& L) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, G = pl.groups >> 1, P2 = pl.vote_p;
  const int P = P2 * W, w0 = (warp / P) * (32 * W) + lane, np = nv >> 1;
  const float4* hb4 = reinterpret_cast<const float4*>(smem + pl.off_hits);
  if (warp < G * P2 && w0 < Wd) {
    VoteArgs<W> v;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int x = w0 + 32 * w;
      v.A[w] = __fmul_rn((float)tc[aw + x], pl.fp_scale);
      v.B[w] = __fmul_rn((float)ts[aw + x], pl.fp_scale);
      v.bs[w] = acc_s + (uint32_t)mp_word(x, 0, pl.rows_phys) * 4u - ((uint32_t)pl.mp_zoff << 7);
    }
    v.c0 = pl.mp_c0;
    v.am = (uint32_t)pl.mp_amask;
    v.p = warp % P;
    v.P = P;
    v.np = np;
    v.hits = pl.off_hits;
    v.tag = (uint32_t)w0;
    v.list = (int)(reinterpret_cast<unsigned char*>(L.e) - smem);
    v.n = (int)((uint32_t)__cvta_generic_to_shared(L.n) - (uint32_t)__cvta_generic_to_shared(smem));
    v.cap = L.cap;
    vote_loop<W, U>(v);
    if ((nv & 1) && warp % P == np % P)
      for (int w = 0; w < W; ++w)
        vote_last(pl, tc, ts, acc_s, aw, w0 + 32 * w, staged_hit(reinterpret_cast<const float*>(hb4), nv - 1));
  }
  __syncthreads();
  // the listed steps' exact rows, a thread a (pair, word); with more steps than the list holds, every one's
  const int nl = *L.n;
  if (nl <= L.cap) {
    for (int it = threadIdx.x; it < nl * (W * U); it += blockDim.x) {
      const uint32_t e = L.e[it / (W * U)];
      const int q = (int)(e >> 10) + (it % U) * P, x = (int)(e & 1023u) + 32 * (it / U % W);
      // a single step at the end of a lane's share stands for one pair
      if (it % U == 0 || (int)(e >> 10) + (U - 1) * P < np)
        pair_fix(pl, hb4[q], tc[aw + x], ts[aw + x], acc_s + (uint32_t)mp_word(x, 0, pl.rows_phys) * 4u);
    }
  } else {
    for (long long it = threadIdx.x; it < (long long)np * Wd; it += blockDim.x) {
      const int q = (int)(it / Wd), x = (int)(it - (long long)q * Wd);
      pair_fix(pl, hb4[q], tc[aw + x], ts[aw + x], acc_s + (uint32_t)mp_word(x, 0, pl.rows_phys) * 4u);
    }
  }
}

// Two words a lane only where every lane has both.
__device__ __forceinline__ void vote_mp32(const Plan& pl, unsigned char* smem, const int16_t* tc, const int16_t* ts,
                                          uint32_t acc_s, int aw, int Wd, int nv, const AmbList& L) {
  if ((Wd & 63) == 0) vote_words<2, 2>(pl, smem, tc, ts, acc_s, aw, Wd, nv, L);
  else vote_words<1, 4>(pl, smem, tc, ts, acc_s, aw, Wd, nv, L);
}

// Halo words of a mirror-pair tile: the words before and after its own (none at the theta wrap or at the
// middle word), each a contiguous column of 4-byte rows (guard rows folded like the accumulator's). Every
// thread of the CTA takes hits, even threads for the word before, odd ones for the word after: a warp
// of its own finished last (the vote of stress events at 512 x 512 took 313 k cycles with it, 207 k without
// any halo).
struct HaloLane {
  bool on;
  int c, s;
  uint32_t col;  // shared address of row 0
};

__device__ __forceinline__ HaloLane halo_lane(const Plan& pl, const int16_t* tc, const int16_t* ts,
                                              const uint32_t* halo, int aw, int Wd) {
  const int side = threadIdx.x & 1, w = side ? aw + Wd : aw - 1;
  HaloLane h;
  h.on = side ? w < ((pl.n_theta + 1) >> 1) : w >= 0;
  h.c = h.on ? tc[w] : 0;
  h.s = h.on ? ts[w] : 0;
  h.col = (uint32_t)__cvta_generic_to_shared(halo) + (uint32_t)(side * pl.rows_phys) * 4u;
  return h;
}

__device__ __forceinline__ void halo_mp32(const Plan& pl, const HaloLane& H, const int2* hb, int nv) {
  if (!H.on) return;
  const float A = __fmul_rn((float)H.c, pl.fp_scale), B = __fmul_rn((float)H.s, pl.fp_scale);
  const uint32_t am = (uint32_t)pl.mp_amask, base2 = H.col - ((uint32_t)pl.mp_k7 >> 5);
  const int F = pl.mp_F;
#pragma unroll 2
  for (int i = threadIdx.x >> 1; i < nv; i += blockDim.x >> 1) {
    const float2 h = staged_hit(reinterpret_cast<const float*>(hb), i);
    const float v0 = __fmaf_rn(h.y, B, pl.mp_c0);
    const uint32_t y0 = __float_as_uint(__fmaf_rn(h.x, A, v0)), y1 = __float_as_uint(__fmaf_rn(-h.x, A, v0));
    if (((y0 & am) != 0u) & ((y1 & am) != 0u)) {
      red_u32(base2 + ((y0 >> F) << 2), 1u);
      red_u32(base2 + ((y1 >> F) << 2), 0x10000u);
    } else {
      const int uc = __float2int_rn(h.x) * H.c, vs = __float2int_rn(h.y) * H.s + (int)kH;
      red_u32(H.col + ((uint32_t)(rho_bin32(vs + uc, pl.magic) + 1) << 2), 1u);
      red_u32(H.col + ((uint32_t)(rho_bin32(vs - uc, pl.magic) + 1) << 2), 0x10000u);
    }
  }
}

__device__ __forceinline__ void halo_mp64(const Plan& pl, const HaloLane& H, const longlong2* hw, int nv) {
  if (!H.on) return;
  for (int i = threadIdx.x >> 1; i < nv; i += blockDim.x >> 1) {
    const long long vs = hw[i].y * H.s + kH, uc = hw[i].x * H.c;
    red_u32(H.col + ((uint32_t)(rho_bin64(vs + uc, pl.magic) + 1) << 2), 1u);
    red_u32(H.col + ((uint32_t)(rho_bin64(vs - uc, pl.magic) + 1) << 2), 0x10000u);
  }
}

__device__ __forceinline__ void vote_mp64(const Plan& pl, const VoteLane& L, const longlong2* hw, int nv) {
  const BinMagic m = pl.magic;
  const long long cj = L.cj, sj = L.sj;
  if (!L.on) return;
  for (int q = L.p; q < nv; q += L.P) {
    const longlong2 h = hw[q];
    const long long vs = h.y * sj + kH, uc = h.x * cj;
    red_u32(L.col1 + ((uint32_t)(rho_bin64(vs + uc, m) + 1) << 7), 1u);
    red_u32(L.col1 + ((uint32_t)(rho_bin64(vs - uc, m) + 1) << 7), 0x10000u);
  }
}

// Guard rows into the edge rows (both halves at once: a column holds at most 32767 votes,
// so the packed add never carries across halves).
__device__ void mp_fold(const Plan& pl, uint32_t* acc, int n_words, uint32_t* halo) {
  const int rp = pl.rows_phys, NR = pl.n_rho;
  for (int w = threadIdx.x; w < n_words; w += blockDim.x) {
    uint32_t* col = acc + mp_word(w, 0, rp);
    col[32] += col[0];
    col[NR << 5] += col[(NR + 1) << 5];
    col[0] = 0u;  // zero guard rows now read as "no neighbour" in the scan
    col[(NR + 1) << 5] = 0u;
  }
  if (halo && threadIdx.x < 2) {  // the tile's two halo words (contiguous rows)
    uint32_t* col = halo + threadIdx.x * rp;
    col[1] += col[0];
    col[NR] += col[NR + 1];
    col[0] = 0u;
    col[NR + 1] = 0u;
  }
}

// Where the word before (side 0) or after (side 1) a 32-word group of the tile lies: its row -1 as a word
// offset into the CTA's shared memory, the words from row to row, and whether its halves are swapped.
struct EdgeWord {
  int at;
  short step, swap;
};

// Edge words of the tile's groups (the CTA's last 2 G threads). Before word 0 lies the theta wrap (word 0, rows mirrored:
// from the top down, halves swapped), after the middle word itself (halves swapped; with an odd N_theta the word
// before it, which holds the column after the middle one), else the halo
// (two contiguous columns of rows_phys words, of the words aw - 1 and aw + half; a tile owns words
// [aw, aw + half), columns aw.. and their mirrors); without a halo, nothing (guard row 0, zero, throughout).
__device__ __forceinline__ void edge_words(const Plan& pl, int aw, int half, bool halo, EdgeWord* ew) {
  const int G = (half + 31) >> 5, i = (int)(blockDim.x - 1 - threadIdx.x), rp = pl.rows_phys, acc0 = pl.off_acc >> 2, halo0 = pl.off_halo >> 2;
  if (i >= 2 * G) return;
  const int w = i & 1 ? min((i >> 1) * 32 + 32, half) : (i >> 1) * 32 - 1;
  EdgeWord e{acc0, 32, 0};
  if (w >= 0 && w < half) {
    e.at += mp_word(w, 0, rp);
  } else if (w < 0 ? aw == 0 : aw + half == ((pl.n_theta + 1) >> 1)) {
    const int at = half - 1 - (pl.n_theta & 1);
    e.at += w < 0 ? mp_word(0, pl.n_rho + 1, rp) : mp_word(at, 0, rp);
    e.step = w < 0 ? -32 : 32;
    e.swap = 1;
    if (w > 0 && at < 0) {  // the middle word alone: the one before it is the halo's
      e.at = halo ? halo0 : acc0;
      e.step = halo ? 1 : 0;
    }
  } else if (halo) {
    e.at = halo0 + (w < 0 ? 0 : rp);
    e.step = 1;
  } else {
    e.step = 0;
  }
  ew[i] = e;
}

constexpr int kFoundGroups = 64;
struct Found {
  uint32_t* key;
  int cap;
  int* n;
};
// tile-local column, row, whether it is a 3x3 local maximum
__device__ __forceinline__ uint32_t found_key(int c, int k, uint32_t lm) { return (uint32_t)(c << 11 | k << 1) | lm; }

// Pass 2 of the peak scan (scan_mp) over nl listed groups; KEYS: with keys.
template <bool CAND, bool KEYS>
__device__ __forceinline__ void scan_groups(const Plan& pl, const uint32_t* sw, const uint32_t* acc, uint32_t TT, int aw, int half,
                                            const EdgeWord* ew, uint32_t* pbits, uint32_t* cand, const uint16_t* list, int nl,
                                            const Found& found) {
  const int NR = pl.n_rho, rp = pl.rows_phys;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  // Raster order runs over theta, then rho: the row above and the preceding column are
  // "before" a cell (strictly below it at a peak), the rest "after" (at most equal). The
  // preceding column of the low half (column aw+w) is lane w-1's low half (the wrapped
  // column N-1 at word 0: after, not before); of the high half (column N-1-aw-w) lane w+1's
  // high half; lane w-1's high half follows it (except at word 0: the wrapped column 0).
  // Strictness becomes +1 on that neighbour, so a cell is a peak iff C >= max(U + 1, D,
  // VU + addU, VD + 0x10000, T) per half.
  const bool mid = 2 * (aw + half) - 1 == pl.n_theta;  // the last word's column is the middle one, which has one place
  const int last = 2 * half - 1 - mid;                  // the tile's last column
  for (int it = warp; it < nl; it += nwarps) {
    const int en = list[it], g = en >> 8, k = (en & 255) << 2, n = min(32, half - 32 * g), w = 32 * g + lane;
    const uint32_t addU = (w != 0 || aw != 0) ? 1u : 0x10000u;
    const uint32_t* ptr = acc + mp_word(w, k, rp);  // row k - 1 (lanes past the last word: zero words)
    const uint32_t R[6] = {ptr[0], ptr[32], ptr[64], ptr[96], ptr[128], ptr[160]};
    uint32_t EV[4] = {0u, 0u, 0u, 0u};  // 3-row maxima of the word beyond the group
    if (lane == 0 || lane == min(n, 31)) {  // (n == 1: lanes 0 and 1)
      const EdgeWord ed = ew[2 * g + (lane != 0)];
      const int st = ed.step;
      const uint32_t* q = sw + ed.at + st * k;
      uint32_t e[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) e[i] = q[st * i];
#pragma unroll
      for (int i = 0; i < 4; ++i) EV[i] = __byte_perm(vmax2(vmax2(e[i], e[i + 1]), e[i + 2]), 0u, ed.swap ? 0x1032u : 0x3210u);
    }
    uint32_t fl = 0u, cf = 0u;  // flags, the low column's in the low half, the newest row at bit 15 of each half
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (CAND) cf = (cf >> 1) | ((R[i + 1] - TT + 0x80008000u) & 0x80008000u);
      uint32_t VM = vmax2(vmax2(R[i], R[i + 1]), R[i + 2]);
      if (n < 32 && lane == n) VM = EV[i];
      uint32_t VU = __shfl_up_sync(kFull, VM, 1), VD = __shfl_down_sync(kFull, VM, 1);
      if (lane == 0) VU = EV[i];
      if (lane == 31 && n == 32) VD = EV[i];
      const uint32_t X = vmax2(vmax2(vmax2(R[i] + 0x00010001u, R[i + 2]), vmax2(VU + addU, VD + 0x10000u)), TT);
      fl = (fl >> 1) | ((R[i + 1] - X + 0x80008000u) & 0x80008000u);
    }
    if (NR - k < 4) {  // rows past the last one
      const uint32_t valid = ((1u << (NR - k)) - 1u) * 0x10001000u;
      fl &= valid;
      cf &= valid;
    }
    if (mid && w == last - w) fl &= 0xffffu, cf &= 0xffffu;
    if (CAND && lane < n) {
      const uint32_t lo = (cf >> 12) & 15u, hi = cf >> 28;
      if (lo) atomicOr(&cand[w * pl.nrb_p + (k >> 5)], lo << (k & 31));
      if (hi) atomicOr(&cand[(last - w) * pl.nrb_p + (k >> 5)], hi << (k & 31));
    }
    if (lane < n) {
      const uint32_t lo = (fl >> 12) & 15u, hi = fl >> 28;
      if (lo) atomicOr(&pbits[w * pl.nrb_p + (k >> 5)], lo << (k & 31));
      if (hi) atomicOr(&pbits[(last - w) * pl.nrb_p + (k >> 5)], hi << (k & 31));
    }
    if (KEYS && lane < n) {
      const uint32_t x = CAND ? cf : fl;  // bits 0-3 the low column's rows, 4-7 the high one's
      uint32_t bits = ((x >> 12) & 15u) | ((x >> 24) & 0xf0u);
      const uint32_t lms = CAND ? ((fl >> 12) & 15u) | ((fl >> 24) & 0xf0u) : 0u;
      if (bits) {
        int at = atomicAdd(found.n, __popc(bits));
        for (; bits && at < found.cap; bits &= bits - 1u, ++at) {
          const int b = __ffs(bits) - 1;
          found.key[at] = found_key(b < 4 ? w : last - w, k + (b & 3), (lms >> b) & 1u);
        }
      }
    }
  }
}

// Peak scan of the mirror-pair layout, both columns of a word at once, in two passes. (1) Row groups (32
// words x 4 rows: one 16-byte load a lane) in which some cell reaches the threshold are listed; about a
// third of them at 256 x 256 and T = 16, a few per cent at 1000 x 1000 and T = 12. (2) Warps take listed
// groups in turn, lane l word l, and set the flags of their peaks in the cleared bitmap.
// For word lane w, lane w-1 holds the left neighbour of column w and the right neighbour of column
// N-1-w; lane w+1 the other two; lane 0 and lane n (lane 31 with a full group of n = 32) also read the
// words beyond the group (edge_words).
// Both passes are bound by the integer ALU, which takes a warp instruction every two cycles of a scheduler (so
// 100 instructions of set-up in each of 32 warps are about 1.3 k cycles): the first takes 11 instructions a
// group, the second about 125. One pass in units of 30 words x 64 rows took 9.3 k cycles an event at 256 x 256
// (the central rows' candidates fell to a few warps) and 10.0 k a tile at 1000 x 1000; units of 8 rows
// 9.6 k and 7.5 k; this form 9.3 k and 3.6 k.
// list: room for (half + 31) / 32 * ((N_rho + 3) / 4) entries; *n_list zero beforehand.
// cand (nullable): a second cleared bitmap for all cells that reach the threshold (the iterative finder's
// candidates, of which the peaks are the 3x3 local maxima).
// found (tiles): with few listed groups, the peaks (CAND: the candidates) also as keys found_key in any order, counted in
// found.n (zero beforehand; past found.cap, or with more groups, the count is and the keys are not complete).
template <bool CAND>
__device__ void scan_mp(const Plan& pl, const unsigned char* smem, int thr, int aw, int half, const EdgeWord* ew,
                        uint32_t* pbits, uint32_t* cand, uint16_t* list, int* n_list, const Found& found) {
  const int NR = pl.n_rho, rp = pl.rows_phys;
  const uint32_t* const sw = reinterpret_cast<const uint32_t*>(smem);
  const uint32_t* const acc = sw + (pl.off_acc >> 2);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int G = (half + 31) >> 5, n4 = (NR + 3) >> 2;  // groups of words, of rows
  const uint32_t TT = (uint32_t)thr | ((uint32_t)thr << 16);
  // (1) A half reaches T iff bit 15 of C - T + 0x8000 is set (cells are at most 32767: no borrow across
  // the halves). Rows past the last one may be read (they only list a group in vain), inside the CTA's
  // shared memory.
  {
    const int per = (n4 - warp + nwarps - 1) / nwarps;  // the warp's row groups of each word group: warp, warp + nwarps, ...
    uint32_t hit = 0;                                   // bit c: its (r0 + c)-th of all
    int c = 0, r0 = 0;
    auto test = [&](const uint4& x) {
      const uint32_t top = vmax2(vmax2(x.x, x.y), vmax2(x.z, x.w));
      if (__any_sync(kFull, ((top - TT + 0x80008000u) & 0x80008000u) != 0u)) hit |= 1u << c;
      ++c;
    };
    auto flush = [&]() {
      if (hit) {
        int at = 0;
        if (lane == 0) at = atomicAdd(n_list, __popc(hit));
        at = __shfl_sync(kFull, at, 0) + __popc(hit & lanemask_lt());
        if ((hit >> lane) & 1u) {
          const int g = (r0 + lane) / per;
          list[at] = (uint16_t)(g << 8 | (warp + (r0 + lane - g * per) * nwarps));
        }
      }
      hit = 0;
      r0 += c;
      c = 0;
    };
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      const uint4* row = reinterpret_cast<const uint4*>(acc + mp_word(32 * g, 1, rp)) + lane + (warp << 5);
      int i = 0;
#pragma unroll 1
      for (; i + 3 < per; i += 4, row += nwarps << 7) {  // independent loads
        const uint4 x0 = row[0], x1 = row[nwarps << 5], x2 = row[nwarps << 6], x3 = row[3 * (nwarps << 5)];
        if (c > 28) flush();
        test(x0);
        test(x1);
        test(x2);
        test(x3);
      }
      if (i + 1 < per) {
        const uint4 x0 = row[0], x1 = row[nwarps << 5];
        if (c > 30) flush();
        test(x0);
        test(x1);
        i += 2;
        row += nwarps << 6;
      }
      if (i < per) {
        if (c > 31) flush();
        test(row[0]);
      }
    }
    flush();
  }
  __syncthreads();
  const int nl = *n_list;  // (2)
  if (found.cap > 0 && nl <= kFoundGroups) {
    scan_groups<CAND, true>(pl, sw, acc, TT, aw, half, ew, pbits, cand, list, nl, found);
  } else {
    if (threadIdx.x == 0) *found.n = INT_MAX;
    scan_groups<CAND, false>(pl, sw, acc, TT, aw, half, ew, pbits, cand, list, nl, found);
  }
}

// ---- peak scan ----

// Row range [k0, k1) of scan range r (word aligned in the packed scan).
// (The number of ranges is a power of two, 2^scan_shift.)
__device__ __forceinline__ void scan_rows(const Plan& pl, bool packed, int r, int& k0, int& k1) {
  const int sh = pl.scan_shift;
  if (packed) {
    const int W2 = pl.n_rho >> 1;
    k0 = 2 * ((W2 * r) >> sh);
    k1 = 2 * ((W2 * (r + 1)) >> sh);
  } else {
    k0 = (pl.n_rho * r) >> sh;
    k1 = (pl.n_rho * (r + 1)) >> sh;
  }
}

// Column source of one scan lane: the tile column itself, a halo column, or the tile's own
// far column mirrored (theta wrap of an untiled event), or nothing.
struct ScanSrc {
  int kind;  // 0 tile column, 1 left halo, 2 right halo, 3 none
  int col;   // tile column for kind 0
  bool mir;  // rows mirrored (k -> N_rho - 1 - k)
};

__device__ __forceinline__ ScanSrc scan_src(int c, int wt, int T, int j0, int NT) {
  ScanSrc s{0, c, false};
  if (c < 0) {
    if (T == 1) {
      s.col = wt - 1;
      s.mir = true;
    } else {
      s.kind = 1;
      s.mir = (j0 == 0);
    }
  } else if (c >= wt) {
    if (c == wt) {
      if (T == 1) {
        s.col = 0;
        s.mir = true;
      } else {
        s.kind = 2;
        s.mir = (j0 + wt == NT);
      }
    } else {
      s.kind = 3;
    }
  }
  return s;
}

// Packed int16 scan (N_rho even): two rows per step, max.u16x2 for the 3-row column maxima,
// one shuffle each way for the neighbour columns, exact tie test only for candidates.
// Missing neighbours (rho edges, no column) read as 0, which never blocks a cell >= T >= 1.
__device__ void scan_packed(const Plan& pl, const uint32_t* acc, const uint32_t* halo, uint32_t* pbits,
                            int wt, int T, int j0, bool do_cs, unsigned long long& csum) {
  const int NT = pl.n_theta, NR = pl.n_rho, W2 = NR >> 1, R = pl.scan_ranges;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nblk = (wt + 29) / 30;
  const uint32_t TT = (uint32_t)pl.threshold | ((uint32_t)pl.threshold << 16);
  for (int u = warp; u < nblk * R; u += nwarps) {
    const int b = u >> pl.scan_shift, r = u & (R - 1);
    int k0, k1;
    scan_rows(pl, true, r, k0, k1);
    const int w0 = k0 >> 1, w1 = k1 >> 1;
    const int c = b * 30 + lane - 1;
    const ScanSrc s = scan_src(c, wt, T, j0, NT);
    const uint32_t* col = nullptr;
    int stride = 32;
    if (s.kind == 0) {
      col = acc + ((s.col >> 5) * W2 << 5) + (s.col & 31);
    } else if (s.kind < 3) {
      col = halo + (s.kind - 1) * W2;
      stride = 1;
    }
    auto fetch = [&](int w) -> uint32_t {
      if (!col || w < 0 || w >= W2) return 0u;
      const uint32_t x = col[(s.mir ? W2 - 1 - w : w) * stride];
      return s.mir ? swap16(x) : x;
    };
    const bool tested = lane >= 1 && lane <= 30 && c >= 0 && c < wt;
    const bool lstrict = !(c == 0 && j0 == 0);
    const bool rstrict = (c == wt - 1) && (j0 + wt == NT);
    // Both rows of a word at once: a cell is a peak iff C >= max(U + 1, D, VL (+1 when the
    // left column precedes it), VR (+1 when the right column is the wrapped column 0), T)
    // per half; cells are at most 32767, so nothing carries across halves.
    const uint32_t addL = lstrict ? 0x00010001u : 0u, addR = rstrict ? 0x00010001u : 0u;
    uint32_t P = fetch(w0 - 1), C = fetch(w0);
    const unsigned long long cell0 = (unsigned long long)(j0 + c) * NR;
    for (int ws = w0; ws < w1;) {
      const int we = min(w1, (ws | 15) + 1);  // row pairs of one bitmap word
      uint32_t bits = 0;                      // peak flags, row k in bit k & 31
      for (int w = ws; w < we; ++w) {
        const uint32_t N = fetch(w + 1);
        // the neighbour test only where some tested cell of the warp reaches T
        const uint32_t cand = (0x80008000u - vmax2(C, TT) + C) & 0x80008000u;
        if (__any_sync(kFull, tested && cand != 0u)) {
          const uint32_t U = __funnelshift_r(P, C, 16);   // rows 2w-1, 2w
          const uint32_t D = __funnelshift_r(C, N, 16);   // rows 2w+1, 2w+2
          const uint32_t VM = vmax2(vmax2(U, C), D);
          const uint32_t VL = __shfl_up_sync(kFull, VM, 1);
          const uint32_t VR = __shfl_down_sync(kFull, VM, 1);
          const uint32_t X = vmax2(vmax2(vmax2(U + 0x00010001u, D), vmax2(VL + addL, VR + addR)), TT);
          const uint32_t Z = 0x80008000u - vmax2(X, C) + C;  // bit 15 of a half: C >= X there
          bits |= (((Z >> 15) & 1u) | ((Z >> 30) & 2u)) << ((2 * w) & 31);  // rows 2w, 2w + 1
        }
        if (do_cs && tested) {
          const unsigned a0 = C & 0xffffu, a1 = C >> 16;
          if (a0) csum += (unsigned long long)a0 * mix64(cell0 + 2 * w + 1);
          if (a1) csum += (unsigned long long)a1 * mix64(cell0 + 2 * w + 2);
        }
        P = C;
        C = N;
      }
      if (tested && bits) atomicOr(&pbits[c * pl.nrb_p + (ws >> 4)], bits);
      ws = we;
    }
  }
}

// Scalar scan for an odd N_rho: one row per step.
__device__ void scan_scalar(const Plan& pl, const uint32_t* acc, const uint32_t* halo, uint32_t* pbits,
                            int wt, int T, int j0, bool do_cs, unsigned long long& csum) {
  const int NT = pl.n_theta, NR = pl.n_rho, nrp = pl.nrho_pad, R = pl.scan_ranges;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nblk = (wt + 29) / 30;
  for (int u = warp; u < nblk * R; u += nwarps) {
    const int b = u >> pl.scan_shift, r = u & (R - 1);
    int k0, k1;
    scan_rows(pl, false, r, k0, k1);
    const int c = b * 30 + lane - 1;
    const ScanSrc s = scan_src(c, wt, T, j0, NT);
    auto fetch = [&](int kk) -> int {
      const int rr = s.mir ? NR - 1 - kk : kk;
      if (s.kind == 3 || rr < 0 || rr >= NR) return -1;
      if (s.kind == 0) return acc_get(acc, s.col, rr, nrp);
      return (int)((halo[(s.kind - 1) * (nrp >> 1) + (rr >> 1)] >> ((rr & 1) << 4)) & 0xffffu);
    };
    const bool tested = lane >= 1 && lane <= 30 && c >= 0 && c < wt;
    const bool lstrict = !(c == 0 && j0 == 0);
    const bool rstrict = (c == wt - 1) && (j0 + wt == NT);
    int vp = fetch(k0 - 1), vc = fetch(k0);
    const unsigned long long cell0 = (unsigned long long)(j0 + c) * NR;
    for (int k = k0; k < k1; ++k) {
      const int vn = fetch(k + 1);
      const int vm = max(max(vp, vc), vn);
      const int vmL = __shfl_up_sync(kFull, vm, 1);
      const int vmR = __shfl_down_sync(kFull, vm, 1);
      if (tested && vc >= pl.threshold && vc > vp && vc >= vn && (lstrict ? vc > vmL : vc >= vmL) &&
          (rstrict ? vc > vmR : vc >= vmR)) {
        atomicOr(&pbits[c * pl.nrb_p + (k >> 5)], 1u << (k & 31));
      }
      if (do_cs && tested && vc > 0) csum += (unsigned long long)vc * mix64(cell0 + k + 1);
      vp = vc;
      vc = vn;
    }
  }
}

// ---- selection: a lane tries the kSelCap most populated peak columns for its hit; hits
// still open go to a whole warp that tests 32 columns per step ----

template <bool WIDE>
__device__ __forceinline__ bool sel_test(const Plan& pl, long long u, long long v, int2 c2, const uint32_t* bmd) {
  const int k = WIDE ? rho_bin64(u * c2.x + v * c2.y + kH, pl.magic)
                     : rho_bin32((int)u * c2.x + ((int)v * c2.y + (int)kH), pl.magic);
  return (bmd[k >> 5] >> (k & 31)) & 1u;
}

template <bool WIDE>
__device__ int select_chunk(const Plan& pl, const void* buf, int cn, long long mbase, uint8_t* __restrict__ mask,
                            const int2* cs, const uint32_t* bm, int D, uint32_t* unres) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int nrb = pl.nrb;
  const int cap = min(D, kSelCap);
  int kept = 0;
  for (int i0 = 0; i0 < cn; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    bool hard = false;
    if (i < cn) {
      long long u, v;
      bool bad;
      if (WIDE) {
        const longlong2 h = reinterpret_cast<const longlong2*>(buf)[i];
        u = h.x;
        v = h.y;
        bad = (h.x == LLONG_MIN);
      } else {
        const int2 h = reinterpret_cast<const int2*>(buf)[i];
        u = h.x;
        v = h.y;
        bad = (h.x == INT_MIN);
      }
      bool m = false;
      if (!bad)
        for (int d = 0; d < cap && !m; ++d) m = sel_test<WIDE>(pl, u, v, cs[d], bm + d * nrb);
      if (m) {
        mask[mbase + i] = 1;
        ++kept;
      } else if (bad || cap == D) {
        mask[mbase + i] = 0;
      } else {
        hard = true;
      }
    }
    const unsigned hb = __ballot_sync(kFull, hard);
    if (lane == 0) unres[(i0 >> 5) + warp] = hb;
  }
  __syncthreads();
  if (D > cap) {
    const int nw = (cn + 31) >> 5;
    for (int wi = warp; wi < nw; wi += nwarps) {
      uint32_t bits = unres[wi];
      while (bits) {
        const int i = (wi << 5) + __ffs(bits) - 1;
        bits &= bits - 1u;
        long long u, v;
        if (WIDE) {
          const longlong2 h = reinterpret_cast<const longlong2*>(buf)[i];
          u = h.x;
          v = h.y;
        } else {
          const int2 h = reinterpret_cast<const int2*>(buf)[i];
          u = h.x;
          v = h.y;
        }
        bool m = false;
        for (int d0 = cap; d0 < D && !m; d0 += 32) {
          const int d = d0 + lane;
          const bool t = d < D && sel_test<WIDE>(pl, u, v, cs[d], bm + d * nrb);
          m = __any_sync(kFull, t);
        }
        if (lane == 0) {
          mask[mbase + i] = m ? 1 : 0;
          kept += m;
        }
      }
    }
  }
  __syncthreads();
  return kept;
}

// Selection over the vote's staged hits (mirror-pair plan, one chunk, no wide hits): floats
// (u, v) in staging order with their original index. The bin comes from the vote's float
// estimate (physical row p = k + 1 read off the bit pattern, exact integer path when
// ambiguous); the dilated bitmaps carry guard bits 0 and N_rho + 1 equal to the edge bins'.
__device__ __forceinline__ bool sel_test_fp(const Plan& pl, float u, float v, int d, const float2* fab,
                                            const int2* cs, const uint32_t* bm) {
  const float2 ab = fab[d];
  const uint32_t y = (uint32_t)__float_as_int(__fmaf_rn(u, ab.x, __fmaf_rn(v, ab.y, pl.mp_c0)));
  int p;
  if ((y & (uint32_t)pl.mp_amask) == 0u) {
    const int2 c2 = cs[d];
    p = rho_bin32(__float2int_rn(u) * c2.x + (__float2int_rn(v) * c2.y + (int)kH), pl.magic) + 1;
  } else {
    p = (int)((y >> pl.mp_F) & (uint32_t)pl.mp_rmask);
  }
  return (bm[d * pl.nrb_g + (p >> 5)] >> (p & 31)) & 1u;
}

// The same for four columns d .. d + 3 (past D: the last four again; with fewer than four, all of them), read and
// tested side by side.
__device__ __forceinline__ bool sel_test4(const Plan& pl, float u, float v, int d, int D, const float2* fab,
                                          const int2* cs, const uint32_t* bm) {
  bool m = false;
  if (D >= 4) {
    d = min(d, D - 4);
    uint32_t hit = 0u;
    bool clear = true;
    const uint32_t* col = bm + d * pl.nrb_g;
#pragma unroll
    for (int i = 0; i < 4; ++i, col += pl.nrb_g) {
      const float2 ab = fab[d + i];
      const uint32_t y = __float_as_uint(__fmaf_rn(u, ab.x, __fmaf_rn(v, ab.y, pl.mp_c0)));
      clear = clear & ((y & (uint32_t)pl.mp_amask) != 0u);
      const uint32_t p = y >> pl.mp_F;  // the row in its low bits
      hit |= __funnelshift_r(col[(p & (uint32_t)pl.mp_rmask) >> 5], 0u, p);  // (shifted by p mod 32)
    }
    if (clear) return (hit & 1u) != 0u;
  }
#pragma unroll 1
  for (int i = 0; i < min(4, D); ++i) m = m || sel_test_fp(pl, u, v, (D >= 4 ? d : 0) + i, fab, cs, bm);
  return m;
}

// Every staged hit against the D peak columns (the most populated first). (A) A lane a hit, the first kSelCap
// columns, four at a time; the hits still open are listed. Then, while many are open, a lane a listed
// hit over the next 24 columns, and again; once they are few, a warp a hit, 64 columns a step. A long list thus
// costs a lane's tests a hit and column, and a short one no more than a few steps. (With a warp for every
// open hit after A: 1000 x 1000 events, whose unkept hits, two fifths, meet all ~95 columns, 50.6 k cycles of 411 k;
// iterative finder at 256 x 256 16.0 k; batched events 5.4 k. So 23.8 k, 10.1 k, 4.2 k.) zeroed: the mask holds 0
// already. list: two lists of lcap entries; with more open hits than that after A, their bits in unres.
__device__ int select_staged(const Plan& pl, const int2* hb, const uint16_t* idx, int nv, long long a,
                             uint8_t* __restrict__ mask, const int2* cs, const float2* fab, const uint32_t* bm, int D,
                             uint32_t* unres, uint16_t* list, int lcap, bool zeroed, int* cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, bd = blockDim.x;
  const int cap = min(D, kSelCap);
  const float* hf = reinterpret_cast<const float*>(hb);
  int kept = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < nv; i0 += bd) {
    const int i = i0 + threadIdx.x;
    const bool on = i < nv;
    const float2 h = staged_hit(hf, on ? i : 0);
    bool open = on;
#pragma unroll 1
    for (int d = 0; d < cap; d += 4) {
      if (open) open = !sel_test4(pl, h.x, h.y, d, D, fab, cs, bm);
      if (!__any_sync(kFull, open)) break;
    }
    if (on && !open) {
      mask[a + idx[i]] = 1;
      ++kept;
    } else if (on && cap == D && !zeroed) {
      mask[a + idx[i]] = 0;
    }
    if (cap < D) {
      const unsigned bal = __ballot_sync(kFull, open);
      if (lane == 0) unres[(i0 >> 5) + warp] = bal;
      const int pos = warp_append(&cnt[0], open);
      if (open && pos < lcap) list[pos] = (uint16_t)i;
    }
  }
  __syncthreads();
  HOUGH_PHASE(HOUGH_PHASE_SEL_A);
  if (cap == D) return kept;
  int n = cnt[0], d0 = cap, cur = 0;
  if (n > lcap) {  // no room: every open hit in its place, all the remaining columns
#pragma unroll 1
    for (int i0 = 0; i0 < nv; i0 += bd) {
      const int i = i0 + threadIdx.x;
      bool open = i < nv && ((unres[(i0 >> 5) + warp] >> lane) & 1u);
      const bool was = open;
      const float2 h = staged_hit(hf, open ? i : 0);
#pragma unroll 1
      for (int d = d0; d < D; d += 4) {
        if (open) open = !sel_test4(pl, h.x, h.y, d, D, fab, cs, bm);
        if (!__any_sync(kFull, open)) break;
      }
      if (was && !(open && zeroed)) mask[a + idx[i]] = open ? 0 : 1;
      kept += was && !open;
    }
    n = 0;
  }
#pragma unroll 1
  while (n >= 4 * nwarps && d0 < D) {  // uniform
    const int d1 = min(D, d0 + 24);
    const uint16_t* from = list + cur * lcap;
    uint16_t* to = list + (cur ^ 1) * lcap;
#pragma unroll 1
    for (int t0 = threadIdx.x - lane; t0 < n; t0 += bd) {  // uniform a warp
      const bool on = t0 + lane < n;
      const int i = from[min(t0 + lane, n - 1)];
      const float2 h = staged_hit(hf, i);
      bool open = on;
#pragma unroll 1
      for (int d = d0; d < d1; d += 4) {
        if (open) open = !sel_test4(pl, h.x, h.y, d, D, fab, cs, bm);
        if (!__any_sync(kFull, open)) break;
      }
      if (on && !open) {
        mask[a + idx[i]] = 1;
        ++kept;
      } else if (on && d1 == D && !zeroed) {
        mask[a + idx[i]] = 0;
      }
      const int pos = warp_append(&cnt[cur + 1], open);
      if (open) to[pos] = (uint16_t)i;
    }
    __syncthreads();
    cur ^= 1;
    d0 = d1;
    n = cnt[cur == 1 ? 1 : 2];
    if (threadIdx.x == 0) cnt[cur + 1] = 0;
    __syncthreads();
  }
  if (d0 < D) {
    const uint16_t* from = list + cur * lcap;
#pragma unroll 1
    for (int t = warp; t < n; t += nwarps) {
      const int i = from[t];
      const float2 h = staged_hit(hf, i);
      bool m = false;
#pragma unroll 1
      for (int d = d0; d < D && !m; d += 64) {
        const bool x = sel_test_fp(pl, h.x, h.y, min(d + lane, D - 1), fab, cs, bm);
        const bool y = sel_test_fp(pl, h.x, h.y, min(d + 32 + lane, D - 1), fab, cs, bm);
        m = __any_sync(kFull, x || y);
      }
      if (lane == 0 && (m || !zeroed)) mask[a + idx[i]] = m ? 1 : 0;
      if (lane == 0) kept += m;
    }
  }
  return kept;
}

constexpr int kFoundMax = 128;  // keys that are ranked one by one

// A work item: tile item % T of event `event`, whose hits are [off[0], off[1]). Two of them in shared
// memory, the current one and the next: in a persistent launch the next is popped while the current one runs, and its
// event's index and offsets are read by asynchronous copies issued between the phases, so that no barrier waits
// for their latency (3.5 k cycles an event in a chain after the last item). It is popped after the vote: the CTAs start with the
// largest events, and those that pop as they start pair them with the next largest; half-way through an item, those
// with small events come first, as they will at its end. (256 x 256, 160 events of 2,022 hits: 83.1 us popped before
// the vote, 63.5 after it; 200 events 84.8 and 70.6; 20,000 events 4,678 and 4,626.) The iterative finder pops before
// the vote (after it 1 % slower, 5,000 events) but for the last two turns (late_items).
struct WorkItem {
  long long off[2];
  int item;  // >= n_items: none
  int event;
  int left;  // items popped together with it and still to come
  int run;   // popped in a run of grab items
};

__device__ __forceinline__ void copy_async(void* smem, const void* gmem, int bytes) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  if (bytes == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(gmem) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct ItemShared {
  WorkItem it[2];
  int nv, flags, wide, last, D, reuse, n_amb, n_low, n_found;
  int staged;  // the event whose hits are staged whole (-1: none)
  unsigned runs;  // of the queue
  int late;       // first of the items after which the next one is popped (late_items)
  int kept_tot;
  int tstart[129], tfrom[128];  // segments of the tile merge (2 a mirror-pair tile): starts, first records
  int tmp[32];
  union {
    struct {
      EdgeWord edge[32];  // of at most 16 word groups, for the scan
      unsigned long long red[32];
    };
    int cnt4[128];  // the merge's counts (after both have been read)
  };
  int it_max, it_ok;  // iterative finder
  // an event's tiles in a cluster: this one's records and low ones, its fingerprint, (tile 0) the hits kept
  int2 cl_cnt;
  unsigned long long cl_cs;
  int cl_kept;
};

// Cluster barrier in two halves: what a thread wrote before `arrive` is seen after `wait`. A shared variable of the
// cluster's CTA `rank` by the address of this CTA's own.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_address(const void* own, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(own)), "r"(rank));
  return a;
}

// Word W of column P's peak rows dilated by +-hw (hw < 32) and cut to [0, N_rho): bit k is
// set iff a peak lies within hw rows of k (0 outside the column's nrb words).
__device__ __forceinline__ uint32_t dilated_word(const uint32_t* P, int W, int nrb, int NR, int hw) {
  if (W < 0 || W >= nrb) return 0u;
  const uint32_t pm = W > 0 ? P[W - 1] : 0u, p0 = P[W], pp = W + 1 < nrb ? P[W + 1] : 0u;
  uint32_t d = p0;
  for (int s = 1; s <= hw; ++s) d |= (p0 << s) | (pm >> (32 - s)) | (p0 >> s) | (pp << (32 - s));
  const int valid = NR - (W << 5);
  return valid < 32 ? d & ((1u << valid) - 1u) : d;
}

// The same with bit k + 1 for row k, and guard bits 0 and N_rho + 1 equal to rows 0 and N_rho - 1.
__device__ __forceinline__ uint32_t dilated_guard_word(const uint32_t* P, int W, int nrb, int NR, int hw) {
  const uint32_t pm = W > 0 ? P[W - 1] : 0u, p0 = W < nrb ? P[W] : 0u, pp = W + 1 < nrb ? P[W + 1] : 0u;
  uint32_t d = (p0 << 1) | (pm >> 31);
  for (int s = 1; s <= hw; ++s)  // rows s above (bits up by s + 1), and s below (down by s - 1); hw <= 31
    d |= (s < 31 ? (p0 << (s + 1)) | (pm >> (31 - s)) : pm) | (s > 1 ? (p0 >> (s - 1)) | (pp << (33 - s)) : p0);
  if (W == 0) d = (d & ~1u) | ((d >> 1) & 1u);
  if (W == ((NR + 1) >> 5)) {
    const int b = (NR + 1) & 31;
    const uint32_t last = b ? (d >> (b - 1)) & 1u : (dilated_word(P, (NR - 1) >> 5, nrb, NR, hw) >> ((NR - 1) & 31)) & 1u;
    d = (d & ~(1u << b)) | (last << b);
  }
  return d;
}

// Back-projection of every hit of event e against its stored peaks pk[0, S). With
// from_bits (one tile, every peak stored, keep_halfwidth < 32) the peak columns and the
// dilated bitmaps come straight from the scan's peak bitmap pbits, which then holds exactly
// the stored peaks.
__device__ int select_event(const Plan& pl, const FusedIO& io, unsigned char* smem, ItemShared& sh,
                            const int16_t* tc, const int16_t* ts, long long a, int n, const hough_peak* pk, int S,
                            bool from_bits) {
  const int NT = pl.n_theta, NR = pl.n_rho, tid = threadIdx.x, bd = blockDim.x;
  int* colcnt = reinterpret_cast<int*>(smem + pl.off_acc);
  int* colidx = colcnt + NT;
  int* hist = colidx + NT;
  int2* cs = reinterpret_cast<int2*>(hist + 64);
  float2* fab = reinterpret_cast<float2*>(cs + NT);
  uint32_t* bm = reinterpret_cast<uint32_t*>(fab + NT);
  uint32_t* unres = reinterpret_cast<uint32_t*>(smem + pl.off_unres);
  const bool staged = sh.reuse != 0;
  const int nrb = staged ? pl.nrb_g : pl.nrb;  // guard-bit bitmaps are one bit wider on each side
  const uint32_t* pbits = reinterpret_cast<const uint32_t*>(smem + pl.off_pbits);
  for (int i = tid; i < 64; i += bd) hist[i] = 0;
  if (from_bits) {
    for (int j = tid; j < NT; j += bd) {
      int cc = 0;
      for (int w = 0; w < pl.nrb; ++w) cc += __popc(pbits[j * pl.nrb_p + w]);
      colcnt[j] = cc;
    }
  } else {
    for (int i = tid; i < NT; i += bd) colcnt[i] = 0;
    __syncthreads();
    for (int q = tid; q < S; q += bd) atomicAdd(&colcnt[pk[q].theta_bin], 1);
  }
  __syncthreads();
  for (int j = tid; j < NT; j += bd)
    if (colcnt[j] > 0) atomicAdd(&hist[63 - min(colcnt[j], 63)], 1);
  __syncthreads();
  if (tid < 32) {
    const int x0 = hist[2 * tid], x1 = hist[2 * tid + 1];
    int x = x0 + x1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, x, o);
      if (tid >= o) x += y;
    }
    const int ex = x - x0 - x1;
    hist[2 * tid] = ex;
    hist[2 * tid + 1] = ex + x0;
    if (tid == 31) sh.D = x;
  }
  __syncthreads();
  for (int j = tid; j < NT; j += bd) {
    const int cc = colcnt[j];
    if (cc > 0) {
      const int pos = atomicAdd(&hist[63 - min(cc, 63)], 1);
      colidx[j] = pos;
      cs[pos] = make_int2(tc[j], ts[j]);
      fab[pos] = make_float2(__fmul_rn((float)tc[j], pl.fp_scale), __fmul_rn((float)ts[j], pl.fp_scale));
    }
  }
  __syncthreads();
  HOUGH_PHASE(HOUGH_PHASE_SEL_COLUMNS);
  const int D = sh.D;
  const int hw = pl.keep_hw;
  if (from_bits) {
    // word W of 32 columns a warp
    const int lane = tid & 31, NG = (NT + 31) >> 5;
#pragma unroll 1
    for (int it = tid >> 5, W = 0; it < NG * nrb; it += bd >> 5) {
      while (it - W * NG >= NG) ++W;
      const int j = 32 * (it - W * NG) + lane;
      if (j >= NT || colcnt[j] == 0) continue;
      const uint32_t* P = pbits + j * pl.nrb_p;
      bm[colidx[j] * nrb + W] = staged ? dilated_guard_word(P, W, pl.nrb, NR, hw) : dilated_word(P, W, pl.nrb, NR, hw);
    }
  } else {
  for (int i = tid; i < D * nrb; i += bd) bm[i] = 0;
  __syncthreads();
  for (int q = tid; q < S; q += bd) {
    const hough_peak pq = pk[q];
    const int d = colidx[pq.theta_bin];
    int lo = max(0, (int)pq.rho_bin - hw), hi = min(NR - 1, (int)pq.rho_bin + hw);
    if (staged) {  // bit k + 1 for row k; guard bits 0 and N_rho + 1 copy rows 0 and N_rho - 1
      lo = (lo == 0) ? 0 : lo + 1;
      hi = (hi == NR - 1) ? NR + 1 : hi + 1;
    }
    for (int w = lo >> 5; w <= (hi >> 5); ++w) {
      const int b0 = max(lo, w << 5) & 31, b1 = min(hi, (w << 5) + 31) & 31;
      const uint32_t bits = (b1 == 31 ? 0xffffffffu : ((1u << (b1 + 1)) - 1u)) & ~((1u << b0) - 1u);
      atomicOr(&bm[d * nrb + w], bits);
    }
  }
  }
  __syncthreads();
  HOUGH_PHASE(HOUGH_PHASE_SEL_BITMAPS);
  int kept = 0;
  if (D == 0) {
    for (int i = tid; i < n; i += bd) io.mask[a + i] = 0;
    return 0;
  }
  if (staged) {
    const bool zeroed = sh.nv < n;  // bad hits are not among the staged ones
    if (zeroed)
      for (int i = tid; i < n; i += bd) io.mask[a + i] = 0;
    if (tid < 3) sh.tmp[tid] = 0;
    __syncthreads();
    // the peak bitmap and what follows it are free now
    return select_staged(pl, reinterpret_cast<const int2*>(smem + pl.off_hits),
                         reinterpret_cast<const uint16_t*>(smem + pl.off_idx), sh.nv, a, io.mask, cs, fab, bm, D, unres,
                         reinterpret_cast<uint16_t*>(smem + pl.off_pbits), (pl.smem_bytes - pl.off_pbits) >> 2, zeroed,
                         sh.tmp);
  }
  int2* hb = reinterpret_cast<int2*>(smem + pl.off_hits);
  longlong2* hw64 = reinterpret_cast<longlong2*>(smem + pl.off_hits);
  for (int h0 = 0; h0 < n; h0 += pl.hit_cap) {
    const int cn = min(pl.hit_cap, n - h0);
    if (tid == 0) sh.wide = 0;
    __syncthreads();
    stage_sel32(io.xy, a + h0, cn, hb, &sh.wide);
    __syncthreads();
    if (!sh.wide) {
      kept += select_chunk<false>(pl, hb, cn, a + h0, io.mask, cs, bm, D, unres);
    } else {
      const int half = pl.hit_cap >> 1;
      for (int s0 = 0; s0 < cn; s0 += half) {
        const int sn = min(half, cn - s0);
        stage_sel64(io.xy, a + h0 + s0, sn, hw64);
        __syncthreads();
        kept += select_chunk<true>(pl, hw64, sn, a + h0 + s0, io.mask, cs, bm, D, unres);
      }
    }
  }
  return kept;
}

// ---- the iterative finder (Sec. 2) on theta tiles ----

// This thread's part of the accumulator checksum over a mirror-pair tile's own cells.
__device__ __noinline__ unsigned long long tile_checksum(const uint32_t* acc, int NT, int NR, int rp, int aw, int half) {
  unsigned long long cs = 0;
#pragma unroll 1
  for (int i = threadIdx.x; i < half * NR; i += blockDim.x) {
    const int k = i / half, w = i - k * half;
    const uint32_t x = acc[mp_word(w, k + 1, rp)];
    cs += (unsigned long long)(x & 0xffffu) * mix64((unsigned long long)(aw + w) * NR + k + 1) +
          (unsigned long long)(x >> 16) * mix64((unsigned long long)(NT - 1 - aw - w) * NR + k + 1);
  }
  if (2 * (aw + half) - 1 == NT)  // the middle column once
    for (int k = threadIdx.x; k < NR; k += blockDim.x)
      cs -= (unsigned long long)(acc[mp_word(half - 1, k + 1, rp)] >> 16) * mix64((unsigned long long)(NT >> 1) * NR + k + 1);
  return cs;
}

// Maximum of a column tile (returned to every thread; *s_max must be 0 beforehand) and, with do_cs, this
// thread's part of the accumulator checksum over the tile's own cells.
__device__ int tile_max_cs(const Plan& pl, const uint32_t* acc, int wt, int j0, bool do_cs, int* s_max,
                           unsigned long long& cs) {
  const int NR = pl.n_rho, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int m = 0;
  for (int k = warp; k < NR; k += nwarps)
    for (int c = lane; c < wt; c += 32) {
      const int v = acc_get(acc, c, k, pl.nrho_pad);
      m = max(m, v);
      if (do_cs && v) cs += (unsigned long long)v * mix64((unsigned long long)(j0 + c) * NR + k + 1);
    }
  m = __reduce_max_sync(kFull, m);
  if (lane == 0 && m) atomicMax(s_max, m);
  __syncthreads();
  return *s_max;
}

// Bit k of word (c, k >> 5) of pbits for every column c of a column tile whose cell k holds >= tq votes.
__device__ void tile_candidate_bits(const Plan& pl, const uint32_t* acc, uint32_t* pbits, int wt, int tq) {
  const int NR = pl.n_rho, nrb = pl.nrb_p, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int k = warp; k < NR; k += nwarps)
    for (int c = lane; c < wt; c += 32)
      if (acc_get(acc, c, k, pl.nrho_pad) >= tq) atomicOr(&pbits[c * nrb + (k >> 5)], 1u << (k & 31));
}

__device__ __forceinline__ uint32_t cand_key(int v, int j, int k) {
  return ((uint32_t)v << 20) | ((uint32_t)(1023 - j) << 10) | (uint32_t)(1023 - k);
}

// The iterative finder's candidates as a list of keys (cand_key) in raster order, colstart[j] the first
// one of column j and colstart[NT] = C, for resolve_kept: ids are places in the list, a window's column is a run of it
// found by binary search over rows, and a key is a rank (votes, then raster order). A column a lane.
struct ListWindow {
  static constexpr int kVotes = 20;
  const uint32_t* keys;
  const int* colstart;
  int NT, NR, R, C;
  uint32_t *alive, *surv;  // a bit a candidate; alive has a word past its last
  __device__ int radius() const { return R; }
  __device__ int lg() const { return 2 * R + 1 <= 8 ? 3 : 2 * R + 1 <= 16 ? 4 : 5; }
  __device__ int words() const { return (C + 31) >> 5; }
  __device__ uint32_t id(int i, int b) const { return (uint32_t)(32 * i + b); }
  __device__ uint32_t bit(uint32_t c, int& w) const {
    w = (int)(c >> 5);
    return 1u << (c & 31u);
  }
  template <class Word>
  __device__ void list_bits(Word&& word, uint32_t* list, int room, int* n) const {
    const int lane = threadIdx.x & 31, nw = words();
#pragma unroll 1
    for (int i0 = threadIdx.x - lane; i0 < nw; i0 += blockDim.x) {  // uniform a warp
      const int i = i0 + lane;
      uint32_t bits = i < nw ? word(i) : 0u;
      int at = warp_positions(__popc(bits), n);
#pragma unroll 1
      while (bits) {
        const int b = 31 - __clz(bits);
        bits ^= 1u << b;
        if (at < room) list[at] = (uint32_t)(32 * i + b);
        ++at;
      }
    }
  }
  __device__ uint32_t key(uint32_t c) const { return keys[c]; }
  __device__ void cell(uint32_t key, int& j, int& k) const {
    j = 1023 - (int)((key >> 10) & 1023u);
    k = 1023 - (int)(key & 1023u);
  }
  __device__ bool live(uint32_t c) const { return (alive[c >> 5] >> (c & 31u)) & 1u; }
  // column j + a of the window of (j, k): its first candidate at or past the window's first row, the last of
  // the window's rows, and the column's end
  __device__ void column(int j, int k, int a, int& lo, int& r1, int& end) const {
    int jj = j + a, r0 = max(0, k - R);
    r1 = min(NR - 1, k + R);
    if ((unsigned)jj >= (unsigned)NT) {  // across the theta wrap: the other end, rho mirrored
      jj += jj < 0 ? NT : -NT;
      const int t0 = NR - 1 - r1;
      r1 = NR - 1 - r0;
      r0 = t0;
    }
    lo = colstart[jj];
    end = colstart[jj + 1];
    int hi = end;
#pragma unroll 1
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (1023 - (int)(keys[mid] & 1023u) < r0) lo = mid + 1;
      else hi = mid;
    }
  }
  __device__ bool look(uint32_t c, bool on, bool& win, uint32_t& at) const {
    const int lane = threadIdx.x & 31, G = 1 << lg(), sub = lane & (G - 1);
    uint32_t m = 0u;
    int j = 0, k = 0, lo = 0, n = 0;  // of this lane's last column: its run in the window
    if (on) {
      cell(keys[c], j, k);
#pragma unroll 1
      for (int a = sub - R; a <= R; a += G) {
        int r1, end;
        column(j, k, a, lo, r1, end);
        n = 0;
#pragma unroll 1
        for (bool in = true; in; n += 4) {  // four independent reads (past the run: not counted)
          const uint32_t f = __funnelshift_r(alive[(lo + n) >> 5], alive[((lo + n) >> 5) + 1], (lo + n) & 31);
          uint32_t x[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = keys[min(lo + n + i, C - 1)];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            in = in && lo + n + i < end && 1023 - (int)(x[i] & 1023u) <= r1;
            if (in && ((f >> i) & 1u) && x[i] > m) {
              m = x[i];
              at = (uint32_t)(lo + n + i);
            }
          }
        }
      }
    }
    uint32_t top = m;
    for (int o = 1; o < G; o <<= 1) top = max(top, __shfl_xor_sync(kFull, top, o));
    win = on && m == top;  // keys are distinct: one lane
    const unsigned self = __ballot_sync(kFull, win && at == c);
    if (!((self >> (lane & ~(G - 1))) & (0xffffffffu >> (32 - G)))) return false;
#pragma unroll 1
    for (int a = sub - R; a <= R; a += G) {
      int r1, end;
      column(j, k, a, lo, r1, end);
#pragma unroll 1
      for (int i = lo; i < end && 1023 - (int)(keys[i] & 1023u) <= r1; ++i)
        if (i != (int)c) atomicAnd(&alive[i >> 5], ~(1u << (i & 31)));
    }
    return true;
  }
};

// The segments that the last tile CTA of an event merges: starts of the low segments in tile order, then
// (mirror-pair tiles) of the high ones in reverse tile order, in sh.tstart (nseg + 1 of them, the last the event's total),
// each segment's first record in its tile's slot in sh.tfrom; the event's checksum in sh.red[0], the tiles' largest
// cell in sh.it_max, and in sh.it_ok whether every tile's records fit its slot. One warp reads all counts
// at once (a thread alone: a chain of 2 to 6 L2 reads a tile).
template <bool MP>
__device__ void merge_segments(const Plan& pl, const FusedIO& io, ItemShared& sh, long long e, bool do_cs) {
  const int T = pl.tiles, nseg = MP ? 2 * T : T, lane = threadIdx.x & 31;
  if (threadIdx.x >= 32) return;
  int ct[4], sum = 0, top = 0;
  bool ok = true;
  unsigned long long cs = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int sg = 4 * lane + i, tt = sg < T ? sg : 2 * T - 1 - sg;
    ct[i] = 0;
    if (sg < nseg) {
      const int2 c = __ldcg(reinterpret_cast<const int2*>(io.tile_cnt) + e * T + tt);  // records, low ones
      ct[i] = sg < T ? c.y : c.x - c.y;
      sh.tfrom[sg] = sg < T ? 0 : c.y;
      ok = ok && c.x <= pl.max_peaks;
      if (sg < T) {
        if (do_cs) cs += __ldcg(io.tile_cs + e * T + tt);
        if (io.tile_max) top = max(top, __ldcg(io.tile_max + e * T + tt));
      }
    }
    sum += ct[i];
  }
  int at = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, at, o);
    if (lane >= o) at += y;
  }
  at -= sum;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (4 * lane + i <= nseg) sh.tstart[4 * lane + i] = at;
    at += ct[i];
  }
  if (lane == 31 && nseg == 128) sh.tstart[128] = at;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cs += __shfl_xor_sync(kFull, cs, o);
  top = __reduce_max_sync(kFull, top);
  ok = __all_sync(kFull, ok);
  if (lane == 0) {
    sh.red[0] = cs;
    sh.it_max = top;
    sh.it_ok = ok;
  }
}

// Record i of the event's merged segments: where it lies in the tiles' slots.
__device__ __forceinline__ const hough_peak* merged_record(const Plan& pl, const FusedIO& io, const ItemShared& sh,
                                                           long long e, int nseg, int i) {
  int lo = 0, hi = nseg - 1;  // the last segment that starts at or before i
#pragma unroll 1
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sh.tstart[mid] <= i) lo = mid;
    else hi = mid - 1;
  }
  const int tt = lo < pl.tiles ? lo : 2 * pl.tiles - 1 - lo;
  return io.tile_peaks + (e * pl.tiles + tt) * (long long)pl.max_peaks + sh.tfrom[lo] + (i - sh.tstart[lo]);
}

// The event's peaks from its tiles' candidate lists, in the last tile CTA of the event (after
// merge_segments). The event's threshold tq = max(T, ceil(rel max)) comes from the tiles' maxima. The
// candidates (cells >= tq) are gathered in raster order, with the first candidate of every column (colstart),
// into the CTA's free shared memory, and their kept set is found and ranked there (resolve_kept; the tiles
// marked the local maxima among them). Returns their count, or -1 (nothing written) when a tile could
// not publish all its candidates, a cell has more votes than a key holds, or there is no room.
// Stress events (512 x 512, 16,100 candidates): 730 k cycles with rounds on two state bits a cell, their ranking included; so
// 389 k.
template <bool MP>
__device__ int merge_iterative(const Plan& pl, const FusedIO& io, unsigned char* smem, ItemShared& sh, long long e) {
  const int T = pl.tiles, NT = pl.n_theta, NR = pl.n_rho, maxp = pl.max_peaks, cap = pl.merge_cap;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bd = blockDim.x, nwarps = bd >> 5;
  const int nseg = MP ? 2 * T : T, total = sh.tstart[nseg], amax = sh.it_max;
  if (!sh.it_ok || amax > 4095) return -1;  // uniform; a key holds votes in 12 bits
  const int tq = (int)max((long long)pl.threshold, ((long long)pl.rel_num * amax + pl.rel_den - 1) / pl.rel_den);
  int* colstart = reinterpret_cast<int*>(smem + pl.off_acc);  // NT + 1
  uint32_t* surv = reinterpret_cast<uint32_t*>(colstart + ((NT + 4) & ~3));
  const int bw = (cap + 63) >> 5;  // bitmap words, one past the last
  uint32_t* alive = surv + bw;
  uint32_t* keys = alive + bw;
  for (int i = tid; i < bw; i += bd) surv[i] = 0u;
  // gather the candidates >= tq, in order, four a thread at a time (their reads go to the L2 together)
  int C = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < total; i0 += 4 * bd) {
    uint32_t key[4];
    bool keep[4], local[4];
    int before[4];
    __syncthreads();  // surv is zero, sh.tmp free
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int i = i0 + m * bd + tid;
      int2 r = make_int2(0, 0);
      if (i < total) r = __ldcg(reinterpret_cast<const int2*>(merged_record(pl, io, sh, e, nseg, i)));
      const int j = r.x & 0xffff, k = (r.x >> 16) & 0xffff, v = r.y & 0xffff;
      keep[m] = i < total && v >= tq;
      local[m] = (r.y >> 16) != 0;
      key[m] = cand_key(v, j, k);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const unsigned bal = __ballot_sync(kFull, keep[m]);
      before[m] = __popc(bal & lanemask_lt());
      if (lane == 0) sh.cnt4[m * 32 + warp] = __popc(bal);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int c = lane < nwarps ? sh.cnt4[m * 32 + lane] : 0;
      const int pos = C + __reduce_add_sync(kFull, lane < warp ? c : 0) + before[m];
      C += __reduce_add_sync(kFull, c);
      if (keep[m] && pos < cap) {
        keys[pos] = key[m];
        if (local[m]) atomicOr(&surv[pos >> 5], 1u << (pos & 31));
      }
    }
  }
  if (C > cap) return -1;  // uniform
  __syncthreads();
  for (int i = tid; i < bw; i += bd) alive[i] = 32 * i + 32 <= C ? 0xffffffffu : 32 * i < C ? (1u << (C & 31)) - 1u : 0u;
  // first candidate of every column (keys are in raster order): where the column changes
  for (int i = tid; i <= C; i += bd) {
    const int j1 = i < C ? 1023 - (int)((keys[i] >> 10) & 1023u) : NT;
    const int j0 = i > 0 ? 1023 - (int)((keys[i - 1] >> 10) & 1023u) : -1;
    for (int j = j0 + 1; j <= j1; ++j) colstart[j] = i;
  }
  __syncthreads();
  uint32_t* list = reinterpret_cast<uint32_t*>((reinterpret_cast<uintptr_t>(keys + C) + 15) & ~(uintptr_t)15);
  // the lists up to the staged hits, which the selection reads again; over them only where they would be short
  int ucap = (int)((smem + pl.off_hits - reinterpret_cast<unsigned char*>(list)) / 10);
  if (ucap < max(1024, C >> 1)) {
    ucap = (int)((smem + pl.smem_bytes - reinterpret_cast<unsigned char*>(list)) / 10);
    if (tid == 0) sh.reuse = 0, sh.staged = -1;  // (read after the barriers below)
  }
  ucap = min(32768, ucap) & ~15;
  const ListWindow lw{keys, colstart, NT, NR, pl.nms_radius, C, alive, surv};
  const int nk = resolve_kept(lw, list, ucap, reinterpret_cast<uint16_t*>(list + 2 * ucap), sh.tmp);
  if (nk > ranked_room(2 * ucap)) return -1;  // uniform
  store_ranked(lw, list, 2 * ucap, nk, amax, tq, maxp, io.peaks + e * (long long)maxp);
  return nk;
}

// Steps 1-2 of a work item: clears the CTA's accumulator of theta tile t (with the halo columns,
// the peak bitmap and the flags) and votes the event's hits [a, a + n) into it, chunk by chunk. The event
// number tells whether its hits are staged already.
template <bool MP, bool ITER, bool WHOLE>
__device__ void vote_tile(const Plan& pl, const FusedIO& io, unsigned char* smem, ItemShared& sh, int event, long long a,
                          int n, int t) {
  uint32_t* acc = reinterpret_cast<uint32_t*>(smem + pl.off_acc);
  uint32_t* halo = reinterpret_cast<uint32_t*>(smem + pl.off_halo);
  int2* hb = reinterpret_cast<int2*>(smem + pl.off_hits);
  longlong2* hw = reinterpret_cast<longlong2*>(smem + pl.off_hits);
  uint32_t* pbits = reinterpret_cast<uint32_t*>(smem + pl.off_pbits);
  const int16_t* tc = reinterpret_cast<const int16_t*>(smem + pl.off_trig);
  const int16_t* ts = tc + pl.n_theta;
  const int T = WHOLE ? 1 : pl.tiles, NT = pl.n_theta, nrp = pl.nrho_pad;
  const int j0 = t * pl.tile_w;
  const int wt = min(pl.tile_w, NT - j0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bd = blockDim.x;
  const int wpad = pl.groups * 32;
  const int rows_w = nrp >> 1;  // words per column
  // mirror-pair tiles: words [aw, aw + Wd), i.e. columns [aw, aw + Wd) and their mirrors
  // (full tiles own tile_w / 2 words, the last one possibly fewer)
  const int Wd = MP ? (wt + 1) >> 1 : 0, aw = t * (pl.tile_w >> 1);

  // lane roles of the vote
  VoteLane L;
  L.halo = !MP && warp >= pl.groups * pl.split;
  L.on = false;
  L.cj = L.sj = 0;
  L.col1 = L.col2 = 0;
  const uint32_t acc_s = (uint32_t)__cvta_generic_to_shared(acc);
  const bool want_halo = !ITER;  // only the 3x3 test reads the halo
  if (L.halo) {
    const int jh = lane < 16 ? (j0 - 1 + NT) % NT : (j0 + wt) % NT;
    L.on = want_halo;
    L.cj = tc[jh];
    L.sj = ts[jh];
    L.col2 = (uint32_t)__cvta_generic_to_shared(halo) + (uint32_t)((lane >> 4) * (nrp >> 1)) * 4u;
    L.p = 0;
    L.P = 1;
  } else if (MP) {
    const int P2 = pl.vote_p, gpair = warp / P2;  // (past the last group: no words)
    L.p = warp % P2;
    L.P = P2;
    const int c1 = gpair * 32 + lane;
    L.on = c1 < Wd;  // lanes past the tile's last word idle
    if (L.on) {
      L.cj = tc[aw + c1];
      L.sj = ts[aw + c1];
    }
    L.col1 = acc_s + (uint32_t)mp_word(c1, 0, pl.rows_phys) * 4u;
  } else {
    const int g = warp / pl.split;
    L.p = warp % pl.split;
    L.P = pl.split;
    const int c1 = g * 32 + lane;
    L.on = c1 < wt;
    if (L.on) {
      L.cj = tc[j0 + c1];
      L.sj = ts[j0 + c1];
    }
    L.col1 = acc_s + (uint32_t)(((g * rows_w) << 5) + lane) * 4u;
  }

  const bool mp_halo = MP && T > 1 && want_halo;
  HaloLane HL{false, 0, 0, 0u};
  if (mp_halo) HL = halo_lane(pl, tc, ts, halo, aw, Wd);
  const AmbList amb{reinterpret_cast<uint32_t*>(smem + pl.off_amb), &sh.n_amb, pl.amb_cap};

  // 1. clear accumulator, halo columns, peak bitmap and counters
  __syncthreads();
  HOUGH_PHASE_START();
  {
    uint4* z = reinterpret_cast<uint4*>(smem + pl.off_acc);
    const int nz = pl.region_bytes >> 4;
    for (int i = tid; i < nz; i += bd) z[i] = make_uint4(0u, 0u, 0u, 0u);
    if (T > 1)
      for (int i = tid; i < (MP ? 2 * pl.rows_phys : nrp); i += bd) halo[i] = 0u;
    for (int i = tid; i < (ITER && MP && T == 1 && pl.iter_cap > 0 ? 2 : 1) * wpad * pl.nrb_p; i += bd) pbits[i] = 0;
    if (tid == 0) {
      sh.flags = 0;
      sh.it_max = 0;
    }
  }

  // 2. map + vote, chunk by chunk. An event's next tile in the same CTA finds its hits staged (a tile of
  // 1000 x 1000 spent 4.5 k of 30 k cycles on mapping them again).
  const bool staged = T > 1 && sh.staged == event;
  if (tid == 0 && !staged) sh.reuse = (MP && n > 0 && n <= pl.hit_cap) ? 1 : 0;
  for (int h0 = 0; h0 < n; h0 += pl.hit_cap) {
    const int cn = min(pl.hit_cap, n - h0);
    __syncthreads();
    HOUGH_PHASE(h0 == 0 ? HOUGH_PHASE_CLEAR : HOUGH_PHASE_VOTE);
    if (tid == 0) {
      if (!staged) sh.nv = sh.wide = 0;
      sh.n_amb = 0;
    }
    __syncthreads();
    if (!staged) {
      stage_vote32(io.xy, a + h0, cn, hb, &sh.nv, &sh.wide, MP ? (unsigned)pl.mp_lsq : 0xffffffffu,
                   MP ? reinterpret_cast<uint16_t*>(smem + pl.off_idx) : nullptr);
      __syncthreads();
      if (tid == 0) {
        if (sh.wide & 2) sh.flags |= HOUGH_F_BAD_HIT;
        if (sh.wide & 1) sh.reuse = 0;  // wide hits are not in the staged list
        sh.staged = sh.reuse ? event : -1;
      }
    }
    HOUGH_PHASE(HOUGH_PHASE_STAGE);
    if (MP && h0 == 0) edge_words(pl, aw, Wd, want_halo, sh.edge);  // for the scan (no hits: no candidates)
    if (!(sh.wide & 1)) {
      if (mp_halo) halo_mp32(pl, HL, hb, sh.nv);
      if (MP)
        vote_mp32(pl, smem, tc, ts, acc_s, aw, Wd, sh.nv, amb);
      else
        vote32_fp(pl, L, hb, sh.nv);
    } else {
      const int half = pl.hit_cap >> 1;
      for (int s0 = 0; s0 < cn; s0 += half) {
        const int sn = min(half, cn - s0);
        __syncthreads();
        if (tid == 0) sh.nv = 0;
        __syncthreads();
        stage_vote64(io.xy, a + h0 + s0, sn, hw, &sh.nv);
        __syncthreads();
        if (mp_halo) halo_mp64(pl, HL, hw, sh.nv);
        if (MP)
          vote_mp64(pl, L, hw, sh.nv);
        else
          vote64(pl, L, hw, sh.nv);
      }
    }
  }
  __syncthreads();
  HOUGH_PHASE(n > 0 ? HOUGH_PHASE_VOTE : HOUGH_PHASE_CLEAR);

}

// The queue hands out runs of pl.grab items (a tiled event's tiles, whose hits are then staged once), the same
// number a CTA, and the rest, at least one a CTA, singly, so that no CTA is left with a run at the end. p: the
// queue's count; runs: how many of them.
__device__ __forceinline__ unsigned queue_runs(const Plan& pl, const FusedIO& io) {
  const unsigned n = (unsigned)io.n_items, g = gridDim.x;
  return pl.grab == 1 ? n : (n - min(n, g)) / g / (unsigned)pl.grab * g;
}

__device__ __forceinline__ void popped(const Plan& pl, const FusedIO& io, unsigned runs, unsigned long long p, int& item,
                                       int& left, int& run) {
  const unsigned q = (unsigned)min(p, (unsigned long long)io.n_items);
  item = (int)min(q < runs ? (unsigned long long)q * pl.grab : (unsigned long long)runs * pl.grab + (q - runs),
                  (unsigned long long)INT_MAX);
  run = q < runs;
  left = run ? pl.grab - 1 : 0;
}

// First of the items at whose end, not after whose vote, the next one is popped. Those of the last two turns on tiles, since
// one of an event's tiles goes on with the merge and the selection, and an item popped before would wait for them instead of
// going to another CTA (512 x 512, events of 4,720 hits: 40 of them 125.5 us popped after the vote, 104.7 so; 449 x 528, 74 of
// them 263.8 and 239.2), but not with more than eight tiles an event, short ones (1000 x 1000, 40 events: 111.1 and 117.1);
// all for the iterative finder on tiles, whose merge takes longest; and those of the last two turns for it on whole
// events, since two thirds of an event come after its vote and not in proportion to its hits (256 x 256, half the maximum, R = 3,
// 160 events of 1,290 hits: 93.4 us popped after the vote, 81.0 so; the chain costs 3.5 k of 119 k cycles an item, in those
// turns alone).
template <bool ITER>
__device__ __forceinline__ int late_items(const Plan& pl, const FusedIO& io) {
  if (!ITER && (pl.tiles == 1 || pl.tiles > 8)) return INT_MAX;
  return pl.tiles > 1 && ITER ? 0 : max(0, (int)io.n_items - 2 * (int)gridDim.x);
}

// The work item sh.it[cur]; with `queue`, sh.it[cur ^ 1] receives the one after it.
// CL: the event's T tiles are the CTAs of a cluster (tile t the CTA of rank t), which exchange their record counts, write their
// records to their places and test a T-th of the hits each: for calls of so few events that SMs would stay idle.
// An event of 256 x 256 alone took 31.7 us in one CTA, 24.5 us in four, of which the two exchanges and the share's
// staging are about 3.
template <bool MP, bool ITER, bool CL, bool WHOLE>
__device__ void run_item(const Plan& pl, const FusedIO& io, unsigned char* smem, ItemShared& sh, int cur, bool queue,
                         bool do_cs) {
  uint32_t* acc = reinterpret_cast<uint32_t*>(smem + pl.off_acc);
  uint32_t* halo = reinterpret_cast<uint32_t*>(smem + pl.off_halo);
  uint32_t* pbits = reinterpret_cast<uint32_t*>(smem + pl.off_pbits);
  int* cnt = reinterpret_cast<int*>(smem + pl.off_cnt);
  const int16_t* tc = reinterpret_cast<const int16_t*>(smem + pl.off_trig);
  const int16_t* ts = tc + pl.n_theta;

  const int T = WHOLE ? 1 : pl.tiles, NT = pl.n_theta, NR = pl.n_rho, nrp = pl.nrho_pad;
  const long long e = sh.it[cur].event;
  const int t = sh.it[cur].item % T;
  const int j0 = t * pl.tile_w;
  const int wt = min(pl.tile_w, NT - j0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bd = blockDim.x;
  const int Wd = MP ? (wt + 1) >> 1 : 0, aw = t * (pl.tile_w >> 1);

  // the next item, in steps whose latencies pass behind the phases between them (thread 0)
  WorkItem& next = sh.it[cur ^ 1];
  const bool fetch = queue && tid == 0 && ((WHOLE && !ITER) || sh.it[cur].item < sh.late);
  unsigned long long pop = 0;
  bool other = false;  // the next item exists and belongs to another event
  auto fetch_pop = [&]() {
    if (fetch && sh.it[cur].left == 0) pop = atomicAdd(io.queue, 1ull);
  };
  auto fetch_event = [&]() {
    if (!fetch) return;
    int more = sh.it[cur].item + 1, left = sh.it[cur].left - 1, run = sh.it[cur].run;
    if (left < 0) popped(pl, io, sh.runs, pop, more, left, run);
    next.item = more;
    next.left = left;
    next.run = run;
    other = more < io.n_items;
    if (other && more - sh.it[cur].item + t < T) {  // items are popped in ascending order
      other = false;
      next.event = sh.it[cur].event;
      next.off[0] = sh.it[cur].off[0];
      next.off[1] = sh.it[cur].off[1];
    }
    if (other) copy_async(&next.event, io.order + (T == 1 ? more : more / T), 4);
  };
  auto fetch_offsets = [&]() {
    if (!fetch || !other) return;
    copy_async_wait();
    copy_async(&next.off[0], io.off + next.event, 8);
    copy_async(&next.off[1], io.off + next.event + 1, 8);
  };
  auto fetch_done = [&]() {
    if (fetch && other) copy_async_wait();
  };

  if (ITER) fetch_pop();
  {
    const long long a = sh.it[cur].off[0], nll = sh.it[cur].off[1] - a;
    vote_tile<MP, ITER, WHOLE>(pl, io, smem, sh, (int)e, a, nll > HOUGH_MAX_EVENT_HITS ? 0 : (int)nll, t);
  }
  if (ITER) fetch_event();
  else fetch_pop();

  // 3-4. peaks
  const int maxp = pl.max_peaks;
  int total = 0, n_low = 0, ev_total = 0;
  unsigned long long cs_tile = 0;
  int tmax = 0;
  if (ITER && T == 1) {
    // the paper's iterative finder on a whole accumulator: the checksum first, then the
    // extraction, which clears the cells it suppresses; records in extraction order
    if (MP) {
      mp_fold(pl, acc, Wd, nullptr);
      if (tid == 0) sh.n_amb = sh.n_found = 0;  // the scan's counts of listed groups and of keys
      __syncthreads();
      HOUGH_PHASE(HOUGH_PHASE_FOLD);
    }
    if (do_cs) {
      unsigned long long cs = 0;
      for (int c = tid; c < NT * NR; c += bd) {
        const int j = c / NR, k = c - j * NR, v = MP ? mp_get(acc, j, k, Wd, wt, pl) : acc_get(acc, j, k, nrp);
        if (v) cs += (unsigned long long)v * mix64((unsigned long long)c + 1);
      }
      cs_tile = block_sum_u64(cs, sh.red);
      __syncthreads();
    }
    HOUGH_PHASE(HOUGH_PHASE_SCAN);
    fetch_offsets();
    hough_peak* dst = io.peaks + e * (long long)maxp;
    total = -1;
    if (MP && pl.iter_cap > 0) {
      // candidates and their 3x3 local maxima as bitmaps (cleared with the accumulator), then the kept set
      const int amax = acc_max_mp(pl, acc, Wd, &sh.it_max);
      HOUGH_PHASE(HOUGH_PHASE_IT_MAX);
      const int tq = (int)max((long long)pl.threshold, ((long long)pl.rel_num * amax + pl.rel_den - 1) / pl.rel_den);
      uint32_t* cand = pbits + pl.groups * 32 * pl.nrb_p;
      uint32_t* list = cand + pl.groups * 32 * pl.nrb_p;
      scan_mp<true>(pl, smem, tq, 0, Wd, sh.edge, pbits, cand, reinterpret_cast<uint16_t*>(list), &sh.n_amb,
                    Found{nullptr, 0, &sh.n_found});
      __syncthreads();
      const WholeWindow ww{acc, Wd, pl.rows_phys, NT, NR, pl.nms_radius, pl.nrb_p, cand, pbits};
      const int nk = resolve_kept(ww, list, pl.iter_cap, reinterpret_cast<uint16_t*>(list + 2 * pl.iter_cap), sh.tmp);
      if (nk <= ranked_room(2 * pl.iter_cap)) {
        store_ranked(ww, list, 2 * pl.iter_cap, nk, amax, tq, maxp, dst);
        total = nk;
      }
    }
    // No bitmaps, or more peaks than the list ranks. (One pass a peak lists a kept set's cells in rank order
    // too: the dropped candidates are zero, the cells that are none below the threshold.)
    if (total < 0) {
      if (MP && (NT & 1)) {  // a middle column's repetition
        for (int k = tid; k < NR; k += bd) reinterpret_cast<uint16_t*>(acc)[2 * mp_word(Wd - 1, k + 1, pl.rows_phys) + 1] = 0;
        __syncthreads();
      }
      FusedCells<MP> cells{acc, Wd, NT, nrp, pl.rows_phys};
      if constexpr (MP) {
        total = extract_iterative_passes(cells, NT, NR, kIterSliceRows, pl.threshold, pl.rel_num, pl.rel_den, pl.nms_radius, maxp,
                                         pbits, dst, sh.tmp);
      } else {
        const int st_words = (((NT * NR + 15) >> 4) + 31) & ~31;  // 2 bits a cell, whole 32-word blocks
        if (pl.iter_cap > 0)
          total = extract_candidates(cells, NT, NR, pl.threshold, pl.rel_num, pl.rel_den, pl.nms_radius, maxp, pbits, pl.iter_cap,
                                     nullptr, st_words, dst, sh.tmp, reinterpret_cast<uint16_t*>(pbits + pl.iter_cap + st_words),
                                     pl.iter_act);
        if (total < 0) total = extract_passes_columns(pl, dst, sh.tmp);
      }
    }
    n_low = total;
  } else {
    // 3. peak scan, or (the iterative finder on theta tiles) the tile's candidates: every cell
    // at or above the tile's own relative threshold, a superset of the cells the event's
    // threshold admits (the event's maximum is at least the tile's)
    // (mirror pairs: with the 3x3 local maxima among them marked; at a tile's edges some that are none, since
    // the neighbour columns of other tiles count as empty there)
    unsigned long long csum = 0;
    const bool packed = !MP && (NR & 1) == 0;
    Found found{nullptr, 0, &sh.n_found};  // after the scan's list of groups
    const int gate = (((Wd + 31) >> 5) * ((NR + 3) >> 2) + 1) >> 1;
    uint32_t* local = pl.off_local ? reinterpret_cast<uint32_t*>(smem + pl.off_local) : pbits;  // no room: none marked
    if (ITER && MP) {
      mp_fold(pl, acc, Wd, nullptr);
      if (tid == 0) sh.n_amb = sh.n_found = 0;  // the scan's counts of listed groups and of keys
      if (pl.off_local)
        for (int i = tid; i < pl.groups * 32 * pl.nrb_p; i += bd) local[i] = 0u;
      __syncthreads();
      HOUGH_PHASE(HOUGH_PHASE_FOLD);
      tmax = acc_max_mp(pl, acc, Wd, &sh.it_max);
      if (do_cs) csum = tile_checksum(acc, NT, NR, pl.rows_phys, aw, Wd);
      const int tq = (int)max((long long)pl.threshold, ((long long)pl.rel_num * tmax + pl.rel_den - 1) / pl.rel_den);
      found = Found{halo + gate, min(kFoundMax, 2 * pl.rows_phys - gate), &sh.n_found};
      scan_mp<true>(pl, smem, tq, aw, Wd, sh.edge, local, pbits, reinterpret_cast<uint16_t*>(halo), &sh.n_amb, found);
    } else if (ITER) {
      tmax = tile_max_cs(pl, acc, wt, j0, do_cs, &sh.it_max, csum);
      tile_candidate_bits(pl, acc, pbits, wt, (int)max((long long)pl.threshold, ((long long)pl.rel_num * tmax + pl.rel_den - 1) / pl.rel_den));
    } else if (MP) {
      mp_fold(pl, acc, Wd, T > 1 ? halo : nullptr);
      if (tid == 0) sh.n_amb = sh.n_found = 0;  // the scan's counts of listed groups and of keys
      __syncthreads();
      HOUGH_PHASE(HOUGH_PHASE_FOLD);
      if (do_cs) csum = tile_checksum(acc, NT, NR, pl.rows_phys, aw, Wd);
      if (T > 1 && !CL)
        found = Found{reinterpret_cast<uint32_t*>(cnt) + gate, min(kFoundMax, pl.groups * 32 * pl.key_groups - gate), &sh.n_found};
      scan_mp<false>(pl, smem, pl.threshold, aw, Wd, sh.edge, pbits, nullptr, reinterpret_cast<uint16_t*>(cnt), &sh.n_amb, found);
    } else if (packed) {
      scan_packed(pl, acc, halo, pbits, wt, T, j0, do_cs, csum);
    } else {
      scan_scalar(pl, acc, halo, pbits, wt, T, j0, do_cs, csum);
    }
    __syncthreads();
    HOUGH_PHASE(HOUGH_PHASE_SCAN);
    fetch_event();

    // 4. raster-order positions and peak records: keys (column, group of key_words bitmap words)
    // in raster order, counted from the peak bitmap
    const int KG = pl.key_groups, G = pl.key_words, nkeys = wt * KG;
    const int nwarps = bd >> 5, kpw = ((nkeys + 32 * nwarps - 1) / (32 * nwarps)) * 32;  // keys a warp
    const int key0 = warp * kpw, key1 = min(nkeys, key0 + kpw);
    auto key_word = [&](int key) {  // one word a key
      const int w = key & (KG - 1);
      return w < pl.nrb ? pbits[(key >> pl.key_shift) * pl.nrb_p + w] : 0u;
    };
    const int key_hi = Wd << pl.key_shift;  // first key of the high columns
    int base = 0;  // records before this warp's keys
    const bool ranked = MP && T > 1 && !CL && sh.n_found <= found.cap;
    if (ranked) {
      total = sh.n_found;
      for (int j = 0; j < total; j += 32)
        n_low += __popc(__ballot_sync(kFull, j + lane < total && found.key[j + lane] < found_key(Wd, 0, 0u)));
    } else if (G == 1) {
      // A warp counts and then writes one run of keys; its first position is the sum of the counts of
      // the warps before it: one barrier, where a block scan of the keys and a second read took five
      // and 3.3 k + 4.7 k cycles an event (batched).
      int np = 0, low = 0;
      for (int key = key0 + lane; key < key1; key += 32) {
        const int x = __popc(key_word(key));
        np += x;
        if (CL && key < key_hi) low += x;
      }
      np = __reduce_add_sync(kFull, np);
      if (CL) low = __reduce_add_sync(kFull, low);
      if (lane == 0) {
        sh.tmp[warp] = np;
        if (CL) sh.tfrom[warp] = low;
      }
      __syncthreads();
      const int x = lane < nwarps ? sh.tmp[lane] : 0;
      base = __reduce_add_sync(kFull, lane < warp ? x : 0);
      total = __reduce_add_sync(kFull, x);
      if (CL) n_low = __reduce_add_sync(kFull, lane < nwarps ? sh.tfrom[lane] : 0);
    } else {
      for (int key = tid; key < nkeys; key += bd) {
        const int c = key >> pl.key_shift, w0 = (key & (KG - 1)) * G, w1 = min(pl.nrb, w0 + G);
        int np = 0;
        for (int w = w0; w < w1; ++w) np += __popc(pbits[c * pl.nrb_p + w]);
        cnt[key] = np;
      }
      __syncthreads();
      total = block_exscan(cnt, nkeys, sh.tmp);
    }
    HOUGH_PHASE(HOUGH_PHASE_EXSCAN);
    fetch_offsets();
    // peaks of the tile's low columns (mirror-pair tiles: the high columns follow them)
    if (!ranked && (!CL || G > 1)) n_low = (MP && Wd < wt && G > 1) ? cnt[key_hi] : total;
    int low_at = 0, high_at = 0;  // CL: of the tile's low and high records, places in the event's less those in the tile's
    if (CL) {
      cs_tile = do_cs ? block_sum_u64(csum, sh.red) : 0ull;
      if (tid == 0) {
        sh.cl_cnt = make_int2(total, n_low);
        sh.cl_cs = cs_tile;
        sh.cl_kept = 0;
      }
      cluster_arrive();
      cluster_wait();
      int all = 0, lo = 0;
      if (lane < T) {
        const uint32_t at = cluster_address(&sh.cl_cnt, lane);
        asm volatile("ld.shared::cluster.v2.s32 {%0, %1}, [%2];" : "=r"(all), "=r"(lo) : "r"(at));
      }
      // raster order: the tiles' low segments, then (mirror pairs) their high ones from the last tile to the first
      low_at = __reduce_add_sync(kFull, lane < t ? lo : 0);
      high_at = __reduce_add_sync(kFull, lane > t ? all : lo) - n_low;
      ev_total = __reduce_add_sync(kFull, all);
    }
    // event column of tile-local column c: mirror-pair tiles hold [aw, aw + Wd) then
    // [N - aw - Wd, N - aw), both ascending; other tiles [j0, j0 + wt)
    const int hi0 = NT - aw - wt;
    hough_peak* dst = (T == 1 || CL) ? io.peaks + e * (long long)maxp : io.tile_peaks + (e * T + t) * (long long)maxp;
    uint2* dst2 = reinterpret_cast<uint2*>(dst);  // records are 8-byte aligned (checked on the host)
    if (ranked) {
      // Few records: a warp a key, its place the number of smaller ones. (A tile of 1000 x 1000 has seven, and the
      // keys of its 2,048 bitmap words took 3.4 k cycles of 23 k: 1,000 events 1405 -> 1357 us, the iterative
      // finder 841 -> 804. Not for whole events: 64 x 64, 126 records, 16.4 us by bitmap words, 18.4 so.)
      for (int i = warp; i < total; i += nwarps) {
        const uint32_t key = found.key[i];
        int pos = 0;
        for (int j = 0; j < total; j += 32)
          pos += __popc(__ballot_sync(kFull, j + lane < total && found.key[j + lane] < key));
        const int c = (int)(key >> 11), k = (int)(key >> 1) & 1023;
        if (lane == 0 && pos < maxp)
          dst2[pos] = make_uint2((uint32_t)(c < Wd ? aw + c : hi0 + c) | ((uint32_t)k << 16),
                                 (uint32_t)mp_get(acc, c, k, Wd, wt, pl) | (pl.off_local ? (key & 1u) << 16 : 0u));
      }
    } else if (G == 1) {
      // a lane takes a key: its word's peaks, one a step, to the positions after the lanes before it
      for (int kb = key0; kb < key1; kb += 32) {
        const int key = kb + lane;
        uint32_t bits = key < key1 ? key_word(key) : 0u;
        if (!__any_sync(kFull, bits != 0u)) {  // (most of a large tile's)
          if (MP && !CL && T > 1 && key == key_hi) sh.n_low = base;
          continue;
        }
        const int np = __popc(bits);
        int pos = np;  // inclusive scan
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kFull, pos, o);
          if (lane >= o) pos += y;
        }
        const int step = __shfl_sync(kFull, pos, 31);
        pos += base - np;
        base += step;
        if (MP && !CL && T > 1 && key == key_hi) sh.n_low = pos;
        if (CL) pos += key < key_hi ? low_at : high_at;
        const int c = key >> pl.key_shift, k0 = (key & (KG - 1)) << 5;
        const int col = MP ? (c < Wd ? aw + c : hi0 + c) : j0 + c;
        while (bits && pos < maxp) {
          const int k = k0 + __ffs(bits) - 1;
          bits &= bits - 1u;
          const int votes = MP ? mp_get(acc, c, k, Wd, wt, pl) : acc_get(acc, c, k, nrp);
          uint32_t lm = 0u;
          if (ITER && MP && pl.off_local) lm = (local[c * pl.nrb_p + (k >> 5)] >> (k & 31)) & 1u;
          dst2[pos++] = make_uint2((uint32_t)col | ((uint32_t)k << 16), (uint32_t)votes | (lm << 16));
        }
      }
    } else {
      for (int key = tid; key < nkeys; key += bd) {
        const int c = key >> pl.key_shift, w0 = (key & (KG - 1)) * G, w1 = min(pl.nrb, w0 + G);
        int pos = cnt[key];
        if (CL) pos += key < key_hi ? low_at : high_at;
        for (int w = w0; w < w1 && pos < maxp; ++w) {
          uint32_t bits = pbits[c * pl.nrb_p + w];
          while (bits && pos < maxp) {
            const int bb = __ffs(bits) - 1;
            bits &= bits - 1u;
            const int k = (w << 5) + bb;
            const int votes = MP ? mp_get(acc, c, k, Wd, wt, pl) : acc_get(acc, c, k, nrp);
            const int col = MP ? (c < Wd ? aw + c : hi0 + c) : j0 + c;
            uint32_t lm = 0u;
            if (ITER && MP && pl.off_local) lm = (local[c * pl.nrb_p + w] >> bb) & 1u;
            dst2[pos] = make_uint2((uint32_t)col | ((uint32_t)k << 16), (uint32_t)votes | (lm << 16));
            ++pos;
          }
        }
      }
    }
    if (!CL) {
      cs_tile = do_cs ? block_sum_u64(csum, sh.red) : 0ull;
      __syncthreads();
      if (!ranked && G == 1 && MP && Wd < wt && T > 1) n_low = sh.n_low;
    }
    HOUGH_PHASE(HOUGH_PHASE_RECORDS);
  }

  fetch_done();

  // 5. tiles: publish, and let the last tile of the event merge
  if (!CL) ev_total = total;
  unsigned long long ev_cs = cs_tile;
  if (T > 1 && !CL) {
    if (tid == 0) {
      io.tile_cnt[2 * (e * T + t)] = total;
      io.tile_cnt[2 * (e * T + t) + 1] = n_low;
      if (do_cs) io.tile_cs[e * T + t] = cs_tile;
      if (io.tile_max) io.tile_max[e * T + t] = tmax;
    }
    // A run is all of an event's tiles in this CTA: they end in order, and what its threads wrote is seen after a
    // barrier. (A fence and a ticket cost each tile of 1000 x 1000 1.4 k cycles of 26.)
    const bool own = sh.it[cur].run && pl.grab == T;
    if (!own) __threadfence();
    __syncthreads();
    if (!own) {
      if (tid == 0) sh.last = (atomicAdd(&io.tickets[e], 1) == T - 1);
      __syncthreads();
    }
    if (own ? t < T - 1 : !sh.last) {
      if (tid == 0 && sh.flags) atomicOr(io.status, sh.flags);
      return;
    }
    if (!own) __threadfence();
    // Raster order of the event: the tiles' low segments in tile order, then (mirror-pair
    // tiles) their high segments in reverse tile order. Segment s < T is tile s's records
    // [0, lo); segment T + i is tile T-1-i's records [lo, all).
    const int nseg = MP ? 2 * T : T;
    merge_segments<MP>(pl, io, sh, e, do_cs);
    __syncthreads();
    ev_cs = sh.red[0];
    if (ITER) {
      ev_total = merge_iterative<MP>(pl, io, smem, sh, e);
      if (ev_total < 0) {  // deferred: the fallback kernel writes this event's outputs
        if (tid == 0) {
          if (io.checksum) io.checksum[e] = ev_cs;
          io.defer_list[atomicAdd(io.defer_count, 1u)] = (int)e;
          if (sh.flags) atomicOr(io.status, sh.flags);
        }
        return;
      }
    } else {
      ev_total = sh.tstart[nseg];
      hough_peak* out = io.peaks + e * (long long)maxp;
      for (int i = tid; i < min(ev_total, maxp); i += bd)
        reinterpret_cast<int2*>(out)[i] = __ldcg(reinterpret_cast<const int2*>(merged_record(pl, io, sh, e, nseg, i)));
      __syncthreads();
    }
  }

  // 6. event outputs and selection (single tile, or the last tile)
  long long a = sh.it[cur].off[0];
  const long long nll = sh.it[cur].off[1] - a;
  const bool too_large = nll > HOUGH_MAX_EVENT_HITS;
  int n = too_large ? 0 : (int)nll;
  if (CL) {
    cluster_arrive();
    // this tile's share of the hits, staged anew while the others write their records
    const int h0 = (int)((long long)n * t / T), cn = (int)((long long)n * (t + 1) / T) - h0;
    a += h0;
    n = cn;
    __syncthreads();  // sh.flags and sh.nv of the vote have been read
    if (tid == 0) sh.nv = sh.wide = sh.reuse = 0;
    __syncthreads();
    if (MP && cn > 0 && cn <= pl.hit_cap) {
      stage_vote32(io.xy, a, cn, reinterpret_cast<int2*>(smem + pl.off_hits), &sh.nv, &sh.wide, (unsigned)pl.mp_lsq,
                   reinterpret_cast<uint16_t*>(smem + pl.off_idx));
      __syncthreads();
      if (tid == 0) sh.reuse = !(sh.wide & 1);
    }
    cluster_wait();
    if (do_cs && t == 0 && warp == 0) {
      unsigned long long x = 0;
      if (lane < T) {
        const uint32_t at = cluster_address(&sh.cl_cs, lane);
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(x) : "r"(at));
      }
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
      ev_cs = x;
    }
  }
  if (tid == 0 && CL && t > 0) {
    if (sh.flags) atomicOr(io.status, sh.flags);
  } else if (tid == 0) {
    io.npeaks[e] = ev_total;
    if (io.checksum) io.checksum[e] = ev_cs;
    if (ev_total > maxp) sh.flags |= HOUGH_F_PEAK_OVERFLOW;
    if (too_large) sh.flags |= HOUGH_F_EVENT_TOO_LARGE;
  }
  __syncthreads();
  HOUGH_PHASE(HOUGH_PHASE_MERGE);
  if (queue && ((WHOLE && !ITER) || sh.it[cur].item < sh.late) && next.item < io.n_items) {  // the next event's hits into the L2 (16 a line)
    const long long i = next.off[0] + 16LL * tid;
    if (i < next.off[1]) asm volatile("prefetch.global.L2 [%0];" ::"l"(io.xy + i));
  }
  int kept = 0;
  if (too_large) {
    for (long long i = tid + (CL ? t * bd : 0); i < nll; i += CL ? T * bd : bd) io.mask[a + i] = 0;
  } else {
    kept = select_event(pl, io, smem, sh, tc, ts, a, n, io.peaks + e * (long long)maxp, min(ev_total, maxp),
                        !ITER && T == 1 && ev_total <= maxp && pl.keep_hw < 32);
  }
  if (tid == 0) sh.kept_tot = 0;
  __syncthreads();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_down_sync(kFull, kept, o);
  if (lane == 0 && kept) atomicAdd(&sh.kept_tot, kept);
  __syncthreads();
  HOUGH_PHASE(HOUGH_PHASE_SEL_B);
  if (CL) {
    if (tid == 0) {
      const uint32_t at = cluster_address(&sh.cl_kept, 0);
      asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(at), "r"(sh.kept_tot) : "memory");
    }
    cluster_arrive();
    cluster_wait();
    if (t > 0) return;
  }
  if (tid == 0) {
    io.nkept[e] = CL ? sh.cl_kept : sh.kept_tot;
    if (sh.flags) atomicOr(io.status, sh.flags);
  }
}

// This thread's share of the check of a batch's offsets: off[0] = 0, none decreasing, off[ne] = nh.
__device__ __forceinline__ int bad_offsets(const long long* off, long long ne, long long nh) {
  int bad = 0;
  for (long long e = threadIdx.x; e < ne; e += blockDim.x) {
    const long long a = off[e], b = off[e + 1];
    if (b < a || a < 0 || b > nh) bad = 1;
  }
  if (threadIdx.x == 0 && (off[0] != 0 || off[ne] != nh)) bad = 1;
  return bad;
}

// Whether a call's events are too uneven for two CTAs an SM instead of one; s: two shared ints, every thread calls it. A large
// event takes longer with 512 threads than with 1,024 (alone on an SM, 128 x 128: 4,000 hits 1.07 times, 8,000 hits 1.15;
// beside another one more), which is worth it only where one CTA an SM would end later anyway: with its share of all
// hits, or after two of the smallest events (an event's fixed part counts as 1,800 hits). 128 x 128, 160 events: of about
// 1,290 hits each 48.0 us in one CTA an SM, 33.8 in two; of 500 to 3,650 hits 42.4 and 46.3 (iterative finder 65 and 78).
__device__ __noinline__ bool is_uneven(const FusedIO& io, int ctas, int* s) {
  constexpr int kFixed = 1800;
  if (threadIdx.x == 0) {
    s[0] = 0;
    s[1] = INT_MAX;
  }
  __syncthreads();
  int most = 0, fewest = HOUGH_MAX_EVENT_HITS;
  for (long long e = threadIdx.x; e < io.n_events; e += blockDim.x) {
    const int n = (int)min(io.off[e + 1] - io.off[e], (long long)HOUGH_MAX_EVENT_HITS);
    most = max(most, n);
    fewest = min(fewest, n);
  }
  most = __reduce_max_sync(kFull, most);
  fewest = __reduce_min_sync(kFull, fewest);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&s[0], most);
    atomicMin(&s[1], fewest);
  }
  __syncthreads();
  const long long top = s[0] + kFixed, share = (io.n_hits + io.n_events * kFixed) / ctas;
  return 23 * top > 20 * max(max(top, share), 2LL * (s[1] + kFixed));
}

// What the validation kernel does for a launch with a queue, by the CTAs of the launch before it: CTA b puts event b at its place
// among the events, largest first, and the first one resets the queue. s: a shared int.
__device__ __noinline__ void order_event(const FusedIO& io, int* s) {
  const long long e = blockIdx.x, c = io.off[e + 1] - io.off[e];
  if (threadIdx.x == 0) *s = 0;
  __syncthreads();
  int before = 0;
  for (long long i = threadIdx.x; i < io.n_events; i += blockDim.x) {
    const long long x = io.off[i + 1] - io.off[i];
    before += x > c || (x == c && i < e);
  }
  before = __reduce_add_sync(kFull, before);
  if ((threadIdx.x & 31) == 0) atomicAdd(s, before);
  __syncthreads();
  if (threadIdx.x != 0) return;
  io.next_order[*s] = (int)e;
  if (e == 0) io.queue[0] = 0ull;
}

// Item `it` of the queue or of the CTA's place, with its event and offsets (thread 0).
__device__ __forceinline__ void fetch_item(const Plan& pl, const FusedIO& io, WorkItem& w, int it, int left, int run) {
  w.item = it;
  w.left = left;
  w.run = run;
  if (it >= io.n_items) return;
  const int e = io.order ? io.order[it / pl.tiles] : it / pl.tiles;
  w.event = e;
  w.off[0] = io.off[e];
  w.off[1] = io.off[e + 1];
}

// The item after sh.it[cur], popped at its end (thread 0).
__device__ __forceinline__ void fetch_late(const Plan& pl, const FusedIO& io, ItemShared& sh, int cur) {
  int it = sh.it[cur].item + 1, left = sh.it[cur].left - 1, run = sh.it[cur].run;
  if (left < 0) popped(pl, io, sh.runs, atomicAdd(io.queue, 1ull), it, left, run);
  fetch_item(pl, io, sh.it[cur ^ 1], it, left, run);
}

// One instance a layout (MP: mirror pairs), peak finder and (CL) use of clusters, so that none carries the others' registers;
// WHOLE: of events in one tile (mirror pairs, local maxima: 20,000 events of 256 x 256 took 4,620 us with the tiles' merge in it and
// 4,731 with their late pops too, 4,501 so; iterative finder, 5,000 events 1,907 and 1,846).
template <bool MP, bool ITER, bool CL, bool WHOLE>
__global__ void __launch_bounds__(1024) fused_kernel(const Plan pl, const FusedIO io, const TrigTable trig) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ItemShared sh;
  int16_t* tc = reinterpret_cast<int16_t*>(smem + pl.off_trig);
  for (int j = threadIdx.x; j < pl.n_theta; j += blockDim.x) {
    tc[j] = trig.c[j];
    tc[pl.n_theta + j] = trig.s[j];
  }
  if (io.solo) {  // no validation kernel before: every CTA looks at all offsets (a few loads a thread)
    const bool first = !CL && io.part == 1;
    if (first) asm volatile("griddepcontrol.launch_dependents;");  // the second launch's CTAs may take SMs that are done
    const int bad = __syncthreads_or(bad_offsets(io.off, io.n_events, io.n_hits));
    const bool uneven = first && !bad && is_uneven(io, io.part_ctas, sh.tmp);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      io.status[1] = bad;
      if (first) io.status[2] = uneven;
      if (bad) atomicOr(io.status, HOUGH_F_BAD_OFFSETS);
    }
    if (uneven) order_event(io, sh.tmp + 2);
    if (bad || uneven) return;
  } else {
    // launched before the validation kernel (or the first launch) has ended: what it writes is read from here on
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (__ldcg(io.status + 1) != 0) return;  // offsets of this call failed validation
    if (!CL && io.part == 2 && __ldcg(io.status + 2) == 0) return;
  }
  __syncthreads();  // the table is read before run_item's first barrier
  const bool do_cs = io.checksum != nullptr;
  const bool queue = io.persistent && io.n_items > gridDim.x;  // else an item a CTA, and none after it
  if (threadIdx.x == 0) {
    sh.staged = -1;
    int it = blockIdx.x, left = 0, run = 0;
    sh.runs = queue_runs(pl, io);
    sh.late = late_items<ITER>(pl, io);
    if (queue) popped(pl, io, sh.runs, atomicAdd(io.queue, 1ull), it, left, run);
    fetch_item(pl, io, sh.it[0], it, left, run);
  }
#pragma unroll 1
  for (int cur = 0;; cur ^= 1) {
    __syncthreads();
    if (sh.it[cur].item >= io.n_items) break;
    run_item<MP, ITER, CL, WHOLE>(pl, io, smem, sh, cur, queue, do_cs);
    if (!queue) break;
    if ((!WHOLE || ITER) && sh.it[cur].item >= sh.late) {
      if (threadIdx.x == 0) fetch_late(pl, io, sh, cur);
    }
  }
}

// Accumulator of one deferred event in HBM (int32 cells, raster order) for the iterative finder;
// suppressed cells are kept in a shared bitmap.
struct SpillCells {
  const int* A;
  uint32_t* gone;
  int NR;
  __device__ int get(int j, int k) const {
    const int c = j * NR + k;
    return ((gone[c >> 5] >> (c & 31)) & 1u) ? 0 : A[c];
  }
  __device__ void clear(int j, int k) {
    const int c = j * NR + k;
    atomicOr(&gone[c >> 5], 1u << (c & 31));
  }
};

// Events the tiled iterative finder deferred (a tile's candidates beyond its record slots, more
// candidates than the merging CTA holds, or a maximum beyond the keys' 12-bit vote field): one
// CTA per HBM accumulator slot takes them in turn, votes every tile of the event in shared
// memory exactly as the fused kernel does and stores the cells to its slot, runs the iterative
// finder there (the stepwise form, any size) and selects the hits. Count and list were written
// by the fused kernel before this launch on the same stream.
template <bool MP>
__global__ void __launch_bounds__(1024) deferred_kernel(const Plan pl, const FusedIO io, const TrigTable trig) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ItemShared sh;
  if (io.status[1] != 0) return;
  const unsigned cnt = *io.defer_count;
  if (blockIdx.x >= cnt) return;
  int16_t* tc = reinterpret_cast<int16_t*>(smem + pl.off_trig);
  for (int j = threadIdx.x; j < pl.n_theta; j += blockDim.x) {
    tc[j] = trig.c[j];
    tc[pl.n_theta + j] = trig.s[j];
  }
  if (threadIdx.x == 0) sh.staged = -1;
  __syncthreads();
  const int T = pl.tiles, NT = pl.n_theta, NR = pl.n_rho, tid = threadIdx.x, bd = blockDim.x, lane = tid & 31;
  const uint32_t* acc = reinterpret_cast<const uint32_t*>(smem + pl.off_acc);
  int* A = io.spill + (long long)blockIdx.x * NT * NR;
  for (unsigned d = blockIdx.x; d < cnt; d += gridDim.x) {
    const long long e = io.defer_list[d];
    const long long a = io.off[e], nll = io.off[e + 1] - a;
    const int n = nll > HOUGH_MAX_EVENT_HITS ? 0 : (int)nll;  // a too-large event is never deferred
    int flags = 0;
    for (int t = 0; t < T; ++t) {
      vote_tile<MP, true, false>(pl, io, smem, sh, (int)e, a, n, t);
      const int j0 = t * pl.tile_w, wt = min(pl.tile_w, NT - j0), Wd = MP ? (wt + 1) >> 1 : 0,
                aw = t * (pl.tile_w >> 1);
      if (MP) {
        mp_fold(pl, const_cast<uint32_t*>(acc), Wd, nullptr);
        __syncthreads();
        for (int i = tid; i < Wd * NR; i += bd) {
          const int w = i / NR, k = i - w * NR;
          const uint32_t x = acc[mp_word(w, k + 1, pl.rows_phys)];
          A[(aw + w) * NR + k] = (int)(x & 0xffffu);
          A[(NT - 1 - aw - w) * NR + k] = (int)(x >> 16);
        }
      } else {
        for (int i = tid; i < wt * NR; i += bd) {
          const int c = i / NR, k = i - c * NR;
          A[(j0 + c) * NR + k] = acc_get(acc, c, k, pl.nrho_pad);
        }
      }
      flags |= sh.flags;
      __syncthreads();
    }
    __threadfence_block();
    // the finder: its scratch first, then the suppression bitmap, after the trig table
    uint32_t* scratch = reinterpret_cast<uint32_t*>(smem + pl.off_unres);
    const int sw = iter_scratch_words(NT, NR, pl.def_sh);
    uint32_t* gone = scratch + (sw > pl.def_cap ? sw : pl.def_cap);
    for (int i = tid; i < (NT * NR + 31) >> 5; i += bd) gone[i] = 0u;
    __syncthreads();
    SpillCells cells{A, gone, NR};
    hough_peak* dst = io.peaks + e * (long long)pl.max_peaks;
    const int total = extract_iterative(cells, NT, NR, pl.def_sh, pl.threshold, pl.rel_num, pl.rel_den,
                                        pl.nms_radius, pl.max_peaks, scratch, pl.def_cap, gone, dst, sh.tmp);
    if (tid == 0) {
      io.npeaks[e] = total;
      if (total > pl.max_peaks) flags |= HOUGH_F_PEAK_OVERFLOW;
      sh.reuse = 0;  // the staged hits were overwritten by the finder
      sh.staged = -1;
    }
    __syncthreads();
    int kept = select_event(pl, io, smem, sh, tc, tc + NT, a, n, dst, min(total, pl.max_peaks), false);
    if (tid == 0) sh.kept_tot = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_down_sync(kFull, kept, o);
    if (lane == 0 && kept) atomicAdd(&sh.kept_tot, kept);
    __syncthreads();
    if (tid == 0) {
      io.nkept[e] = sh.kept_tot;
      if (flags) atomicOr(io.status, flags);
    }
    __syncthreads();
  }
}

// Validates offsets (sets status word 1 for the following kernels), resets the persistent
// queue and the per-event tickets, and orders events by decreasing hit count.
__global__ void __launch_bounds__(1024) prep_kernel(const long long* off, long long ne, long long nh, int* status,
                                                    unsigned long long* queue, int* tickets, int* order) {
  __shared__ int hist[2048];
  __shared__ int s_tmp[32];
  asm volatile("griddepcontrol.launch_dependents;");  // the fused kernel's start overlaps with this one
  const int bad = __syncthreads_or(bad_offsets(off, ne, nh));
  if (threadIdx.x == 0) {
    status[1] = bad;
    if (bad) atomicOr(status, HOUGH_F_BAD_OFFSETS);
    if (queue) {
      queue[0] = 0ull;  // the persistent queue's item counter
      queue[1] = 0ull;  // the count of deferred events (tiled iterative finder)
    }
  }
  if (bad) return;
  if (tickets)
    for (long long e = threadIdx.x; e < ne; e += blockDim.x) tickets[e] = 0;
  if (!order) return;
  for (int i = threadIdx.x; i < 2048; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  for (long long e = threadIdx.x; e < ne; e += blockDim.x) {
    const long long c = off[e + 1] - off[e];
    atomicAdd(&hist[2047 - (int)min(c >> 4, 2047LL)], 1);
  }
  __syncthreads();
  block_exscan(hist, 2048, s_tmp);
  for (long long e = threadIdx.x; e < ne; e += blockDim.x) {
    const long long c = off[e + 1] - off[e];
    const int pos = atomicAdd(&hist[2047 - (int)min(c >> 4, 2047LL)], 1);
    order[pos] = (int)e;
  }
}

// Random (u, v, column) tuples in the int32 fast-path range: the float bin (with its exact
// fallback) against plain 64-bit floor division. Counts disagreements and fallbacks.
__global__ void selftest_fpbin_kernel(const Plan pl, const TrigTable trig, unsigned long long seed, long long n,
                                      unsigned long long* out) {
  unsigned long long bad = 0, amb = 0, bad_mp = 0, amb_mp = 0, n_mp = 0;
  const FpBin K{pl.fp_khi, pl.fp_dlo, pl.fp_dhi};
  const long long NR = pl.n_rho;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const unsigned long long z = mix64(seed + 0x9E3779B97F4A7C15ULL * (unsigned long long)(i + 1));
    const int u = (int)(z % (2ULL * kFast32 + 1)) - kFast32;
    const int v = (int)((z >> 20) % (2ULL * kFast32 + 1)) - kFast32;
    const int j = (int)((z >> 44) % (unsigned long long)pl.n_theta);
    const int c = trig.c[j], s = trig.s[j];
    const float uf = (float)u, vf = (float)v;
    const float A = __fmul_rn((float)c, pl.fp_scale), B = __fmul_rn((float)s, pl.fp_scale);
    const float kf = __fmaf_rn(uf, A, __fmaf_rn(vf, B, pl.fp_c0));
    const int k = bin_fp(kf, K, uf, vf, c, s, pl.magic);
    const float kc = fminf(fmaxf(kf, 0.5f), K.khi);
    amb += __fadd_rn(__fadd_rn(kc, K.dlo), 12582912.0f) != __fadd_rn(__fadd_rn(kc, K.dhi), 12582912.0f);
    const long long t = (long long)u * c + (long long)v * s + kH;
    const long long ref = t < 0 ? 0 : min(NR - 1, (t * NR) / (2 * kH));
    bad += (k != ref);
    // mirror-pair estimate: physical row from the bit pattern (guard rows 0 and N_rho + 1
    // stand for the clamped edge bins), exact path inside the ambiguous window
    if ((long long)u * u + (long long)v * v <= pl.mp_lsq) {
      ++n_mp;
      const uint32_t y = (uint32_t)__float_as_int(__fmaf_rn(uf, A, __fmaf_rn(vf, B, pl.mp_c0)));
      long long p;
      if ((y & (uint32_t)pl.mp_amask) == 0u) {
        ++amb_mp;
        p = rho_bin32(u * c + (v * s + (int)kH), pl.magic) + 1;
      } else {
        p = (long long)((y >> pl.mp_F) & (uint32_t)pl.mp_rmask);
        bad_mp += (((y >> pl.mp_F) << 7) - (uint32_t)pl.mp_k7) != ((uint32_t)p << 7);
      }
      bad_mp += (p < 0 || p > NR + 1 || min(max(p - 1, 0LL), NR - 1) != ref);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    bad += __shfl_down_sync(kFull, bad, o);
    amb += __shfl_down_sync(kFull, amb, o);
    bad_mp += __shfl_down_sync(kFull, bad_mp, o);
    amb_mp += __shfl_down_sync(kFull, amb_mp, o);
    n_mp += __shfl_down_sync(kFull, n_mp, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (bad) atomicAdd(out, bad);
    if (amb) atomicAdd(out + 1, amb);
    if (bad_mp) atomicAdd(out + 2, bad_mp);
    if (amb_mp) atomicAdd(out + 3, amb_mp);
    if (n_mp) atomicAdd(out + 4, n_mp);
  }
}

}  // namespace

cudaError_t launch_selftest_fpbin(const Plan& pl, const TrigTable& trig, unsigned long long seed, long long n,
                                  unsigned long long* out, cudaStream_t st) {
  selftest_fpbin_kernel<<<152 * 8, 256, 0, st>>>(pl, trig, seed, n, out);
  return cudaGetLastError();
}

cudaError_t launch_prep(const long long* off, long long n_events, long long n_hits, int* status,
                        unsigned long long* queue, int* tickets, int* order, cudaStream_t st) {
  prep_kernel<<<1, 1024, 0, st>>>(off, n_events, n_hits, status, queue, tickets, order);
  return cudaGetLastError();
}

// Raises the kernel's dynamic shared-memory limit to the largest size requested so far
// (per kernel and device; never lowers it), so that no attribute call happens while a
// stream is being captured into a graph once a shape has been used.
static cudaError_t set_smem(const void* fn, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int> limit;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  int& cur = limit[std::make_pair(fn, dev)];
  if (bytes <= cur) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}

namespace {
using FusedKernel = void (*)(const Plan, const FusedIO, const TrigTable);
FusedKernel fused_of(const Plan& pl) {
  const bool it = pl.peak_mode == HOUGH_PEAK_ITERATIVE;
  if (pl.cluster) return fused_kernel<true, false, true, false>;
  if (!pl.mp) return it ? fused_kernel<false, true, false, false> : fused_kernel<false, false, false, false>;
  if (it) return pl.tiles == 1 ? fused_kernel<true, true, false, true> : fused_kernel<true, true, false, false>;
  return pl.tiles == 1 ? fused_kernel<true, false, false, true> : fused_kernel<true, false, false, false>;
}
}  // namespace

int fused_max_ctas_per_sm(const Plan& pl) {
  const void* fn = (const void*)fused_of(pl);
  if (set_smem(fn, pl.smem_bytes) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, pl.threads, pl.smem_bytes) != cudaSuccess) return 0;
  return n;
}

bool fused_solo(const Plan& pl, long long n_items, int grid) {
  return pl.cluster || (pl.tiles == 1 && n_items > 0 && n_items <= grid && n_items <= pl.threads);
}

cudaError_t launch_fused(const Plan& pl, const FusedIO& io, const TrigTable& trig, int grid, cudaStream_t st,
                         bool overlap) {
  const bool deferred = pl.peak_mode == HOUGH_PEAK_ITERATIVE && pl.tiles > 1;
  const FusedKernel fused = fused_of(pl), def = pl.mp ? deferred_kernel<true> : deferred_kernel<false>;
  cudaError_t err = set_smem((const void*)fused, pl.smem_bytes);
  if (err == cudaSuccess && deferred) err = set_smem((const void*)def, pl.smem_bytes);
  if (err != cudaSuccess) return err;
  cudaLaunchAttribute at{};
  if (pl.cluster) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)pl.tiles;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
  } else {
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)pl.threads);
  cfg.dynamicSmemBytes = (size_t)pl.smem_bytes;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = overlap || pl.cluster ? 1 : 0;
  err = cudaLaunchKernelEx(&cfg, fused, pl, io, trig);
  if (err != cudaSuccess) return err;
  if (deferred) def<<<io.n_spill, pl.threads, pl.smem_bytes, st>>>(pl, io, trig);
  return cudaGetLastError();
}

CallGrid call_grid(const CallPlan& cp, long long n_items, int sms) {
  auto grid = [&](const Plan& pl) {
    const long long g = (long long)sms * fused_max_ctas_per_sm(pl);
    if (g < 1) return 0;
    return (int)std::max(1LL, g > n_items || pl.cluster ? n_items : g);  // clusters are whole and take no queue
  };
  return CallGrid{grid(cp.pl), cp.two ? grid(cp.one) : 0};
}

cudaError_t launch_call(const CallPlan& cp, FusedIO io, const TrigTable& trig, const CallGrid& g, int* order, cudaStream_t st,
                        Mark before, Mark after) {
  cudaError_t e = cudaSuccess;
  io.solo = fused_solo(cp.pl, io.n_items, g.grid);
  if (!io.solo) e = launch_prep(io.off, io.n_events, io.n_hits, io.status, io.queue, io.tickets, order, st);
  if (e != cudaSuccess || io.n_items == 0) return e;
  if (before) e = before(st);
  const bool two = cp.two && io.solo && g.one > 0;
  io.order = io.solo ? nullptr : order;
  io.part = two;
  io.part_ctas = g.one;
  io.next_order = order;
  // the validation kernel stands right before only without a mark between
  if (e == cudaSuccess) e = launch_fused(cp.pl, io, trig, g.grid, st, !io.solo && !before);
  if (e == cudaSuccess && two) {
    io.part = 2;
    io.solo = 0;
    io.order = order;
    e = launch_fused(cp.one, io, trig, g.one, st, true);
  }
  if (e == cudaSuccess && after) e = after(st);
  return e;
}

}  // namespace hgpu

extern "C" int hough_phase_cycles(uint64_t* host_cycles, int32_t n, int32_t reset, int32_t* enabled) {
  if (!host_cycles || n < 0) return HOUGH_EINVAL;
  const int m = n < HOUGH_PHASE_COUNT ? n : HOUGH_PHASE_COUNT;
#ifdef HOUGH_PHASE_TIMERS
  if (enabled) *enabled = 1;
  unsigned long long buf[HOUGH_PHASE_COUNT];
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpyFromSymbol(buf, hgpu::g_phase_cycles, sizeof(buf));
  if (e == cudaSuccess && reset) {
    const unsigned long long zero[HOUGH_PHASE_COUNT] = {};
    e = cudaMemcpyToSymbol(hgpu::g_phase_cycles, zero, sizeof(zero));
  }
  if (e != cudaSuccess) {
    hgpu::note_cuda_error(e);
    return HOUGH_ECUDA;
  }
  for (int i = 0; i < m; ++i) host_cycles[i] = buf[i];
#else
  (void)reset;
  if (enabled) *enabled = 0;
  for (int i = 0; i < m; ++i) host_cycles[i] = 0;
#endif
  return HOUGH_OK;
}
