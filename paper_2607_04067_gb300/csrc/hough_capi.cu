// C ABI of libhough.so: argument checks, launch planning, workspace layout, CUDA-graph
// replay of the batched path, status words. See include/hough.h for the contract.
#include <cmath>
#include <atomic>
#include <climits>
#include <cstring>
#include <algorithm>
#include <list>
#include <map>
#include <mutex>

#include "hough_internal.h"

namespace hgpu {

static thread_local int g_last_cuda = 0;
static thread_local cudaEvent_t g_ev_begin = nullptr, g_ev_end = nullptr;

static int cuda_fail(cudaError_t e) {
  g_last_cuda = (int)e;
  return HOUGH_ECUDA;
}

// Lets other files of the library report a CUDA error through hough_last_cuda_error.
void note_cuda_error(cudaError_t e) { g_last_cuda = (int)e; }

// th_j = (j + 1/2) pi / N_theta; c_j = round(2^14 cos th_j) (half away from zero).
void host_trig(int n_theta, TrigTable* t) {
  std::memset(t, 0, sizeof(*t));
  const double pi = 3.14159265358979323846;
  for (int j = 0; j < n_theta; ++j) {
    const double th = (j + 0.5) * pi / n_theta;
    t->c[j] = (int16_t)std::llround(16384.0 * std::cos(th));
    t->s[j] = (int16_t)std::llround(16384.0 * std::sin(th));
  }
}

// M = ceil(2^64 N_rho / 2H), split into 32-bit halves (M < 2^44 for N_rho <= 1024).
BinMagic host_magic(int n_rho) {
  const unsigned __int128 two_h = (unsigned __int128)(2 * kH);
  const unsigned __int128 num = ((unsigned __int128)1 << 64) * (unsigned __int128)n_rho;
  const unsigned __int128 M = (num + two_h - 1) / two_h;
  BinMagic m;
  m.lo = (uint32_t)(M & 0xffffffffu);
  m.hi = (uint32_t)(M >> 32);
  return m;
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

WsLayout ws_layout(const Plan& pl, long long n_events) {
  WsLayout w{};
  size_t o = 0;
  w.queue = o;
  o = align256(o + 64);
  const long long T = pl.ws_tiles;
  w.tickets = o;
  if (T > 1) o = align256(o + 4 * (size_t)n_events);
  w.tile_cnt = o;  // per tile: record count and low-segment count
  if (T > 1) o = align256(o + 8 * (size_t)(n_events * T));
  w.tile_cs = o;
  if (T > 1) o = align256(o + 8 * (size_t)(n_events * T));
  w.tile_peaks = o;
  if (T > 1) o = align256(o + sizeof(hough_peak) * (size_t)(n_events * T) * (size_t)pl.max_peaks);
  const bool it_tiled = T > 1 && pl.peak_mode == HOUGH_PEAK_ITERATIVE;
  w.n_spill = it_tiled ? (int)std::min<long long>(std::max<long long>(n_events, 1), kSpillSlots) : 0;
  w.tile_max = o;
  if (it_tiled) o = align256(o + 4 * (size_t)(n_events * T));
  w.defer_list = o;
  if (it_tiled) o = align256(o + 4 * (size_t)(n_events > 0 ? n_events : 1));
  w.spill = o;
  if (it_tiled) o = align256(o + 4 * (size_t)w.n_spill * (size_t)pl.n_theta * (size_t)pl.n_rho);
  w.order = o;
  o = align256(o + 4 * (size_t)(n_events > 0 ? n_events : 1));
  w.total = o;
  return w;
}

void bind_workspace(const Plan& pl, const WsLayout& wl, char* ws, FusedIO& io) {
  const bool tiled = pl.tiles > 1 && !pl.cluster, it_tiled = tiled && pl.peak_mode == HOUGH_PEAK_ITERATIVE;
  io.queue = (unsigned long long*)(ws + wl.queue);
  io.defer_count = (unsigned*)(ws + wl.queue + 8);  // reset with the queue counter by the validation kernel
  io.tickets = tiled ? (int*)(ws + wl.tickets) : nullptr;
  io.tile_cnt = tiled ? (int*)(ws + wl.tile_cnt) : nullptr;
  io.tile_cs = tiled ? (unsigned long long*)(ws + wl.tile_cs) : nullptr;
  io.tile_peaks = tiled ? (hough_peak*)(ws + wl.tile_peaks) : nullptr;
  io.tile_max = it_tiled ? (int*)(ws + wl.tile_max) : nullptr;
  io.defer_list = it_tiled ? (int*)(ws + wl.defer_list) : nullptr;
  io.spill = it_tiled ? (int*)(ws + wl.spill) : nullptr;
  io.n_spill = it_tiled ? wl.n_spill : 0;
}

static constexpr int kSmemStatic = 2048;  // static shared memory stays below
static constexpr int kSmemBudget = 227 * 1024 - kSmemStatic;  // dynamic bytes
static constexpr int kSmemPerSm = 228 * 1024, kSms = 152;

static int round16(int x) { return (x + 15) & ~15; }

// Shared-memory layout for a shape; returns false if it does not fit.
static bool layout(Plan& pl, bool local);

// The layout with more hits staged whole (up to 7,168, so that events above 4,096 hits take one chunk and their
// selection reads the staged ones) where a CTA fills an SM in any case.
static void stage_more(Plan& pl, bool local) {
  if (pl.hit_cap != 4096 || pl.smem_bytes * 2 <= kSmemBudget || pl.tiles == 1 && pl.peak_mode == HOUGH_PEAK_ITERATIVE) return;
  for (int cap = 7168; cap >= 4096; cap -= 1024) {
    pl.hit_cap = cap;
    if (layout(pl, local)) return;
  }
}

static bool layout(Plan& pl, bool local) {
  const int wpad = pl.groups * 32;
  // mirror-pair: groups / 2 word groups of 32 lanes (the last may be part idle) x rows_phys
  const int acc_bytes = pl.mp ? (pl.groups / 2) * 32 * pl.rows_phys * 4 : wpad * pl.nrho_pad * 2;
  const int sel_bytes = (2 * pl.n_theta + 64) * 4 + pl.n_theta * 16 + pl.n_theta * pl.nrb_g * 4;
  int o = 0;
  pl.off_trig = o;
  o += round16(2 * pl.n_theta * 2);
  pl.off_unres = o;
  o += round16((pl.hit_cap + 1024) / 32 * 4);
  if (pl.mp) o = std::max(o, 384);  // the scan of a wrapped word may read up to three rows (of 128 bytes) below row 0
  pl.off_acc = o;
  pl.region_bytes = round16(acc_bytes > sel_bytes ? acc_bytes : sel_bytes);
  o += pl.region_bytes;
  pl.off_halo = o;
  if (pl.tiles > 1) o += round16(2 * (pl.mp ? pl.rows_phys : pl.nrho_pad) * 4);
  pl.off_hits = o;
  o += round16(pl.hit_cap * 8);
  pl.off_idx = o;
  if (pl.mp) o += round16(pl.hit_cap * 2);
  pl.off_pbits = o;  // also the iterative finder's slice and column maxima
  const bool it_whole = pl.peak_mode == HOUGH_PEAK_ITERATIVE && pl.tiles == 1;
  {
    int iter_words = 0;
    if (it_whole) {
      iter_words = iter_scratch_words(pl.n_theta, pl.n_rho, kIterSliceRows);
      // Mirror pairs: the candidates' and the local maxima's bitmaps, then three lists (undecided
      // candidates, the cells that block them, those to look at again). Columns: candidate keys, 2 state bits a cell (also room for
      // the walk's 1-bit bitmap), two lists of undecided candidates (16-bit indices).
      const int cand_words = pl.mp ? 2 * wpad * pl.nrb_p + 2 * pl.iter_cap + pl.iter_cap / 2
                                   : pl.iter_cap + (((pl.n_theta * pl.n_rho + 15) / 16 + 31) & ~31) + pl.iter_act;
      if (pl.iter_cap > 0 && cand_words > iter_words) iter_words = cand_words;
    }
    o += round16((wpad * pl.nrb_p > iter_words ? wpad * pl.nrb_p : iter_words) * 4);
  }
  pl.off_cnt = o;  // record keys of the local-maximum scan or of a tile's candidates
  if (!it_whole) o += round16(wpad * pl.key_groups * 4);
  // the record keys' counts are not needed where a key is one word: the local maxima's bitmap may lie there
  const bool it_tiled = pl.peak_mode == HOUGH_PEAK_ITERATIVE && pl.tiles > 1;
  pl.off_local = it_tiled && pl.mp && local ? (pl.key_words == 1 ? pl.off_cnt : o) : 0;
  if (pl.off_local) o = std::max(o, pl.off_local + round16(wpad * pl.nrb_p * 4));
  // the vote's list lies in a region that is first written after the vote
  pl.off_amb = !it_whole ? pl.off_cnt : pl.off_pbits + (pl.mp && pl.iter_cap > 0 ? 8 * wpad * pl.nrb_p : 0);
  pl.amb_cap = std::min(1024, (o - pl.off_amb) / 4);
  pl.smem_bytes = o;
  if (o > kSmemBudget) return false;
  if (pl.peak_mode == HOUGH_PEAK_ITERATIVE && pl.tiles > 1) {
    // the merging CTA's candidates (a key and a state byte each, after the column starts) in
    // [off_acc, smem_bytes); the deferred kernel's finder (scratch, then a bitmap of every cell)
    // after the trig table
    const int free_bytes = pl.smem_bytes - pl.off_acc - 4 * ((pl.n_theta + 4) & ~3);
    pl.merge_cap = std::min(65520, free_bytes / 5) & ~15;  // key and state a candidate (16-bit indices)
    const int avail = (pl.smem_bytes - pl.off_unres) / 4, gone = (pl.n_theta * pl.n_rho + 31) / 32;
    int sh = kIterSliceRows;
    while (sh < pl.n_rho && iter_scratch_words(pl.n_theta, pl.n_rho, sh) + gone > avail) sh *= 2;
    const int sw = iter_scratch_words(pl.n_theta, pl.n_rho, sh);
    if (sw + gone > avail || pl.merge_cap < 64) return false;
    int cap = 16384;
    while (cap > 0 && (cap > sw ? cap : sw) + gone > avail) cap = cap > 1024 ? cap / 2 : 0;
    pl.def_sh = sh;
    pl.def_cap = cap;
  }
  return true;
}

static int check_params(const hough_params* p) {
  if (!p) return HOUGH_EINVAL;
  if (p->n_theta < 4 || p->n_theta > 1024 || p->n_rho < 4 || p->n_rho > 1024) return HOUGH_EPARAM;
  if (p->threshold < 1 || p->threshold > 32767) return HOUGH_EPARAM;
  if (p->keep_halfwidth < 0 || p->keep_halfwidth > 1024) return HOUGH_EPARAM;
  if (p->max_peaks < 1 || p->max_peaks > 65536) return HOUGH_EPARAM;
  if (p->theta_tiles < 0 || p->theta_tiles > 64 || p->theta_tiles > p->n_theta) return HOUGH_EPARAM;
  if (p->events_per_cta < 0 || p->events_per_cta > 1024) return HOUGH_EPARAM;
  if (p->block < 0 || p->block > 1024 || (p->block % 32) != 0) return HOUGH_EPARAM;
  if (p->peak_mode != HOUGH_PEAK_LOCAL_MAX && p->peak_mode != HOUGH_PEAK_ITERATIVE) return HOUGH_EPARAM;
  if (p->peak_mode == HOUGH_PEAK_ITERATIVE &&
      (p->rel_den < 1 || p->rel_num < 0 || p->rel_num > p->rel_den || p->nms_radius < 0 || p->nms_radius > 64 ||
       2 * p->nms_radius >= p->n_theta))
    return HOUGH_EPARAM;
  return HOUGH_OK;
}

// Constants of the mirror-pair vote's float row estimate k_f + 1 + 2^b + e (k_f = u A + v B +
// N_rho/2, 2^b > N_rho + 1, F = 23 - b fraction bits). Error bound of the estimate, in bins:
// A = fl(c fl(N_rho/2H)) is within 2^-23 (1 + 2^-24) of c N_rho/2H relative, and |u c| N_rho/2H
// <= (N_rho + 1)/2 for hits of the fast path (u^2 + v^2 <= lsq), so each product is off by
// at most (N_rho + 1) 2^-24 (1 + 2^-23); each of the two fused multiply-adds rounds a value
// in [2^b, 2^(b+1)) by at most 2^-(F+1). e (in units of 2^-F) is at least that bound and the
// ambiguous window [0, 2e) a power of two wide.
static void mp_consts(Plan& pl, int n_rho) {
  int b = 0;
  while ((1 << b) < n_rho + 2) ++b;
  const int F = 23 - b;
  pl.rows_phys = n_rho + 2;
  pl.mp_F = F;
  pl.mp_rmask = (1 << b) - 1;
  pl.mp_zoff = 0x4B400000 + (1 << b);
  const double E = (n_rho + 1) * std::ldexp(1.0, F - 23) * (1.0 + std::ldexp(1.0, -20)) + 1.0;
  const int e_min = (int)std::ceil(E);
  int W = 2;
  while (W < 2 * e_min) W <<= 1;
  pl.mp_amask = ((1 << F) - 1) & ~(W - 1);
  pl.mp_k7 = (int)((uint32_t)((127 + b) << b) << 7);
  pl.mp_c0 = (float)(0.5 * n_rho + 1.0 + (double)(1 << b) + std::ldexp((double)(W / 2), -F));
  const double L = (double)kH * (1.0 + 1.0 / n_rho) / 16385.0;
  pl.mp_lsq = (long long)std::floor(L * L);
}

// Whether the table of n_theta columns has c[N-1-j] = -c[j], s[N-1-j] = s[j]; looked at once each.
static bool table_symmetric(int n_theta) {
  static std::atomic<signed char> known[kMaxNTheta + 1];
  signed char k = known[n_theta].load(std::memory_order_relaxed);
  if (!k) {
    TrigTable tt;
    host_trig(n_theta, &tt);
    k = 1;
    for (int j = 0; j < n_theta && k > 0; ++j)
      if (tt.c[n_theta - 1 - j] != -tt.c[j] || tt.s[n_theta - 1 - j] != tt.s[j]) k = -1;
    known[n_theta].store(k, std::memory_order_relaxed);
  }
  return k > 0;
}

// make_plan with T theta tiles, in mirror pairs or (mp false) columns; with `threads`, of so many (a multiple of 32).
static int plan_tiles(const hough_params* p, int T, bool mp, int max_cap, Plan& pl, int threads = 0) {
  // A mirror-pair tile owns WD = ceil(N/2 / T) words (columns [a, a + WD) and their mirrors;
  // the last tile fewer), in word groups of 32 lanes; other tiles W = ceil(N / T) columns.
  int W;
  if (mp) {
    const int NW = (p->n_theta + 1) / 2, WD = (NW + T - 1) / T;
    if ((T - 1) * WD >= NW) return HOUGH_ESMEM;  // every tile must own at least one word
    W = 2 * WD;
    pl.groups = 2 * ((WD + 31) / 32);
  } else {
    W = (p->n_theta + T - 1) / T;
    if ((T - 1) * W >= p->n_theta) return HOUGH_ESMEM;  // every tile must own at least one column
    pl.groups = (W + 31) / 32;
  }
  pl.tiles = pl.ws_tiles = T;
  pl.tile_w = W;
  if (p->events_per_cta == 0) pl.grab = T;  // a run of an event's tiles, whose hits are staged once
  pl.nrho_pad = (p->n_rho + 1) & ~1;
  const int halo = T > 1 ? 32 : 0;
  if (threads) {
    pl.split = 1;
  } else if (p->block) {
    const int work = p->block - halo;
    if (work <= 0 || work % (pl.groups * 32)) {
      return p->theta_tiles ? HOUGH_EPARAM : HOUGH_ESMEM;  // this tile count cannot use the requested block
    }
    pl.split = work / (pl.groups * 32);
  } else {
    // as many warps as fit 1024 threads: with one CTA per SM (large accumulators) the
    // extra warps hide the latency of the vote chains, the scan and the selection
    int s = (1024 - halo) / (pl.groups * 32);
    if (s < 1) s = 1;
    pl.split = s;
  }
  pl.threads = threads ? threads : pl.groups * 32 * pl.split + halo;
  if (pl.threads > 1024) {
    return p->theta_tiles ? HOUGH_EPARAM : HOUGH_ESMEM;
  }
  pl.mp = mp ? 1 : 0;
  if (mp) {
    pl.vote_p = (pl.threads - halo) / 32 / (pl.groups / 2);
    if (pl.vote_p < 1) return HOUGH_ESMEM;
  }
  if (pl.mp) mp_consts(pl, p->n_rho);
  if (!pl.mp)
  // Column layout: the power of two of row ranges that minimises the slowest warp's row steps, each
  // unit (30 columns x one range) paying two extra rows to prime its window and about 16 rows' worth
  // of setup.
  {
    const bool packed = (p->n_rho & 1) == 0;
    const int nblk = (pl.tile_w + 29) / 30, nwarps = pl.threads / 32;
    const int rows = packed ? p->n_rho / 2 : p->n_rho;
    long best = -1;
    for (int Rs = 0; (1 << Rs) <= 64 && (rows >> Rs) >= 2; ++Rs) {
      const long R = 1L << Rs;
      const long cost = ((nblk * R + nwarps - 1) / nwarps) * ((rows + R - 1) / R + 18);
      if (best < 0 || cost < best) {
        best = cost;
        pl.scan_ranges = (int)R;
        pl.scan_shift = Rs;
      }
    }
  }
  // keys of the peak records: (column, group of bitmap words), at most 4096 per CTA
  {
    int kg = 1, ks = 0;
    while (kg < pl.nrb) {
      kg <<= 1;
      ++ks;
    }
    int gw = 1;
    while (pl.groups * 32 * kg > 4096) {
      kg >>= 1;
      --ks;
      gw <<= 1;
    }
    pl.key_groups = kg;
    pl.key_shift = ks;
    pl.key_words = gw;
  }
  // the most staged hits, then (iterative finder on a whole accumulator) the longest lists: mirror pairs,
  // 4,096 to 256 undecided candidates; columns, 8,192 to 1,024 candidate keys and 2,048 to 256 undecided
  // ones. No lists (one pass a peak) only where no number of staged hits leaves room for any.
  const bool whole = pl.peak_mode == HOUGH_PEAK_ITERATIVE && T == 1;
  for (int lists = whole ? 1 : 0; lists >= 0; --lists) {
    for (int cap = max_cap; cap >= 512; cap >>= 1) {
      pl.hit_cap = cap;
      for (int icap = !lists ? 0 : pl.mp ? 4096 : 8192; icap >= (!lists ? 0 : pl.mp ? 256 : 1024);
           icap = pl.mp && icap > 1024 ? icap - 512 : icap > 0 ? icap / 2 : -1) {
        pl.iter_cap = icap;
        for (int act = icap > 0 && !pl.mp ? 2048 : 0; act >= 0;
             act = act > 1024 ? act - 512 : act > 256 ? act / 2 : act - 256) {  // 2048, 1536, 1024, 512, 256, 0
          pl.iter_act = act;
          // odd bitmap strides and the tiles' local maxima where there is room
          for (bool local : {true, false})
            for (pl.nrb_p = pl.nrb | 1; pl.nrb_p >= pl.nrb; --pl.nrb_p)
              if (layout(pl, local)) {
                stage_more(pl, local);
                return HOUGH_OK;
              }
        }
      }
    }
  }
  return HOUGH_ESMEM;
}

// Launch shape for parameters p, with at most max_cap staged hits a chunk (more where a CTA fills an SM in any case).
int make_plan(const hough_params* p, Plan& pl, int max_cap = 4096) {
  int rc = check_params(p);
  if (rc) return rc;
  std::memset(&pl, 0, sizeof(pl));
  pl.n_theta = p->n_theta;
  pl.n_rho = p->n_rho;
  pl.threshold = p->threshold;
  pl.keep_hw = p->keep_halfwidth;
  pl.max_peaks = p->max_peaks;
  pl.peak_mode = p->peak_mode;
  pl.rel_num = p->rel_num;
  pl.rel_den = p->rel_den;
  pl.nms_radius = p->nms_radius;
  pl.nrb = (p->n_rho + 31) / 32;
  pl.nrb_g = ((p->n_rho + 2 + 31) / 32) | 1;
  pl.magic = host_magic(p->n_rho);
  pl.grab = p->events_per_cta > 0 ? p->events_per_cta : 1;
  {
    const double nr = p->n_rho, delta = nr * std::ldexp(1.0, -20);
    pl.fp_scale = (float)(nr / (2.0 * (double)kH));
    pl.fp_c0 = (float)(0.5 * nr);
    pl.fp_khi = (float)(nr - 0.5);
    pl.fp_dlo = (float)(delta - 0.5);
    pl.fp_dhi = (float)(-delta - 0.5);
  }
  // Mirror pairs (columns j and N-1-j in one word) need a table with c[N-1-j] = -c[j], s[N-1-j] = s[j] (true for
  // round-half-away-from-zero). An odd N_theta takes them in the tiles and threads that its columns take (so
  // that a shape is accepted, and reported, as a column shape), else columns. (101 x 63, 500 events 118 -> 60 us; 199 x 200,
  // 1,000 events 335 -> 204 us; iterative finder, 553 x 54, 196 events 529 -> 280 us.)
  const bool sym = table_symmetric(p->n_theta), odd = p->n_theta % 2 != 0;
  for (int T = (p->theta_tiles ? p->theta_tiles : 1); T <= (p->theta_tiles ? p->theta_tiles : 64); ++T) {
    rc = plan_tiles(p, T, sym && !odd, max_cap, pl);
    if (rc == HOUGH_OK && odd && sym) {
      Plan mp = pl;
      // not where a whole accumulator leaves the iterative finder no room for lists
      if (plan_tiles(p, T, true, max_cap, mp, pl.threads) == HOUGH_OK &&
          !(mp.peak_mode == HOUGH_PEAK_ITERATIVE && T == 1 && mp.iter_cap == 0))
        pl = mp;
    }
    if (rc == HOUGH_OK || p->theta_tiles) return rc;
  }
  return HOUGH_ESMEM;
}
// Launch shape of a call: make_plan's, but for few events or many.
// (1) Where tiles and block are the library's to choose and all CTAs of 2, 4 or 8 tiles an event find an SM at once, an
// event's tiles are a cluster. (A cluster lies in one group of 16 to 20 SMs: 15 events of 8 tiles, 36 of 4 and 76 of
// 2 were the most that ran together, and 48 us after 31.5 the step beyond; the line stays below them.) A tile
// takes more than half a word group of 32 lanes, since fewer cost the vote the same (256 x 256 in 8 tiles 31.5, in 4
// 31.8 us). Up to 20,000 cells the exchange costs what the tiles save (128 x 128: 21.6 us an event in one CTA, 23.1 in two).
// 256 x 256: one event 31.7 -> 24.5 us, 16 46.8 -> 31.9, 64 52 -> 43.8; 512 x 512, 8 events 69 -> 44.
// (2) Fewer threads a CTA where the block is the library's to choose and
// several CTAs fit an SM. One CTA of 1,024 threads fills an SM's registers, and on a small accumulator it spends
// most of its time on barriers and on chains that 32 warps wait for together; CTAs of other events run in those
// gaps. c CTAs of 1024 / c threads take kTurn[c] times as long as one (in twentieths; measured from 64 x 64 to
// 160 x 160), so the c with the shortest time for all the events' turns is taken. Where events have few hits, fewer
// staged hits (half as many again as the mean; an event with more takes several chunks) make room for more CTAs; but not for
// more than two in a single turn of events of more than 1,500 hits (128 x 128, events of 500 to 3,650 hits, 400 of them: three
// CTAs 72.4 us, two 60.8; 64 x 64, 608 of them: four 61.0, three 63.9; 100 x 100, 500 of about 1,290: four 57.7, 66.5 with 4,096 staged hits).
// One CTA -> this rule, us: 64 x 64, 616 hits, 5,000 events 424 -> 177 and 500 events 59 -> 30; 100 x 100, 1,290
// hits, 5,000 events 640 -> 365; 128 x 128, 2,022 hits, 1,000 events 167 -> 131, iterative finder 286 -> 218.
// An accumulator of at most 8,192 cells with up to 1,024 hits an event takes half the threads in any case (64 x 64, 616
// hits, 100 events: 18.2 -> 16.5; 64 x 74, 4,720 hits, two events: 45.2 -> 51.6, hence the line): its phases are shorter
// than what 32 warps add to each barrier.
// A call's sizes do not tell how even its events are, and one event with many times the others' hits takes longer in a CTA of
// fewer threads (8,000 hits: 1.2 times with 512, 1.9 times with 256; 64 x 64, 608 events of 600 hits, ten of 8,000: 113 us,
// 75 with a block of 1,024). Among events of 500 to 3,650 hits that loses only where one CTA an SM has a few events left after the
// first turn, the smallest ones: so calls of at most one and a half turns, with more than 1,500 hits an event (with fewer its
// fixed part counts most) and more than one word group (64 columns: 35.8 us in two CTAs an SM, 37.9 in one), launch both
// shapes, and the events choose (is_uneven). The launch that finds nothing to do costs 2.2 us; behind the validation
// kernel of larger calls it would be 4.
int make_plan(const hough_params* p, long long n_hits, long long n_events, CallPlan& cp) {
  cp.two = false;
  Plan& pl = cp.pl;
  const int rc = make_plan(p, pl);
  if (rc || p->block || n_events < 1) return rc;
  if (!p->theta_tiles && pl.mp && pl.peak_mode == HOUGH_PEAK_LOCAL_MAX && p->n_theta * p->n_rho > 20000) {
    hough_params q = *p;
    for (int T = 8; T >= 2 && T >= pl.tiles; T >>= 1) {
      if (n_events > (T == 8 ? 12 : T == 4 ? 32 : 72) || (p->n_theta + 1) / 2 <= 32 * (T / 2)) continue;
      Plan x;
      q.theta_tiles = T;
      if (make_plan(&q, x) != HOUGH_OK || !x.mp) continue;
      x.cluster = 1;
      x.ws_tiles = pl.ws_tiles;
      pl = x;
      return rc;
    }
  }
  if (pl.tiles > 1) return rc;
  static constexpr int kTurn[5] = {0, 20, 27, 38, 42};
  hough_params q = *p;
  q.theta_tiles = 1;
  const bool small = pl.n_theta * pl.n_rho <= 8192 && pl.peak_mode == HOUGH_PEAK_LOCAL_MAX && n_hits <= 1024 * n_events;
  long long best = small ? LLONG_MAX : (n_events + kSms - 1) / kSms * kTurn[1] * 1024 / pl.threads;
  int best_cap = 0;
  Plan x = pl;
  for (int cap = 4096; cap >= 2048; cap -= 1024) {
    if (cap < 4096) {
      hough_params w = q;
      w.block = 0;
      if (n_hits * 3 > n_events * cap * 2 || make_plan(&w, x, cap) != HOUGH_OK) break;
    }
    const int fit = kSmemPerSm / (x.smem_bytes + kSmemStatic + 1024);  // 1 KB a CTA is the system's
    for (int c = 2; c <= std::min(fit, 4); ++c) {
      const int block = 1024 / c / (x.groups * 32) * (x.groups * 32);
      if (!block) break;
      // in one turn the largest events end the call, and those above the staged hits take chunks
      if (c > 2 && cap < 4096 && n_events <= kSms * c && n_hits > 1500 * n_events) continue;
      const long long t = (n_events + kSms * c - 1) / (kSms * c) * kTurn[c] * (1024 / c) / block;
      if (t < best) {
        best = t;
        best_cap = cap;
        q.block = block;
      }
    }
    if (fit >= 4) break;
  }
  if (!best_cap || make_plan(&q, x, best_cap) != HOUGH_OK) return rc;
  cp.two = n_events > kSms && n_events * 2 <= kSms * 3 && n_hits > 1500 * n_events && pl.groups > 2;
  cp.one = pl;
  pl = x;
  return rc;
}

// ---- CUDA graph cache of the batched path ----

struct GraphKey {
  const void *xy, *off, *npeaks, *peaks, *mask, *nkept, *checksum, *ws, *status;
  long long n_hits, n_events;
  size_t ws_bytes;
  hough_params p;
  cudaStream_t stream;
  cudaEvent_t ev_begin, ev_end;
  int device;
  bool operator==(const GraphKey& o) const { return std::memcmp(this, &o, sizeof(GraphKey)) == 0; }
};

struct GraphEntry {
  GraphKey key;
  cudaGraphExec_t exec;
};

static std::mutex g_graph_mu;
static std::list<GraphEntry> g_graphs;

}  // namespace hgpu

using namespace hgpu;

namespace {

// External records become real event-record nodes when the stream is being captured.
cudaError_t mark_begin(cudaStream_t st) { return cudaEventRecordWithFlags(g_ev_begin, st, cudaEventRecordExternal); }
cudaError_t mark_end(cudaStream_t st) { return cudaEventRecordWithFlags(g_ev_end, st, cudaEventRecordExternal); }

struct Common {
  CallPlan cp;
  WsLayout wl;
  FusedIO io;
};

int prepare_fused(const int32_t* d_xy, int64_t n_hits, const int64_t* d_off, int64_t n_events, const hough_params* p,
                  int32_t* d_npeaks, hough_peak* d_peaks, uint8_t* d_mask, int32_t* d_nkept, uint64_t* d_checksum,
                  void* d_ws, size_t ws_bytes, int32_t* d_status, Common& cm) {
  if (!d_off || !d_ws || !d_status) return HOUGH_EINVAL;
  if (n_hits < 0 || n_events < 0) return HOUGH_EINVAL;
  if (n_events > 0 && (!d_npeaks || !d_peaks || !d_nkept)) return HOUGH_EINVAL;
  if (n_hits > 0 && (!d_xy || !d_mask)) return HOUGH_EINVAL;
  if (((uintptr_t)d_xy & 7) || ((uintptr_t)d_peaks & 7) || ((uintptr_t)d_ws & 255)) return HOUGH_EINVAL;
  int rc = make_plan(p, n_hits, n_events, cm.cp);
  if (rc) return rc;
  const Plan& pl = cm.cp.pl;
  if ((long long)n_events * pl.tiles > 0x7fffffffLL) return HOUGH_EINVAL;
  cm.wl = ws_layout(pl, n_events);
  if (ws_bytes < cm.wl.total) return HOUGH_EWORKSPACE;
  char* ws = (char*)d_ws;
  FusedIO& io = cm.io;
  std::memset(&io, 0, sizeof(io));
  io.xy = (const int2*)d_xy;
  io.n_hits = n_hits;
  io.off = (const long long*)d_off;
  io.n_events = n_events;
  io.npeaks = d_npeaks;
  io.peaks = d_peaks;
  io.mask = d_mask;
  io.nkept = d_nkept;
  io.checksum = (unsigned long long*)d_checksum;
  io.status = d_status;
  bind_workspace(pl, cm.wl, ws, io);
  io.n_items = n_events * (long long)pl.tiles;
  return HOUGH_OK;
}

}  // namespace

extern "C" {

int hough_map(const int32_t* d_xy, int64_t n_hits, const int64_t* d_off, int64_t n_events, int64_t* d_uq,
              int64_t* d_vq, int32_t* d_status, void* stream) {
  if (!d_off || !d_status || n_hits < 0 || n_events < 0) return HOUGH_EINVAL;
  if (n_hits > 0 && (!d_xy || !d_uq || !d_vq)) return HOUGH_EINVAL;
  if ((uintptr_t)d_xy & 7) return HOUGH_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = launch_prep((const long long*)d_off, n_events, n_hits, d_status, nullptr, nullptr, nullptr, st);
  if (e != cudaSuccess) return cuda_fail(e);
  if (n_hits == 0) return HOUGH_OK;
  e = launch_map((const int2*)d_xy, n_hits, (long long*)d_uq, (long long*)d_vq, d_status, st);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_vote(const int64_t* d_uq, const int64_t* d_vq, int64_t n_hits, const int64_t* d_off, int64_t n_events,
               const hough_params* p, int16_t* d_acc, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc) return rc;
  if (!d_off || !d_status || n_hits < 0 || n_events < 0) return HOUGH_EINVAL;
  if (n_events > 0 && !d_acc) return HOUGH_EINVAL;
  if (n_hits > 0 && (!d_uq || !d_vq)) return HOUGH_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = launch_prep((const long long*)d_off, n_events, n_hits, d_status, nullptr, nullptr, nullptr, st);
  if (e != cudaSuccess) return cuda_fail(e);
  TrigTable trig;
  host_trig(p->n_theta, &trig);
  e = launch_vote((const long long*)d_uq, (const long long*)d_vq, (const long long*)d_off, n_events, *p, d_acc,
                  d_status, trig, st);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_peaks(const int16_t* d_acc, int64_t n_events, const hough_params* p, int32_t* d_npeaks,
                hough_peak* d_peaks, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc) return rc;
  if (!d_status || n_events < 0) return HOUGH_EINVAL;
  if (n_events > 0 && (!d_acc || !d_npeaks || !d_peaks)) return HOUGH_EINVAL;
  cudaError_t e = launch_peaks(d_acc, n_events, *p, d_npeaks, d_peaks, d_status, (cudaStream_t)stream);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_select(const int64_t* d_uq, const int64_t* d_vq, int64_t n_hits, const int64_t* d_off, int64_t n_events,
                 const hough_params* p, const int32_t* d_npeaks, const hough_peak* d_peaks, uint8_t* d_mask,
                 int32_t* d_nkept, int32_t* d_status, void* stream) {
  int rc = check_params(p);
  if (rc) return rc;
  if (!d_off || !d_status || n_hits < 0 || n_events < 0) return HOUGH_EINVAL;
  if (n_events > 0 && (!d_npeaks || !d_peaks || !d_nkept)) return HOUGH_EINVAL;
  if (n_hits > 0 && (!d_uq || !d_vq || !d_mask)) return HOUGH_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = launch_prep((const long long*)d_off, n_events, n_hits, d_status, nullptr, nullptr, nullptr, st);
  if (e != cudaSuccess) return cuda_fail(e);
  TrigTable trig;
  host_trig(p->n_theta, &trig);
  e = launch_select((const long long*)d_uq, (const long long*)d_vq, (const long long*)d_off, n_events, *p, d_npeaks,
                    d_peaks, d_mask, d_nkept, d_status, trig, st);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_circles(const int32_t* d_npeaks, const hough_peak* d_peaks, int64_t n_events, const hough_params* p,
                  double b_tesla, float* d_circles, void* stream) {
  int rc = check_params(p);
  if (rc) return rc;
  if (n_events < 0) return HOUGH_EINVAL;
  if (n_events > 0 && (!d_npeaks || !d_peaks || !d_circles)) return HOUGH_EINVAL;
  if (((uintptr_t)d_peaks & 7) || ((uintptr_t)d_circles & 15)) return HOUGH_EINVAL;
  const cudaError_t e = launch_circles(d_npeaks, d_peaks, n_events, p->n_theta, p->n_rho, p->max_peaks, b_tesla,
                                       d_circles, (cudaStream_t)stream);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

size_t hough_workspace_size(const hough_params* p, int64_t n_events) {
  Plan pl;
  if (make_plan(p, pl) != HOUGH_OK || n_events < 0) return 256;
  return ws_layout(pl, n_events).total;
}

int hough_resolve_params(hough_params* p) {
  Plan pl;
  int rc = make_plan(p, pl);
  if (rc) return rc;
  p->theta_tiles = pl.tiles;
  p->events_per_cta = pl.grab;
  p->block = pl.threads;
  return HOUGH_OK;
}

// (grid 0: not to be had)
static CallGrid batched_grid(const Common& cm) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return CallGrid{};
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CallGrid{};
  return call_grid(cm.cp, cm.io.n_items, sms);
}

static int enqueue(const Common& cm, const hough_params* p, const CallGrid& g, int* order, cudaStream_t st) {
  TrigTable trig;
  if (cm.io.n_items > 0) host_trig(p->n_theta, &trig);
  const bool timed = g_ev_begin && g_ev_end;
  const cudaError_t e = launch_call(cm.cp, cm.io, trig, g, order, st, timed ? mark_begin : nullptr, timed ? mark_end : nullptr);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

static int enqueue_batched(Common cm, const hough_params* p, void* d_ws, const CallGrid& g, cudaStream_t st) {
  cm.io.persistent = 1;
  return enqueue(cm, p, g, (int*)((char*)d_ws + cm.wl.order), st);
}

int hough_run(const int32_t* d_xy, int64_t n_hits, const int64_t* d_off, int64_t n_events, const hough_params* p,
              int32_t* d_npeaks, hough_peak* d_peaks, uint8_t* d_mask, int32_t* d_nkept, uint64_t* d_checksum,
              void* d_ws, size_t ws_bytes, int32_t* d_status, void* stream) {
  Common cm;
  int rc = prepare_fused(d_xy, n_hits, d_off, n_events, p, d_npeaks, d_peaks, d_mask, d_nkept, d_checksum, d_ws,
                         ws_bytes, d_status, cm);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if (cm.cp.two) {
    const CallGrid g = batched_grid(cm);
    return g.grid < 1 || g.one < 1 ? HOUGH_ESMEM : enqueue_batched(cm, p, d_ws, g, st);
  }
  return enqueue(cm, p, CallGrid{(int)cm.io.n_items, 0}, nullptr, st);
}

// ---- autotuner ----

namespace {

// Everything but the launch shape that the work depends on, so that a cached shape is reused
// only for the same kind of work (the peak finder included).
struct TuneKey {
  int n_theta, n_rho, threshold, keep_hw, max_peaks, peak_mode, rel_num, rel_den, nms_radius, device, sms,
      hits_bucket, events_bucket;
  bool operator<(const TuneKey& o) const { return std::memcmp(this, &o, sizeof(TuneKey)) < 0; }
};

// The launch shape the autotuner picks; the rest of the caller's parameters is left alone.
struct TuneShape {
  int theta_tiles, events_per_cta, block;
};

std::mutex g_tune_mu;
std::map<TuneKey, TuneShape> g_tune_cache;

struct TuneScratch {
  size_t npeaks, peaks, mask, nkept, ws, total;
};

TuneScratch tune_scratch(const hough_params* p, int64_t n_hits, int64_t n_events) {
  TuneScratch L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    const size_t at = o;
    o = (o + (b ? b : 1) + 255) & ~(size_t)255;
    return at;
  };
  L.npeaks = take(4 * (size_t)n_events);
  L.peaks = take(sizeof(hough_peak) * (size_t)n_events * (size_t)p->max_peaks);
  L.mask = take((size_t)n_hits);
  L.nkept = take(4 * (size_t)n_events);
  size_t ws = 0;
  for (int T = 1; T <= 16; T *= 2) {
    hough_params q = *p;
    q.theta_tiles = T;
    q.block = 0;
    Plan pl;
    if (make_plan(&q, pl) == HOUGH_OK) ws = std::max(ws, ws_layout(pl, n_events).total);
  }
  L.ws = take(ws);
  L.total = o;
  return L;
}

}  // namespace

size_t hough_autotune_scratch_size(const hough_params* p, int64_t n_hits, int64_t n_events) {
  if (check_params(p) != HOUGH_OK || n_hits < 0 || n_events < 0) return 256;
  return tune_scratch(p, n_hits, n_events).total;
}

int hough_autotune(hough_params* p, const int32_t* d_xy, int64_t n_hits, const int64_t* d_off, int64_t n_events,
                   void* d_scratch, size_t scratch_bytes, int32_t* d_status, void* stream, float* best_ms) {
  int rc = check_params(p);
  if (rc) return rc;
  if (!d_off || !d_scratch || !d_status || n_events < 1 || n_hits < 0 || ((uintptr_t)d_scratch & 255))
    return HOUGH_EINVAL;
  const TuneScratch L = tune_scratch(p, n_hits, n_events);
  if (scratch_bytes < L.total) return HOUGH_EWORKSPACE;
  TuneKey key;
  std::memset(&key, 0, sizeof(key));
  key.n_theta = p->n_theta;
  key.n_rho = p->n_rho;
  key.threshold = p->threshold;
  key.keep_hw = p->keep_halfwidth;
  key.max_peaks = p->max_peaks;
  key.peak_mode = p->peak_mode;
  key.rel_num = p->peak_mode == HOUGH_PEAK_ITERATIVE ? p->rel_num : 0;
  key.rel_den = p->peak_mode == HOUGH_PEAK_ITERATIVE ? p->rel_den : 0;
  key.nms_radius = p->peak_mode == HOUGH_PEAK_ITERATIVE ? p->nms_radius : 0;
  cudaGetDevice(&key.device);
  cudaDeviceGetAttribute(&key.sms, cudaDevAttrMultiProcessorCount, key.device);
  {
    const double hpe = (double)n_hits / (double)n_events;  // hit density in octaves
    int b = 0;
    while (b < 20 && (double)(1 << (b + 1)) <= hpe) ++b;
    key.hits_bucket = b;
    // a call of few events takes clusters, one of a few turns several CTAs an SM
    const long long turns = (n_events + kSms - 1) / kSms;
    key.events_bucket = n_events <= 12 ? 0 : n_events <= 32 ? 1 : n_events <= 72 ? 2 : (int)std::min(turns, 16LL) + 2;
  }
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      p->theta_tiles = it->second.theta_tiles;
      p->events_per_cta = it->second.events_per_cta;
      p->block = it->second.block;
      if (best_ms) *best_ms = -1.0f;
      return HOUGH_OK;
    }
  }
  char* s = (char*)d_scratch;
  cudaStream_t st = (cudaStream_t)stream;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return cuda_fail(cudaGetLastError());
  hough_params best = *p;
  float best_t = 1e30f;
  bool found = false;
  auto time_shape = [&](const hough_params& q) {
    Common cm;
    if (prepare_fused(d_xy, n_hits, d_off, n_events, &q, (int32_t*)(s + L.npeaks), (hough_peak*)(s + L.peaks),
                      (uint8_t*)(s + L.mask), (int32_t*)(s + L.nkept), nullptr, s + L.ws, scratch_bytes - L.ws, d_status,
                      cm) != HOUGH_OK)
      return;
    const CallGrid grid = batched_grid(cm);
    if (grid.grid < 1) return;
    if (enqueue_batched(cm, &q, s + L.ws, grid, st) != HOUGH_OK) return;
    cudaEventRecord(e0, st);
    for (int r = 0; r < 2; ++r) enqueue_batched(cm, &q, s + L.ws, grid, st);
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess) return;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    ms *= 0.5f;
    if (ms < best_t) {
      best_t = ms;
      best = q;
      found = true;
    }
  };
  for (int T = 1; T <= 16; T *= 2) {
    for (int threads : {256, 512, 1024}) {
      bool have_t = false;
      for (int grab : {1, 2, 4, T}) {  // (T: an event's tiles in a run)
        if (grab == T && T <= 4 && have_t) continue;
        have_t = have_t || grab == T;
        hough_params q = *p;
        q.theta_tiles = T;
        q.events_per_cta = grab;
        Plan probe;
        q.block = 0;
        if (make_plan(&q, probe) != HOUGH_OK) continue;
        q.block = threads;
        Plan exact;
        if (make_plan(&q, exact) != HOUGH_OK) {
          if (threads != 1024) continue;
          q.block = probe.threads;  // the widest block this tiling allows
        }
        time_shape(q);
      }
    }
  }
  // the shape of zero fields, where no explicit ones give it: clusters, fewer staged hits, a choice by the events' sizes
  hough_params q = *p;
  q.theta_tiles = q.block = q.events_per_cta = 0;
  CallPlan cp;
  if (make_plan(&q, n_hits, n_events, cp) == HOUGH_OK) {
    hough_params w = *p;
    w.theta_tiles = cp.pl.tiles;
    w.block = cp.pl.threads;
    w.events_per_cta = 0;
    Plan x;
    if (cp.two || cp.pl.cluster || make_plan(&w, x) != HOUGH_OK || x.hit_cap != cp.pl.hit_cap) time_shape(q);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!found) return HOUGH_ESMEM;
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = TuneShape{best.theta_tiles, best.events_per_cta, best.block};
  }
  p->theta_tiles = best.theta_tiles;
  p->events_per_cta = best.events_per_cta;
  p->block = best.block;
  if (best_ms) *best_ms = best_t;
  return HOUGH_OK;
}

int hough_run_batched(const int32_t* d_xy, int64_t n_hits, const int64_t* d_off, int64_t n_events,
                      const hough_params* p, int32_t* d_npeaks, hough_peak* d_peaks, uint8_t* d_mask,
                      int32_t* d_nkept, uint64_t* d_checksum, void* d_ws, size_t ws_bytes, int32_t* d_status,
                      void* stream) {
  Common cm;
  int rc = prepare_fused(d_xy, n_hits, d_off, n_events, p, d_npeaks, d_peaks, d_mask, d_nkept, d_checksum, d_ws,
                         ws_bytes, d_status, cm);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const CallGrid grid = batched_grid(cm);
  if (grid.grid < 1 || (cm.cp.two && grid.one < 1)) return HOUGH_ESMEM;
  if (st == nullptr) return enqueue_batched(cm, p, d_ws, grid, st);  // legacy stream: no capture
  GraphKey key;
  std::memset(&key, 0, sizeof(key));
  key.xy = d_xy;
  key.off = d_off;
  key.npeaks = d_npeaks;
  key.peaks = d_peaks;
  key.mask = d_mask;
  key.nkept = d_nkept;
  key.checksum = d_checksum;
  key.ws = d_ws;
  key.status = d_status;
  key.n_hits = n_hits;
  key.n_events = n_events;
  key.ws_bytes = ws_bytes;
  key.p = *p;
  key.stream = st;
  key.ev_begin = g_ev_begin;
  key.ev_end = g_ev_end;
  cudaGetDevice(&key.device);
  std::lock_guard<std::mutex> lk(g_graph_mu);
  for (auto it = g_graphs.begin(); it != g_graphs.end(); ++it) {
    if (it->key == key) {
      g_graphs.splice(g_graphs.begin(), g_graphs, it);
      cudaError_t e = cudaGraphLaunch(it->exec, st);
      return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
    }
  }
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return cuda_fail(e);
  rc = enqueue_batched(cm, p, d_ws, grid, st);
  e = cudaStreamEndCapture(st, &graph);
  if (rc) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(e);
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return cuda_fail(e);
  g_graphs.push_front(GraphEntry{key, exec});
  while (g_graphs.size() > 64) {
    cudaGraphExecDestroy(g_graphs.back().exec);
    g_graphs.pop_back();
  }
  e = cudaGraphLaunch(exec, st);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

void hough_set_stage_events(void* begin, void* end) {
  g_ev_begin = (begin && end) ? (cudaEvent_t)begin : nullptr;
  g_ev_end = (begin && end) ? (cudaEvent_t)end : nullptr;
}

namespace {
constexpr int kHostChunks = 16;  // most event chunks of one hough_run_host call (measured: 4, 8, 16, 32)

struct HostLayout {
  size_t xy, off, npeaks, peaks, mask, nkept, peak_off, dense, ws, ws_bytes, total;
};

bool host_layout(const hough_params* p, int64_t n_hits, int64_t n_events, HostLayout& L) {
  Plan pl;
  if (make_plan(p, pl) != HOUGH_OK || n_hits < 0 || n_events < 0) return false;
  const size_t ne = (size_t)n_events, nh = (size_t)n_hits, mp = (size_t)p->max_peaks;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = (o + (bytes ? bytes : 1) + 255) & ~(size_t)255;
    return at;
  };
  L.xy = take(8 * nh);
  L.off = take(8 * (ne + 1 + kHostChunks));  // per chunk its own rebased offsets
  L.npeaks = take(4 * ne);
  L.peaks = take(sizeof(hough_peak) * ne * mp);
  L.mask = take(nh);
  L.nkept = take(4 * ne);
  L.peak_off = take(8 * (ne + 1 + kHostChunks));
  L.dense = take(sizeof(hough_peak) * ne * mp);
  L.ws_bytes = ws_layout(pl, n_events).total;
  L.ws = take(L.ws_bytes);
  L.total = o;
  return true;
}
}  // namespace

size_t hough_host_buffer_size(const hough_params* p, int64_t n_hits, int64_t n_events) {
  HostLayout L;
  return host_layout(p, n_hits, n_events, L) ? L.total : 256;
}

// Timing events of one chunk, on the streams of their stages: copy-in [0, 1], kernels [2, 3],
// packing [3, 4], copy-out of counts, masks and offsets [5, 6], copy-out of the peaks [7, 8].
constexpr int kStageEvents = 9;

// Streams and events of the pipelined host path, per host thread and device.
struct HostPipe {
  int device = -1;
  cudaStream_t in = nullptr, out = nullptr, peaks = nullptr;
  cudaEvent_t ev[3 * kHostChunks] = {};
  bool ok = false;
  bool timing = false;  // per-stage timing of the calls on this thread (hough_set_host_timing)
  bool tev_ok = false;
  cudaEvent_t t_start = nullptr;
  cudaEvent_t tev[kStageEvents * kHostChunks] = {};
  float stage_ms[HOUGH_HOST_STAGES] = {};
  bool stage_valid = false;
};

static HostPipe& host_pipe_raw() {
  thread_local HostPipe hp;
  return hp;
}

static HostPipe& host_pipe() {
  HostPipe& hp = host_pipe_raw();
  int dev = 0;
  cudaGetDevice(&dev);
  if (!hp.ok || hp.device != dev) {
    hp.ok = cudaStreamCreateWithFlags(&hp.in, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&hp.out, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&hp.peaks, cudaStreamNonBlocking) == cudaSuccess;
    for (int i = 0; i < 3 * kHostChunks && hp.ok; ++i)
      hp.ok = cudaEventCreateWithFlags(&hp.ev[i], cudaEventDisableTiming) == cudaSuccess;
    hp.device = dev;
    hp.tev_ok = false;
  }
  if (hp.ok && hp.timing && !hp.tev_ok) {
    hp.tev_ok = cudaEventCreate(&hp.t_start) == cudaSuccess;
    for (int i = 0; i < kStageEvents * kHostChunks && hp.tev_ok; ++i) hp.tev_ok = cudaEventCreate(&hp.tev[i]) == cudaSuccess;
  }
  return hp;
}

// The batch is cut into up to kHostChunks event ranges that flow through four streams:
// copy-in (hits and offsets, rebased to the chunk), compute on `stream` (the batched path
// and the peak packing), copy-out (counts, mask, offsets) and, once a chunk's counts are on
// the host, a peak stream that copies exactly its stored peaks, so every transfer overlaps
// the kernels of other chunks.
int hough_run_host(const int32_t* h_xy, int64_t n_hits, const int64_t* h_off, int64_t n_events, const hough_params* p,
                   int32_t* h_npeaks, int64_t* h_peak_off, hough_peak* h_peaks, int64_t h_peaks_cap, uint8_t* h_mask,
                   int32_t* h_nkept, void* d_buf, size_t d_buf_bytes, int32_t* d_status, void* stream) {
  if (!h_off || !h_npeaks || !h_peak_off || !h_nkept || !d_buf || !d_status || n_hits < 0 || n_events < 0 ||
      h_peaks_cap < 0)
    return HOUGH_EINVAL;
  if (n_hits > 0 && (!h_xy || !h_mask)) return HOUGH_EINVAL;
  if (h_peaks_cap > 0 && !h_peaks) return HOUGH_EINVAL;
  if ((uintptr_t)d_buf & 255) return HOUGH_EINVAL;
  int rc = check_params(p);
  if (rc) return rc;
  HostLayout L;
  if (!host_layout(p, n_hits, n_events, L)) return HOUGH_EPARAM;
  if (d_buf_bytes < L.total) return HOUGH_EWORKSPACE;
  if (h_off[0] != 0 || h_off[n_events] != n_hits) return HOUGH_EINVAL;
  for (int64_t e = 0; e < n_events; ++e)
    if (h_off[e + 1] < h_off[e]) return HOUGH_EINVAL;
  HostPipe& hp = host_pipe();
  if (!hp.ok) return cuda_fail(cudaGetLastError());
  const bool timed = hp.timing && hp.tev_ok;
  hp.stage_valid = false;
  auto mark = [&](int c, int k, cudaStream_t s) {
    return timed ? cudaEventRecord(hp.tev[kStageEvents * c + k], s) : cudaSuccess;
  };
  char* b = (char*)d_buf;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t mp = (size_t)p->max_peaks;
  // chunk c: events [ce[c], ce[c + 1])
  const int K = (int)std::max<int64_t>(1, std::min<int64_t>(kHostChunks, n_events / 2048));
  int64_t ce[kHostChunks + 1];
  for (int c = 0; c <= K; ++c) ce[c] = n_events * c / K;
  cudaError_t e = cudaSuccess;
  int32_t* d_npk = (int32_t*)(b + L.npeaks);
  int32_t* d_nk = (int32_t*)(b + L.nkept);
  int64_t* d_off = (int64_t*)(b + L.off);
  int64_t* d_poff = (int64_t*)(b + L.peak_off);
  hough_peak* d_pk = (hough_peak*)(b + L.peaks);
  hough_peak* d_dense = (hough_peak*)(b + L.dense);
  uint8_t* d_mask = (uint8_t*)(b + L.mask);
  const int32_t* d_xy = (const int32_t*)(b + L.xy);
  // the compute stream's earlier work must not see half-written inputs: copy-in starts after it
  e = cudaEventRecord(hp.ev[0], st);
  if (e == cudaSuccess && timed) e = cudaEventRecord(hp.t_start, st);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(hp.in, hp.ev[0], 0);
  for (int c = 0; c < K && e == cudaSuccess; ++c) {
    const int64_t e0 = ce[c], n = ce[c + 1] - ce[c], a0 = h_off[e0], nh = h_off[ce[c + 1]] - a0;
    int64_t* roff = d_off + e0 + c;
    cudaEvent_t ev_in = hp.ev[3 * c], ev_comp = hp.ev[3 * c + 1], ev_out = hp.ev[3 * c + 2];
    e = mark(c, 0, hp.in);
    if (e == cudaSuccess) e = cudaMemcpyAsync(roff, h_off + e0, 8 * (size_t)(n + 1), cudaMemcpyHostToDevice, hp.in);
    if (e == cudaSuccess && nh)
      e = cudaMemcpyAsync((char*)d_xy + 8 * (size_t)a0, h_xy + 2 * a0, 8 * (size_t)nh, cudaMemcpyHostToDevice, hp.in);
    if (e == cudaSuccess) e = launch_rebase((long long*)roff, n + 1, a0, hp.in);
    if (e == cudaSuccess) e = mark(c, 1, hp.in);
    if (e == cudaSuccess) e = cudaEventRecord(ev_in, hp.in);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev_in, 0);
    if (e == cudaSuccess) e = mark(c, 2, st);
    if (e != cudaSuccess) break;
    rc = hough_run_batched(d_xy + 2 * a0, nh, roff, n, p, d_npk + e0, d_pk + e0 * mp, d_mask + a0, d_nk + e0,
                           nullptr, b + L.ws, L.ws_bytes, d_status, stream);
    if (rc) {  // nothing may still read or write the caller's host buffers after the return
      cudaStreamSynchronize(hp.in);
      cudaStreamSynchronize(hp.out);
      cudaStreamSynchronize(st);
      return rc;
    }
    e = mark(c, 3, st);
    if (e == cudaSuccess)
      e = launch_pack_peaks(d_npk + e0, d_pk + e0 * mp, n, p->max_peaks, (long long*)(d_poff + e0 + c),
                            d_dense + e0 * mp, st);
    if (e == cudaSuccess) e = mark(c, 4, st);
    if (e == cudaSuccess) e = cudaEventRecord(ev_comp, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(hp.out, ev_comp, 0);
    if (e == cudaSuccess) e = mark(c, 5, hp.out);
    if (e == cudaSuccess && n) e = cudaMemcpyAsync(h_npeaks + e0, d_npk + e0, 4 * (size_t)n, cudaMemcpyDeviceToHost, hp.out);
    if (e == cudaSuccess && n) e = cudaMemcpyAsync(h_nkept + e0, d_nk + e0, 4 * (size_t)n, cudaMemcpyDeviceToHost, hp.out);
    if (e == cudaSuccess && nh) e = cudaMemcpyAsync(h_mask + a0, d_mask + a0, (size_t)nh, cudaMemcpyDeviceToHost, hp.out);
    if (e == cudaSuccess && n)
      e = cudaMemcpyAsync(h_peak_off + e0, d_poff + e0 + c, 8 * (size_t)n, cudaMemcpyDeviceToHost, hp.out);
    if (e == cudaSuccess) e = mark(c, 6, hp.out);
    if (e == cudaSuccess) e = cudaEventRecord(ev_out, hp.out);
  }
  // stored peaks, chunk by chunk, as each chunk's counts arrive
  int64_t base = 0;
  bool over = false;
  for (int c = 0; c < K && e == cudaSuccess; ++c) {
    const int64_t e0 = ce[c], n = ce[c + 1] - ce[c];
    e = cudaEventSynchronize(hp.ev[3 * c + 2]);
    if (e != cudaSuccess) break;
    int64_t tot = 0;
    for (int64_t i = e0; i < e0 + n; ++i) {
      h_peak_off[i] += base;
      tot += std::min<int64_t>(h_npeaks[i], (int64_t)mp);
    }
    if (base + tot > h_peaks_cap) over = true;
    // the chunk's packing finished before its counts were copied, which the host has seen
    e = mark(c, 7, hp.peaks);
    if (e == cudaSuccess && !over && tot > 0)
      e = cudaMemcpyAsync(h_peaks + base, d_dense + e0 * mp, sizeof(hough_peak) * (size_t)tot,
                          cudaMemcpyDeviceToHost, hp.peaks);
    if (e == cudaSuccess) e = mark(c, 8, hp.peaks);
    base += tot;
  }
  h_peak_off[n_events] = base;
  int32_t flags = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&flags, d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, hp.out);
  // every stream is drained on every exit: no copy touches the caller's buffers afterwards
  const cudaError_t s1 = cudaStreamSynchronize(hp.in), s2 = cudaStreamSynchronize(hp.out);
  const cudaError_t s3 = cudaStreamSynchronize(hp.peaks), s4 = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = s1 != cudaSuccess ? s1 : s2 != cudaSuccess ? s2 : s3 != cudaSuccess ? s3 : s4;
  if (e != cudaSuccess) return cuda_fail(e);
  if (timed) {  // stage busy times summed over the chunks, and the span of the whole call
    float acc[HOUGH_HOST_STAGES] = {};
    float last = 0.f;
    bool ok = true;
    auto el = [&](cudaEvent_t a, cudaEvent_t z) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, a, z) != cudaSuccess) ok = false;
      return ms;
    };
    for (int c = 0; c < K && ok; ++c) {
      cudaEvent_t* t = hp.tev + kStageEvents * c;
      acc[HOUGH_HOST_STAGE_H2D] += el(t[0], t[1]);
      acc[HOUGH_HOST_STAGE_KERNELS] += el(t[2], t[3]);
      acc[HOUGH_HOST_STAGE_PACK] += el(t[3], t[4]);
      acc[HOUGH_HOST_STAGE_D2H] += el(t[5], t[6]);
      acc[HOUGH_HOST_STAGE_PEAKS_D2H] += el(t[7], t[8]);
      last = std::max(last, std::max(el(hp.t_start, t[6]), el(hp.t_start, t[8])));
    }
    acc[HOUGH_HOST_STAGE_SPAN] = last;
    cudaGetLastError();  // a failed elapsed-time query only invalidates the stage times
    if (ok) {
      std::memcpy(hp.stage_ms, acc, sizeof(acc));
      hp.stage_valid = true;
    }
  }
  if (over) return HOUGH_EWORKSPACE;
  return flags ? HOUGH_EDEVICE : HOUGH_OK;
}

void hough_set_host_timing(int32_t on) { host_pipe_raw().timing = on != 0; }

int hough_host_stage_ms(float* ms, int32_t n) {
  if (!ms || n < 0) return HOUGH_EINVAL;
  HostPipe& hp = host_pipe_raw();
  if (!hp.stage_valid) return HOUGH_EINVAL;
  for (int i = 0; i < n && i < HOUGH_HOST_STAGES; ++i) ms[i] = hp.stage_ms[i];
  return HOUGH_OK;
}

int hough_status(const int32_t* d_status, void* stream, int32_t* host_flags) {
  if (!d_status || !host_flags) return HOUGH_EINVAL;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail(e);
  e = cudaMemcpy(host_flags, d_status, sizeof(int32_t), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e);
  return *host_flags ? HOUGH_EDEVICE : HOUGH_OK;
}

const char* hough_strerror(int code) {
  switch (code) {
    case HOUGH_OK: return "ok";
    case HOUGH_EINVAL: return "invalid argument (null pointer, negative count or misaligned buffer)";
    case HOUGH_EPARAM: return "parameters out of range";
    case HOUGH_ESMEM: return "shape does not fit shared memory";
    case HOUGH_ECUDA: return "CUDA runtime error";
    case HOUGH_EWORKSPACE: return "workspace too small";
    case HOUGH_ETIMEDOUT: return "bounded wait timed out";
    case HOUGH_EFULL: return "no free serving slot";
    case HOUGH_EDEVICE: return "device status flags set";
    case HOUGH_F_BAD_HIT: return "hit at r = 0 or beyond 2^24 um";
    case HOUGH_F_BAD_OFFSETS: return "event offsets invalid";
    case HOUGH_F_PEAK_OVERFLOW: return "more peaks than max_peaks";
    case HOUGH_F_EVENT_TOO_LARGE: return "event has more than HOUGH_MAX_EVENT_HITS hits";
    case HOUGH_F_TIMEOUT: return "micro-batch did not complete in time";
    case HOUGH_F_LAUNCH_FAILED: return "micro-batch could not be enqueued or failed on the device";
    default: return "unknown code";
  }
}

int hough_last_cuda_error(void) { return g_last_cuda; }

int hough_selftest_bin(int32_t n_rho, int64_t rho_lo, int64_t rho_hi, unsigned long long* d_mismatch,
                       void* stream) {
  if (!d_mismatch || n_rho < 4 || n_rho > 1024 || rho_hi < rho_lo) return HOUGH_EINVAL;
  cudaError_t e = launch_selftest_bin(n_rho, rho_lo, rho_hi, d_mismatch, (cudaStream_t)stream);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_selftest_fpbin(int32_t n_theta, int32_t n_rho, uint64_t seed, int64_t n_samples, unsigned long long* d_out,
                         void* stream) {
  hough_params p{n_theta, n_rho, 1, 1, 1, 0, 0, 0, HOUGH_PEAK_LOCAL_MAX, 0, 1, 0};
  Plan pl;
  if (!d_out || n_samples < 0 || make_plan(&p, pl) != HOUGH_OK) return HOUGH_EINVAL;
  mp_consts(pl, n_rho);  // the mirror-pair estimate is checked whatever layout the plan chose
  TrigTable trig;
  host_trig(n_theta, &trig);
  cudaError_t e = launch_selftest_fpbin(pl, trig, seed, n_samples, d_out, (cudaStream_t)stream);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

int hough_probe_smem_atomics(int32_t mode, int32_t ctas_per_sm, int32_t threads, int32_t smem_bytes, int32_t iters,
                             unsigned long long* d_sink, void* stream) {
  if (!d_sink || mode < 0 || mode > 4 || ctas_per_sm < 1 || threads < 32 || threads > 1024 || (threads % 32) ||
      smem_bytes < 4096 || smem_bytes > kSmemBudget || iters < 1)
    return HOUGH_EINVAL;
  cudaError_t e = launch_probe_atomics(mode, ctas_per_sm, threads, smem_bytes, iters, d_sink, (cudaStream_t)stream);
  return e == cudaSuccess ? HOUGH_OK : cuda_fail(e);
}

}  // extern "C"
