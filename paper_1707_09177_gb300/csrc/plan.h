// Host-side planning of the FFT passes, shared by every entry point that
// launches them (the context-owning solvers and the allocation-free filter):
// the radix decomposition of a transform length, the Stockham stage table,
// and the tile width / block size / shared-memory row stride of a pass. The
// pass kernels take their fixed-plan fast path only when a plan equals the
// compile-time plan for its length, so every launcher must build plans the
// same way; keeping one copy here guarantees that.
#pragma once

#include <cmath>
#include <cstddef>

#include "args.h"

namespace gad {

// Padded shared-memory index of element i (one pad slot every 16 elements).
inline int phys_h(int i) { return i + (i >> 4); }

inline bool smooth23(long long n) {
  if (n < 1) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  return n == 1;
}

// Largest power of two dividing n (capped at 2^20).
inline int pow2_part(long long n) {
  int p = 1;
  while (n % 2 == 0 && p < (1 << 20)) { n /= 2; p *= 2; }
  return p;
}

// Elements per FFT thread: 24 when the length has a factor 3, else 16.
inline int pick_E(int L) { return (L % 3 == 0) ? 24 : 16; }

constexpr int kMaxStages = 5;       // the kernels unroll at most 5 stages

// Elements per FFT thread on a grid too small to fill the GPU (choose_pass):
// two or four times as many threads, each with a shorter chain; 0: the default.
// A batch of the same grid takes the same count (see choose_pass), so it must
// not be the slower one there. 12 elements, and 4 in float64, whose passes are
// bound by arithmetic, are not; float32 passes of powers of two are bound by
// shared memory, which the radices of 4 elements (4 and 2) pass through up to
// twice as often: one 64^3 field filters in 39 us with 4 elements and in 51 with
// 16, but 64 of them in 279 and 237, 32 fields of 512^2 in 136 and 72.
inline int small_E(int L, size_t csize) { return (L % 3 == 0) ? 12 : csize == 16 ? 4 : 0; }

// Balanced radix list for a length L and E elements per thread: the factors 3
// first, then the power of two split into as few stages of at most 2^4 (E =
// 16), 2^3 (E = 24) or 2^2 (E = 4, 12) as possible, the larger radices first. Writes at most
// kMaxStages radices into rad and returns their number, or 0 when L is not
// 2^a 3^b, a radix does not divide E, or more stages would be needed.
inline int radices_for(int L, int E, int* rad) {
  int n = L, a = 0, b = 0;
  while (n > 1 && n % 2 == 0) { n /= 2; ++a; }
  while (n > 1 && n % 3 == 0) { n /= 3; ++b; }
  if (n != 1 || (a == 0 && b == 0)) return 0;
  if (b > 0 && E % 3 != 0) return 0;
  const int maxlog = (E % 16 == 0) ? 4 : (E % 8 == 0) ? 3 : 2;
  const int ns = a > 0 ? (a + maxlog - 1) / maxlog : 0;
  if (b + ns > kMaxStages) return 0;
  int k = 0;
  for (int i = 0; i < b; ++i) rad[k++] = 3;
  for (int i = 0; i < ns; ++i) rad[k++] = 1 << (a / ns + (i < a % ns ? 1 : 0));
  for (int i = 0; i < k; ++i)
    if (E % rad[i] != 0) return 0;
  return k;
}

// Radices of the float32 plans of lengths with a factor 3 (E = 12): the fewest
// stages from 12, 6, 4, 3 and 2 (ties go to the smaller sum), so that a factor
// 3 shares a stage with a power of two instead of taking one of its own (288:
// 4 6 12 instead of 3 3 8 4). Powers of two
// come first: the first stage writes with a stride of its radix, which is free
// of bank conflicts for them. n = 0 when there is no such plan.
struct RadixSeq {
  int n = 0, sum = 0;
  int r[kMaxStages] = {};
};

constexpr RadixSeq fused_search(int L, int E, int top, int depth) {
  RadixSeq best{};
  if (L == 1 || depth == kMaxStages) return best;
  const int cand[5] = {12, 6, 4, 3, 2};
  for (int i = 0; i < 5; ++i) {
    const int c = cand[i];
    if (c > top || E % c != 0 || L % c != 0) continue;
    RadixSeq s = fused_search(L / c, E, c, depth + 1);
    if (L / c != 1 && s.n == 0) continue;
    s.r[s.n] = c;
    s.n += 1;
    s.sum += c;
    if (best.n == 0 || s.n < best.n || (s.n == best.n && s.sum < best.sum)) best = s;
  }
  return best;
}

constexpr RadixSeq fused_radices(int L, int E) {
  RadixSeq s = fused_search(L, E, 12, 0), o{};
  for (int pow2 = 1; pow2 >= 0; --pow2)
    for (int i = 0; i < s.n; ++i)                 // s.r ascends
      if ((s.r[i] % 3 != 0) == (pow2 != 0)) o.r[o.n++] = s.r[i];
  return o;
}

// Lengths of those plans, at 12 elements per thread: 64 registers and 4 blocks
// per SM, with nothing spilled in the kernels compiled for 2^a 3 and 2^a 9
// (kernels_fused.cu) and 64 bytes in the filter pass of the general stages that
// the other lengths (108, 162, 216, 324, 432, 648, 864, ..) run; at 24 elements
// it spills 900 bytes per thread at 80 registers. The general stages gain from
// the fewer stages too, 24 separate against 12 fused elements, us: filter of
// 216^3 x 3 783 / 545, 324^3 x 3 2539 / 2009, 864^2 x 8 142 / 88, 1728^2 x 8
// 471 / 383. A transposed tile of more than 768 elements per row would hold
// fewer than the four rows of a 32-byte sector in 256 threads and keeps 24
// elements.
constexpr bool fused_length(int L) { return L % 3 == 0 && L >= 36 && L <= 2304 && fused_radices(L, 12).n > 0; }

// Key of a plan: its element count, odd for the fused radices.
inline int plan_E(int L, int E, size_t csize) { return csize == 8 && E == 12 && fused_length(L) ? 13 : E; }

// Stockham stage table for the radices rad[0..nrad) (in that order) over the
// plan's twiddle table `tab` (see FftPlan; fill it with plan_twiddles).
inline bool make_fft_from(int L, const int* rad, int nrad, const void* tab, FftPlan& fp) {
  if (nrad < 1 || nrad > kMaxStages) return false;
  fp = FftPlan{};
  fp.L = L;
  fp.nst = nrad;
  fp.tw = tab;
  long long ns = 1, off = 0;
  for (int q = 0; q < nrad; ++q) {
    FftStage& s = fp.st[q];
    s.radix = rad[q];
    s.ns = (int)ns;
    s.tw_off = (int)off;
    s.rcp_lr = 1.0f / (float)(L / rad[q]);
    s.rcp_ns = 1.0f / (float)ns;
    off += (long long)(rad[q] - 1) * ns;
    ns *= rad[q];
  }
  return ns == L;
}

// Radices of the plan of length L for E elements per thread; `reversed` gives
// them in reverse order (the filter pass's inverse transform, whose first
// stage meets the forward transform's last stage in registers). Returns the
// number of stages, 0 when there is no plan.
inline int plan_radices(int L, int E, bool reversed, int* rad) {
  int n;
  if (E & 1) {
    const RadixSeq s = fused_radices(L, E - 1);
    n = s.n;
    for (int i = 0; i < n; ++i) rad[i] = s.r[i];
  } else {
    n = radices_for(L, E, rad);
  }
  if (reversed)
    for (int i = 0; i < n / 2; ++i) {
      const int t = rad[i];
      rad[i] = rad[n - 1 - i];
      rad[n - 1 - i] = t;
    }
  return n;
}

inline bool make_fft(int L, int E, const void* tab, FftPlan& fp, bool reversed = false) {
  int rad[kMaxStages];
  const int n = plan_radices(L, E, reversed, rad);
  return n > 0 && make_fft_from(L, rad, n, tab, fp);
}

// The plan's twiddle table (L - 1 complex entries, interleaved re, im) in
// long double, rounded to T: stage q, factor r, butterfly k at
// tw_off(q) + (r - 1) ns(q) + k holds exp(-2 pi i r k / (rad[q] ns(q))); the
// quarter and half turns are exact.
template <typename T>
inline void plan_twiddles(const int* rad, int nrad, T* out) {
  const long double two_pi = 6.283185307179586476925286766559005768L;
  long long ns = 1, off = 0;
  for (int q = 0; q < nrad; ++q) {
    const long long len = (long long)rad[q] * ns;
    for (int r = 1; r < rad[q]; ++r)
      for (long long k = 0; k < ns; ++k) {
        const long long m = ((long long)r * k) % len;
        long double c, sn;
        if (m == 0) { c = 1; sn = 0; }
        else if (4 * m == len) { c = 0; sn = -1; }
        else if (2 * m == len) { c = -1; sn = 0; }
        else if (4 * m == 3 * len) { c = 0; sn = 1; }
        else {
          const long double ang = two_pi * (long double)m / (long double)len;
          c = cosl(ang);
          sn = -sinl(ang);
        }
        const long long e = off + (long long)(r - 1) * ns + k;
        out[2 * e] = (T)c;
        out[2 * e + 1] = (T)sn;
      }
    off += (long long)(rad[q] - 1) * ns;
    ns *= rad[q];
  }
}

// Odd shared-memory row stride (complex units) of a tile row of `slots`
// elements.
inline int tile_ld(int slots) {
  int ld = phys_h(slots - 1) + 1;
  if ((ld & 1) == 0) ++ld;
  return ld;
}

struct TileShape {
  int E = 0, W = 0, T = 0, ld = 0;
  size_t smem = 0;
};

// Picks the tile width W (a power of two dividing `div`, or any power of two
// when div = 0) whose block size T = W*L/E is closest to 256 threads, with at
// most 100 KB of shared memory (rows of `slots` elements of csize bytes).
inline bool choose_tile(int L, int E, int slots, int div, size_t csize, TileShape& ts) {
  const int ld = tile_ld(slots);
  int bestW = 0, bestT = 0;
  double bestScore = 1e30;
  for (int W = 1; W <= 4096; W *= 2) {
    if (div > 0 && div % W != 0) break;
    const long long tot = (long long)W * L;
    if (tot % E != 0) continue;
    const long long T = tot / E;
    if (T < 1 || T > 256) continue;
    const size_t smem = (size_t)W * ld * csize;
    if (smem > 100 * 1024) continue;
    const double score = std::fabs(std::log2((double)T / 256.0));
    if (score < bestScore - 1e-9) { bestScore = score; bestW = W; bestT = (int)T; }
  }
  if (!bestW) return false;
  ts.E = E;
  ts.W = bestW;
  ts.T = bestT;
  ts.ld = ld;
  ts.smem = (size_t)bestW * ld * csize;
  return true;
}

// Blocks below which a launch cannot fill the GPU with the default tile: of one
// field where it has dots, of all its fields where it has none. Two blocks per
// SM for the launches without dots: with one, 32 fields of 192^2 float64 filter
// in 259 us, with two in 198, with four 64^3 float32 x 4 takes 54 against 51 us.
// Four for float64 powers of two, bound by the float64 rate of the busiest SM
// (16 fields of 256^2 148 us against 154, four of 64^3 159 against 177); lengths
// with a factor 3 lose by it there (16 fields of 288^2 270 against 214).
constexpr int kWantBlocks = 152;
inline int want_launch(int L, size_t csize) { return (csize == 16 && L % 3 != 0 ? 4 : 2) * 152; }
// Complex elements per field below which a pass takes small_E: with the default
// count less than a third of the GPU's threads would have work. For powers of
// two (float64) a quarter of that: one 64^3 field (135,168 elements) filters in
// 68 us with 4 elements and 111 with 16, but the closure of 32 such velocities
// takes 6.6 against 6.1 ms; 256^2 (33,024): 39 against 88 us for one, 2.10
// against 1.93 ms for 256 (2.06 before narrow tiles); 32^3 (17,408): 49 against
// 95 us for one, closure of 128 velocities 3.06 against 2.75 ms (2.89 before).
constexpr long long kSmallElems = 152 * 64 * 16, kSmallElemsPow2 = kSmallElems / 4;

// Row stride of a tile of W rows that is stored or loaded transposed (the W
// values of one wavenumber by consecutive threads): the 128 bytes that a
// shared-memory phase moves are then W rows of 128/csize/W consecutive
// elements, which fall into distinct banks when the stride is that count
// modulo 128/csize (an odd stride when a phase holds one element per row).
// With the odd stride of tile_ld, W = 4 rows of float2 met in 7 of 16 bank pairs.
inline int transposed_ld(int ld, int W, size_t csize) {
  const int B = (int)(128 / csize);
  if (W >= B || W < 2) return ld;
  while (ld % B != B / W) ++ld;
  return ld;
}

// Elements per thread and tile of a pass over `nseq` sequences of length L
// per field. Default: 12 (fused_length) or pick_E(L) elements and choose_tile's
// blocks narrowed to about `want_T` threads. Small grids get small_E(L) and
// narrower tiles, the widest that still gives enough blocks, down to rows of 32
// bytes (one sector) in the transposed spectra and to one warp.
// A field's result must not depend on the batch it is solved in. The element
// count (it sets the radices and with them the rounding) and the tile of a
// launch with dots (it sets the order of their sums) therefore follow the
// field alone; `batch` = 0 asks for that tile. The tile of a launch without
// dots changes no result and follows the blocks of all its `batch` fields:
// narrow tiles cost a launch that fills the GPU without them (float64 closure
// of four 72 x 72 x 96 velocities 2.81 ms with the field's tiles, 2.60 with the
// launch's, filter of 32 fields 96 x 72 x 72 3.79 and 3.54 ms).
inline bool choose_pass(int L, int slots, int div, long long nseq, bool transposed, size_t csize, TileShape& ts,
                        int want_T = 256, int batch = 0) {
  const int E0 = csize == 8 && fused_length(L) && !(transposed && L > 768) ? 12 : pick_E(L);
  if (!choose_tile(L, E0, slots, div, csize, ts)) return false;
  auto done = [&]() {
    if (transposed) {
      ts.ld = transposed_ld(ts.ld, ts.W, csize);
      ts.smem = (size_t)ts.W * ts.ld * csize;
    }
    return true;
  };
  // the default tile narrowed to about `want_T` threads, rows of 32 bytes at least
  while (ts.T > want_T && ts.W > 1 && (!transposed || ts.W * csize > 32)) {
    ts.W /= 2;
    ts.T /= 2;
    ts.smem /= 2;
  }
  auto enough = [&](int W) {
    const long long n = (nseq + W - 1) / W;
    return batch > 0 ? n * batch >= want_launch(L, csize) : n >= kWantBlocks;
  };
  int rad[kMaxStages];
  int E = E0;
  if ((nseq + ts.W - 1) / ts.W < kWantBlocks && nseq * L < (L % 3 == 0 ? kSmallElems : kSmallElemsPow2) &&
      small_E(L, csize) > 0 && radices_for(L, small_E(L, csize), rad) > 0)
    E = small_E(L, csize);
  if (E == E0 && enough(ts.W)) return done();
  TileShape best;
  for (int W = 4096; W >= 1; W /= 2) {
    if (div > 0 && div % W != 0) continue;
    const long long tot = (long long)W * L;
    if (tot % E != 0 || tot / E > 256) continue;
    const size_t smem = (size_t)W * ts.ld * csize;
    if (smem > 100 * 1024) continue;
    const bool narrow = tot / E < 32 || (transposed && W * csize < 32);
    if (best.W && narrow) break;
    best.E = E;
    best.W = W;
    best.T = (int)(tot / E);
    best.ld = ts.ld;
    best.smem = smem;
    if (enough(W) && (batch == 0 || best.T <= want_T)) break;
  }
  if (best.W) ts = best;
  return done();
}

// The tiles of every pass of a grid: forward x, inverse x and filter with and
// without dots, both y passes (3D).
struct GridTiles {
  TileShape xf, xi, xi_nodots, fl, fl_nodots, y;
};

inline bool grid_tiles(int nx, int ny, int nz, int batch, size_t csize, GridTiles& t) {
  const int M = nx / 2, kxn = M + 1, L = nz > 1 ? nz : ny, dx = pow2_part(ny);
  const long long rows = (long long)ny * nz, seqs = nz > 1 ? (long long)kxn * ny : kxn;
  return choose_pass(M, M + 1, dx, rows, true, csize, t.xf, M % 3 == 0 ? 128 : 64, batch) &&
         choose_pass(M, M + 1, dx, rows, true, csize, t.xi, 256) &&
         choose_pass(M, M + 1, dx, rows, true, csize, t.xi_nodots, 256, batch) &&
         choose_pass(L, L, 0, seqs, false, csize, t.fl, 128) &&
         choose_pass(L, L, 0, seqs, false, csize, t.fl_nodots, 128, batch) &&
         (nz == 1 || choose_pass(ny, ny, pow2_part(nz), (long long)kxn * nz, true, csize, t.y, 256, batch));
}

// Shared-memory layout of a cluster solve (cluster.cuh): the rows of a 2D field
// and its sequences along y spread over `csize` CTAs.
struct ClusterShape {
  int csize = 0, threads = 0, buf = 0, ldx = 0, ldl = 0, kc = 0;
  size_t smem = 0;
};

constexpr size_t kClusterSmem = 224 * 1024;   // dynamic shared memory a CTA may take
constexpr int kClusterE = 24;                 // element count whose plans have radices of at most 8

// Rounds of clusters that a batch may take (the GPU holds 14 of 16 CTAs at a
// time); more fields take the pass kernels. A cluster is a chain of latencies
// and a further round of them as long again, where the pass kernels hardly
// notice more fields. 3 BiCGSTAB passes, cluster / pass kernels, us: 256^2
// float32 1 field 197 / 334, 14 223 / 351, 16 356 / 326, 40 545 / 414; 128^2
// float32 16 to 28 fields 290 / 400, 40 400 / 403; 64^2 float64 14 fields
// 343 / 431, 16 604 / 431, 128 2660 / 825.
inline int cluster_rounds(long long points, size_t csize) { return csize == 8 && points <= 128 * 128 ? 2 : 1; }

// False when the grid is not one for a cluster: it takes the pass kernels.
// Measured per pass of a single field, cluster against pass kernels: CG float32
// 256^2 18 against 40 us; Van Cittert float64 128^2 36 against 53 us (the
// float64 rate of 16 SMs, two lanes per clock each, is the larger part of it and
// grows with the points). The float64 limit lies where powers of two stop
// gaining (10 CG passes, us: 128^2 545 / 685, 128 x 256 766 / 706, 256^2 1324 /
// 719); float32 gains up to about 400^2 (256^2 265 / 508, 288^2 320 / 422, 384^2
// 401 / 459), its limit is where the gain is largest. 3D fields have four more transposing steps through
// shared memory and gain nothing (64^3 float32 CG: 53 against 50 us).
constexpr long long kClusterPoints32 = 256 * 256, kClusterPoints64 = 128 * 128;

inline bool cluster_shape(int nx, int ny, int nz, size_t csize, ClusterShape& cs) {
  const int M = nx / 2, kxn = M + 1;
  const long long P = (long long)nx * ny;
  if (nz > 1 || P > (csize == 16 ? kClusterPoints64 : kClusterPoints32)) return false;
  int rad[kMaxStages];
  if (radices_for(M, kClusterE, rad) == 0 || radices_for(ny, kClusterE, rad) == 0) return false;
  // as many CTAs as divide the rows, at most 16, each with at least 1024 bytes of them
  int C = 1;
  while (C < 16 && ny % (2 * C) == 0 && P * (long long)csize / (4 * C) >= 1024) C *= 2;
  const int own = ny / C;
  cs.csize = C;
  cs.kc = (kxn + C - 1) / C;
  cs.ldx = tile_ld(M);
  cs.ldl = tile_ld(ny);
  long long buf = (long long)own * cs.ldx;
  const long long bl = (long long)cs.kc * cs.ldl, by = (long long)kxn * own;
  if (bl > buf) buf = bl;
  if (by > buf) buf = by;
  const long long tabs = M / 2 + 1 + M - 1 + ny - 1;
  const long long bytes = (3 * buf + tabs) * (long long)csize + (csize == 16 ? (long long)cs.kc * ny * 8 : 0);
  if (bytes > (long long)kClusterSmem) return false;
  cs.buf = (int)buf;
  cs.smem = (size_t)bytes;
  cs.threads = own * M > 2048 ? 512 : 256;
  return true;
}

}  // namespace gad
