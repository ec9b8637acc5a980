// Launch rules that are arithmetic alone: which tile of a kernel a launch of
// given sizes takes.  Plain C++ (no CUDA), so that they can be checked on any
// host.
#pragma once
#include <limits.h>
#include <stddef.h>

namespace wmg {

// ------------------------------------------------------------------ CUDA-core coarse stencil
// A unit is a group of bv consecutive sites (one 16-byte load of the operator)
// and ir consecutive rows; a CTA takes lb consecutive units and rb right-hand
// sides.  Units are numbered with `pitch` of them per ir rows: as many as there
// are site groups, or rounded up to whole CTAs (units without sites are idle).
struct CoarseShape {
  int ir, rb, lb;
  long pitch;
};
constexpr long kCoarseLarge = 65536;
// The tiles that have a kernel, for elements of `elem` bytes.
constexpr bool coarse_has(int elem, int bv, int ir, int rb, int lb) {
  if (elem == 16) return ir == 1 ? rb <= 2 : ir == 4 && rb == 1 && lb == 32;
  if (rb == 2 && bv == 1) return false;
  if (lb == 32) return ir == (rb > 1 ? rb : (bv == 1 ? 4 : 2));
  return ir == 1 || (lb == 16 && (ir == 2 || rb == 4));
}
inline int coarse_bv(size_t elem, long V) {
  const int bv = (int)(16 / elem);
  return V % bv ? 1 : bv;  // a row of sites that does not start on 16 bytes: element by element
}
inline long coarse_ctas(long n, int ir, int lb, long pitch) { return ((n + ir - 1) / ir * pitch + lb - 1) / lb; }

// CTAs of a launch per right-hand side, at most (sizes the reduction partials;
// not below the count this function has always given).
inline long coarse_blocks(long n, long V, int nrhs) {
  const long outs = n * V;
  long G = 1;
  while (G < 32 && outs * G < 65536) G *= 2;
  const long most = (outs * G + 127) / 128;
  const long per16 = (V + 15) / 16 * n, per32 = (V + 31) / 32 * n;
  const long four = (V + 31) / 32 * ((n + 3) / 4), two = V % 2 ? 0 : (V + 63) / 64 * ((n + 1) / 2);
  const long c = outs < kCoarseLarge ? per16 : (nrhs > 1 ? per32 : (four > two ? four : two));
  return c > most ? c : most;
}

// FP64 is bound by its arithmetic pipe, which a warp's instruction occupies for 16
// cycles, so the shape is the one whose fullest SM issues the fewest: those of a
// CTA's eight warps over their slices of the 9 n terms, the additions that join
// the slices, and about 15 more per CTA, times the CTAs of the fullest SM.  That
// is within 5 % of the times measured above 20 us.  Near ties go to the larger
// tile, which reads the operator less often.  (Tiles of 16 or 32 sites of one
// row, chosen by the CTA count alone, left 28 of 64 lanes idle on 36 sites and 30
// of 32 on two: n = 64, 24 right-hand sides, 409 and 225 us.)
//
// FP32 and 16 bits: the most rows (4, 2, 1) that leave two CTAs per SM -- rows
// share the vector's loads, but few CTAs leave the GPU idle (32 sites, n = 48, 12
// right-hand sides, FP32: 10.6 us with one row, 16.7 with four; 512 sites: 103
// with two, 76 with four; one right-hand side 20.7 with two, 27.8 with one); with
// one row the tile narrows while not even a quarter of the SMs has a CTA.  A row
// fills whole CTAs, which keeps a warp's loads contiguous, unless that makes half
// as many units again (two sites, n = 64, 64 right-hand sides: 43 us in whole
// CTAs).  From kCoarseLarge outputs on 32 units, and for one right-hand side rows
// enough to keep the reduction partials few.
inline CoarseShape coarse_shape(size_t elem, long n, long V, int nrhs, int sms) {
  const int bv = coarse_bv(elem, V);
  const long groups = V / bv;
  const bool large = n * V >= kCoarseLarge;
  auto pitch = [&](int lb) {
    const long whole = (groups + lb - 1) / lb * lb;
    return 2 * whole >= 3 * groups ? groups : whole;
  };
  if (large && nrhs == 1) return {bv == 1 ? 4 : 2, 1, 32, groups};
  const long bound = coarse_blocks(n, V, nrhs);
  if (elem == 16) {
    CoarseShape best = {1, 1, 32, groups};
    double least = 0;
    for (int rb = nrhs > 1 ? 2 : 1; rb >= 1; --rb)
      for (int lb = 32, lg = 0; lb >= 4; lb /= 2, ++lg) {
        const long ctas = coarse_ctas(n, 1, lb, groups);
        if (ctas > bound) break;
        const long per_sm = (ctas * ((nrhs + rb - 1) / rb) + sms - 1) / sms;
        const double cost = (double)per_sm * (rb * (32 * ((9 * n * lb + 255) / 256) + 16 * lg + 24) + 15);
        if (least == 0 || cost < 0.97 * least) {
          best = {1, rb, lb, groups};
          least = cost;
        }
      }
    return best;
  }
  const int rb = nrhs == 1 ? 1 : (nrhs == 2 && bv > 1 ? 2 : 4);
  if (large) return {rb, rb, 32, pitch(32)};
  const long gy = (nrhs + rb - 1) / rb;
  for (int ir = rb == 4 ? 4 : 2; ir > 1; ir /= 2)
    if (coarse_ctas(n, ir, 16, pitch(16)) * gy >= 2L * sms) return {ir, rb, 16, pitch(16)};
  int lb = 16;
  while (lb > 4 && coarse_ctas(n, 1, lb, pitch(lb)) * gy * 4 < sms && coarse_ctas(n, 1, lb / 2, pitch(lb / 2)) <= bound)
    lb /= 2;
  return {1, rb, lb, pitch(lb)};
}

// ------------------------------------------------------------------ coarsest product
// Right-hand sides up to which the row form runs: it reads the matrix once for
// each, the tiled product once for all.  FP32, N = 1536: 16 right-hand sides 37 us
// against 50, 24 53 against 56; N = 4096 (a matrix as large as the L2): 12 279
// against 321, 16 368 against 338; N = 8192: 12 1053 against 1259, 16 1393 against
// 1327.  FP64: both are bound by arithmetic, of which the tiled product does 64
// right-hand sides' in any case (N = 1536, 24: 420 against 1320).
inline int matvec_most(int prec, long N) { return prec == 0 || N <= 3584 ? 16 : 12; }
// FP64: rows of a CTA, four or two, by the fuller of the SMs (N = 2048: 512 CTAs of four are four on some SMs).
inline int matvec_rows_per_cta(long N, int nrhs, int sms) {
  auto time = [&](long rows) { return ((N + rows - 1) / rows * nrhs + sms - 1) / sms * rows; };
  return 100 * time(2) < 97 * time(4) ? 2 : 4;
}

// ------------------------------------------------------------------ fine stencil
// Threads an SM is to hold, one thread per site, for elements of `elem` bytes,
// i.e. the register budget (65,536 / threads).  Measured (us per launch; "-":
// the compiler's own choice of 96-102, 144 in FP64, 180 for two right-hand sides
// per thread):
//   FP32 plain, 32^3 x 64: - 168, 512 170, 640 158, 768 162
//   FP32 plain, 16^3 x 32, 12 right-hand sides: - 115, 640 103 (wide loads included)
//   16-bit plain: 512 135 (384 152, 640 136, 768 138) at 32^3 x 64
//   two right-hand sides per thread, FP16, 12: - 105, 384 90.5, 512 90.3 (spills)
//   fused dots, FP16, 12, in several tiles per CTA: - 134, 512 129, 640 134
//   FP64, 9 x 7 x 5 x 11, 12 right-hand sides (336 CTAs): 256 114 (a second wave), 384 101; bound by its arithmetic
//   pipe, 16^3 x 32 takes 233 with either
constexpr int stencil_threads(int elem, int nr, bool dots) {
  return elem == 16 ? 384 : (nr == 2 ? 384 : (elem == 8 && !dots ? 640 : 512));
}

// Tiles of 128 sites per CTA of a launch with fused dots: `lanes` rows of `tiles`
// tiles (a row is one or two right-hand sides), `per_sm` CTAs on an SM.  Each tile
// keeps its own partial sums, so the result does not depend on the choice.
//
// FP32: a CTA's start and its last reduction step take about 0.3 tile times
// whatever its tiles, and a wave as long as its longest CTA: the largest number
// within 3 % of the shortest waves, at most 24, or 32 in a single wave.  16 x 8 x
// 8 x 16, 64 right-hand sides: 88 us (one tile per CTA 109, fourteen, which are
// 640 CTAs on 608 places, 123); 24^4, 24 right-hand sides: one tile 792, eighteen
// 658; 16^3 x 32, 12, two right-hand sides per thread: 184 -> 129 with its own
// lanes and places instead of those of one per thread.
// 16 bits, where a tile is longer: one below eight waves, else about four, in
// whole waves on average (16^3 x 32, FP16, 12: 134 with one tile, 127; the rule
// above 124, but 112 instead of 108 on 12^4 with 64).
inline int dot_tiles(long tiles, long lanes, int per_sm, int sms, int elem) {
  const long total = tiles * lanes, places = (long)per_sm * sms;
  if (elem != 8) {
    if (total < places * 8) return 1;
    const long waves = total / (places * 4);
    return (int)((total + places * waves - 1) / (places * waves));
  }
  auto time = [&](int k) {
    const long waves = ((tiles + k - 1) / k * lanes + places - 1) / places;
    return k > 24 && waves > 1 ? LONG_MAX / 100 : waves * (10 * k + 3);
  };
  const int most = 32;
  long least = time(1);
  for (int k = 2; k <= most; ++k) least = time(k) < least ? time(k) : least;
  int best = most;
  while (100 * time(best) > 103 * least) --best;
  return best;
}

// ------------------------------------------------------------------ Gram-Schmidt dots
// Blocks per lane (a chunk of eight vectors and a right-hand side) for `tiles`
// tiles of 256 elements: at least four tiles each, one block per SM; where few
// lanes leave the SMs with less than four FP32 or two FP64 blocks, more of them as
// long as each has eight (FP32) or sixteen tiles.  25 M elements, up to 8 vectors,
// one right-hand side: FP32 701 -> 272 us, FP64 1877 -> 1350 (four blocks on
// 393,216 elements: 43 us instead of 29).  FP32 blocks stay whole waves of four
// per SM (1.5 M elements, 40 vectors, five lanes: 88 us with a block per SM and lane, 77).
inline int multidot_grid(long tiles, int lanes, int elem, int sms, int most) {
  const long few = (tiles + 3) / 4, each = elem == 16 ? 16 : 8;
  const long want = elem == 16 ? 2 : 4, cap = sms * ((want + lanes - 1) / lanes);
  long b = few;
  if (b > sms) {
    b = tiles / each > sms ? tiles / each : sms;
    b = b > cap ? cap : b;
    if (elem != 16 && lanes > 4) b = 4L * sms * (lanes / 4) / lanes;
  }
  b = b > most ? most : b;
  return (int)(b < 1 ? 1 : b);
}

// ------------------------------------------------------------------ chained launches
// Whether a launch may start early (launch_chain) without crowding.  The CTAs of
// an early launch take the places that its predecessor leaves.  A second grid of
// the same size fits beside the first up to half of the GPU's places; above, its
// last CTAs go wherever a CTA of the predecessor ends first, and where even
// placement means two or three per SM, some SMs get one more than the others
// (`per_sm` places of an SM; FP64 prolongation, 512 CTAs on 6 x 152 places: 23.0
// -> 29.9 us; FP64 restriction, 432 on 5 x 152: 8.4 -> 10.1; 486 to 576: no
// difference).  Nearly full grids have the most CTAs on every SM anyway.
inline bool chain_fits(long ctas, int per_sm, int sms) {
  const long places = (long)per_sm * sms;
  return 2 * ctas <= places || 4 * ctas > 3 * places;
}

}  // namespace wmg
