// irs_brute.cu -- plain ("ordinary GPU IRS") ray pass: every ray sums every
// lens (arXiv:2204.10871, Sec. 1 and the "ordinary GPU-based IRS code" of
// Sec. 3.1), with the rectangular negative sheet of Eq. (alpha1) / Appendix A.
//
// Layout of the work: the ray lattice is cut into tiles of 32 x 64 rays.  A
// CTA of 64/R warps owns one tile at a time (persistent grid); lane l takes
// column i0 + l and each warp R consecutive rows (R = 16 in the default
// variant), so a thread carries R rays that share their x offset.  Lenses stream through shared memory 256 at a
// time as FP32 positions relative to the tile centre (converted from the
// caller's FP64 once per tile and stage) and are broadcast to all warps.
//
// Precision plan: per pair FP32 with rcp.approx on the SFU (one reciprocal
// per ray, or one per two or four rows of a column through products of
// their squared distances); each 256-lens
// stage is summed in FP32 and folded into a TwoSum (hi, lo) accumulator; the
// sheet, the smooth terms and the pixel base of the tile centre are FP64 in
// the setup kernel and reach the rays as double-float constants plus an
// FP32 Taylor series of the sheet's analytic part in the ray's offset t.
#include <math.h>

#include <type_traits>

#include "irs_common.cuh"

namespace irs {

// ------------------------------------------------------------ mass sum (FP64)
// Deterministic sum of the masses: fixed strides per thread, fixed reduction
// tree, fixed order of the block partials.  With lens positions
// given, the same pass checks that every lens lies in the plan's lens region
// (the rectangle that is both image and lens plane, Sec. 2.2, or the
// circumscribed circle), with a margin of 1e-9 of the plane's extent for
// positions drawn on its edges: a lens outside it (or a NaN position) sets
// IRS_ERR_ARG in the plan's status word unless an earlier error is there.
struct LensRegion {
  double x0, x1, y0, y1;  // rectangle, margin included
  double cx, cy, r2;      // circle: centre and squared radius, margin included
  int32_t circle;
  int32_t check;          // 0: positions not given, no check
};

__device__ __forceinline__ bool lens_inside(const LensRegion& L, double2 p) {
  if (L.circle) {
    const double dx = p.x - L.cx, dy = p.y - L.cy;
    return dx * dx + dy * dy <= L.r2;  // false for NaN
  }
  return p.x >= L.x0 && p.x <= L.x1 && p.y >= L.y0 && p.y <= L.y1;
}

// The sum of up to MSUM_THREADS lenses is one block's; more blocks leave partial
// sums that a second launch adds in block order.  (Letting the block that
// finishes last add them saves that launch, but it needs a count of blocks that
// is zero at the start: one that lives across calls stays wrong for good once two
// calls on the same workspace have overlapped.)  Blocks past the last lens would
// only add zeros and are not launched; the stride between a thread's lenses is
// that of all MSUM_BLOCKS either way, so the sum is the same bits.
__global__ void k_mass_sum(const double* __restrict__ mass, const double2* __restrict__ xy, int64_t n,
                           LensRegion region, int* __restrict__ status, double* __restrict__ part,
                           bool whole, double* __restrict__ out, unsigned long long* __restrict__ queue,
                           int32_t* __restrict__ zero, int64_t nzero) {
  __shared__ double sh[MSUM_THREADS];
  after_ready();
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nzero; k += (int64_t)gridDim.x * blockDim.x)
    zero[k] = 0;
  double s = 0.0;
  bool outside = false;
  const int64_t stride = (int64_t)MSUM_BLOCKS * MSUM_THREADS;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
    s += mass[k];
    if (region.check) outside |= !lens_inside(region, xy[k]);
  }
  if (__syncthreads_or(outside) && threadIdx.x == 0) atomicCAS(status, 0, (int)IRS_ERR_ARG);
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = MSUM_THREADS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  if (!whole) {
    part[blockIdx.x] = sh[0];
  } else if (blockIdx.x == 0) {  // its lenses are all there are
    out[0] = sh[0];
    if (queue) *queue = 0ull;  // the ray pass's work counter
  }
}

__global__ void __launch_bounds__(MSUM_BLOCKS) k_mass_final(const double* part, int nblocks, double* __restrict__ out,
                                                            unsigned long long* __restrict__ queue) {
  __shared__ double sh[MSUM_BLOCKS];
  after_ready();
  after_wait();
  if ((int)threadIdx.x < nblocks) sh[threadIdx.x] = part[threadIdx.x];
  __syncthreads();
  if (threadIdx.x != 0) return;
  double t = 0.0;
#pragma unroll 4
  for (int b = 0; b < nblocks; ++b) t += sh[b];
  out[0] = t;
  if (queue) *queue = 0ull;
}

cudaError_t launch_mass_sum(const irs_plan_t* P, const double* mass, int64_t n, cudaStream_t s,
                            const double* xy) {
  LensRegion L{};
  const Geo& g = P->g;
  const double ext = fmax(fmax(fabs(g.a1), fabs(g.a2)), fmax(fmax(fabs(g.b1), fabs(g.b2)),
                                                             fmax(g.a2 - g.a1, g.b2 - g.b1)));
  const double tol = 1e-9 * ext;
  L.x0 = g.a1 - tol;
  L.x1 = g.a2 + tol;
  L.y0 = g.b1 - tol;
  L.y1 = g.b2 + tol;
  L.cx = g.cx;
  L.cy = g.cy;
  L.r2 = (P->circle_r + tol) * (P->circle_r + tol);
  L.circle = g.plane == IRS_PLANE_CIRCLE;
  L.check = xy != nullptr && n > 0;
  const bool whole = mass_sum_launches(n) == 1;
  const int64_t lens_blocks = (n + MSUM_THREADS - 1) / MSUM_THREADS;
  const int64_t nzero = P->d_zero ? P->n_zero : 0, zblocks = (nzero + 16 * MSUM_THREADS - 1) / (16 * MSUM_THREADS);
  auto clip = [](int64_t b) { return (int)(b < 1 ? 1 : b < MSUM_BLOCKS ? b : MSUM_BLOCKS); };
  k_mass_sum<<<(unsigned)clip(lens_blocks > zblocks ? lens_blocks : zblocks), MSUM_THREADS, 0, s>>>(
      mass, reinterpret_cast<const double2*>(xy), n, L, P->d_status, P->d_mpart, whole, P->d_msum, P->d_queue, P->d_zero,
      nzero);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || whole) return e;
  return launch_after(k_mass_final, 1, MSUM_BLOCKS, 0, s, P->d_mpart, clip(lens_blocks), P->d_msum, P->d_queue);
}

// ------------------------------------------------------------ FP64 complex
struct cd {
  double re, im;
};
__device__ __forceinline__ cd cmul(cd a, cd b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ cd crecip(cd a) {
  const double d = a.re * a.re + a.im * a.im;
  return {a.re / d, -a.im / d};
}
// principal Log
__device__ __forceinline__ cd clog_p(cd a) {
  return {0.5 * log(a.re * a.re + a.im * a.im), atan2(a.im, a.re)};
}

// ------------------------------------------------------------ tile setup
// Analytic part of the positive rectangle sheet (complex form derived from the
// appendix integrals): inside the rectangle,
//   conj(alpha_sheet)(z) = kappa_* conj(z) + g(z),
//   g(z) = kappa_* (z - 2 a2) + sum_c phi_c(z),
//   phi_c(z) = -i a_c (z - c) Log(z - c),   a_c = (kappa_*/pi) s_c,
// with corner signs s = +1 at (a1,b1) and (a2,b2), -1 at (a2,b1) and (a1,b2).
// Derivatives: phi_c' = -i a_c (Log(z-c) + 1),
//              phi_c^(n) = -i a_c (-1)^n (n-2)! / (z-c)^(n-1)  (n >= 2).
// Corners closer than 6 tile half-diagonals are left out of the series and
// evaluated per ray instead (the series would converge slowly there).
//
// Bound by FP64 latency and issue (GB300 runs FP64 at 1/64 of FP32), so a CTA
// of four warps takes 32 tiles: first one thread per (tile, corner) for the
// logarithm, arctangent and powers, then one warp sums the corners of each
// tile in order and adds the centre's terms.  With one thread per tile for all
// of it 5,120 tiles and 224 tiles took 32 us each, now 20 and 16 us.
constexpr int SETUP_TILES = 32;
constexpr int SETUP_VALUES = 4 + 2 * (SHEET_TERMS - 1);  // Log w, w Log w, w^-1 ... w^-7

__global__ void __launch_bounds__(4 * SETUP_TILES)
k_brute_setup(Geo g, const double* msum, int64_t ntx, int64_t tile0, int64_t tile1, bool early,
              TileRec* __restrict__ recs) {
  __shared__ double val_s[4][SETUP_VALUES][SETUP_TILES];
  __shared__ bool near_s[4][SETUP_TILES];
  if (early) after_ready();
  const int lt = threadIdx.x & 31;  // a warp per corner
  const int64_t tile = min(tile0 + (int64_t)blockIdx.x * SETUP_TILES + lt, tile1 - 1);
  const TileGeo tg = tile_geo(g, tile, ntx);
  const double zx = g.a1 + tg.ci * g.dx3, zy = g.b1 + tg.cj * g.dx3;
  auto corner = [&](int c) { return cd{zx - ((c & 1) ? g.a2 : g.a1), zy - ((c & 2) ? g.b2 : g.b1)}; };
  if (g.plane != IRS_PLANE_CIRCLE) {
    const int c = threadIdx.x >> 5;
    const cd w = corner(c);
    // the exact test only where a cheap upper bound of the radius leaves it open
    const double ub = 6.0 * fmax(0.5 * g.dx3 * (double)((tg.i1 - tg.i0) + (tg.j1 - tg.j0)), g.dx3);
    bool near = fmax(fabs(w.re), fabs(w.im)) < ub;
    if (near) {
      const double half_diag = 0.5 * g.dx3 * hypot((double)(tg.i1 - tg.i0), (double)(tg.j1 - tg.j0));
      near = hypot(w.re, w.im) < 6.0 * fmax(half_diag, g.dx3);
    }
    near_s[c][lt] = near;
    if (!near) {
      cd L = clog_p(w);
      // branch continuous with the rectangle's interior (tile centres are
      // inside it, so this only guards the two right-hand corners' cuts)
      if (c == 3 && w.re < 0.0 && w.im > 0.0) L.im -= 2.0 * M_PI;
      if (c == 1 && w.re < 0.0 && w.im < 0.0) L.im += 2.0 * M_PI;
      const cd wl = cmul(w, L);
      val_s[c][0][lt] = L.re;
      val_s[c][1][lt] = L.im;
      val_s[c][2][lt] = wl.re;
      val_s[c][3][lt] = wl.im;
      const cd inv = crecip(w);
      cd pw = inv;
#pragma unroll
      for (int k = 0; k < SHEET_TERMS - 1; ++k) {
        val_s[c][4 + 2 * k][lt] = pw.re;
        val_s[c][5 + 2 * k][lt] = pw.im;
        pw = cmul(pw, inv);
      }
    }
  }
  after_wait();  // the corners need the plan's geometry alone
  __syncthreads();
  if (threadIdx.x >= SETUP_TILES || tile0 + (int64_t)blockIdx.x * SETUP_TILES + lt >= tile1) return;

  const double ks = g.kstar_scale * msum[0];  // kappa_*^act = pi sum(m) / A of the lenses passed in
  const double kap = g.kappa_s + ks;
  // base pixel from the mean lens map of the tile centre
  const double m1 = (1.0 - kap - g.gamma) * zx, m2 = (1.0 - kap + g.gamma) * zy;
  double fx = floor((m1 - g.src_x0) / g.sx), fy = floor((m2 - g.src_y0) / g.sy);
  fx = fmin(fmax(fx, -1.0e9), 1.0e9);
  fy = fmin(fmax(fy, -1.0e9), 1.0e9);
  const double base_x = g.src_x0 + fx * g.sx, base_y = g.src_y0 + fy * g.sy;
  TileRec r;
  r.ix = (int32_t)fx;
  r.iy = (int32_t)fy;
  r.n_near = 0;
  r.pad_ = 0;
  for (int k = 0; k < SHEET_TERMS; ++k) r.T[k][0] = r.T[k][1] = 0.f;
  for (int k = 0; k < MAX_NEAR; ++k) r.near[k][0] = r.near[k][1] = r.near[k][2] = r.near[k][3] = 0.f;
  double cre, cim;  // conj(beta) of the centre without the lens sum
  if (g.plane == IRS_PLANE_CIRCLE) {
    // Eq. (alpha) + k_* theta_c:  conj(beta) = (1-k_s) conj(z) - g z - k_* conj(z_c) - L
    cre = (1.0 - g.kappa_s - g.gamma) * zx - ks * g.cx;
    cim = -(1.0 - g.kappa_s + g.gamma) * zy + ks * g.cy;
  } else {
    // Eq. (alpha1): conj(beta) = (1-k) conj(z) - g z - L + conj(alpha_sheet,+)
    cd T0 = {ks * (2.0 * zx - 2.0 * g.a2), 0.0};  // kappa_* (conj z + z - 2 a2)
    cd T[SHEET_TERMS];
#pragma unroll
    for (int k = 0; k < SHEET_TERMS; ++k) T[k] = {0.0, 0.0};
    T[0].re = ks;  // derivative of kappa_* (z - 2 a2)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double ac = ks / M_PI * ((c == 0 || c == 3) ? 1.0 : -1.0);
      if (ac == 0.0) continue;
      if (near_s[c][lt]) {
        const cd w = corner(c);
        r.near[r.n_near][0] = (float)w.re;
        r.near[r.n_near][1] = (float)w.im;
        r.near[r.n_near][2] = (float)ac;
        r.n_near++;
        continue;
      }
      auto v = [&](int k) { return val_s[c][k][lt]; };
      T0.re += ac * v(3);  // -i a_c (w L)
      T0.im -= ac * v(2);
      T[0].re += ac * v(1);  // -i a_c (L + 1)
      T[0].im -= ac * (v(0) + 1.0);
#pragma unroll
      for (int n = 2; n <= SHEET_TERMS; ++n) {
        const double coef = ((n & 1) ? -1.0 : 1.0) / (double)(n * (n - 1));
        T[n - 1].re += ac * coef * v(2 * n + 1);
        T[n - 1].im -= ac * coef * v(2 * n);
      }
    }
    cre = (1.0 - kap - g.gamma) * zx + T0.re;
    cim = -(1.0 - kap + g.gamma) * zy + T0.im;
#pragma unroll
    for (int k = 0; k < SHEET_TERMS; ++k) {
      r.T[k][0] = (float)T[k].re;
      r.T[k][1] = (float)T[k].im;
    }
  }
  split_df(cre - base_x, r.cx_hi, r.cx_lo);
  split_df(-cim - base_y, r.cy_hi, r.cy_lo);
  recs[tile] = r;
}

// Tile constants of the tile rows that cover lattice rows [row0, row1).
//
// The pass that follows may start beside this kernel (`early`), which hides the
// set-up behind its lens sums: 5 to 10 % of a map of up to half a millisecond
// (110 lenses, 4960 tiles: 305 against 325 us).  But CTAs placed around these
// find the registers in pieces, and an SM then keeps two of k_brute's three
// for a long time (124 lenses, 16150 tiles: 1,442 against 1,071 us; a band of
// 1296 tiles with 14297 lenses 4.4 against 3.5 ms), and the few CTAs of chosen
// rays crowd onto few SMs (472 rays: 254 against 88 us).  So: early for maps of
// up to 2^20 tile-lens products (about 0.5 ms) whose set-up is at most two CTAs
// per SM.
constexpr int64_t EARLY_WORK = (int64_t)1 << 20;
cudaError_t launch_brute_setup(const irs_plan_t* P, int64_t row0, int64_t row1, int64_t n, cudaStream_t s) {
  const int64_t t0 = row0 / BR_TY * P->br_ntx, t1 = (row1 + BR_TY - 1) / BR_TY * P->br_ntx;
  if (t1 <= t0) return cudaSuccess;
  const int64_t blocks = (t1 - t0 + SETUP_TILES - 1) / SETUP_TILES;
  const bool early = n >= 0 && blocks <= 2 * (int64_t)P->num_sms && (double)n * (double)(t1 - t0) <= (double)EARLY_WORK;
  return launch_after(k_brute_setup, (unsigned)blocks, 4 * SETUP_TILES, 0, s, P->g, P->d_msum, P->br_ntx, t0, t1, early,
                      P->d_tiles);
}

// ------------------------------------------------------------ ray pass
// Source position of a ray relative to its tile's base pixel corner, from its
// offset (tx, ty) to the tile centre and its lens sums: the sheet's series
// P(t) = sum_n T_n t^n, corners near the tile, the smooth terms and the centre.
// The rounding of every step is explicit: the map's and the chosen-ray kernels
// must agree bit for bit.
__device__ __forceinline__ void brute_corner(const float* near, float tx, float ty, float& pr, float& pi) {
  const float wr = __fadd_rn(near[0], tx), wi = __fadd_rn(near[1], ty);
  const float lr = __fmul_rn(0.5f, logf(__fmaf_rn(wr, wr, __fmul_rn(wi, wi)))), li = atan2f(wi, wr);
  const float plr = __fmaf_rn(wr, lr, -__fmul_rn(wi, li)), pli = __fmaf_rn(wi, lr, __fmul_rn(wr, li));  // w Log w
  pr = __fmaf_rn(near[2], pli, pr);  // -i a_c (w Log w)
  pi = __fmaf_rn(-near[2], plr, pi);
}
__device__ __forceinline__ void brute_sum(const Geo& g, const TileRec& rec, float tx, float ty, float pr, float pi,
                                          float axh, float axl, float ayh, float ayl, float& b1, float& b2) {
  float s1, e1, s2, e2;
  two_sum(rec.cx_hi, -axh, s1, e1);
  two_sum(rec.cy_hi, -ayh, s2, e2);
  b1 = __fadd_rn(s1, __fadd_rn(__fsub_rn(__fadd_rn(e1, rec.cx_lo), axl), __fmaf_rn(g.lam_s1, tx, pr)));
  b2 = __fadd_rn(s2, __fadd_rn(__fsub_rn(__fadd_rn(e2, rec.cy_lo), ayl), __fmaf_rn(g.lam_s2, ty, -pi)));
}
__device__ __forceinline__ void brute_beta(const Geo& g, const TileRec& rec, float tx, float ty, float axh, float axl,
                                           float ayh, float ayl, float& b1, float& b2) {
  float pr = 0.f, pi = 0.f;
#pragma unroll
  for (int k = SHEET_TERMS - 1; k >= 0; --k) {  // Horner, complex FP32
    const float ar = __fadd_rn(rec.T[k][0], pr), ai = __fadd_rn(rec.T[k][1], pi);
    pr = __fmaf_rn(ar, tx, -__fmul_rn(ai, ty));
    pi = __fmaf_rn(ar, ty, __fmul_rn(ai, tx));
  }
  for (int c = 0; c < rec.n_near; ++c) brute_corner(rec.near[c], tx, ty, pr, pi);
  brute_sum(g, rec, tx, ty, pr, pi, axh, axl, ayh, ayl, b1, b2);
}

// Variants: R rows per thread (the tile stays 32 x 64: 64/R warps per CTA),
// PAIRED rows per thread that share one reciprocal per two rows, QUAD groups
// of four packed rows that share one reciprocal per four rows, and PACK: the
// other rows go two at a time through the packed FP32x2 instructions (the two
// rows share dx and dx^2; fewer issue slots, the same FP32-pipe work).  The
// TwoSum accumulators live in shared memory (updated once per 256-lens stage).
// TPSM: resident threads per SM the register budget is sized for.
//
// Balance of the pair sum per lens and warp (32 lanes x R rows): the MUFU
// unit takes 8 cycles per warp-wide reciprocal, the FP32 pipe 1 cycle per
// scalar and 2 per packed instruction.  An unshared packed row pair costs 5
// packed instructions (10 FP32 cycles) and 2 reciprocals (16 MUFU cycles); a
// quad, two row pairs, 12 packed and 2 scalar instructions (26 FP32 cycles)
// and 1 reciprocal (8 MUFU cycles):
//   variant 11 (2 paired rows x 2, 6 packed pairs): MUFU 112, FP32  88 cycles
//   variant 0 (1 quad, 6 packed pairs):             MUFU 104, FP32  90 cycles
//   variant 10 (2 quads, 4 packed pairs):           MUFU  80, FP32  96 cycles
// bounding the pair sum at 71, 77 and 83 % of the FP32 peak.  Measured on
// the 1e5-lens band (one GB300, 2070 MHz): 59.7 % (variant 11), 62.3 %
// (variant 0, the default), 60.6 % (variant 10), all with four CTAs per SM and
// two lenses an iteration: with two quads the FP32 pipe's longer dependent
// chains cost more than the MUFU cycles they save.
//
// Variant 0 runs three CTAs per SM (160 registers) and eight lenses an
// iteration: more independent chains per warp keep the MUFU busier than more
// warps do.  The 64-row band of the 1e5-lens lattice takes 415 ms (64 %, 83 %
// of the MUFU's bound); four CTAs and 2, 4 or 8 lenses took 437, 437 and 436,
// three CTAs and 2, 4, 6, 16 or 32 lenses 432, 431, 421, 415 and 418, two CTAs
// and 4, 8 or 16 lenses 426, 430 and 433.  CTAs of one or two warps, each with
// its own copy of the lenses, take 452 and 447 us where this form takes 411 (128^2
// map, 150 lenses).
#define BR_VARIANTS(X)                                                                         \
  X(0, 16, 0, 1, 1, 384) X(1, 16, 8, 0, 0, 512) X(2, 8, 4, 0, 0, 512) X(3, 8, 2, 0, 0, 512)      \
  X(4, 16, 4, 0, 0, 512) X(5, 16, 2, 0, 0, 512) X(6, 16, 8, 0, 1, 512) X(7, 16, 6, 0, 1, 512)     \
  X(8, 16, 2, 0, 1, 512) X(9, 16, 4, 0, 1, 640) X(10, 16, 0, 2, 1, 512) X(11, 16, 4, 0, 1, 512)  \
  X(12, 16, 0, 3, 1, 512) X(13, 8, 0, 1, 1, 512) X(14, 16, 2, 1, 1, 512) X(15, 16, 4, 1, 1, 512)
constexpr int BR_NVARIANT = 16;

// Plane diagonal (theta_E) up to which the four-row products of squared
// distances stay inside the FP32 range with a wide margin ((1e4)^8 = 1e32).
constexpr double BR_QUAD_MAX_DIAG = 1.0e4;

template <int R, int PAIRED, int QUAD, int PACK, int TPSM>
__global__ void __launch_bounds__(32 * (BR_TY / R), TPSM / (32 * (BR_TY / R)))
k_brute(Geo g, const double2* __restrict__ xy, const double* __restrict__ mass, int64_t n,
        const TileRec* recs, int64_t ntx, int64_t nwork, int64_t row0, int64_t row1,
        uint32_t* __restrict__ counts) {
  constexpr int NT = 32 * (BR_TY / R);
  static_assert(PAIRED % 2 == 0 && (!PACK || (R - PAIRED) % 2 == 0), "rows go in pairs");
  static_assert(QUAD == 0 || PACK, "quads are packed");
  static_assert(PAIRED + 4 * QUAD <= R, "rows");
  // packed row pairs after the PAIRED scalar rows: the first 2 QUAD of them
  // form the quads
  constexpr int NPK = PACK ? (R - PAIRED) / 2 : 0;
  // lens records: (x, y, m, 0) for the scalar form; with PACK, (-x, -x, -y, -y)
  // and (m, m) -- the duplicates feed the packed instructions and the scalar
  // rows read one half (t + (-x) == t - x)
  __shared__ float4 lens_s[BR_LT];
  __shared__ float2 lensm_s[PACK ? BR_LT : 1];
  __shared__ float acc_s[4][R][NT];  // x hi, x lo, y hi, y lo
  __shared__ float2 ty_s[BR_TY / 2];  // row offsets to the tile centre, in pairs
  __shared__ TileRec rec;
  const int tid = threadIdx.x, lane = tid & 31;
  bool waited = false;
  after_ready();

  for (int64_t work = blockIdx.x; work < nwork; work += gridDim.x) {
    const int64_t tile = (row0 / BR_TY) * ntx + work;  // tile rows covering [row0, row1)
    const TileGeo tg = tile_geo(g, tile, ntx);
    // A warp whose rows lie outside the band or the lattice sums nothing.  Which
    // warp takes which rows varies from tile to tile: the warps of a CTA go to
    // the SM's four schedulers in turn, and rows that the band leaves out would
    // idle the same schedulers in every CTA (a 64-row band across two tile rows
    // sums 64 to 80 rows instead of 128).
    const int warp = ((tid >> 5) + (int)((uint32_t)work * 0x9E3779B1u >> 30)) & (BR_TY / R - 1);
    const bool live = tg.j0 + warp * R < min(row1, tg.j1) && tg.j0 + (warp + 1) * R > row0;
    const double zx = g.a1 + tg.ci * g.dx3, zy = g.b1 + tg.cj * g.dx3;
    const int64_t col = tg.i0 + lane;
    const float tx = (float)(((double)col + 0.5 - tg.ci) * g.dx3);
    const float2 TX2 = make_float2(tx, tx);
    __syncthreads();  // previous tile's readers of rec / lens_s / ty_s are done
    if (tid < BR_TY)
      reinterpret_cast<float*>(ty_s)[tid] = (float)(((double)(tg.j0 + tid) + 0.5 - tg.cj) * g.dx3);
    __syncthreads();
    float ty[R];
#pragma unroll
    for (int r = 0; r < R; r += 2) {
      const float2 t = ty_s[(warp * R + r) / 2];
      ty[r] = t.x;
      ty[r + 1] = t.y;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) acc_s[0][r][tid] = acc_s[1][r][tid] = acc_s[2][r][tid] = acc_s[3][r][tid] = 0.f;
    float2 TYP[NPK > 0 ? NPK : 1];
#pragma unroll
    for (int q = 0; q < NPK; ++q) TYP[q] = make_float2(ty[PAIRED + 2 * q], ty[PAIRED + 2 * q + 1]);

    for (int64_t base = 0; base < n; base += BR_LT) {
      float4 v[BR_LT / NT];
#pragma unroll
      for (int q = 0; q < BR_LT / NT; ++q) {
        const int64_t k = base + q * NT + tid;
        // padding: massless, and far enough that it is never on a ray, near
        // enough that products of four squared distances stay finite (a
        // product overflowing to inf would turn 0 x inf into NaN)
        v[q] = make_float4(4096.f, 4096.f, 0.f, 0.f);
        if (k < n) {
          const double2 p = xy[k];
          v[q] = make_float4((float)(p.x - zx), (float)(p.y - zy), (float)mass[k], 0.f);
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < BR_LT / NT; ++q) {
        if (PACK) {
          lens_s[q * NT + tid] = make_float4(-v[q].x, -v[q].x, -v[q].y, -v[q].y);
          lensm_s[q * NT + tid] = make_float2(v[q].z, v[q].z);
        } else {
          lens_s[q * NT + tid] = v[q];
        }
      }
      __syncthreads();
      float pax[R], pay[R];
      float2 PAX[NPK > 0 ? NPK : 1], PAY[NPK > 0 ? NPK : 1];
#pragma unroll
      for (int r = 0; r < R; ++r) pax[r] = pay[r] = 0.f;
#pragma unroll
      for (int q = 0; q < NPK; ++q) PAX[q] = PAY[q] = make_float2(0.f, 0.f);
      // lenses in this stage, rounded up to the unroll (padding is massless)
      const int cnt = live ? (int)min((int64_t)BR_LT, ((n - base) + 7) & ~(int64_t)7) : 0;
      constexpr int UNROLL = TPSM == 384 ? 8 : 2;
#pragma unroll UNROLL
      for (int jl = 0; jl < cnt; ++jl) {
        float4 L = lens_s[jl];
        float2 M, DX, DX2;
        float dx, dx2;
        if (PACK) {
          M = lensm_s[jl];
          DX = __fadd2_rn(TX2, make_float2(L.x, L.y));
          DX2 = __fmul2_rn(DX, DX);
          dx = DX.x;
          dx2 = DX2.x;
        } else {  // scalar layout: (x, y, m, 0) -> the same quantities
          M = make_float2(L.z, L.z);
          dx = tx - L.x;
          dx2 = dx * dx;
          L.z = -L.y;
        }
        // rows 0..PAIRED-1: one reciprocal for two rows, 1/(r_a^2 r_b^2), to move
        // work from the SFU (MUFU) to the FP32 pipe; remaining rows: one each
#pragma unroll
        for (int r = 0; r < PAIRED; r += 2) {
          const float dya = ty[r] + L.z, dyb = ty[r + 1] + L.z;
          const float r2a = fmaf(dya, dya, dx2), r2b = fmaf(dyb, dyb, dx2);
          const float mR = M.x * rcp_approx(r2a * r2b);
          const float wa = r2b * mR, wb = r2a * mR;
          pax[r] = fmaf(wa, dx, pax[r]);
          pay[r] = fmaf(wa, dya, pay[r]);
          pax[r + 1] = fmaf(wb, dx, pax[r + 1]);
          pay[r + 1] = fmaf(wb, dyb, pay[r + 1]);
        }
        // quads: rows (a, b) and (c, d) as two packed pairs sharing one
        // reciprocal of r_a^2 r_b^2 r_c^2 r_d^2; with P = (r_a^2 r_c^2, r_b^2 r_d^2)
        // and Q = m/(r_a^2 r_b^2 r_c^2 r_d^2) (P.y, P.x), m/r^2 of (a, b) is
        // Q (r_c^2, r_d^2) and of (c, d) is Q (r_a^2, r_b^2)
#pragma unroll
        for (int g4 = 0; g4 < QUAD; ++g4) {
          const float2 DYa = __fadd2_rn(TYP[2 * g4], make_float2(L.z, L.w));
          const float2 DYc = __fadd2_rn(TYP[2 * g4 + 1], make_float2(L.z, L.w));
          const float2 R2a = __ffma2_rn(DYa, DYa, DX2), R2c = __ffma2_rn(DYc, DYc, DX2);
          const float2 P4 = __fmul2_rn(R2a, R2c);
          const float mR = M.x * rcp_approx(P4.x * P4.y);
          const float2 Q4 = __fmul2_rn(make_float2(mR, mR), make_float2(P4.y, P4.x));
          const float2 Wa = __fmul2_rn(Q4, R2c), Wc = __fmul2_rn(Q4, R2a);
          PAX[2 * g4] = __ffma2_rn(Wa, DX, PAX[2 * g4]);
          PAY[2 * g4] = __ffma2_rn(Wa, DYa, PAY[2 * g4]);
          PAX[2 * g4 + 1] = __ffma2_rn(Wc, DX, PAX[2 * g4 + 1]);
          PAY[2 * g4 + 1] = __ffma2_rn(Wc, DYc, PAY[2 * g4 + 1]);
        }
        if (PACK) {
#pragma unroll
          for (int q = 2 * QUAD; q < NPK; ++q) {
            const float2 DY = __fadd2_rn(TYP[q], make_float2(L.z, L.w));
            const float2 R2 = __ffma2_rn(DY, DY, DX2);
            const float2 W = __fmul2_rn(M, make_float2(rcp_approx(R2.x), rcp_approx(R2.y)));
            PAX[q] = __ffma2_rn(W, DX, PAX[q]);
            PAY[q] = __ffma2_rn(W, DY, PAY[q]);
          }
        } else {
#pragma unroll
          for (int r = PAIRED; r < R; ++r) {
            const float dy = ty[r] + L.z;
            const float r2 = fmaf(dy, dy, dx2);
            const float w = M.x * rcp_approx(r2);
            pax[r] = fmaf(w, dx, pax[r]);
            pay[r] = fmaf(w, dy, pay[r]);
          }
        }
      }
      if (PACK) {
#pragma unroll
        for (int q = 0; q < NPK; ++q) {
          pax[PAIRED + 2 * q] = PAX[q].x;
          pax[PAIRED + 2 * q + 1] = PAX[q].y;
          pay[PAIRED + 2 * q] = PAY[q].x;
          pay[PAIRED + 2 * q + 1] = PAY[q].y;
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float s, e;
        two_sum(acc_s[0][r][tid], pax[r], s, e);
        acc_s[0][r][tid] = s;
        acc_s[1][r][tid] += e;
        two_sum(acc_s[2][r][tid], pay[r], s, e);
        acc_s[2][r][tid] = s;
        acc_s[3][r][tid] += e;
      }
    }
    // ---- per-ray: smooth terms, sheet series, near corners, pixel; two rows at
    // a time through the packed instructions, the roundings of brute_beta.  The
    // lens sums above need the caller's lenses alone; the tile's constants and
    // the map are the set-up's.
    if (!waited) {
      after_wait();
      waited = true;
    }
    if (tid == 0) rec = recs[tile];
    __syncthreads();
    const bool colok = col < tg.i1;
    const uint32_t npx = (uint32_t)g.npix_x, npy = (uint32_t)g.npix_y;
#pragma unroll 1
    for (int r = live ? 0 : R; r < R; r += 2) {
      const int64_t row = tg.j0 + warp * R + r;
      const float2 TY = ty_s[(warp * R + r) / 2], NTY = make_float2(-TY.x, -TY.y);
      float2 PR = make_float2(0.f, 0.f), PI = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = SHEET_TERMS - 1; k >= 0; --k) {
        const float2 AR = __fadd2_rn(make_float2(rec.T[k][0], rec.T[k][0]), PR);
        const float2 AI = __fadd2_rn(make_float2(rec.T[k][1], rec.T[k][1]), PI);
        PR = __ffma2_rn(AR, TX2, __fmul2_rn(AI, NTY));
        PI = __ffma2_rn(AR, TY, __fmul2_rn(AI, TX2));
      }
      float p1[2] = {PR.x, PR.y}, p2[2] = {PI.x, PI.y};
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float tyr = j ? TY.y : TY.x;
        for (int c = 0; c < rec.n_near; ++c) brute_corner(rec.near[c], tx, tyr, p1[j], p2[j]);
        float b1, b2;
        brute_sum(g, rec, tx, tyr, p1[j], p2[j], acc_s[0][r + j][tid], acc_s[1][r + j][tid], acc_s[2][r + j][tid],
                  acc_s[3][r + j][tid], b1, b2);
        const bool inside = colok && row + j < tg.j1 && row + j >= row0 && row + j < row1;
        // pixel_from_rel in 32 bits: base pixels are within 1e9 (k_brute_setup)
        const float f1 = floorf(b1 * g.inv_sx), f2 = floorf(b2 * g.inv_sy);
        const uint32_t px = (uint32_t)rec.ix + (uint32_t)(int)f1, py = (uint32_t)rec.iy + (uint32_t)(int)f2;
        const bool ok = inside && fabsf(f1) < 1.0e9f && fabsf(f2) < 1.0e9f && px < npx && py < npy;
        bin_warp(counts, ok, py * npx + px);
      }
    }
  }
}

#define BR_DECL_OCC(V, R, PAIRED, QUAD, PACK, TPSM)                                             \
  case V:                                                                                       \
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm,                                  \
                                                      k_brute<R, PAIRED, QUAD, PACK, TPSM>, \
                                                      32 * (BR_TY / R), 0) != cudaSuccess)      \
      per_sm = 1;                                                                               \
    break;
int brute_num_variants() { return BR_NVARIANT; }

#define BR_DECL_QUAD(V, R, PAIRED, QUAD, PACK, TPSM) \
  case V:                                            \
    return QUAD;
static int brute_quads(int variant) {
  switch (variant) { BR_VARIANTS(BR_DECL_QUAD) default: break; }
  return 0;
}

// A variant with four-row reciprocals multiplies four squared distances: it
// serves planes whose diagonal (the largest ray-lens distance; every lens is
// inside the plane) keeps that product in the FP32 range.
bool brute_variant_fits(int variant, double plane_diag) {
  if (variant < 0 || variant >= BR_NVARIANT) return false;
  return brute_quads(variant) == 0 || plane_diag <= BR_QUAD_MAX_DIAG;
}

int brute_grid_size(int num_sms, int variant) {
  int per_sm = 0;
  switch (variant) { BR_VARIANTS(BR_DECL_OCC) default: break; }
  return num_sms * (per_sm < 1 ? 1 : per_sm);
}

#define BR_DECL_LAUNCH(V, R, PAIRED, QUAD, PACK, TPSM)                                              \
  case V:                                                                                           \
    return launch_after(k_brute<R, PAIRED, QUAD, PACK, TPSM>, (unsigned)grid, 32 * (BR_TY / R), 0, s, P->g, xy2, mass, \
                        n, P->d_tiles, P->br_ntx, nwork, row0, row1, counts);
cudaError_t launch_brute_map(const irs_plan_t* P, const double* xy, const double* mass, int64_t n,
                             int64_t row0, int64_t row1, uint32_t* counts, cudaStream_t s) {
  if (row1 <= row0) return cudaSuccess;
  const int64_t tr0 = row0 / BR_TY, tr1 = (row1 + BR_TY - 1) / BR_TY;
  const int64_t nwork = (tr1 - tr0) * P->br_ntx;
  const int64_t grid = nwork < P->br_grid ? nwork : P->br_grid;
  const double2* xy2 = reinterpret_cast<const double2*>(xy);
  switch (P->p.kernel_variant) {
    BR_VARIANTS(BR_DECL_LAUNCH)
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------ chosen rays
// irs_shoot_rays: each ray by itself, in the arithmetic of k_brute -- lens
// positions relative to the ray's tile centre, FP32 sums of 256 lenses in
// order folded by TwoSum, and the reciprocal shared with the rows that the
// variant groups it with (their squared distances are computed for that
// alone).  The sums of different stages of 256 lenses are independent, so a
// CTA runs several stages of a ray at once and folds them in order.  The form
// before shot the ray's whole tile, 2048 rays.
//
// Two layouts.  BY_TILE: a CTA serves the chosen rays of one tile (a share of
// them), found by a scan over the indices, and converts each lens to the
// tile's frame once for all of them.  Otherwise a CTA takes 32 rays wherever
// they lie and every ray converts for itself, bound by the FP64 subtractions
// (GB300 issues two a clock per SM).  5e4 rays of a 923^2 lattice with 1e4 lenses
// take 0.50 ms by tile and 3.93 ms by ray, and took 209 ms before (0.76 by tile
// with both kinds of rays in most warps).  Which is the faster depends on the
// scan, which passes every index once per tile (rays_by_tile).
constexpr int BD_THREADS = 256;
constexpr int BD_STAGES = BD_THREADS / 32;  // stages at once where every ray converts for itself
constexpr int BD_LIST = 256;                // rays of a tile served at once
constexpr int BD_PARTS = 8;                 // CTAs per tile

struct RowGroup {  // rows that share a ray's reciprocal
  int kind;        // 0: none, 1: one row (a), 2: three rows; a the row two on, b and c the others
  float ta, tb, tc;
};

struct BruteForm {  // the variant's row groups (BR_VARIANTS)
  int R, paired, quad;
};

__device__ __forceinline__ RowGroup row_group(const BruteForm& f, const TileGeo& tg, double dx3, int64_t row) {
  RowGroup q{0, 0.f, 0.f, 0.f};
  const int64_t slab = tg.j0 + (row - tg.j0) / f.R * f.R;
  const int r = (int)(row - slab);
  auto ty = [&](int i) { return (float)(((double)(slab + i) + 0.5 - tg.cj) * dx3); };
  if (r < f.paired) {
    q.kind = 1;
    q.ta = ty(r ^ 1);
  } else if (r - f.paired < 4 * f.quad) {
    const int b = f.paired + ((r - f.paired) & ~3), i = (r - f.paired) & 3;
    q.kind = 2;
    q.ta = ty(b + (i ^ 2));
    q.tb = ty(b + (i ^ 1));
    q.tc = ty(b + (i ^ 3));
  }
  return q;
}

// one lens (offset x, y to the tile centre, mass m) into a ray's stage sums
__device__ __forceinline__ void ray_pair(float tx, float ty, const RowGroup& q, float x, float y, float m, float& px,
                                         float& py) {
  const float dx = __fsub_rn(tx, x), dx2 = __fmul_rn(dx, dx), dy = __fsub_rn(ty, y);
  const float r2 = __fmaf_rn(dy, dy, dx2);
  float w;
  if (q.kind == 0) {
    w = __fmul_rn(m, rcp_approx(r2));
  } else {
    const float da = __fsub_rn(q.ta, y), ra = __fmaf_rn(da, da, dx2);
    if (q.kind == 1) {
      w = __fmul_rn(ra, __fmul_rn(m, rcp_approx(__fmul_rn(r2, ra))));
    } else {
      const float db = __fsub_rn(q.tb, y), dc = __fsub_rn(q.tc, y);
      const float own = __fmul_rn(r2, ra);
      const float other = __fmul_rn(__fmaf_rn(db, db, dx2), __fmaf_rn(dc, dc, dx2));
      w = __fmul_rn(__fmul_rn(__fmul_rn(m, rcp_approx(__fmul_rn(own, other))), other), ra);
    }
  }
  px = __fmaf_rn(w, dx, px);
  py = __fmaf_rn(w, dy, py);
}

__device__ __forceinline__ void fold(float& hi, float& lo, float p) {
  float s, e;
  two_sum(hi, p, s, e);
  hi = s;
  lo = __fadd_rn(lo, e);
}

__device__ __forceinline__ void write_ray(const Geo& g, const TileRec& rec, float tx, float ty, float axh, float axl,
                                          float ayh, float ayl, int64_t slot, double* beta_out, int64_t* pix_out) {
  float b1, b2;
  brute_beta(g, rec, tx, ty, axh, axl, ayh, ayl, b1, b2);
  beta_out[2 * slot] = (g.src_x0 + (double)rec.ix * g.sx) + (double)b1;
  beta_out[2 * slot + 1] = (g.src_y0 + (double)rec.iy * g.sy) + (double)b2;
  if (pix_out) {
    uint32_t key = 0;
    int64_t pix = -1;
    pixel_from_rel(g, rec.ix, rec.iy, b1, b2, key, pix);
    pix_out[slot] = pix;
  }
}

template <bool BY_TILE>
__global__ void __launch_bounds__(BD_THREADS)
k_brute_rays(Geo g, BruteForm form, const double2* __restrict__ xy, const double* __restrict__ mass, int64_t n,
             const TileRec* recs, int64_t ntx, const int64_t* __restrict__ idx, int64_t nidx,
             double* __restrict__ beta_out, int64_t* __restrict__ pix_out) {
  // a stage's lenses: by tile as FP32 offsets (x, y, m), else as given
  __shared__ double2 pos_s[BY_TILE ? 1 : BD_STAGES * BR_LT];
  __shared__ float m_s[BY_TILE ? 1 : BD_STAGES * BR_LT];
  __shared__ float4 lens_s[BY_TILE ? BD_STAGES * BR_LT : 1];
  __shared__ float2 part_s[BD_THREADS];
  __shared__ int64_t list_s[BY_TILE ? BD_LIST : 1];
  __shared__ int found_s, grouped_s;
  const int tid = threadIdx.x;
  const int64_t tile = BY_TILE ? (int64_t)blockIdx.x / BD_PARTS : 0;
  const int64_t n_rays = g.nrx * g.nry;
  after_wait();
  int64_t scan = BY_TILE ? (int64_t)(blockIdx.x % BD_PARTS) * BD_THREADS : (int64_t)blockIdx.x * 32;
  while (scan < nidx) {
    // ---- the rays of this round: `live` of them, ray k's slot in the caller's arrays
    int live, nplain = 32, ngrouped = 0;  // of them sharing no reciprocal, and the others
    if (BY_TILE) {
      __syncthreads();
      if (tid == 0) found_s = grouped_s = 0;
      __syncthreads();
      for (; scan < nidx; scan += (int64_t)BD_PARTS * BD_THREADS) {
        const int64_t i = scan + tid;
        bool mine = false, grouped = false;
        if (i < nidx) {
          const int64_t f = idx[i];
          if (f < 0 || f >= n_rays) {
            mine = tile == 0;  // not a lattice ray: reported by the first tile's CTAs
          } else {
            const bool small = n_rays < ((int64_t)1 << 32);
            const int64_t j = small ? (int64_t)((uint32_t)f / (uint32_t)g.nrx) : f / g.nrx;
            mine = (j / BR_TY) * ntx + (f - j * g.nrx) / BR_TX == tile;
            grouped = (int)(j % BR_TY) % form.R < form.paired + 4 * form.quad;
          }
        }
        const int have = found_s + grouped_s;  // read before the barrier: nobody adds until everyone has passed it
        const int hits = __syncthreads_count(mine);
        if (have + hits > BD_LIST) break;  // next round starts here (a scan step adds at most BD_THREADS)
        // rays that share reciprocals from the list's end
        if (mine) list_s[grouped ? BD_LIST - 1 - atomicAdd(&grouped_s, 1) : atomicAdd(&found_s, 1)] = i;
        __syncthreads();
      }
      nplain = found_s;
      ngrouped = grouped_s;
      live = nplain + ngrouped;
      if (live == 0) continue;
    } else {
      live = (int)min((int64_t)32, nidx - scan);
    }
    // thread (ray, stage group): rays fastest; S groups of the rays that share
    // no reciprocal, then S of those that do, from a warp of their own where that
    // fits: a warp of both kinds runs both loops (8 and 19 instructions a pair)
    const int S = BY_TILE ? min(BD_STAGES, BD_THREADS / live) : BD_STAGES;
    int first = nplain * S;  // first thread of the second kind
    if (((first + 31) & ~31) + ngrouped * S <= BD_THREADS) first = (first + 31) & ~31;
    const bool second = tid >= first;
    const int step = second ? ngrouped : nplain, from = second ? tid - first : tid;
    const int grp = step > 0 ? from / step : S, ray = from - grp * step;
    const bool on = grp < S && ray < live;
    int64_t slot = 0, f = -1;
    if (on) {
      slot = BY_TILE ? list_s[second ? BD_LIST - ngrouped + ray : ray] : scan + ray;
      f = idx[slot];
    }
    const bool ok = f >= 0 && f < n_rays;
    const int64_t col = ok ? f % g.nrx : 0, row = ok ? f / g.nrx : 0;
    const int64_t mytile = (row / BR_TY) * ntx + col / BR_TX;
    const TileGeo tg = tile_geo(g, BY_TILE ? tile : mytile, ntx);
    const double zx = g.a1 + tg.ci * g.dx3, zy = g.b1 + tg.cj * g.dx3;
    const float tx = (float)(((double)col + 0.5 - tg.ci) * g.dx3), ty = (float)(((double)row + 0.5 - tg.cj) * g.dx3);
    const RowGroup q = ok ? row_group(form, tg, g.dx3, row) : RowGroup{0, 0.f, 0.f, 0.f};
    float axh = 0.f, axl = 0.f, ayh = 0.f, ayl = 0.f;
    for (int64_t base = 0; base < n; base += (int64_t)S * BR_LT) {
      const int total = (int)min((int64_t)S * BR_LT, n - base);
      __syncthreads();  // the stages and partial sums before are used up
      for (int t = tid; t < total; t += BD_THREADS) {
        const double2 p = xy[base + t];
        if (BY_TILE) {
          lens_s[t] = make_float4((float)(p.x - zx), (float)(p.y - zy), (float)mass[base + t], 0.f);
        } else {
          pos_s[t] = p;
          m_s[t] = (float)mass[base + t];
        }
      }
      __syncthreads();
      float px = 0.f, py = 0.f;
      if (on && ok) {
        const int e = min((grp + 1) * BR_LT, total);
        auto pairs = [&](auto kind) {
          RowGroup r = q;
          r.kind = kind;
#pragma unroll 4
          for (int t = grp * BR_LT; t < e; ++t) {
            if (BY_TILE) {
              const float4 L = lens_s[t];
              ray_pair(tx, ty, r, L.x, L.y, L.z, px, py);
            } else {
              const double2 p = pos_s[t];
              ray_pair(tx, ty, r, (float)(p.x - zx), (float)(p.y - zy), m_s[t], px, py);
            }
          }
        };
        if (!BY_TILE) pairs(q.kind);  // a loop per kind would convert every lens once for each
        else if (q.kind == 0) pairs(std::integral_constant<int, 0>{});
        else if (q.kind == 1) pairs(std::integral_constant<int, 1>{});
        else pairs(std::integral_constant<int, 2>{});
      }
      part_s[tid] = make_float2(px, py);
      __syncthreads();
      if (on && grp == 0) {  // fold the stages in order
        const int ns = (total + BR_LT - 1) / BR_LT;
        for (int k = 0; k < ns; ++k) {
          const float2 p = part_s[tid + k * step];
          fold(axh, axl, p.x);
          fold(ayh, ayl, p.y);
        }
      }
    }
    if (on && grp == 0) {
      if (ok) {
        write_ray(g, recs[mytile], tx, ty, axh, axl, ayh, ayl, slot, beta_out, pix_out);
      } else {  // not a lattice ray: report it, touch nothing else
        beta_out[2 * slot] = beta_out[2 * slot + 1] = nan("");
        if (pix_out) pix_out[slot] = -1;
      }
    }
    if (!BY_TILE) scan = nidx;  // one round of 32 rays
  }
}

#define BR_DECL_FORM(V, R, PAIRED, QUAD, PACK, TPSM) \
  case V:                                            \
    return BruteForm{R, PAIRED, QUAD};
static BruteForm brute_form(int variant) {
  switch (variant) { BR_VARIANTS(BR_DECL_FORM) default: break; }
  return BruteForm{16, 0, 0};
}

// Whether chosen rays go by tile: from 8 rays per tile on average, where the
// times below say so.  In picoseconds (one GB300, 6 to 63,000 tiles, 3 to 1e4
// lenses, 8 to 512 rays per tile): an index scanned for a tile costs 4.4, a pair
// by tile 0.75 and a lens converted for a tile's eight CTAs 46; a pair by ray
// costs 7.4, and fewer than 5000 rays take as long as those.  1e6 rays of 16,000
// tiles with 100 lenses take 72 ms by tile and 1.5 by ray, 2.6e5 rays of 4000 tiles
// with 1e4 lenses 8.4 and 18.8.
static bool rays_by_tile(int64_t ntiles, int64_t nidx, int64_t n) {
  if (nidx < 8 * ntiles || ntiles * BD_PARTS >= ((int64_t)1 << 31)) return false;
  const double T = (double)ntiles, k = (double)nidx, m = (double)n;
  return 4.4 * T * k + m * (0.75 * k + 46.0 * T) < 7.4 * m * fmax(k, 5000.0);
}

cudaError_t launch_brute_dump(const irs_plan_t* P, const double* xy, const double* mass, int64_t n,
                              const int64_t* idx, int64_t nidx, double* beta, int64_t* pix,
                              cudaStream_t s) {
  const double2* xy2 = reinterpret_cast<const double2*>(xy);
  const BruteForm form = brute_form(P->p.kernel_variant);
  if (rays_by_tile(P->br_ntiles, nidx, n))
    return launch_after(k_brute_rays<true>, (unsigned)(P->br_ntiles * BD_PARTS), BD_THREADS, 0, s, P->g, form, xy2,
                        mass, n, P->d_tiles, P->br_ntx, idx, nidx, beta, pix);
  return launch_after(k_brute_rays<false>, (unsigned)((nidx + 31) / 32), BD_THREADS, 0, s, P->g, form, xy2, mass, n,
                      P->d_tiles, P->br_ntx, idx, nidx, beta, pix);
}

// ------------------------------------------------------------ magnification
// Mag_ij = N_ij * S_I / S_S with S_I = dx3^2 and S_S = s_x s_y ("Calculate the
// magnification of each pixel", Sec. 2.4).
__global__ void k_magnify(const uint32_t* counts, float* __restrict__ mag, int64_t npix,
                          float ratio) {
  after_wait();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < npix; k += stride)
    mag[k] = (float)counts[k] * ratio;
}

cudaError_t launch_magnify(const irs_plan_t* P, const uint32_t* counts, float* mag, bool chained, cudaStream_t s) {
  const int64_t npix = (int64_t)P->g.npix_x * P->g.npix_y;
  const float ratio = (float)(P->g.dx3 * P->g.dx3 / (P->g.sx * P->g.sy));
  int64_t blocks = (npix + 255) / 256;
  const int64_t cap = (int64_t)P->num_sms * 8;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  if (chained) return launch_after(k_magnify, (unsigned)blocks, 256, 0, s, counts, mag, npix, ratio);
  k_magnify<<<(unsigned)blocks, 256, 0, s>>>(counts, mag, npix, ratio);
  return cudaGetLastError();
}

}  // namespace irs
