// irs_interp.cu -- the interpolated method of arXiv:2204.10871, Sec. 2.4
// ("Interpolation algorithm" and the flow chart's level-1/2/3 grids),
// re-designed for GB300.
//
//  level 1  square cells of k x k rays, side h = k Delta x3 with k from the
//           paper's Delta x1 = min(L0, min(I_x, I_y)/10), L0 = sqrt(A/N_*).
//           Lenses are binned into cells (counting sort, CSR, deterministic
//           order inside a cell).  A ray's "nearby lenses" are those of its own
//           cell and the 8 neighbours; they are summed directly per ray.
//  far      every other lens and the negative sheet are summed once per cell
//           into a Taylor series G_C(t) = sum_k c_k t^k about the cell centre:
//             cells at Chebyshev distance 2..W: each lens directly (P2L);
//             beyond W: multipole moments of each cell (P2M) translated to the
//             target cell by a convolution over the regular cell grid (M2L),
//             evaluated with FFTs, double-float for the low multipole and
//             local orders and FP32 for the rest (IP_PD, IP_KD below);
//             the rectangle sheet: its analytic part g(z), whose Taylor
//             coefficients are closed-form (rational for order >= 2).
//           The per-cell sums (window lenses, sheet, first series terms)
//           accumulate in FP64.
//  level 2  each cell's series is re-centred on Q x Q sub-cells (the paper's
//           level-2 grid points) with K2 terms, in shared memory per CTA.
//  level 3  the rays: one CTA per cell; near lenses broadcast from shared
//           memory, FP32 pair sums, sub-cell Horner, pixel, warp-aggregated
//           atomic binning.
//
// Per ray, with t = z - z_C (complex) and tau = t / h:
//   conj(beta) = B_C + (1 - kappa_s) conj(t) - gamma t - L_near(t) + sum_{k>=1} c_k tau^k
// where B_C = (1-kappa_s) conj(z_C) - gamma z_C + c_0 (rectangle), and
// L_near(t) = sum_near m_i / (t - t_i).  The kappa_* conj(z) parts of the
// matrix term and of the sheet cancel exactly and never appear.
#include <math.h>
#include <string.h>

#include <new>
#include <type_traits>

#include "irs_df.cuh"
#include "irs_fft.cuh"
#include "irs_interp.cuh"
#include "irs_mlp.cuh"

namespace irs {

namespace {

constexpr int IP_KMAX = 32;        // local series terms (max)
constexpr int IP_P = 18;           // multipole terms per cell
constexpr int IP_KF = 14;          // local terms produced by the M2L (cells >= 4 apart:
                                   // truncation (0.71 / 3.29)^14 ~ 5e-10 of a cell's field)
// Precision split of the convolution.  Multipole order j reaches the local
// term k through kernels of order j + k, each cell >= 4 cells away, so its
// share of term k is at most (0.71 / 4)^j = 0.18^j of the monopole's; local
// term k moves a ray by at most 0.71^k times its value.  Only the low orders
// carry sums that FP32 cannot hold to 1e-7 theta_E (term 0 is a potential-like
// sum over the whole plane, term 1 grows with its logarithm): multipole
// planes j < IP_PD and local planes k < IP_KD, with the kernel planes their
// products need, are transformed and multiplied in double-float; every other
// plane and product in FP32 (the j >= 4 share of term 0 is below 1e-3 of it,
// so FP32 adds ~1e-10 relative; terms k >= 3 are stored as FP32 anyway).
constexpr int IP_PD = 4;
constexpr int IP_KD = 3;
constexpr int IP_NKD = IP_PD + IP_KD - 1;  // kernel orders n = j + k of the double-float products
constexpr int IP_NEAR_MAX = 1024;  // lenses of a 3x3 block held in shared memory
constexpr int IP_KMAX_RAYS = 1024;  // rays along a cell side (row table in shared memory)
constexpr int IP_THREADS = 256;     // largest CTA of the ray pass
constexpr int IP_MAX_CORNER = 4;

constexpr int DEFAULT_K = 24;
constexpr int DEFAULT_W = 3;

struct __align__(16) CellRec {
  float bx_hi, bx_lo, by_hi, by_lo;  // beta of the centre (without L_near) relative to the base pixel
  int32_t ix, iy;                    // base pixel
  int32_t n_corner;
  float off;                         // how far off the map every ray of the cell lands for the smooth
                                     // terms and the centre's far field alone (theta_E; < 0: it may land)
  float corner[IP_MAX_CORNER][4];    // (z_C - c).re, .im, a_c, 0: corners evaluated per ray
};

static_assert(sizeof(CellRec) % 4 == 0 && sizeof(CellRec) / 4 <= 32, "a warp copies a cell record word by word");

struct IpGeo {
  int64_t k;           // rays per cell side
  double h;            // cell side
  int32_t ncx, ncy;    // cell grid
  int32_t ox, oy;      // first ray cell
  int32_t nrcx, nrcy;  // ray cells
  double gx0, gy0;     // grid origin (lower-left corner of cell (0,0))
  int K, P, W;
  int variant;  // ray-pass kernel variant (R, Q, K2)
  float hf;     // (float) h
  float inv_k;  // 1 / k in FP32 (correctly rounded)
  int32_t nrow;  // row-pair entries of the ray pass's row table: (k + 1)/2 + IP_ROW_PAD
  int32_t pad_;
  // blocks of a cell that map into about one binning box of the ray pass:
  // columns and 8-row groups; the cell's pixel extents under the mean lens map
  int32_t blk_col, blk_rg;
  float cell_px, cell_py;
};

struct InterpState {
  IpGeo ig;
  double rule_rays;  // the flow chart's Delta x1 in ray spacings, before the multiplier
  Fft2d fft;
  void* ws;
  size_t ws_bytes;
  void* lens_ws;
  size_t lens_ws_bytes;
  int64_t cap;
  int32_t* cell_count;
  int32_t* cell_start;
  int32_t* cell_cursor;
  int32_t* scan_blocks;
  int32_t* lens_cell;
  int32_t* sorted_idx;
  float4* lens_rel;
  double2* lens_pos;
  double* lens_m;
  float4* lens_pdf;  // positions as complex double-float
  float2* lens_mdf;  // masses as double-float
  // far-field convolution: complex double-float (float4, irs_df.cuh) for
  // the low orders, FP32 (float2) for the rest
  float4* mpole_d;  // [PD][ncells]    multipoles j < PD
  float2* mpole_f;  // [P-PD][ncells]  multipoles j >= PD
  float4* spec_d;   // [PD][Ny][Nx]    their spectra; then local spectra k < KD
  float2* spec_f;   // [P-PD][Ny][Nx]  their spectra; then local spectra KD <= k < KF
  float4* kspec_d;  // [NKD][Ny][Nx]   kernel spectra n < NKD, normalised by 1/(Nx Ny)
  float2* kspec_f;  // [P+KF-1][Ny][Nx] every kernel spectrum in FP32
  float4* conv_d;   // [KD][ncells]    local terms k < KD
  float2* conv_f;   // [KF-KD][ncells] local terms KD <= k < KF
  CellRec* recs;   // [nray cells]
  float2* coef;    // [nray cells][K]
  // the rectangle sheet's corner series per ray cell divided by kappa_*
  // (geometry only; k_ip_sheet_table), rectangular planes only
  double2* sheet_d;     // [nray cells][FIN_K64] terms k < FIN_K64
  float2* sheet_f;      // [nray cells][K - FIN_K64] the rest
  uint8_t* sheet_near;  // [nray cells] bit q: corner q evaluated per ray instead
  int64_t n_last;  // lenses of the last cell lists built
};

InterpState* S_(irs_plan_t* P) { return static_cast<InterpState*>(P->interp); }
const InterpState* S_(const irs_plan_t* P) { return static_cast<const InterpState*>(P->interp); }

// ------------------------------------------------------------ complex FP64
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

// ------------------------------------------------------------ cell lists
__device__ __forceinline__ int cell_of(const IpGeo& ig, double x, double y) {
  long long cx = (long long)floor((x - ig.gx0) / ig.h);
  long long cy = (long long)floor((y - ig.gy0) / ig.h);
  cx = cx < 0 ? 0 : (cx >= ig.ncx ? ig.ncx - 1 : cx);  // lenses off the grid: edge cell
  cy = cy < 0 ? 0 : (cy >= ig.ncy ? ig.ncy - 1 : cy);
  return (int)(cy * ig.ncx + cx);
}

__global__ void k_ip_count(IpGeo ig, const double2* __restrict__ xy, int64_t n,
                           int32_t* __restrict__ lens_cell, int32_t* __restrict__ count) {
  after_ready();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  if (i < n) {
    const double2 p = xy[i];
    c = cell_of(ig, p.x, p.y);
    lens_cell[i] = c;
  }
  after_wait();  // the counts are zeroed by the mass sum
  if (i < n) atomicAdd(count + c, 1);
}

// Exclusive scan of the cell counts into `start` (n + 1 entries) and a copy of it
// that the scatter advances: each block of SCAN_B cells scans its own and,
// unless it is the only one, leaves its sum; a second launch adds to each block
// the sums of those before it (which it adds up by itself; a third launch that
// scanned the sums on one thread took 50 us at 1.9e6 cells).
constexpr int SCAN_B = 1024;
__global__ void k_scan_local(const int32_t* in, int32_t* __restrict__ out, int32_t* __restrict__ copy,
                             int64_t n, int32_t* __restrict__ block_sums) {
  __shared__ int32_t warp_s[32];
  after_ready();
  after_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * SCAN_B + threadIdx.x;
  const int32_t v = i < n ? in[i] : 0;
  int32_t inc = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, d);
    if (lane >= d) inc += t;
  }
  if (lane == 31) warp_s[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int32_t w = warp_s[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t t = __shfl_up_sync(0xFFFFFFFFu, w, d);
      if (lane >= d) w += t;
    }
    warp_s[lane] = w;
  }
  __syncthreads();
  inc += warp ? warp_s[warp - 1] : 0;
  if (i < n) {
    out[i] = inc - v;
    if (gridDim.x == 1) {
      copy[i] = inc - v;
      if (i == n - 1) out[n] = inc;
    }
  }
  if (gridDim.x > 1 && threadIdx.x == SCAN_B - 1) block_sums[blockIdx.x] = inc;
}
__global__ void k_scan_add(int32_t* __restrict__ out, int32_t* __restrict__ copy, int64_t n,
                           const int32_t* block_sums) {
  __shared__ int32_t warp_s[32];
  after_ready();
  after_wait();
  int32_t s = 0;
  for (int64_t b = threadIdx.x; b < blockIdx.x; b += SCAN_B) s += block_sums[b];
  s = __reduce_add_sync(0xFFFFFFFFu, s);
  if ((threadIdx.x & 31) == 0) warp_s[threadIdx.x >> 5] = s;
  __syncthreads();
  s = __reduce_add_sync(0xFFFFFFFFu, warp_s[threadIdx.x & 31]);
  const int64_t i = (int64_t)blockIdx.x * SCAN_B + threadIdx.x;
  if (i < n) {
    const int32_t v = out[i] + s;
    out[i] = v;
    copy[i] = v;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[n] = s + block_sums[blockIdx.x];
}

__global__ void k_ip_scatter(const int32_t* lens_cell, int64_t n,
                             int32_t* __restrict__ cursor, int32_t* __restrict__ sorted_idx) {
  after_ready();
  after_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int pos = atomicAdd(cursor + lens_cell[i], 1);
  sorted_idx[pos] = (int32_t)i;
}

// Per cell, for the lenses of its list:
// - insertion sort of the indices: the order inside a cell no longer depends on
//   the atomics, so every map is bitwise reproducible;
// - the sorted records: position relative to the cell centre (FP32), position
//   and mass in double-float, and in FP64 where the network form wants them;
// - P2M (series form): a_j = sum_i m_i ((z_i - z_S)/h)^j; orders j < IP_PD in
//   FP64 (stored double-float), the rest in FP32 from the FP32 offset (|d| <=
//   0.71; they are stored and convolved in FP32).
//
// A CTA takes CELLS_B cells, whose lenses are contiguous.  Cells hold half a lens on
// average, so the FP64 work (GB300 issues two a clock per SM) is done with one
// thread per lens, a chunk of CELLS_B lenses at a time through shared memory, and
// one thread per cell only adds, in list order.  As three kernels (sort, fill,
// P2M with one thread per cell) this took 14.6 us at 250 cells and 474 us at the
// high-res map's 1.9e6; now 8.7 and 311 us.
constexpr int CELLS_B = 128;
__global__ void __launch_bounds__(CELLS_B)
k_ip_cells(IpGeo ig, const int32_t* start, const double2* __restrict__ xy,
           const double* __restrict__ mass, const int32_t* lens_cell, int32_t* __restrict__ sorted_idx,
           float4* __restrict__ rel, double2* __restrict__ pos, double* __restrict__ m_out,
           float4* __restrict__ pos_df, float2* __restrict__ m_df, float4* __restrict__ mpole_d,
           float2* __restrict__ mpole_f) {
  __shared__ double pw_s[2 * IP_PD][CELLS_B];  // m d^j, j < PD, of the chunk's lenses
  __shared__ float2 d_s[CELLS_B], pf_s[CELLS_B];  // d and m d^PD in FP32
  after_ready();
  after_wait();
  const int64_t ncells = (int64_t)ig.ncx * ig.ncy, c0 = (int64_t)blockIdx.x * CELLS_B;
  const int64_t c = c0 + threadIdx.x;
  const bool on = c < ncells;
  const int b = on ? start[c] : 0, e = on ? start[c + 1] : 0;
  for (int i = b + 1; i < e; ++i) {
    const int32_t v = sorted_idx[i];
    int j = i - 1;
    while (j >= b && sorted_idx[j] > v) {
      sorted_idx[j + 1] = sorted_idx[j];
      --j;
    }
    sorted_idx[j + 1] = v;
  }
  cd a[IP_PD];
  float2 af[IP_P - IP_PD];
#pragma unroll
  for (int j = 0; j < IP_PD; ++j) a[j] = {0.0, 0.0};
#pragma unroll
  for (int j = 0; j < IP_P - IP_PD; ++j) af[j] = make_float2(0.f, 0.f);
  const double inv_h = 1.0 / ig.h;
  const int first = start[c0], last = start[min(c0 + CELLS_B, ncells)];
  for (int chunk = first; chunk < last; chunk += CELLS_B) {
    __syncthreads();  // lists sorted; the chunk before is used up
    const int p = chunk + threadIdx.x;
    if (p < last) {
      const int32_t i = sorted_idx[p];
      const int cell = lens_cell[i], cx = cell % ig.ncx, cy = cell / ig.ncx;
      const double zx = ig.gx0 + (cx + 0.5) * ig.h, zy = ig.gy0 + (cy + 0.5) * ig.h;
      const double2 q = xy[i];
      const double m = mass[i];
      rel[p] = make_float4((float)(q.x - zx), (float)(q.y - zy), (float)m, 0.f);
      pos_df[p] = dfc_from_double(q.x, q.y);
      m_df[p] = df_from_double(m);
      if (pos) {
        pos[p] = q;
        m_out[p] = m;
      }
      if (mpole_d) {
        const cd d = {(q.x - zx) * inv_h, (q.y - zy) * inv_h};
        cd pw = {m, 0.0};
#pragma unroll
        for (int j = 0; j < IP_PD; ++j) {
          pw_s[2 * j][threadIdx.x] = pw.re;
          pw_s[2 * j + 1][threadIdx.x] = pw.im;
          pw = cmul(pw, d);
        }
        d_s[threadIdx.x] = make_float2((float)d.re, (float)d.im);
        pf_s[threadIdx.x] = make_float2((float)pw.re, (float)pw.im);  // m d^PD
      }
    }
    if (!mpole_d) continue;
    __syncthreads();
    for (int k = max(b, chunk); k < min(e, chunk + CELLS_B); ++k) {
      const int t = k - chunk;
#pragma unroll
      for (int j = 0; j < IP_PD; ++j) {
        a[j].re += pw_s[2 * j][t];
        a[j].im += pw_s[2 * j + 1][t];
      }
      const float2 df = d_s[t];
      float2 pf = pf_s[t];
#pragma unroll
      for (int j = 0; j < IP_P - IP_PD; ++j) {
        af[j].x += pf.x;
        af[j].y += pf.y;
        pf = make_float2(fmaf(pf.x, df.x, -pf.y * df.y), fmaf(pf.x, df.y, pf.y * df.x));
      }
    }
  }
  if (!mpole_d || !on) return;
#pragma unroll
  for (int j = 0; j < IP_PD; ++j)
    mpole_d[(int64_t)j * ncells + c] = b == e ? make_float4(0.f, 0.f, 0.f, 0.f) : dfc_from_double(a[j].re, a[j].im);
#pragma unroll
  for (int j = 0; j < IP_P - IP_PD; ++j) mpole_f[(int64_t)j * ncells + c] = af[j];
}

// ------------------------------------------------------------ far field
// Translation kernels on the padded grid, scaled by n! / (Nx Ny):
// K'_n[e] = n! (-e)^-(n+1) / (Nx Ny) for offsets e (cell units, wrapped) with
// Chebyshev norm > W, else 0 (the n! is one factor of the M2L's binomial,
// below; the 1/(Nx Ny) normalises the inverse FFT and keeps every spectrum
// far inside the FP32 exponent range).  Orders n < nkd in double-float (kg_d),
// every order in FP32 (kg_f).
__global__ void k_ip_kernel_grid(int Nx, int Ny, int W, int nker, int nkd, float4* __restrict__ kg_d,
                                 float2* __restrict__ kg_f) {
  const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t G = (int64_t)Nx * Ny;
  if (f >= G) return;
  const int ex = (int)(f % Nx), ey = (int)(f / Nx);
  const int sx = ex < Nx / 2 ? ex : ex - Nx, sy = ey < Ny / 2 ? ey : ey - Ny;
  const bool far = abs(sx) > W || abs(sy) > W;
  cd inv = {0.0, 0.0};
  if (far) inv = crecip(cd{-(double)sx, -(double)sy});
  cd pw = inv;
  double fact = 1.0 / (double)G;  // n! / (Nx Ny)
  for (int n = 0; n < nker; ++n) {
    if (n > 0) fact *= (double)n;
    const double re = far ? pw.re * fact : 0.0, im = far ? pw.im * fact : 0.0;
    if (n < nkd) kg_d[(int64_t)n * G + f] = dfc_from_double(re, im);
    kg_f[(int64_t)n * G + f] = make_float2((float)re, (float)im);
    pw = cmul(pw, inv);
  }
}

// Pointwise M2L in frequency space:
//   C_k = sum_j (-1)^j binom(j+k, k) A_j Kh_{j+k},  j < P, k < KF,
// with binom(j+k, k) = (j+k)! / (j! k!): the (j+k)! sits in the kernel
// spectra, so each term is one complex multiply-add of (-1)^j A_j / j! and
// the scaled kernel, and C_k takes the 1/k! at the end.  Products with
// j < PD and k < KD in double-float, the others in FP32 (the FP32 operands
// of the double-float planes are their high parts); the FP32 share of
// C_k, k < KD, joins the double-float sum before the scaling.
__global__ void __launch_bounds__(128) k_ip_m2l_freq(int64_t G, float4* __restrict__ spec_d,
                                                     float2* __restrict__ spec_f,
                                                     const float4* __restrict__ kspec_d,
                                                     const float2* __restrict__ kspec_f) {
  after_ready();
  after_wait();
  const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= G) return;
  float4 Ad[IP_PD], Cd[IP_KD];
  float2 Af[IP_P], Cf[IP_KF];
  double ifact = 1.0;  // 1/j!, folded at compile time
#pragma unroll
  for (int j = 0; j < IP_P; ++j) {
    if (j > 0) ifact /= (double)j;
    const double sc = ((j & 1) ? -1.0 : 1.0) * ifact;
    if (j < IP_PD) {
      Ad[j] = dfc_scale(spec_d[(int64_t)j * G + f], df_from_double(sc));
      Af[j] = dfc_hi(Ad[j]);
    } else {
      const float2 v = spec_f[(int64_t)(j - IP_PD) * G + f];
      Af[j] = make_float2(v.x * (float)sc, v.y * (float)sc);
    }
  }
#pragma unroll
  for (int k = 0; k < IP_KD; ++k) Cd[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < IP_KF; ++k) Cf[k] = make_float2(0.f, 0.f);
#pragma unroll
  for (int nn = 0; nn < IP_P + IP_KF - 1; ++nn) {
    const float2 kf = kspec_f[(int64_t)nn * G + f];
    const float4 kd = nn < IP_NKD ? kspec_d[(int64_t)nn * G + f] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < IP_P; ++j) {
      const int k = nn - j;
      if (k < 0 || k >= IP_KF) continue;
      if (j < IP_PD && k < IP_KD) {
        Cd[k] = dfc_add(Cd[k], dfc_mul(Ad[j], kd));
      } else {
        Cf[k].x = fmaf(Af[j].x, kf.x, fmaf(-Af[j].y, kf.y, Cf[k].x));
        Cf[k].y = fmaf(Af[j].x, kf.y, fmaf(Af[j].y, kf.x, Cf[k].y));
      }
    }
  }
  double kfact = 1.0;  // 1/k!
#pragma unroll
  for (int k = 0; k < IP_KF; ++k) {
    if (k > 0) kfact /= (double)k;
    if (k < IP_KD) {
      const float4 c = dfc_add(Cd[k], make_float4(Cf[k].x, Cf[k].y, 0.f, 0.f));
      spec_d[(int64_t)k * G + f] = dfc_scale(c, df_from_double(kfact));
    } else {
      spec_f[(int64_t)(k - IP_KD) * G + f] = make_float2(Cf[k].x * (float)kfact, Cf[k].y * (float)kfact);
    }
  }
}

// Series terms of the per-cell finalize accumulated in FP64; the others in
// FP32.  A window lens sits >= 1.5 cells from the cell centre and a ray
// <= 0.71 cells from it, so term k of a lens contributes at most
// (m/d) 0.47^k: FP32 rounding of the terms k >= 3 moves a ray's deflection by
// <= 1e-7 x 0.1 of that lens's field, and every term k >= 1 is stored as FP32
// for the ray pass anyway.  Terms 0..2 (the constant, which sets the ray's
// beta, and the two largest slopes) keep FP64.
constexpr int FIN_K64 = 3;
constexpr int FIN_K32 = IP_KMAX - FIN_K64;
static_assert(IP_KD == FIN_K64, "the M2L's double-float terms are the FP64 ones");

// 1/a for complex a, |a| >~ 1e-19 (cell or theta_E units): an FP32 seed for
// 1/|a|^2 refined by one FP64 Newton step (relative error ~1e-14), instead of
// two FP64 divisions.
__device__ __forceinline__ cd crecip_nr(cd a) {
  const double q = a.re * a.re + a.im * a.im;
  double r = (double)rcp_approx((float)q);
  r = r * fma(-q, r, 2.0);
  return {a.re * r, -a.im * r};
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// 1/(re + i im) in double-float: conj / |.|^2, the reciprocal of |.|^2 from
// the FP32 reciprocal of its high part and one Newton step r + r (1 - q r)
// (quadratic convergence: ~2^-47 relative).  |.| >= 1 here (window lenses
// are at least a cell away, in cell units).
__device__ __forceinline__ float4 dfc_recip(float2 re, float2 im) {
  const float2 q = df_add(df_mul(re, re), df_mul(im, im));
  const float2 r0 = make_float2(__frcp_rn(q.x), 0.f);
  const float2 e = df_sub(make_float2(1.f, 0.f), df_mul(q, r0));
  const float2 r = df_add(r0, df_mul(r0, e));
  return dfc_make(df_mul(re, r), df_neg(df_mul(im, r)));
}

// Corners of the lens rectangle (a1, b1), (a2, b1), (a1, b2), (a2, b2) and
// the signs of their a_c / kappa_* * pi.
__device__ __forceinline__ double sheet_corner_x(const Geo& g, int q) { return (q & 1) ? g.a2 : g.a1; }
__device__ __forceinline__ double sheet_corner_y(const Geo& g, int q) { return (q & 2) ? g.b2 : g.b1; }
__device__ __forceinline__ double sheet_corner_sign(int q) { return (q == 0 || q == 3) ? 1.0 : -1.0; }

// Per ray cell: the four corner terms of the sheet's analytic part,
// sum_c -i (a_c / kappa_*) (z - c) Log(z - c), as a series in tau = (z -
// z_C)/h: terms k < FIN_K64 in FP64, the next K - FIN_K64 in FP32.  They
// depend on the plan's geometry alone, so a plan builds them once and each
// map scales them by its kappa_*.  A corner within 4 x 0.71 h of the centre
// is left out (bit q of `near`): the ray pass evaluates it per ray.
__global__ void k_ip_sheet_table(Geo g, IpGeo ig, double2* __restrict__ sheet_d, float2* __restrict__ sheet_f,
                                 uint8_t* __restrict__ sheet_near, int64_t nrc) {
  const int64_t rc = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (rc >= nrc) return;
  const int cx = (int)(rc % ig.nrcx) + ig.ox, cy = (int)(rc / ig.nrcx) + ig.oy;
  const double zx = ig.gx0 + (cx + 0.5) * ig.h, zy = ig.gy0 + (cy + 0.5) * ig.h;
  const double h = ig.h;
  const int nsf = ig.K - FIN_K64;
  cd acc[FIN_K64];
  float2 accf[FIN_K32];
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) acc[k] = {0.0, 0.0};
#pragma unroll
  for (int k = 0; k < FIN_K32; ++k) accf[k] = make_float2(0.f, 0.f);
  unsigned near = 0;
  const double rho = 4.0 * 0.70710678118654752 * h;
  for (int q = 0; q < 4; ++q) {
    const double ac = sheet_corner_sign(q) / M_PI;
    const cd w = {zx - sheet_corner_x(g, q), zy - sheet_corner_y(g, q)};
    if (hypot(w.re, w.im) < rho) {
      near |= 1u << q;
      continue;
    }
    // Log(z - c) on the branch that is continuous with the rectangle's
    // interior: the principal cuts of the two right-hand corners run along
    // the top and bottom edges, so a cell centre beyond those edges (a
    // ragged last cell row) takes the argument across the cut.
    double arg = atan2(w.im, w.re);
    if (q == 3 && w.re < 0.0 && w.im > 0.0) arg -= 2.0 * M_PI;  // (a2, b2), centre above b2
    if (q == 1 && w.re < 0.0 && w.im < 0.0) arg += 2.0 * M_PI;  // (a2, b1), centre below b1
    const cd L = {0.5 * log(w.re * w.re + w.im * w.im), arg};
    const cd wl = cmul(w, L);
    acc[0].re += ac * wl.im;
    acc[0].im -= ac * wl.re;
    acc[1].re += ac * L.im * h;
    acc[1].im -= ac * (L.re + 1.0) * h;
    const cd inv = crecip_nr(w);
    const cd ih = {inv.re * h, inv.im * h};
    cd pw = {inv.re * h * h, inv.im * h * h};  // h^n / w^(n-1) at n = 2
    // n = 2 in FP64 (FIN_K64 = 3), n >= 3 in FP32
    acc[2].re += ac * 0.5 * pw.im;
    acc[2].im -= ac * 0.5 * pw.re;
    pw = cmul(pw, ih);
    const float2 ihf = make_float2((float)ih.re, (float)ih.im);
    float2 pf = make_float2((float)pw.re, (float)pw.im);
    const float acf = (float)ac;
#pragma unroll
    for (int k = 0; k < FIN_K32; ++k) {
      const int n = k + FIN_K64;
      const float cf = ((n & 1) ? -1.0f : 1.0f) / (float)(n * (n - 1));
      accf[k].x += acf * cf * pf.y;
      accf[k].y -= acf * cf * pf.x;
      pf = cmulf(pf, ihf);
    }
  }
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) sheet_d[rc * FIN_K64 + k] = make_double2(acc[k].re, acc[k].im);
#pragma unroll
  for (int k = 0; k < FIN_K32; ++k) {
    if (k >= nsf) break;
    sheet_f[rc * nsf + k] = accf[k];
  }
  sheet_near[rc] = (uint8_t)near;
}

// Centre term and base pixel of a cell from its series' first terms: acc[0..2]
// (FP64, before the sheet's share when `sheet`), written to the record and the
// first coefficients.
__device__ __forceinline__ void finish_cell(const Geo& g, const IpGeo& ig, double ks, double zx, double zy, int64_t rc,
                                            cd* acc, bool sheet, const double2* __restrict__ sheet_d,
                                            const uint8_t* __restrict__ sheet_near, CellRec* __restrict__ recs,
                                            float2* __restrict__ coef) {
  const double kap = g.kappa_s + ks, h = ig.h;
  CellRec r;
  r.n_corner = 0;
  for (int q = 0; q < IP_MAX_CORNER; ++q) r.corner[q][0] = r.corner[q][1] = r.corner[q][2] = r.corner[q][3] = 0.f;
  cd B;
  if (sheet && g.plane == IRS_PLANE_CIRCLE) {
    B = {(1.0 - g.kappa_s - g.gamma) * zx - ks * g.cx, -(1.0 - g.kappa_s + g.gamma) * zy + ks * g.cy};
  } else {
    if (sheet) {
      // sheet: g(z) = kappa_* (z - 2 a2) + sum_c -i a_c (z - c) Log(z - c); adds
      // g_k h^k.  a_c = +-kappa_* / pi, so the corner sums are kappa_* times a
      // per-plan table (k_ip_sheet_table); corners near the cell go to the rays.
      acc[0].re += ks * (zx - 2.0 * g.a2);
      acc[0].im += ks * zy;
      acc[1].re += ks * h;
      if (ks != 0.0) {
        const unsigned near = sheet_near[rc];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (!((near >> q) & 1u)) continue;
          r.corner[r.n_corner][0] = (float)(zx - sheet_corner_x(g, q));
          r.corner[r.n_corner][1] = (float)(zy - sheet_corner_y(g, q));
          r.corner[r.n_corner][2] = (float)(ks / M_PI * sheet_corner_sign(q));
          r.n_corner++;
        }
#pragma unroll
        for (int k = 0; k < FIN_K64; ++k) {
          const double2 t = sheet_d[rc * FIN_K64 + k];
          acc[k].re += ks * t.x;
          acc[k].im += ks * t.y;
        }
      }
    }
    B = {(1.0 - g.kappa_s - g.gamma) * zx, -(1.0 - g.kappa_s + g.gamma) * zy};
  }
  B.re += acc[0].re;
  B.im += acc[0].im;
  const double m1 = (1.0 - kap - g.gamma) * zx, m2 = (1.0 - kap + g.gamma) * zy;
  double fx = floor((m1 - g.src_x0) / g.sx), fy = floor((m2 - g.src_y0) / g.sy);
  fx = fmin(fmax(fx, -1.0e9), 1.0e9);
  fy = fmin(fmax(fy, -1.0e9), 1.0e9);
  r.ix = (int32_t)fx;
  r.iy = (int32_t)fy;
  split_df(B.re - (g.src_x0 + fx * g.sx), r.bx_hi, r.bx_lo);
  split_df(-B.im - (g.src_y0 + fy * g.sy), r.by_hi, r.by_lo);
  // distance of the centre's beta from the map along each axis, less what the
  // smooth terms add over half a cell
  const double d1 = fmax(g.src_x0 - B.re, B.re - (g.src_x0 + g.npix_x * g.sx)) - 0.5 * h * fabs(1.0 - g.kappa_s - g.gamma);
  const double d2 = fmax(g.src_y0 + B.im, -B.im - (g.src_y0 + g.npix_y * g.sy)) - 0.5 * h * fabs(1.0 - g.kappa_s + g.gamma);
  r.off = (float)fmax(d1, d2);
  recs[rc] = r;
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) coef[rc * ig.K + k] = make_float2((float)acc[k].re, (float)acc[k].im);
}

// Per ray cell of [rc0, rc1): window P2L, M2L result, sheet series, centre
// term, base pixel (series mode).  NF: FP32 series terms computed (k = FIN_K64
// ... FIN_K64 + NF - 1; at least K - FIN_K64).
//
// A warp takes four cells at a time, eight lanes each.  A cell's window lenses,
// which lie in a few contiguous ranges of the sorted lists, are dealt to its
// lanes, each of which computes one lens's powers (double-float reciprocal,
// first terms, FP32 terms) into shared memory; then the lanes change places
// and each sums some (cell, term) components over the eight lenses, in list
// order -- the sums come out as if one thread had walked the window.  One
// thread per cell was bound by that walk where cells are few (40 lenses of
// ~500 instructions in a row): 67 us for 250 cells, 83 us for 2.1e4, 355 us for
// 3.0e5 (paper-mid); now 20, 39 and 333 us.
constexpr int FG_WARPS = 4;                 // warps per CTA
constexpr int FG_CELLS = 32;                // cells per CTA: the FP64 end runs on one full warp (fewer for few cells)
constexpr int FG_LANES = 8;                 // lanes per cell
constexpr int FG_WMAX = 16;                 // largest direct window
constexpr int FG_RANGES = 2 * FG_WMAX + 4;  // list ranges of a window

template <int NF>
__global__ void __launch_bounds__(32 * FG_WARPS, 6)
k_ip_finalize_group(Geo g, IpGeo ig, const double* msum, const int32_t* start, const float4* pos_df,
                    const float2* m_df, const float4* conv_d, const float2* conv_f,
                    const double2* __restrict__ sheet_d, const float2* __restrict__ sheet_f,
                    const uint8_t* __restrict__ sheet_near, CellRec* __restrict__ recs, float2* __restrict__ coef,
                    int64_t rc0, int64_t rc1, int cta_cells) {
  constexpr int NV = 2 * NF + 4 * FIN_K64;  // values per lens
  constexpr int NS = (4 * 2 * NF + 31) / 32;  // FP32 sums per lane
  __shared__ float val_s[FG_WARPS][NV][33];
  __shared__ int from_s[FG_WARPS][4][FG_RANGES], off_s[FG_WARPS][4][FG_RANGES + 1];
  __shared__ float2 sum_s[FG_CELLS][2 * FIN_K64];
  // No after_ready: the ray pass that follows is a grid of CTAs that stay, six
  // to an SM.  Started beside this kernel's CTAs they found its shared memory
  // in pieces and 100 of 152 SMs kept only five of them to the end (paper-mid
  // map 12.0 ms, 11.5 this way; high-res 128.7 and 123.0; 128^2 149 and 148 us).
  after_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t base = rc0 + (int64_t)blockIdx.x * cta_cells;
  const int64_t ncells = (int64_t)ig.ncx * ig.ncy;
  const double h = ig.h, inv_h = 1.0 / h;
  const double ks = g.kstar_scale * msum[0];
  const float inv_hf = (float)inv_h, ksf = (float)ks;
  const bool table = g.plane != IRS_PLANE_CIRCLE && ks != 0.0;
  const int K = ig.K, nsf = K - FIN_K64, W = ig.W, nr = 2 * W + 4;
  const float2 ih_df = df_from_double(inv_h);
  for (int grp = warp; grp < cta_cells / 4; grp += FG_WARPS) {
    if (base + 4 * grp >= rc1) break;  // uniform over the warp
    // ---- this lane's cell and the list ranges of its window: rows dy = -W ... W
    // of cells x - W ... x + W, the middle three without their near columns
    const int ci = lane >> 3, sub = lane & 7;
    const int64_t rc = base + 4 * grp + ci;
    const bool cell_on = rc < rc1;
    const int cx = (int)(rc % ig.nrcx) + ig.ox, cy = (int)(rc / ig.nrcx) + ig.oy;
    int total = 0;
    for (int r0 = 0; r0 < nr; r0 += FG_LANES) {
      const int r = r0 + sub;
      int from = 0, len = 0;
      if (cell_on && r < nr) {
        int dy, xa = cx - W, xb = cx + W;
        if (r < W - 1) dy = r - W;
        else if (r < W + 5) {
          dy = (r - (W - 1)) / 2 - 1;
          if ((r - (W - 1)) & 1) xa = cx + 2; else xb = cx - 2;
        } else dy = r - (W + 5) + 2;
        const int y = cy + dy;
        xa = max(xa, 0);
        xb = min(xb, ig.ncx - 1);
        if (y >= 0 && y < ig.ncy && xa <= xb) {
          from = start[(int64_t)y * ig.ncx + xa];
          len = start[(int64_t)y * ig.ncx + xb + 1] - from;
        }
      }
      int inc = len;
#pragma unroll
      for (int d = 1; d < FG_LANES; d <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, inc, d, FG_LANES);
        if (sub >= d) inc += v;
      }
      if (r < nr) {
        from_s[warp][ci][r] = from;
        off_s[warp][ci][r] = total + inc - len;
      }
      total += __shfl_sync(0xFFFFFFFFu, inc, FG_LANES - 1, FG_LANES);
    }
    if (sub == 0) off_s[warp][ci][nr] = total;
    __syncwarp();
    const double zx = ig.gx0 + (cx + 0.5) * h, zy = ig.gy0 + (cy + 0.5) * h;
    const float2 zx_df = df_from_double(zx), zy_df = df_from_double(zy);
    // ---- sums this lane keeps: FP32 component j of cell c for index lane + 32 i,
    // and one double-float component of a cell for lanes < 24
    float accf[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) accf[i] = 0.f;
    float2 accd = make_float2(0.f, 0.f);
    const int dc = lane / (2 * FIN_K64), dj = lane % (2 * FIN_K64);  // double-float sum: cell, component
    int steps = (total + FG_LANES - 1) / FG_LANES;
#pragma unroll
    for (int d = FG_LANES; d < 32; d <<= 1) steps = max(steps, __shfl_xor_sync(0xFFFFFFFFu, steps, d));
    int r = 0;
    float4 next_q = make_float4(0.f, 0.f, 0.f, 0.f);  // the lane's next lens, loaded a step ahead
    float2 next_m = make_float2(0.f, 0.f);
    auto load = [&](int t) {
      if (t >= total) return;
      while (t >= off_s[warp][ci][r + 1]) ++r;
      const int p = from_s[warp][ci][r] + (t - off_s[warp][ci][r]);
      next_q = pos_df[p];
      next_m = m_df[p];
    };
    load(sub);
    for (int step = 0; step < steps; ++step) {
      const int t = step * FG_LANES + sub;
      const float4 q4 = next_q;
      const float2 m2 = next_m;
      load(t + FG_LANES);
      if (t < total) {
        const float2 dre = df_mul(df_sub(dfc_re(q4), zx_df), ih_df);
        const float2 dim = df_mul(df_sub(dfc_im(q4), zy_df), ih_df);
        const float4 inv = dfc_recip(dre, dim);
        float4 pw = dfc_scale(inv, m2);  // + m d^-(k+1)
#pragma unroll
        for (int k = 0; k < FIN_K64; ++k) {
          val_s[warp][4 * k][lane] = pw.x;
          val_s[warp][4 * k + 1][lane] = pw.z;
          val_s[warp][4 * k + 2][lane] = pw.y;
          val_s[warp][4 * k + 3][lane] = pw.w;
          pw = dfc_mul(pw, inv);
        }
        const float2 invf = dfc_hi(inv);
        float2 pf = dfc_hi(pw);
#pragma unroll
        for (int k = 0; k < NF; ++k) {
          val_s[warp][4 * FIN_K64 + 2 * k][lane] = pf.x;
          val_s[warp][4 * FIN_K64 + 2 * k + 1][lane] = pf.y;
          pf = cmulf(pf, invf);
        }
      } else {  // no lens: zeros leave every sum as it is
#pragma unroll
        for (int v = 0; v < NV; ++v) val_s[warp][v][lane] = 0.f;
      }
      __syncwarp();
      if (lane < 4 * 2 * FIN_K64) {
#pragma unroll
        for (int i = 0; i < FG_LANES; ++i)
          accd = df_add(accd, make_float2(val_s[warp][2 * dj][dc * FG_LANES + i], val_s[warp][2 * dj + 1][dc * FG_LANES + i]));
      }
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int idx = lane + 32 * s, c = idx / (2 * NF), j = idx - c * (2 * NF);
        if (4 * 2 * NF % 32 == 0 || c < 4) {
          const float* v = &val_s[warp][4 * FIN_K64 + j][c * FG_LANES];
#pragma unroll
          for (int i = 0; i < FG_LANES; ++i) accf[s] += v[i];
        }
      }
      __syncwarp();
    }
    if (lane < 4 * 2 * FIN_K64) sum_s[4 * grp + dc][dj] = accd;
    // ---- terms k >= FIN_K64: M2L result, 1/h, sheet
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int idx = lane + 32 * s, c = idx / (2 * NF), j = idx - c * (2 * NF), k = FIN_K64 + (j >> 1);
      const int64_t crc = base + 4 * grp + c;
      if (c < 4 && crc < rc1 && k < K) {
        float v = accf[s];
        const int64_t cell = (int64_t)((int)(crc / ig.nrcx) + ig.oy) * ig.ncx + (int)(crc % ig.nrcx) + ig.ox;
        if (k < IP_KF) v += reinterpret_cast<const float*>(conv_f + (int64_t)(k - IP_KD) * ncells + cell)[j & 1];
        v *= inv_hf;
        if (table) v = fmaf(ksf, reinterpret_cast<const float*>(sheet_f + crc * nsf + (k - FIN_K64))[j & 1], v);
        reinterpret_cast<float*>(coef + crc * K + k)[j & 1] = v;
      }
    }
  }
  __syncthreads();
  // ---- the FP64 end, one lane per cell
  const int64_t rc = base + threadIdx.x;
  if ((int)threadIdx.x >= cta_cells || rc >= rc1) return;
  const int cx = (int)(rc % ig.nrcx) + ig.ox, cy = (int)(rc / ig.nrcx) + ig.oy;
  const int64_t c = (int64_t)cy * ig.ncx + cx;
  const double zx = ig.gx0 + (cx + 0.5) * h, zy = ig.gy0 + (cy + 0.5) * h;
  cd acc[FIN_K64];
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) {
    acc[k] = {df_to_double(sum_s[threadIdx.x][2 * k]), df_to_double(sum_s[threadIdx.x][2 * k + 1])};
    const float4 v = conv_d[(int64_t)k * ncells + c];
    acc[k].re += df_to_double(dfc_re(v));
    acc[k].im += df_to_double(dfc_im(v));
    acc[k].re *= inv_h;
    acc[k].im *= inv_h;
  }
  finish_cell(g, ig, ks, zx, zy, rc, acc, true, sheet_d, sheet_near, recs, coef);
}

// The same for learned far fields and for windows wider than FG_WMAX cells: one
// thread per cell.
template <int NF>
__global__ void __launch_bounds__(64)
k_ip_finalize(Geo g, IpGeo ig, const double* msum, const int32_t* start, const double2* pos, const double* m,
              const float4* pos_df, const float2* m_df, const float4* conv_d, const float2* conv_f, MlpFar far,
              const double2* __restrict__ sheet_d,
              const float2* __restrict__ sheet_f, const uint8_t* __restrict__ sheet_near,
              CellRec* __restrict__ recs, float2* __restrict__ coef, int64_t rc0, int64_t rc1) {
  after_wait();  // no after_ready, as above
  const int64_t rc = rc0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (rc >= rc1) return;
  const int cx = (int)(rc % ig.nrcx) + ig.ox, cy = (int)(rc / ig.nrcx) + ig.oy;
  const int64_t ncells = (int64_t)ig.ncx * ig.ncy;
  const int64_t c = (int64_t)cy * ig.ncx + cx;
  const double zx = ig.gx0 + (cx + 0.5) * ig.h, zy = ig.gy0 + (cy + 0.5) * ig.h;
  const double h = ig.h, inv_h = 1.0 / h;
  const int K = ig.K;

  // coefficients of tau^k before the 1/h of the lens parts: k < FIN_K64 in
  // FP64, the rest in FP32 (terms past K are computed and dropped)
  cd acc[FIN_K64];
  float2 accf[NF];
  float4 accd[FIN_K64];  // the window's terms k < FIN_K64 in double-float (series mode)
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) {
    acc[k] = {0.0, 0.0};
    accd[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int k = 0; k < NF; ++k) accf[k] = make_float2(0.f, 0.f);
  const float2 zx_df = df_from_double(zx), zy_df = df_from_double(zy), ih_df = df_from_double(inv_h);
  // direct ring: lenses of cells at Chebyshev distance 2..W (series mode), or
  // every lens outside the near block weighted by w(r) out to R_f (network
  // mode).  The (cell, lens) pairs are walked as one sequence per thread, one
  // lens per step, so that the lanes of a warp, whose windows hold different
  // numbers of lenses per cell, stay busy until their own lenses run out.
  const int Wd = far.active ? (int)ceil(far.rf) + 1 : ig.W;
  const int side = 2 * Wd + 1, nwin = side * side;
  int q = -1, p = 0, pend = 0;  // window cell (row-major), lens range left in it
  while (true) {
    while (p >= pend && ++q < nwin) {
      const int dy = q / side - Wd, dx = q % side - Wd;
      const int x = cx + dx, y = cy + dy;
      if ((abs(dx) <= 1 && abs(dy) <= 1) || x < 0 || x >= ig.ncx || y < 0 || y >= ig.ncy) continue;
      const int64_t s = (int64_t)y * ig.ncx + x;
      p = start[s];
      pend = start[s + 1];
    }
    if (q >= nwin) break;
    const int pl = p++;  // this step's lens (the step always advances)
    float2 invf, pf;
    if (far.active) {  // network mode: the ring weight wants |d| in FP64
      const cd d = {(pos[pl].x - zx) * inv_h, (pos[pl].y - zy) * inv_h};
      const double wm = m[pl] * mlp_ring_weight(hypot(d.re, d.im), far.rf);
      if (wm == 0.0) continue;
      const cd inv = crecip_nr(d);
      cd pw = {wm * inv.re, wm * inv.im};  // + m d^-(k+1)
#pragma unroll
      for (int k = 0; k < FIN_K64; ++k) {
        acc[k].re += pw.re;
        acc[k].im += pw.im;
        pw = cmul(pw, inv);
      }
      invf = make_float2((float)inv.re, (float)inv.im);
      pf = make_float2((float)pw.re, (float)pw.im);
    } else {  // series mode: the same terms in double-float on the FP32 pipes
      const float4 q4 = pos_df[pl];
      const float2 dre = df_mul(df_sub(dfc_re(q4), zx_df), ih_df);
      const float2 dim = df_mul(df_sub(dfc_im(q4), zy_df), ih_df);
      const float4 inv = dfc_recip(dre, dim);
      float4 pw = dfc_scale(inv, m_df[pl]);  // + m d^-(k+1)
#pragma unroll
      for (int k = 0; k < FIN_K64; ++k) {
        accd[k] = dfc_add(accd[k], pw);
        pw = dfc_mul(pw, inv);
      }
      invf = dfc_hi(inv);
      pf = dfc_hi(pw);
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      accf[k].x += pf.x;
      accf[k].y += pf.y;
      pf = cmulf(pf, invf);
    }
  }
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) {
    acc[k].re += df_to_double(dfc_re(accd[k]));
    acc[k].im += df_to_double(dfc_im(accd[k]));
  }
  // outer cells through the FFT convolution (series mode)
  if (!far.active) {
#pragma unroll
    for (int k = 0; k < IP_KF; ++k) {
      if (k >= K) break;
      if (k < FIN_K64) {
        const float4 v = conv_d[(int64_t)k * ncells + c];
        acc[k].re += df_to_double(dfc_re(v));
        acc[k].im += df_to_double(dfc_im(v));
      } else {
        const float2 v = conv_f[(int64_t)(k - IP_KD) * ncells + c];
        accf[k - FIN_K64].x += v.x;
        accf[k - FIN_K64].y += v.y;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < FIN_K64; ++k) {
    acc[k].re *= inv_h;
    acc[k].im *= inv_h;
  }
  const float inv_hf = (float)inv_h;
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    accf[k].x *= inv_hf;
    accf[k].y *= inv_hf;
  }
  // network mode away from corners: G = -L_ring - U - kappa_* conj(z_C); the
  // sheet's g cancels against the definition of U
  const bool learned = far.active && far.corner[rc] < 0;
  if (far.active && !learned) {  // corner zone: exact far-far sum, then the sheet as usual
    const double2* ex = far.exact + (int64_t)far.corner[rc] * MLP_KEXACT;
#pragma unroll
    for (int k = 0; k < MLP_KEXACT; ++k) {
      if (k >= K) break;
      if (k < FIN_K64) {
        acc[k].re -= ex[k].x;
        acc[k].im -= ex[k].y;
      } else {
        accf[k - FIN_K64].x -= (float)ex[k].x;
        accf[k - FIN_K64].y -= (float)ex[k].y;
      }
    }
  }

  const double ks = g.kstar_scale * msum[0];
  if (learned) {
#pragma unroll
    for (int k = 0; k < MLP_KFF; ++k) {
      if (k >= K) break;
      const float2 u = far.U[rc * MLP_KFF + k];
      if (k < FIN_K64) {
        acc[k].re -= (double)u.x;
        acc[k].im -= (double)u.y;
      } else {
        accf[k - FIN_K64].x -= u.x;
        accf[k - FIN_K64].y -= u.y;
      }
    }
    acc[0].re -= ks * zx;  // kappa_* conj(z_C)
    acc[0].im += ks * zy;
  } else if (g.plane != IRS_PLANE_CIRCLE && ks != 0.0) {
    const int nsf = K - FIN_K64;
    const float ksf = (float)ks;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      if (k >= nsf) break;
      const float2 t = sheet_f[rc * nsf + k];
      accf[k].x = fmaf(ksf, t.x, accf[k].x);
      accf[k].y = fmaf(ksf, t.y, accf[k].y);
    }
  }
  finish_cell(g, ig, ks, zx, zy, rc, acc, !learned, sheet_d, sheet_near, recs, coef);
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    if (FIN_K64 + k >= K) break;
    coef[rc * K + FIN_K64 + k] = accf[k];
  }
}

// ------------------------------------------------------------ ray pass
struct IpRayArgs {
  const int32_t* start;
  const float4* rel;
  const CellRec* recs;
  const float2* coef;
  uint32_t* counts;
  int* status;
  int64_t row0, row1;
  int64_t rc_base;  // first ray cell of the work range
  const int64_t* idx;
  double* beta_out;
  int64_t* pix_out;
  int64_t nwork;
  unsigned long long* queue;  // work counter of the launch, zero before it
  int32_t near_cap;           // lenses of a 3x3 block the CTA's shared memory holds
  int32_t parts;              // work items per cell, each a share of its row groups
};

// Kernel variants of the ray pass (the autotuner picks one per plan):
// level-2 sub-cells per side Q, sub-cell series terms K2, and NPR: how many of
// a thread's four row pairs share one reciprocal per lens, 1/(r_a^2 r_b^2)
// (the MUFU's 16 reciprocals per SM per clock bound the near sum; a shared
// reciprocal trades one MUFU op for FP32 work).  The truncation is (sub-cell
// half-diagonal / distance to the nearest far lens)^K2 of that lens's field:
// Q = 8, 10, 12, 16 give ratios 0.083, 0.067, 0.057, 0.042, so 8, 7, 6 and 6
// terms stay at or below ~3e-8; variants 11, 14 and 15 trade one Horner step
// per ray for bounds of 1.7e-7 (16 sub-cells, 5 terms), 3.3e-7 (14) and 7.3e-7
// (12), the last with fewer sub-cells to re-centre per cell; variant 16 takes
// one more step off with 4 terms on 16 sub-cells (3.1e-6, more sub-cells to
// re-centre).  Variant numbers that differ only in launch shape or binning
// share one kernel: every launch is shaped from the cell (ip_launch_shape).
#define IP_VARIANTS(X)                                                                     \
  X(0, 12, 6, 0) X(1, 10, 7, 0) X(2, 16, 6, 2) X(3, 16, 6, 4) X(5, 16, 6, 0) X(9, 8, 8, 0) \
  X(11, 16, 5, 0) X(14, 12, 5, 0) X(15, 14, 5, 0) X(16, 16, 4, 0)
constexpr int IP_NVARIANT = 17;
// the variant whose kernel serves variant v
constexpr int ip_kernel_of(int v) {
  return v == 4 || v == 7 || v == 8 ? 5 : v == 6 ? 2 : v == 10 ? 0 : v == 12 || v == 13 ? 11 : v;
}

constexpr int IP_R = 8;  // rays per thread and unit: one lattice column, four row pairs

// Row pairs of the row table past the cell's last: a thread's four pairs are
// read without clamping the index.
constexpr int IP_ROW_PAD = 4;
static_assert(IP_R <= 2 * IP_ROW_PAD, "row table padding");

// Row stride (float2) of the per-cell table of scaled series coefficients:
// odd, so that the K2 rows a warp reads at once fall in distinct banks.
constexpr int IP_CB_STRIDE = IP_KMAX + 1;

// Binning box: a CTA counts its cell's rays in a shared-memory histogram of
// 32 x 64 pixels placed
// around the block's position under the near lenses' softened pull and adds the
// non-empty bins to the map once per box (87-98 % of the rays fall inside).  An increment by one of a shared word is a single instruction that
// the hardware resolves for all lanes at once, equal addresses included:
// 1.25 SM cycles per warp whatever the number of distinct pixels, against 2.1
// per distinct pixel for __match_any_sync, which the binning used before.  The
// paper-mid ray pass took 28.0 ms with match-and-add into the map and 26.0 ms
// with this histogram (same loop otherwise; 64 x 64 pixels: 26.6 ms, the
// larger flush costs more than the fewer rays outside save).
constexpr int IP_BOX_W = 32, IP_BOX_H = 64;
constexpr int IP_HS = IP_BOX_W;  // row stride in words
constexpr int IP_HIST = IP_HS * IP_BOX_H;

// Dynamic shared memory of the ray pass: the level-2 series as conj duplicated
// (c.re, c.re, -c.im, -c.im), the histogram, the level-1 series scaled for the
// re-centring with its scale factors, the row table, and the near lenses.  Tables
// of fixed size come first, so that the addresses of the hot ones are constants.
struct __align__(16) IpRowPair {  // one entry per pair of cell rows (2l, 2l + 1)
  float4 sg;      // (sigma_y, sigma_y', -sigma_y, -sigma_y'), sigma_y = (l + 1/2) Q/k - v - 1/2
  float4 ty;      // (tau_y h, tau_y' h, y0, y0'), y0 = by_lo + lambda_2 tau_y h: the row's share of beta_2
  int q4;         // byte offset of the level-2 row shared by this pair and the next, or -1
  uint16_t v[2];  // the two rows' level-2 rows times Q
  int pad[2];
};
struct __align__(16) IpNear {  // a lens of the 3x3 block
  float4 xy;  // (-x, -x, -y, -y)
  float2 m;   // (-m, -m)
  float pad[2];
};
// float4s per level-2 sub-cell: odd, so that the eight sub-cells that a quarter
// of a warp reads or writes at once lie in distinct banks (with 4, 6 or 8
// terms back to back, 2, 2 and 8 of them share one)
__host__ __device__ constexpr int ip_sub_stride(int k2) { return k2 | 1; }
template <int Q, int K2>
struct IpSmem {
  static constexpr int sub = 0;
  static constexpr int hist = sub + 16 * Q * Q * ip_sub_stride(K2);
  static constexpr int cb = hist + 4 * IP_HIST;
  static constexpr int sc = cb + 8 * K2 * IP_CB_STRIDE;
  static constexpr int keep = sc + 4 * K2 * IP_CB_STRIDE;  // a bit per work unit of a cell
  static constexpr int row = (keep + (IP_KMAX_RAYS / 32) * (IP_KMAX_RAYS / IP_R) / 8 + 15) & ~15;
  int near, bytes;
  __host__ __device__ IpSmem(int nrow, int near_cap) {
    near = row + (int)sizeof(IpRowPair) * nrow;
    bytes = near + (int)sizeof(IpNear) * near_cap;
  }
};

// A CTA's tables that depend on the plan's geometry alone: written once per
// launch (per map in a batch), with y0 and x0 left to each cell.
template <int Q, int K2>
__device__ __forceinline__ void ip_tables(const IpGeo& ig, const IpSmem<Q, K2>& L, unsigned char* sm) {
  IpRowPair* row_s = reinterpret_cast<IpRowPair*>(sm + L.row);
  float* sc_s = reinterpret_cast<float*>(sm + L.sc);
  constexpr int SUB = 16 * ip_sub_stride(K2);  // bytes per sub-cell
  const int tid = threadIdx.x, nt = blockDim.x;
  const float hf = ig.hf, inv_k = ig.inv_k;
  const float qk = __fmul_rn((float)Q, inv_k);  // sub-cell index = floor((l + 1/2) Q / k)
  auto level2 = [&](int l, float& s) {
    s = __fmul_rn(__fadd_rn((float)l, 0.5f), qk);
    return min(__float2int_rd(s), Q - 1);
  };
  // rows of the whole cell side and IP_ROW_PAD pairs past it (rows past the
  // cell side are never binned; their sub-cell row is clamped to Q - 1)
  for (int pr = tid; pr < ig.nrow; pr += nt) {
    float t[2], s[2];
    int v[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int l = 2 * pr + j;
      float sv;
      v[j] = level2(l, sv);
      t[j] = __fmul_rn(fmaf((float)l, inv_k, fmaf(0.5f, inv_k, -0.5f)), hf);
      s[j] = __fsub_rn(__fsub_rn(sv, (float)v[j]), 0.5f);
    }
    float s3;
    const int v3 = level2(2 * pr + 3, s3);
    row_s[pr].sg = make_float4(s[0], s[1], -s[0], -s[1]);
    row_s[pr].ty = make_float4(t[0], t[1], 0.f, 0.f);
    row_s[pr].q4 = v[0] == v3 ? v[0] * Q * SUB : -1;
    row_s[pr].v[0] = (uint16_t)(v[0] * Q);
    row_s[pr].v[1] = (uint16_t)(v[1] * Q);
  }
  // Q^-n binom(kk, n) (binomials exact in FP32 for kk < 32)
  const float inv_q = __fdiv_rn(1.0f, (float)Q);
  for (int t = tid; t < K2 * IP_CB_STRIDE; t += nt) {
    const int nn = t / IP_CB_STRIDE, kk = t % IP_CB_STRIDE;
    float sc = 0.f;
    if (kk >= nn && kk >= 1) {
      int b = 1;  // binom(kk, nn), exact integer steps
      for (int i = 1; i <= nn; ++i) b = b * (kk - nn + i) / i;
      sc = (float)b;
      for (int i = 0; i < nn; ++i) sc = __fmul_rn(sc, inv_q);
    }
    sc_s[t] = sc;
  }
  uint32_t* hist_s = reinterpret_cast<uint32_t*>(sm + L.hist);
  for (int t = tid; t < IP_HIST; t += nt) hist_s[t] = 0u;
}

// A sheet corner near the cell, for one ray: -i a_c (z - c) Log(z - c) added to
// the conjugate series (qr, qi); corner = ((z_C - c).re, .im, a_c).
__device__ __forceinline__ void sheet_corner_ray(const float* corner, float tx, float ty, float& qr, float& qi) {
  const float wr = __fadd_rn(corner[0], tx), wi = __fadd_rn(corner[1], ty);
  const float lr = __fmul_rn(0.5f, logf(fmaf(wr, wr, __fmul_rn(wi, wi)))), li = atan2f(wi, wr);
  const float plr = fmaf(wr, lr, -__fmul_rn(wi, li)), pli = fmaf(wr, li, __fmul_rn(wi, lr));
  qr = fmaf(corner[2], pli, qr);
  qi = fmaf(corner[2], plr, qi);
}

// Shared-memory words at four byte addresses incremented by one where `on`.
__device__ __forceinline__ void shared_inc4(uint32_t a, uint32_t b, uint32_t c, uint32_t d, bool on) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n @p red.shared.add.u32 [%0], 1;\n"
      " @p red.shared.add.u32 [%1], 1;\n @p red.shared.add.u32 [%2], 1;\n @p red.shared.add.u32 [%3], 1;\n}" ::"r"(a),
      "r"(b), "r"(c), "r"(d), "r"((uint32_t)on)
      : "memory");
}

// Re-centring: pairs of sub-cells per thread.  They share each coefficient read
// from shared memory, and their Horner chains interleave.
constexpr int IP_RC = 4;

// One level-1 cell: gather the 3x3 block's lenses, re-centre the series on the
// sub-cells, then every ray of rows [row0, row1) of the cell.
//
// Each thread takes one lattice column and eight rows; rows go in pairs through
// the packed FP32x2 instructions (two rows share the column's dx and sigma_x),
// which round exactly as the scalar ones.  The accumulators hold -alpha (the
// masses are stored negated) and the level-2 Horner runs on the conjugate, so
// no negation is issued per ray.  The pass is bound by instruction issue (0.69
// of the slots, FP32 pipe 51 %, MUFU 29 %), so
// what is the same for a row comes from a table, four rows that share a level-2
// row read its series once, the sheet's corners sit on the general path of the
// tail only, and a last strip of few columns takes several row groups at once
// (a 45-ray cell: 83 % of the lanes busy instead of 70 %).  Ray pass, one
// GB300, every ray evaluated, against the form with match-and-add binning, fixed
// cells per CTA and one set-up chain per thread: paper-mid 20.2 ms (28.0), high-res 204 ms (275),
// a 500^2 map of 1e4 lenses 0.28 ms (0.44), 128^2 with 150 lenses 0.078 (0.088).
template <int Q, int K2, int NPR>
__device__ __forceinline__ void ip_cell(const Geo& g, const IpGeo& ig, const IpRayArgs& a, int64_t rc,
                                        int part, const IpSmem<Q, K2>& L, unsigned char* sm, long long next,
                                        long long* next_s) {
  static_assert(NPR >= 0 && NPR <= IP_R / 2, "paired row pairs");
  constexpr int SUB = 16 * ip_sub_stride(K2);  // bytes per sub-cell
  float4* sub_s = reinterpret_cast<float4*>(sm + L.sub);
  uint32_t* hist_s = reinterpret_cast<uint32_t*>(sm + L.hist);
  float2* cb_s = reinterpret_cast<float2*>(sm + L.cb);
  const float* sc_s = reinterpret_cast<const float*>(sm + L.sc);
  IpRowPair* row_s = reinterpret_cast<IpRowPair*>(sm + L.row);
  IpNear* near_s = reinterpret_cast<IpNear*>(sm + L.near);
  __shared__ CellRec rec_s;
  __shared__ int blk_start[9], blk_off[10];
  __shared__ float series_s;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);  // uniform
  // Every FP32 step of the cell's ray geometry below is written with explicit
  // rounding (__fadd_rn, __fmul_rn, __fdiv_rn, fmaf): implicit contraction
  // would depend on how the compiler places the code in each kernel that
  // inlines this function, and the single-map and batched ray passes must
  // give the same maps bit for bit.
  const float hf = ig.hf;
  const int k = (int)ig.k;
  const int rcx = (int)(rc % ig.nrcx), rcy = (int)(rc / ig.nrcx);
  const int cx = rcx + ig.ox, cy = rcy + ig.oy;
  const int64_t i0 = (int64_t)rcx * k, j0 = (int64_t)rcy * k;
  const int64_t jlo = max(j0, a.row0), jhi = min(min(j0 + k, g.nry), a.row1);
  // cell-local lattice indices: columns [0, kx), rows [ylo, yhi), of these the
  // row groups [grg0, nrg) of this part; units start on an even row so that row
  // pairs line up with the table, and on a multiple of R where only some of a
  // unit's pairs share a reciprocal, so that a band's rays round as the map's do
  constexpr int R = IP_R;
  constexpr int ANCHOR = NPR > 0 && NPR < R / 2 ? R : 2;
  const int kx = (int)(min(i0 + k, g.nrx) - i0), ylo = (int)(jlo - j0), yhi = (int)(jhi - j0);
  const int ylo2 = ylo & ~(ANCHOR - 1);
  int grg0 = 0, nrg = jlo < jhi ? (yhi - ylo2 + R - 1) / R : 0;
  if (a.parts > 1) {
    const int all = nrg;
    grg0 = all * part / a.parts;
    nrg = all * (part + 1) / a.parts;
  }
  if (grg0 >= nrg) {  // nothing to shoot; uniform over the CTA
    __syncthreads();  // everyone has read the item before
    if (tid == 0) *next_s = next;
    __syncthreads();
    return;
  }
  if (warp == 0) {
    // lane q < 9 takes cell q of the 3x3 block (row-major from the lower
    // left); the block's lens offsets are the exclusive prefix sum of the counts
    int s0 = 0, cnt = 0;
    if (lane < 9) {
      const int x = cx + (lane % 3) - 1, y = cy + (lane / 3) - 1;
      if (x >= 0 && x < ig.ncx && y >= 0 && y < ig.ncy) {
        const int64_t s = (int64_t)y * ig.ncx + x;
        s0 = a.start[s];
        cnt = a.start[s + 1] - s0;
      }
    }
    int inc = cnt;
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
      const int v = __shfl_up_sync(0xFFFFFFFFu, inc, d);
      if (lane >= d) inc += v;
    }
    if (lane < 9) {
      blk_start[lane] = s0;
      blk_off[lane] = inc - cnt;
    }
    if (lane == 8) {
      int off = inc;
      if (off > IP_NEAR_MAX) {
        atomicCAS(a.status, 0, (int)IRS_ERR_OVERFLOW);  // the first error stays
        off = IP_NEAR_MAX;
      }
      blk_off[9] = off;
    }
  } else if (warp == 1 && lane < (int)(sizeof(CellRec) / 4)) {
    reinterpret_cast<uint32_t*>(&rec_s)[lane] = reinterpret_cast<const uint32_t*>(a.recs + rc)[lane];
  }
  else if (warp == 2) {
    // bound of |sum_kk c_kk w^kk| over the cell, |w| <= 1/sqrt(2), which also
    // bounds the re-centred, truncated form (its terms expand the same powers
    // of |eps| + |sigma|/Q <= 1/sqrt(2))
    float v = 0.f;
    if (lane >= 1 && lane < ig.K) {
      const float2 c = a.coef[rc * ig.K + lane];
      v = (fabsf(c.x) + fabsf(c.y)) * exp2f(-0.4999f * (float)lane);
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    if (lane == 0) series_s = v;
  }
  // Level 2 re-centres the cell series sum_kk c_kk w^kk (w in cell units,
  // terms from 1: term 0 sits in the cell's base) on the sub-cell centres
  // eps: with w = eps + sigma / Q the coefficient of sigma^n is
  // Q^-n sum_kk binom(kk, n) c_kk eps^(kk - n).  First the per-cell table
  // cb[n][kk] = Q^-n binom(kk, n) c_kk.
  for (int t = tid; t < K2 * IP_KMAX; t += nt) {
    const int nn = t / IP_KMAX, kk = t % IP_KMAX;
    if (kk < ig.K) {
      const float2 c = a.coef[rc * ig.K + kk];
      const float sc = sc_s[nn * IP_CB_STRIDE + kk];
      cb_s[nn * IP_CB_STRIDE + kk] =
          kk >= 1 ? make_float2(__fmul_rn(c.x, sc), __fmul_rn(c.y, sc)) : make_float2(0.f, 0.f);
    }
  }
  __syncthreads();
  const int n_near = __shfl_sync(0xFFFFFFFFu, blk_off[9], 0);
  const bool near_fits = n_near <= a.near_cap;
  // lens t of the block relative to the cell's centre
  auto near_lens = [&](int t) {
    int q = 0;
#pragma unroll
    for (int i = 1; i < 9; ++i) q += t >= blk_off[i] ? 1 : 0;
    float4 v = a.rel[blk_start[q] + (t - blk_off[q])];
    v.x = __fadd_rn(v.x, __fmul_rn((float)((q % 3) - 1), hf));
    v.y = __fadd_rn(v.y, __fmul_rn((float)((q / 3) - 1), hf));
    return v;
  };
  // this thread's first lens is in flight during the re-centring
  float4 lens0 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (near_fits && tid < n_near) lens0 = near_lens(tid);
  auto store_lenses = [&]() {
    if (!near_fits) return;
    if (tid < n_near) {
      near_s[tid].xy = make_float4(-lens0.x, -lens0.x, -lens0.y, -lens0.y);
      near_s[tid].m = make_float2(-lens0.z, -lens0.z);
    }
    for (int t = tid + nt; t < n_near; t += nt) {
      const float4 v = near_lens(t);
      near_s[t].xy = make_float4(-v.x, -v.x, -v.y, -v.y);
      near_s[t].m = make_float2(-v.z, -v.z);
    }
  };
  // Rays that cannot reach the map.  A cell whose smooth and far-field beta lies
  // off the map by more than `room` sends a ray onto it only where the near
  // lenses pull by `room`, sum_i |m_i| / |t - t_i| >= room: in small discs
  // around them.  Work units (32 columns x 8 rows) that touch no disc are left
  // out, and so is the set-up of a cell with none left.  The protective border
  // makes most cells of a plane such cells: 40 % of the paper-mid units are
  // left (48 % at high-res, 32 % of a 500^2 map, 24 % of a circular plane) and
  // the pass takes 10.2 instead of 20.3 ms (115 for 205, 0.20 for 0.28, 0.47
  // for 0.85).  `room` keeps a margin of 2 % of the series' bound, two pixels
  // and 1e-3 of a cell, far above the FP32 error of a ray; a NaN anywhere keeps
  // the unit.  Maps are the same bits.
  const int nstrip = (kx + 31) / 32, ngrp = nrg - grg0;
  const float room = rec_s.off - 1.02f * series_s - 2.0f * fmaxf(__frcp_rn(g.inv_sx), __frcp_rn(g.inv_sy)) - 1e-3f * hf;
  const bool cull = room > 0.f && rec_s.n_corner == 0;
  uint32_t* keep_s = reinterpret_cast<uint32_t*>(sm + L.keep);  // bit per unit, strip-major
  if (cull) {
    store_lenses();
    __syncthreads();
    const float dxr = hf * ig.inv_k;
    bool any = false;
    for (int u = tid; u - lane < nstrip * ngrp; u += nt) {
      const int st = u / ngrp, gr = u - st * ngrp + grg0;
      const int w = min(32, kx - 32 * st);
      const float hx = 0.501f * (float)w * dxr + 1e-5f * hf, hy = 0.501f * (float)R * dxr + 1e-5f * hf;
      const float xc = ((float)(32 * st) + 0.5f * (float)w) * dxr - 0.5f * hf;
      const float yc = ((float)(ylo2 + gr * R) + 0.5f * (float)R) * dxr - 0.5f * hf;
      float pull = 0.f;
      auto add_pull = [&](float nx, float ny, float nm) {
        const float dx = fmaxf(fabsf(xc + nx) - hx, 0.f), dy = fmaxf(fabsf(yc + ny) - hy, 0.f);
        pull += fabsf(nm) * rsqrtf(dx * dx + dy * dy);
      };
      if (near_fits) {
        for (int q = 0; q < n_near; ++q) add_pull(near_s[q].xy.x, near_s[q].xy.z, near_s[q].m.x);
      } else {  // a lane fetches one of every 32 lenses, which pass from lane to lane
#pragma unroll 1
        for (int b0 = 0; b0 < n_near; b0 += 32) {
          const float4 v = b0 + lane < n_near ? near_lens(b0 + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
          for (int q = 0; q < min(32, n_near - b0); ++q)
            add_pull(-__shfl_sync(0xFFFFFFFFu, v.x, q), -__shfl_sync(0xFFFFFFFFu, v.y, q), __shfl_sync(0xFFFFFFFFu, v.z, q));
        }
      }
      const unsigned word = __ballot_sync(0xFFFFFFFFu, u < nstrip * ngrp && !(1.01f * pull < room));
      if (lane == 0) keep_s[u >> 5] = word;
      any = any || word != 0u;
    }
    if (tid == 0) *next_s = next;
    if (!__syncthreads_or(any)) return;  // the cell sends nothing onto the map
  }
  // then per (sub-cell, n) the polynomial sum_j cb[n][n + j] eps^j by Horner,
  // two sub-cells of one sub-cell row at a time (Q is even) through packed
  // FP32x2 instructions: the same roundings as two scalar Horner chains.  A
  // thread runs IP_RC of these chains at once.
  static_assert(Q % 2 == 0, "sub-cells go in pairs along a row");
  constexpr int NPAIR = Q * Q / 2;
  constexpr int NB = (NPAIR + IP_RC - 1) / IP_RC;  // batches of pairs per n
  const float inv_q = __fdiv_rn(1.0f, (float)Q);
  for (int t = tid; t < NB * K2; t += nt) {
    const int nn = t / NB, b = t - nn * NB;
    float2 ER[IP_RC], EI[IP_RC], NEI[IP_RC], SR[IP_RC], SI[IP_RC];
#pragma unroll
    for (int i = 0; i < IP_RC; ++i) {
      const int sa = 2 * min(b + i * NB, NPAIR - 1);  // sub-cells sa, sa + 1: same row, adjacent columns
      ER[i] = make_float2(__fmaf_rn(__fadd_rn((float)(sa % Q), 0.5f), inv_q, -0.5f),
                          __fmaf_rn(__fadd_rn((float)(sa % Q + 1), 0.5f), inv_q, -0.5f));
      const float ei = __fmaf_rn(__fadd_rn((float)(sa / Q), 0.5f), inv_q, -0.5f);
      EI[i] = make_float2(ei, ei);
      NEI[i] = make_float2(-ei, -ei);
      SR[i] = SI[i] = make_float2(0.f, 0.f);
    }
    const float2* cb = cb_s + nn * IP_CB_STRIDE;
#pragma unroll 2
    for (int kk = ig.K - 1; kk >= nn; --kk) {
      const float2 c = cb[kk];
#pragma unroll
      for (int i = 0; i < IP_RC; ++i) {
        const float2 NR = __ffma2_rn(SR[i], ER[i], __ffma2_rn(SI[i], NEI[i], make_float2(c.x, c.x)));
        SI[i] = __ffma2_rn(SR[i], EI[i], __ffma2_rn(SI[i], ER[i], make_float2(c.y, c.y)));
        SR[i] = NR;
      }
    }
#pragma unroll
    for (int i = 0; i < IP_RC; ++i) {
      const int sp = b + i * NB;
      if (NPAIR % IP_RC == 0 || sp < NPAIR) {
        sub_s[(2 * sp) * ip_sub_stride(K2) + nn] = make_float4(SR[i].x, SR[i].x, -SI[i].x, -SI[i].x);
        sub_s[(2 * sp + 1) * ip_sub_stride(K2) + nn] = make_float4(SR[i].y, SR[i].y, -SI[i].y, -SI[i].y);
      }
    }
  }
  // the rows' shares of beta
  for (int pr = tid; pr < ig.nrow; pr += nt) {
    float4 t = row_s[pr].ty;
    t.z = __fmaf_rn(g.lam_s2, t.x, rec_s.by_lo);
    t.w = __fmaf_rn(g.lam_s2, t.y, rec_s.by_lo);
    row_s[pr].ty = t;
  }
  if (!cull) store_lenses();
  __syncthreads();

  // base pixel of this cell for the 32-bit pixel test, folded with the
  // floor's bit pattern offset (pixel_keys2)
  const int32_t rix = rec_s.ix, riy = rec_s.iy;
  // the cell centre's beta (hi parts) in pixel units
  const float bxs = __fmul_rn(rec_s.bx_hi, g.inv_sx), bys = __fmul_rn(rec_s.by_hi, g.inv_sy);
  const float2 BXS = make_float2(bxs, bxs), BYS = make_float2(bys, bys);
  const float2 ISX = make_float2(g.inv_sx, g.inv_sx), ISY = make_float2(g.inv_sy, g.inv_sy);
  const int n_corner = __shfl_sync(0xFFFFFFFFu, rec_s.n_corner, 0);
  const int corner = n_corner ? -1 : 0;  // cells with sheet corners take the general path of the tail
  const float fnan = __int_as_float(0x7fffffff);
  const float ulp0 = __uint_as_float(1u);  // the smallest denormal, 2^-149
  const float2 ULP = make_float2(ulp0, ulp0);
  const float hist_f = __uint_as_float((uint32_t)__cvta_generic_to_shared(hist_s));
  const float c_tau = fmaf(0.5f, ig.inv_k, -0.5f);  // tau = (l + 1/2)/k - 1/2
  const float qk = __fmul_rn((float)Q, ig.inv_k);   // sub-cell index = floor((l + 1/2) Q / k)
  // blocks of the cell that map into about one box each; nearly always the
  // whole cell
  for (int g0 = grg0; g0 < nrg; g0 += ig.blk_rg) {
    for (int c0 = 0; c0 < kx; c0 += ig.blk_col) {
      const int w = min(ig.blk_col, kx - c0), ng = min(ig.blk_rg, nrg - g0);
      // box origin: the block centre's beta under the mean lens map plus the
      // near lenses' pull on it (softened), the same in every warp
      int box_x, box_y;
      {
        const float fx = w == k ? 0.f : ((float)c0 + 0.5f * (float)w) * ig.inv_k - 0.5f;
        const float fy = ng * R >= k ? 0.f : ((float)(ylo2 + g0 * R) + 0.5f * (float)(ng * R)) * ig.inv_k - 0.5f;
        float sx = 0.f, sy = 0.f;
        const float eps = 0.15f * hf * hf;
        for (int t = lane; t < n_near; t += 32) {
          float nx, ny, nm;
          if (near_fits) {
            nx = near_s[t].xy.x;
            ny = near_s[t].xy.z;
            nm = near_s[t].m.x;
          } else {
            const float4 v = near_lens(t);
            nx = -v.x;
            ny = -v.y;
            nm = -v.z;
          }
          const float x = fx * hf + nx, y = fy * hf + ny;
          const float wgt = nm / (x * x + y * y + eps);
          sx += wgt * x;
          sy += wgt * y;
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
          sx += __shfl_xor_sync(0xFFFFFFFFu, sx, d);
          sy += __shfl_xor_sync(0xFFFFFFFFu, sy, d);
        }
        const float ox = (rec_s.bx_hi + sx) * g.inv_sx + fx * ig.cell_px - 0.5f * IP_BOX_W;
        const float oy = (rec_s.by_hi + sy) * g.inv_sy + fy * ig.cell_py - 0.5f * IP_BOX_H;
        box_x = (int)fminf(fmaxf(ox, -1048576.f), 1048576.f);
        box_y = (int)fminf(fmaxf(oy, -1048576.f), 1048576.f);
      }
      // A ray's bin: floor(T) - box in units of the smallest denormal, whose
      // bit pattern is that integer when it is not negative.  One packed
      // multiply-add rounded toward -inf does both rays of a pair exactly; a
      // negative, infinite or NaN value has a pattern above every bin.  Two
      // more give the shared-memory addresses of the bins (their sums stay
      // below 2^23 units, hence exact).
      float mgx = -(float)box_x * ulp0, mgy = -(float)box_y * ulp0;
      asm volatile("" : "+f"(mgx), "+f"(mgy));  // kept, not converted again for every group
      const float2 MGX = make_float2(mgx, mgx), MGY = make_float2(mgy, mgy);
      const float2 HA = make_float2(hist_f, hist_f);

      // strips of 32 columns, walked down their row groups by the warps in
      // turn; in a last strip of w <= 16 columns the lanes take 32 / w row
      // groups at once
      int ru = warp;
      for (int cs = 0; cs < w; cs += 32) {
        const int ws = min(32, w - cs), par = 32 / ws, nru = (ng + par - 1) / par;
        if (ru >= nru) {
          ru -= nru;
          continue;
        }
        const int sub = lane / ws, c = c0 + cs + lane - sub * ws;
        const bool lane_on = sub < par;
        const float su = __fmul_rn(__fadd_rn((float)c, 0.5f), qk);
        const int u = min(__float2int_rd(su), Q - 1);
        const float sgx = __fsub_rn(__fsub_rn(su, (float)u), 0.5f);
        const float tx = __fmul_rn(fmaf((float)c, ig.inv_k, c_tau), hf);
        const float x0 = __fmaf_rn(g.lam_s1, tx, rec_s.bx_lo);  // the column's share of beta_1
        const float2 TX = make_float2(tx, tx), X0 = make_float2(x0, x0), SGR = make_float2(sgx, sgx);
        const char* sub_u = reinterpret_cast<const char*>(sub_s) + u * SUB;
#pragma unroll 1
        for (; ru < nru; ru += nt >> 5) {
        const int rg = ru * par + sub;
        bool live = lane_on && rg < ng;
        if (cull) {  // uniform over the CTA
          const int u = ((c0 + cs) >> 5) * ngrp + (g0 - grg0) + min(rg, ng - 1);
          live = live && ((keep_s[u >> 5] >> (u & 31)) & 1u);
          if (!__any_sync(0xFFFFFFFFu, live)) continue;
        }
        const int rl0 = ylo2 + (g0 + min(rg, ng - 1)) * R;
        const IpRowPair* rows = row_s + (rl0 >> 1);
        float2 TY[R / 2], NAX[R / 2], NAY[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) TY[i] = *reinterpret_cast<const float2*>(&rows[i].ty);
        // FIRST: the accumulators start from this lens (0 + w d is w d)
        auto near_step = [&](auto first, float2 NLX, float2 NLY, float2 NM) {
          const float2 DX = __fadd2_rn(TX, NLX);
          const float2 DX2 = __fmul2_rn(DX, DX);
#pragma unroll
          for (int i = 0; i < R / 2; ++i) {
            const float2 DY = __fadd2_rn(TY[i], NLY);
            const float2 R2 = __ffma2_rn(DY, DY, DX2);
            float2 W;
            if (i < NPR) {  // -m/r_a^2 = -m r_b^2 / (r_a^2 r_b^2), and the same for b
              const float mi = NM.x * rcp_approx(R2.x * R2.y);
              W = __fmul2_rn(make_float2(R2.y, R2.x), make_float2(mi, mi));
            } else {
              W = __fmul2_rn(NM, make_float2(rcp_approx(R2.x), rcp_approx(R2.y)));
            }
            NAX[i] = first ? __fmul2_rn(W, DX) : __ffma2_rn(W, DX, NAX[i]);
            NAY[i] = first ? __fmul2_rn(W, DY) : __ffma2_rn(W, DY, NAY[i]);
          }
        };
        if (n_near == 0 || !near_fits) {
#pragma unroll
          for (int i = 0; i < R / 2; ++i) NAX[i] = NAY[i] = make_float2(0.f, 0.f);
        }
        if (near_fits) {
          if (n_near > 0)
            near_step(std::true_type{}, make_float2(near_s[0].xy.x, near_s[0].xy.y),
                      make_float2(near_s[0].xy.z, near_s[0].xy.w), near_s[0].m);
#pragma unroll 2
          for (int q = 1; q < n_near; ++q) {
            const float4 v = near_s[q].xy;
            near_step(std::false_type{}, make_float2(v.x, v.y), make_float2(v.z, v.w), near_s[q].m);
          }
        } else {
          // more lenses than the shared buffer holds (a clump): each warp takes them
          // through its share of the buffer, a lane fetching one lens of a turn.
          // Every thread fetching every lens took 102 ms for a 2000^2 map with its 1e5
          // lenses in 4 % of the plane (75 with a buffer of 1024 for every block,
          // 42 now).
          const int slots = min(a.near_cap / (nt >> 5), 32);
          IpNear* mine = near_s + (tid >> 5) * slots;
#pragma unroll 1
          for (int b0 = 0; b0 < n_near; b0 += slots) {
            const int cnt = min(slots, n_near - b0);
            __syncwarp();
            if (lane < cnt) {
              const float4 v = near_lens(b0 + lane);
              mine[lane].xy = make_float4(-v.x, -v.x, -v.y, -v.y);
              mine[lane].m = make_float2(-v.z, -v.z);
            }
            __syncwarp();
#pragma unroll 1
            for (int q = 0; q < cnt; ++q) {
              const float4 v = mine[q].xy;
              near_step(std::false_type{}, make_float2(v.x, v.y), make_float2(v.z, v.w), mine[q].m);
            }
          }
        }
        // a group at the band's edge, the first or the last: rays outside its
        // rows get a NaN, which reaches beta and fails the pixel test
        if (ru == 0 || ru == nru - 1) {
#pragma unroll
          for (int i = 0; i < R / 2; ++i) {
            const int ra = rl0 + 2 * i;
            NAY[i].x = ra >= ylo && ra < yhi ? NAY[i].x : fnan;
            NAY[i].y = (ANCHOR == 2 || ra + 1 >= ylo) && ra + 1 < yhi ? NAY[i].y : fnan;
          }
        }
        // tail in groups of two row pairs: level-2 series (conj, in sigma),
        // sheet corners, beta and its bin; the chains of a group interleave
#pragma unroll
        for (int h = 0; h < R / 2; h += 2) {
          float2 QR[2], QI[2];
          const float4 sga = rows[h].sg, sgb = rows[h + 1].sg;
          const float2 SG[2] = {make_float2(sga.x, sga.y), make_float2(sgb.x, sgb.y)};
          const float2 NSG[2] = {make_float2(sga.z, sga.w), make_float2(sgb.z, sgb.w)};
          const int q4 = rows[h].q4 | corner;
          if (__all_sync(0xFFFFFFFFu, q4 >= 0)) {  // four rows of one level-2 row
            const float4* sp = reinterpret_cast<const float4*>(sub_u + q4);
            const float4 dl = sp[K2 - 1];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              QR[i] = make_float2(dl.x, dl.y);
              QI[i] = make_float2(dl.z, dl.w);
            }
#pragma unroll
            for (int nn = K2 - 2; nn >= 0; --nn) {
              const float4 dn = sp[nn];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const float2 t1 = __ffma2_rn(QI[i], SG[i], make_float2(dn.x, dn.y));
                const float2 t2 = __ffma2_rn(QI[i], SGR, make_float2(dn.z, dn.w));
                const float2 nr = __ffma2_rn(QR[i], SGR, t1);
                QI[i] = __ffma2_rn(QR[i], NSG[i], t2);
                QR[i] = nr;
              }
            }
          } else {
            const float4 *ea[2], *eb[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              ea[i] = reinterpret_cast<const float4*>(sub_u + rows[h + i].v[0] * SUB);
              eb[i] = reinterpret_cast<const float4*>(sub_u + rows[h + i].v[1] * SUB);
              QR[i] = make_float2(ea[i][K2 - 1].x, eb[i][K2 - 1].x);
              QI[i] = make_float2(ea[i][K2 - 1].z, eb[i][K2 - 1].z);
            }
#pragma unroll
            for (int nn = K2 - 2; nn >= 0; --nn) {
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const float4 xa = ea[i][nn], xb = eb[i][nn];
                const float2 t1 = __ffma2_rn(QI[i], SG[i], make_float2(xa.x, xb.x));
                const float2 t2 = __ffma2_rn(QI[i], SGR, make_float2(xa.z, xb.z));
                const float2 nr = __ffma2_rn(QR[i], SGR, t1);
                QI[i] = __ffma2_rn(QR[i], NSG[i], t2);
                QR[i] = nr;
              }
            }
            if (n_corner) {  // corners of the sheet near this cell, per ray (uniform over the CTA)
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                float qr[2] = {QR[i].x, QR[i].y}, qi[2] = {QI[i].x, QI[i].y};
                const float4 t = rows[h + i].ty;
                const float tyr[2] = {t.x, t.y};
#pragma unroll
                for (int j = 0; j < 2; ++j)
                  for (int c = 0; c < n_corner; ++c) sheet_corner_ray(rec_s.corner[c], tx, tyr[j], qr[j], qi[j]);
                QR[i] = make_float2(qr[0], qr[1]);
                QI[i] = make_float2(qi[0], qi[1]);
              }
            }
          }
          // beta relative to the base pixel, (by_hi, by_hi) + ((x0, y0) + L_local -
          // alpha_near), in pixel units
          float2 T1[2], T2[2], U[2], V[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float2 y0 = *(reinterpret_cast<const float2*>(&rows[h + i].ty) + 1);
            const float2 SX = __fadd2_rn(X0, __fadd2_rn(NAX[h + i], QR[i]));
            const float2 SY = __fadd2_rn(y0, __fadd2_rn(NAY[h + i], QI[i]));
            T1[i] = __ffma2_rn(SX, ISX, BXS);
            T2[i] = __ffma2_rn(SY, ISY, BYS);
            U[i] = __ffma2_rd(T1[i], ULP, MGX);
            V[i] = __ffma2_rd(T2[i], ULP, MGY);
          }
          const uint32_t ux = __float_as_uint(U[0].x) | __float_as_uint(U[0].y) | __float_as_uint(U[1].x) |
                              __float_as_uint(U[1].y);
          const uint32_t uy = __float_as_uint(V[0].x) | __float_as_uint(V[0].y) | __float_as_uint(V[1].x) |
                              __float_as_uint(V[1].y);
          if (!__any_sync(0xFFFFFFFFu, live && (ux >= (uint32_t)IP_BOX_W || uy >= (uint32_t)IP_BOX_H))) {
            uint32_t ad[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float2 A = __ffma2_rn(V[i], make_float2(4.f * IP_HS, 4.f * IP_HS),
                                          __ffma2_rn(U[i], make_float2(4.f, 4.f), HA));
              ad[2 * i] = __float_as_uint(A.x);
              ad[2 * i + 1] = __float_as_uint(A.y);
            }
            shared_inc4(ad[0], ad[1], ad[2], ad[3], live);
          } else if (live) {  // some ray of the warp outside the box: each on its own
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t key[2];
              pixel_keys2(T1[i], T2[i], (uint32_t)rix - PIX_MAGIC_BITS, (uint32_t)riy - PIX_MAGIC_BITS,
                          (uint32_t)g.npix_x, (uint32_t)g.npix_y, key[0], key[1]);
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const uint32_t u = __float_as_uint(j ? U[i].y : U[i].x), v = __float_as_uint(j ? V[i].y : V[i].x);
                if (u < (uint32_t)IP_BOX_W && v < (uint32_t)IP_BOX_H)
                  atomicAdd(hist_s + v * IP_HS + u, 1u);
                else if (key[j] != 0xFFFFFFFFu)
                  atomicAdd(a.counts + key[j], 1u);
              }
            }
          }
        }
      }
        ru -= nru;
      }
      // flush the box, four bins of a row at a time, and leave it zero; bins
      // off the map are dropped
      if (tid == 0) *next_s = next;  // the counter's answer has arrived by now
      __syncthreads();
      const int ox = rix + box_x, oy = riy + box_y;
      for (int t = tid; t < IP_HIST / 2; t += nt) {
        const uint2 v = reinterpret_cast<const uint2*>(hist_s)[t];
        if (v.x | v.y) {
          reinterpret_cast<uint2*>(hist_s)[t] = make_uint2(0u, 0u);
          const int y = t / (IP_HS / 2), x = 2 * (t - y * (IP_HS / 2));
          const uint32_t px = (uint32_t)(ox + x), py = (uint32_t)(oy + y), nx = (uint32_t)g.npix_x;
          if (py < (uint32_t)g.npix_y) {
            uint32_t* c = a.counts + ((int64_t)py * g.npix_x + (ox + x));
            if (v.x && px < nx) atomicAdd(c, v.x);
            if (v.y && px + 1u < nx) atomicAdd(c + 1, v.y);
          }
        }
      }
      if (g0 + ng < nrg || c0 + w < kx) __syncthreads();  // another block of this cell
    }
  }
}

// One map: a persistent grid over its ray cells.  CTAs take cells from a
// counter: with a fixed share each, the CTAs that the SM's scheduler favours
// ran out early and left it with 5.3 of 6 warps per scheduler on average.
template <int Q, int K2, int NPR>
__global__ void __launch_bounds__(IP_THREADS, 3) k_ip_ray(Geo g, IpGeo ig, IpRayArgs a) {
  extern __shared__ __align__(16) unsigned char ip_smem[];
  __shared__ long long next_s;
  const IpSmem<Q, K2> L(ig.nrow, a.near_cap);
  after_ready();
  ip_tables<Q, K2>(ig, L, ip_smem);
  after_wait();
  __syncthreads();
  long long next = 0;
  for (long long work = blockIdx.x; work < a.nwork * a.parts; work = next_s) {
    if (threadIdx.x == 0) next = (long long)gridDim.x + (long long)atomicAdd(a.queue, 1ull);
    const unsigned cell = a.parts == 1 ? (unsigned)work : (unsigned)work / (unsigned)a.parts;
    ip_cell<Q, K2, NPR>(g, ig, a, a.rc_base + cell, (int)((unsigned)work - cell * (unsigned)a.parts), L, ip_smem, next,
                        &next_s);
  }
}

// Many maps: one persistent launch; CTAs pull (map, cell) items from a global
// counter, so maps of any size and cost share the GPU without a tail per map.
struct MapDesc {
  Geo g;
  IpGeo ig;
  IpRayArgs a;
  int64_t item0;  // index of the map's first item in the concatenated list
};

// CUT: the cells of these maps are cut into shares (the other instance knows that
// an item is a whole cell, and spills less: 24 uneven maps 28.1 instead of 28.6 ms).
template <int Q, int K2, int NPR, bool CUT>
__global__ void __launch_bounds__(IP_THREADS, 3)
k_ip_ray_batch(const MapDesc* __restrict__ maps, int nmaps, int64_t nitems,
               unsigned long long* __restrict__ queue, int near_cap) {
  extern __shared__ __align__(16) unsigned char ip_smem[];
  __shared__ MapDesc md;
  __shared__ long long next_s, end_s;  // end_s: one past the loaded map's last item
  long long next = 0, end = -1;
  for (long long it = blockIdx.x; it < nitems; it = next_s) {
    if (it >= end) {  // items of one map are contiguous: reload on change only
      __syncthreads();  // everyone is done with md and the tables
      if (threadIdx.x == 0) {
        int lo = 0, hi = nmaps - 1;  // last map with item0 <= it
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (maps[mid].item0 <= it) lo = mid; else hi = mid - 1;
        }
        md = maps[lo];
        md.a.near_cap = near_cap;
        end_s = lo + 1 < nmaps ? maps[lo + 1].item0 : nitems;
      }
      __syncthreads();
      end = end_s;
      ip_tables<Q, K2>(md.ig, IpSmem<Q, K2>(md.ig.nrow, near_cap), ip_smem);
      __syncthreads();
    }
    if (threadIdx.x == 0) next = (long long)gridDim.x + (long long)atomicAdd(queue, 1ull);
    const IpSmem<Q, K2> L(md.ig.nrow, near_cap);
    if (CUT) {
      const unsigned item = (unsigned)(it - md.item0), parts = (unsigned)md.a.parts, cell = item / parts;
      ip_cell<Q, K2, NPR>(md.g, md.ig, md.a, md.a.rc_base + cell, (int)(item - cell * parts), L, ip_smem, next, &next_s);
    } else {
      ip_cell<Q, K2, NPR>(md.g, md.ig, md.a, md.a.rc_base + (it - md.item0), 0, L, ip_smem, next, &next_s);
    }
  }
}

// Chosen rays (irs_shoot_rays): one thread per ray, the arithmetic of ip_cell
// for that ray alone -- the same operations in the same order and roundings,
// so the beta written is the one the map's ray pass bins.  A thread re-centres
// only its ray's level-2 series and walks its 3x3 block in memory; the form
// before gave each ray a whole cell's pass (all k^2 rays of it).
template <int Q, int K2, int NPR>
__global__ void __launch_bounds__(128) k_ip_dump(Geo g, IpGeo ig, IpRayArgs a) {
  after_wait();
  const int64_t work = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (work >= a.nwork) return;
  const int64_t f = a.idx[work];
  if (f < 0 || f >= g.nrx * g.nry) {  // not a lattice ray: report it, touch nothing else
    a.beta_out[2 * work] = a.beta_out[2 * work + 1] = nan("");
    if (a.pix_out) a.pix_out[work] = -1;
    return;
  }
  const int64_t wi = f % g.nrx, wj = f / g.nrx;
  const int rcx = (int)(wi / ig.k), rcy = (int)(wj / ig.k);
  const int c = (int)(wi - rcx * ig.k), l = (int)(wj - rcy * ig.k);
  const int64_t rc = (int64_t)rcy * ig.nrcx + rcx;
  const CellRec& rec = a.recs[rc];
  const float hf = ig.hf, inv_k = ig.inv_k, qk = __fmul_rn((float)Q, inv_k);
  auto tau_h = [&](int i) { return __fmul_rn(fmaf((float)i, inv_k, fmaf(0.5f, inv_k, -0.5f)), hf); };
  const float tx = tau_h(c), ty = tau_h(l);
  // the row that shares this row's reciprocal, where the variant pairs them:
  // pairs (2p, 2p + 1) with p mod 4 < NPR
  const bool paired = ((l >> 1) & (IP_R / 2 - 1)) < NPR;
  const float typ = tau_h(l ^ 1);
  float nax = 0.f, nay = 0.f;
  int left = IP_NEAR_MAX;
  for (int q = 0; q < 9; ++q) {
    const int x = rcx + ig.ox + (q % 3) - 1, y = rcy + ig.oy + (q / 3) - 1;
    if (x < 0 || x >= ig.ncx || y < 0 || y >= ig.ncy) continue;
    const int64_t s = (int64_t)y * ig.ncx + x;
    const int b = a.start[s];
    int e = a.start[s + 1];
    if (e - b > left) {
      atomicCAS(a.status, 0, (int)IRS_ERR_OVERFLOW);  // the first error stays
      e = b + left;
    }
    left -= e - b;
    const float ox = __fmul_rn((float)((q % 3) - 1), hf), oy = __fmul_rn((float)((q / 3) - 1), hf);
    for (int p = b; p < e; ++p) {
      const float4 v = a.rel[p];
      const float dx = __fadd_rn(tx, -__fadd_rn(v.x, ox)), ly = -__fadd_rn(v.y, oy);
      const float dx2 = __fmul_rn(dx, dx), dy = __fadd_rn(ty, ly);
      const float r2 = __fmaf_rn(dy, dy, dx2);
      float wgt;
      if (NPR > 0 && paired) {
        const float dyp = __fadd_rn(typ, ly), r2p = __fmaf_rn(dyp, dyp, dx2);
        wgt = __fmul_rn(r2p, __fmul_rn(-v.z, rcp_approx(__fmul_rn(r2, r2p))));
      } else {
        wgt = __fmul_rn(-v.z, rcp_approx(r2));
      }
      nax = __fmaf_rn(wgt, dx, nax);
      nay = __fmaf_rn(wgt, dy, nay);
    }
  }
  // the level-2 series of the ray's sub-cell, then its Horner on the conjugate
  const float inv_q = __fdiv_rn(1.0f, (float)Q);
  auto level2 = [&](int i, float& sig) {
    const float s = __fmul_rn(__fadd_rn((float)i, 0.5f), qk);
    const int v = min(__float2int_rd(s), Q - 1);
    sig = __fsub_rn(__fsub_rn(s, (float)v), 0.5f);
    return v;
  };
  float sgx, sgy;
  const int u = level2(c, sgx), v = level2(l, sgy);
  const float er = __fmaf_rn(__fadd_rn((float)u, 0.5f), inv_q, -0.5f);
  const float ei = __fmaf_rn(__fadd_rn((float)v, 0.5f), inv_q, -0.5f);
  const float2* coef = a.coef + rc * ig.K;
  float qr = 0.f, qi = 0.f;
#pragma unroll 1
  for (int nn = K2 - 1; nn >= 0; --nn) {
    float sr = 0.f, si = 0.f;
    for (int kk = ig.K - 1; kk >= nn; --kk) {
      float2 cc = make_float2(0.f, 0.f);
      if (kk >= 1) {
        int b = 1;
        for (int i = 1; i <= nn; ++i) b = b * (kk - nn + i) / i;
        float sc = (float)b;
        for (int i = 0; i < nn; ++i) sc = __fmul_rn(sc, inv_q);
        cc = make_float2(__fmul_rn(coef[kk].x, sc), __fmul_rn(coef[kk].y, sc));
      }
      const float nr = __fmaf_rn(sr, er, __fmaf_rn(si, -ei, cc.x));
      si = __fmaf_rn(sr, ei, __fmaf_rn(si, er, cc.y));
      sr = nr;
    }
    if (nn == K2 - 1) {
      qr = sr;
      qi = -si;
    } else {
      const float nr = __fmaf_rn(qr, sgx, __fmaf_rn(qi, sgy, sr));
      qi = __fmaf_rn(qr, -sgy, __fmaf_rn(qi, sgx, -si));
      qr = nr;
    }
  }
  for (int n = 0; n < rec.n_corner; ++n) sheet_corner_ray(rec.corner[n], tx, ty, qr, qi);
  const float x0 = __fmaf_rn(g.lam_s1, tx, rec.bx_lo), y0 = __fmaf_rn(g.lam_s2, ty, rec.by_lo);
  const float sx = __fadd_rn(x0, __fadd_rn(nax, qr)), sy = __fadd_rn(y0, __fadd_rn(nay, qi));
  a.beta_out[2 * work] = (g.src_x0 + (double)rec.ix * g.sx) + ((double)rec.bx_hi + (double)sx);
  a.beta_out[2 * work + 1] = (g.src_y0 + (double)rec.iy * g.sy) + ((double)rec.by_hi + (double)sy);
  if (a.pix_out) {
    const float t1 = __fmaf_rn(sx, g.inv_sx, __fmul_rn(rec.bx_hi, g.inv_sx));
    const float t2 = __fmaf_rn(sy, g.inv_sy, __fmul_rn(rec.by_hi, g.inv_sy));
    uint32_t ka, kb;
    pixel_keys2(make_float2(t1, t1), make_float2(t2, t2), (uint32_t)rec.ix - PIX_MAGIC_BITS,
                (uint32_t)rec.iy - PIX_MAGIC_BITS, (uint32_t)g.npix_x, (uint32_t)g.npix_y, ka, kb);
    a.pix_out[work] = ka != 0xFFFFFFFFu ? (int64_t)ka : -1;
  }
}

// Dynamic shared memory above the 48 KB default: set once per instantiation,
// before any launch or graph capture that uses it.
#define IP_DECL_ATTR(V, Q, K2, NPR)                                                                          \
  case V:                                                                                                    \
    e = cudaFuncSetAttribute(k_ip_ray<Q, K2, NPR>, cudaFuncAttributeMaxDynamicSharedMemorySize, IP_SMEM_MAX); \
    if (e == cudaSuccess)                                                                                    \
      e = cudaFuncSetAttribute(k_ip_ray_batch<Q, K2, NPR, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                               IP_SMEM_MAX);                                                                 \
    if (e == cudaSuccess)                                                                                    \
      e = cudaFuncSetAttribute(k_ip_ray_batch<Q, K2, NPR, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                               IP_SMEM_MAX);                                                                 \
    break;
constexpr int IP_SMEM_MAX = 160 * 1024;
cudaError_t ip_ray_attributes(int variant) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (ip_kernel_of(variant)) { IP_VARIANTS(IP_DECL_ATTR) default: break; }
  return e;
}

#define IP_DECL_BYTES(V, Q, K2, NPR) \
  case V:                            \
    return IpSmem<Q, K2>(nrow, near_cap).bytes;
int ip_ray_smem(int variant, int nrow, int near_cap) {
  switch (ip_kernel_of(variant)) { IP_VARIANTS(IP_DECL_BYTES) default: break; }
  return 0;
}

// Launch shape of the ray pass: the register budget (80 per thread) holds 24
// warps per SM, as six CTAs of 128 threads where their shared memory fits and
// three of 256 otherwise.  Six small CTAs hide each other's per-cell set-up
// better: 204 against 217 ms at the high-res map (224-ray cells).
struct IpShape {
  int threads, grid, smem;
};
IpShape ip_launch_shape(int variant, int nrow, int near_cap, int num_sms) {
  constexpr int SM_BYTES = 228 * 1024, CTA_RESERVED = 1024, STATIC = 256;
  const int b = ip_ray_smem(variant, nrow, near_cap);
  int best = 0;
  IpShape s{};
  for (int threads : {128, 256}) {
    const int fit = SM_BYTES / (b + CTA_RESERVED + STATIC), regs = 24 * 32 / threads;
    const int per_sm = fit < regs ? (fit < 1 ? 1 : fit) : regs;
    if (per_sm * threads > best) {
      best = per_sm * threads;
      s.threads = threads;
      s.grid = num_sms * per_sm;
      s.smem = b;
    }
  }
  return s;
}

// Lenses of a 3x3 block kept in shared memory: the mean of n lenses over the
// cell grid and six deviations; fuller blocks take theirs through it in turns.
int ip_near_cap(const IpGeo& ig, int64_t n) {
  const double mean = 9.0 * (double)n / ((double)ig.ncx * (double)ig.ncy);
  double cap = mean + 6.0 * sqrt(mean) + 8.0;
  if (cap > (double)n) cap = (double)n;
  int c = cap >= (double)IP_NEAR_MAX ? IP_NEAR_MAX : (int)ceil(cap);
  c = (c + 15) & ~15;
  return c < 16 ? 16 : c;
}

#define IP_DECL_LAUNCH(V, Q, K2, NPR)                                                             \
  case V:                                                                                         \
    return launch_after(k_ip_ray<Q, K2, NPR>, (unsigned)grid, sh.threads, sh.smem, s, g, ig, a);
// A map of few cells is cut into more work items, each a share of a cell's row
// groups (with the cell's set-up of its own), until every CTA slot has four or
// an item is down to four groups a strip.  With two items per slot the pass
// over a 300^2 map of 3000 lenses at 50 rays per pixel took 274 us, with three,
// four and six 264, 227 and 233; items of two groups 235.
int32_t ip_parts(int64_t ncells, int64_t k, int grid) {
  if (ncells <= 0) return 1;
  const int64_t want = (4 * (int64_t)grid + ncells - 1) / ncells, most = (k + 4 * IP_R - 1) / (4 * IP_R);
  return (int32_t)(want < most ? want : most);
}
cudaError_t launch_ip_ray(int num_sms, cudaStream_t s, const Geo& g, const IpGeo& ig, IpRayArgs a) {
  if (a.nwork <= 0) return cudaSuccess;
  const IpShape sh = ip_launch_shape(ig.variant, ig.nrow, a.near_cap, num_sms);
  a.parts = ip_parts(a.nwork, ig.k, sh.grid);
  const int64_t items = a.nwork * a.parts, grid = items < sh.grid ? items : sh.grid;
  switch (ip_kernel_of(ig.variant)) { IP_VARIANTS(IP_DECL_LAUNCH) default: return cudaErrorInvalidValue; }
  return cudaGetLastError();
}

#define IP_DECL_DUMP(V, Q, K2, NPR)                                                    \
  case V:                                                                              \
    return launch_after(k_ip_dump<Q, K2, NPR>, (unsigned)((a.nwork + 127) / 128), 128, 0, s, g, ig, a);
cudaError_t launch_ip_dump(cudaStream_t s, const Geo& g, const IpGeo& ig, const IpRayArgs& a) {
  switch (ip_kernel_of(ig.variant)) { IP_VARIANTS(IP_DECL_DUMP) default: return cudaErrorInvalidValue; }
  return cudaGetLastError();
}

#define IP_DECL_BATCH(V, Q, K2, NPR)                                                                            \
  case V:                                                                                                       \
    if (cut)                                                                                                    \
      k_ip_ray_batch<Q, K2, NPR, true><<<(unsigned)grid, sh.threads, sh.smem, s>>>(maps, nmaps, nitems, queue, near_cap); \
    else                                                                                                        \
      k_ip_ray_batch<Q, K2, NPR, false><<<(unsigned)grid, sh.threads, sh.smem, s>>>(maps, nmaps, nitems, queue, near_cap); \
    break;
cudaError_t launch_ip_ray_batch(int variant, const IpShape& sh, cudaStream_t s, const MapDesc* maps, int nmaps,
                                int64_t nitems, bool cut, unsigned long long* queue, int near_cap) {
  const int64_t grid = nitems < sh.grid ? nitems : sh.grid;
  switch (ip_kernel_of(variant)) { IP_VARIANTS(IP_DECL_BATCH) default: return cudaErrorInvalidValue; }
  return cudaGetLastError();
}

// ------------------------------------------------------------ host helpers
irs_status alloc_lens_buffers(irs_plan_t* P, InterpState* S, int64_t cap) {
  ++P->ws_gen;  // the lens buffers move: graphs captured on the old ones are stale
  if (S->lens_ws) cudaFree(S->lens_ws);
  S->lens_ws = nullptr;
  cap = cap < 256 ? 256 : cap;
  size_t off = 0;
  auto take = [&](size_t b) {
    size_t o = off;
    off += (b + 255) & ~(size_t)255;
    return o;
  };
  const size_t o_cell = take(sizeof(int32_t) * cap), o_sidx = take(sizeof(int32_t) * cap);
  const size_t o_rel = take(sizeof(float4) * cap), o_pos = take(sizeof(double2) * cap);
  const size_t o_m = take(sizeof(double) * cap);
  const size_t o_pdf = take(sizeof(float4) * cap), o_mdf = take(sizeof(float2) * cap);
  if (cudaMalloc(&S->lens_ws, off) != cudaSuccess) {
    cudaGetLastError();
    S->lens_ws = nullptr;
    S->cap = 0;
    return IRS_ERR_OOM;
  }
  char* b = static_cast<char*>(S->lens_ws);
  S->lens_cell = reinterpret_cast<int32_t*>(b + o_cell);
  S->sorted_idx = reinterpret_cast<int32_t*>(b + o_sidx);
  S->lens_rel = reinterpret_cast<float4*>(b + o_rel);
  S->lens_pos = reinterpret_cast<double2*>(b + o_pos);
  S->lens_m = reinterpret_cast<double*>(b + o_m);
  S->lens_pdf = reinterpret_cast<float4*>(b + o_pdf);
  S->lens_mdf = reinterpret_cast<float2*>(b + o_mdf);
  S->lens_ws_bytes = off;
  S->cap = cap;
  return IRS_OK;
}

void mark(irs_plan_t* P, int slot, cudaStream_t s) {
  if (P->timing) cudaEventRecord(P->ev[slot], s);
}

#define IP_TRY(expr)                                                     \
  do {                                                                   \
    cudaError_t e_ = (expr);                                             \
    if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? IRS_ERR_OOM : IRS_ERR_CUDA; \
  } while (0)

// kernel launches of one map, reported through irs_plan_timings
int far_launches(const InterpState* S, int64_t n) {  // series mode
  const int64_t ncells = (int64_t)S->ig.ncx * S->ig.ncy;
  return (n > 0 ? 2 : 0) + (ncells > SCAN_B ? 2 : 1) + 1 + 2 * fft2d_launches(S->fft) + 1 + 1;
}

// Cell lists and far field; the per-cell finalize covers ray cells
// [rc0, rc1) only (rc1 < 0: all of them).  Follows the mass sum, which zeroes
// the cell counts.
irs_status build_cells_and_far(irs_plan_t* P, const double* xy, const double* mass, int64_t n,
                               cudaStream_t s, int64_t rc0 = 0, int64_t rc1 = -1) {
  InterpState* S = S_(P);
  const IpGeo& ig = S->ig;
  const int64_t ncells = (int64_t)ig.ncx * ig.ncy;
  if (n > S->cap) {
    cudaStreamSynchronize(s);
    irs_status st = alloc_lens_buffers(P, S, n + n / 4);
    if (st != IRS_OK) return st;
  }
  const double2* xy2 = reinterpret_cast<const double2*>(xy);
  const bool learned = P->p.method == IRS_MLP && mlp_trained(P);
  S->n_last = n;
  const unsigned lens_blocks = (unsigned)((n + 255) / 256);
  if (n > 0) IP_TRY(launch_after(k_ip_count, lens_blocks, 256, 0, s, ig, xy2, n, S->lens_cell, S->cell_count));
  const unsigned nb = (unsigned)((ncells + SCAN_B - 1) / SCAN_B);
  IP_TRY(launch_after(k_scan_local, nb, SCAN_B, 0, s, S->cell_count, S->cell_start, S->cell_cursor, ncells,
                      S->scan_blocks));
  if (nb > 1)
    IP_TRY(launch_after(k_scan_add, nb, SCAN_B, 0, s, S->cell_start, S->cell_cursor, ncells, S->scan_blocks));
  if (n > 0) IP_TRY(launch_after(k_ip_scatter, lens_blocks, 256, 0, s, S->lens_cell, n, S->cell_cursor, S->sorted_idx));
  IP_TRY(launch_after(k_ip_cells, (unsigned)((ncells + CELLS_B - 1) / CELLS_B), CELLS_B, 0, s, ig, S->cell_start, xy2,
                      mass, S->lens_cell, S->sorted_idx, S->lens_rel, learned ? S->lens_pos : nullptr, S->lens_m, S->lens_pdf, S->lens_mdf,
                      learned ? nullptr : S->mpole_d, S->mpole_f));
  mark(P, EV_CELLS, s);
  // far field: the network (trained IRS_MLP plans) or the FFT series
  MlpFar far{};
  if (learned) {
    irs_status st = mlp_prepare(P, xy, mass, n, ig.gx0, ig.gy0, ig.h, ig.nrcx, ig.nrcy, ig.ox, ig.oy, &far, s);
    if (st != IRS_OK) return st;
  } else {
    IP_TRY(fft2d_forward(S->mpole_d, S->spec_d, IP_PD, S->mpole_f, S->spec_f, IP_P - IP_PD, ig.ncx, ig.ncy, ncells,
                         S->fft, s));
    const int64_t G = (int64_t)S->fft.Nx * S->fft.Ny;
    IP_TRY(launch_after(k_ip_m2l_freq, (unsigned)((G + 127) / 128), 128, 0, s, G, S->spec_d, S->spec_f, S->kspec_d,
                        S->kspec_f));
    IP_TRY(fft2d_inverse(S->spec_d, S->conv_d, IP_KD, S->spec_f, S->conv_f, IP_KF - IP_KD, S->fft, ig.ncx, ig.ncy,
                         ncells, s));
  }
  const int64_t nrc = (int64_t)ig.nrcx * ig.nrcy;
  if (rc1 < 0 || rc1 > nrc) rc1 = nrc;
  mark(P, EV_FIN, s);
  if (rc1 > rc0) {
    // the default K = 24 needs 21 FP32 terms; larger K the full FIN_K32
    const bool few = ig.K - FIN_K64 <= 21;
    if (!far.active && ig.W <= FG_WMAX) {
      const int cta_cells = rc1 - rc0 <= 4 * FG_CELLS * (int64_t)P->num_sms ? FG_CELLS / 2 : FG_CELLS;
      const unsigned nb = (unsigned)((rc1 - rc0 + cta_cells - 1) / cta_cells);
      auto* kern = few ? k_ip_finalize_group<21> : k_ip_finalize_group<FIN_K32>;
      IP_TRY(launch_after(kern, nb, 32 * FG_WARPS, 0, s, P->g, ig, P->d_msum, S->cell_start, S->lens_pdf, S->lens_mdf,
                          S->conv_d, S->conv_f, S->sheet_d, S->sheet_f, S->sheet_near, S->recs, S->coef, rc0, rc1,
                          cta_cells));
    } else {
      const unsigned nb = (unsigned)((rc1 - rc0 + 63) / 64);
      auto* kern = few ? k_ip_finalize<21> : k_ip_finalize<FIN_K32>;
      IP_TRY(launch_after(kern, nb, 64, 0, s, P->g, ig, P->d_msum, S->cell_start, S->lens_pos, S->lens_m, S->lens_pdf,
                          S->lens_mdf, S->conv_d, S->conv_f, far, S->sheet_d, S->sheet_f, S->sheet_near, S->recs,
                          S->coef, rc0, rc1));
    }
  }
  IP_TRY(cudaGetLastError());
  mark(P, EV_FAR, s);
  return IRS_OK;
}

IpRayArgs ray_args(irs_plan_t* P) {
  InterpState* S = S_(P);
  IpRayArgs a{};
  a.start = S->cell_start;
  a.rel = S->lens_rel;
  a.recs = S->recs;
  a.coef = S->coef;
  a.status = P->d_status;
  a.queue = P->d_queue;
  a.near_cap = ip_near_cap(S->ig, S->n_last);
  return a;
}

}  // namespace

// ------------------------------------------------------------ entry points
irs_status interp_plan(irs_plan_t* P) {
  InterpState* S = new (std::nothrow) InterpState();
  if (!S) return IRS_ERR_OOM;
  memset(S, 0, sizeof(*S));
  P->interp = S;
  IpGeo& ig = S->ig;
  const irs_params& p = P->p;
  const Geo& g = P->g;
  const double Ix = P->ix, Iy = P->iy;
  int64_t nstar = p.n_star > 0 ? p.n_star : P->n_star_suggested;
  if (nstar < 1) nstar = 1;
  // level-1 resolution, flow chart: Delta x1 = min(L0, min(I_x, I_y)/10)
  const double L0 = sqrt(Ix * Iy / (double)nstar);
  const double dx1_rule = fmin(L0, fmin(Ix, Iy) / 10.0);
  S->rule_rays = dx1_rule / g.dx3;
  double dx1 = dx1_rule * (p.cell_mult > 0 ? p.cell_mult : 1.0);
  int64_t k = (int64_t)ceil(dx1 / g.dx3 - 1e-9);
  if (k < 4) k = 4;
  if (k > IP_KMAX_RAYS) k = IP_KMAX_RAYS;  // the ray pass keeps a row table per cell
  ig.k = k;
  ig.nrow = (int32_t)((k + 1) / 2) + IP_ROW_PAD;
  ig.h = (double)k * g.dx3;
  // under the mean lens map (declared kappa_*) a cell covers (1 - kappa -+
  // gamma) h; a block of it is kept to three quarters of a binning box
  ig.cell_px = (float)(P->lambda1 * ig.h / g.sx);
  ig.cell_py = (float)(P->lambda2 * ig.h / g.sy);
  const double bc = 0.75 * IP_BOX_W * (double)k / fabs((double)ig.cell_px);
  const double br = 0.75 * IP_BOX_H * (double)k / fabs((double)ig.cell_py);
  ig.blk_col = bc >= (double)k ? (int32_t)k : (bc < 64.0 ? 32 : (int32_t)bc & ~31);
  ig.blk_rg = br >= (double)k ? (int32_t)k : (br < 16.0 ? 1 : (int32_t)(br / IP_R));
  ig.hf = (float)ig.h;
  ig.inv_k = 1.0f / (float)k;
  ig.nrcx = (int32_t)((g.nrx + k - 1) / k);
  ig.nrcy = (int32_t)((g.nry + k - 1) / k);
  // lens region: the rectangle, or the circumscribed circle's bounding box
  int64_t ox = 0, oy = 0, ex = 0, ey = 0;
  if (p.plane == IRS_PLANE_CIRCLE) {
    const double R = P->circle_r;
    ox = (int64_t)ceil((g.a1 - (g.cx - R)) / ig.h);
    oy = (int64_t)ceil((g.b1 - (g.cy - R)) / ig.h);
    ex = (int64_t)ceil(((g.cx + R) - (g.a1 + ig.nrcx * ig.h)) / ig.h);
    ey = (int64_t)ceil(((g.cy + R) - (g.b1 + ig.nrcy * ig.h)) / ig.h);
    ox = ox < 0 ? 0 : ox;
    oy = oy < 0 ? 0 : oy;
    ex = ex < 0 ? 0 : ex;
    ey = ey < 0 ? 0 : ey;
  }
  // the ray pass's pixel keys (pixel_keys2) need every ray that lands to be
  // within 2^22 pixels of its cell's base pixel: maps below 2^21 pixels per
  // side and protective borders below 2^20 pixels
  if (g.npix_x >= (1 << 21) || g.npix_y >= (1 << 21) || P->border >= 1048576.0 * fmin(g.sx, g.sy))
    return IRS_ERR_OVERFLOW;
  const int64_t ncx = ox + ig.nrcx + ex, ncy = oy + ig.nrcy + ey;
  if (ncx > FFT_MAX_LEN / 2 || ncy > FFT_MAX_LEN / 2) return IRS_ERR_OVERFLOW;
  ig.ncx = (int32_t)ncx;
  ig.ncy = (int32_t)ncy;
  ig.ox = (int32_t)ox;
  ig.oy = (int32_t)oy;
  ig.gx0 = g.a1 - (double)ox * ig.h;
  ig.gy0 = g.b1 - (double)oy * ig.h;
  ig.K = p.far_order > 0 ? p.far_order : DEFAULT_K;
  // `window` is the direct window of the series form; an IRS_MLP plan reads it
  // as the learned split's radius R_f instead (its untrained fallback keeps
  // the default window)
  ig.W = (p.window > 0 && p.method != IRS_MLP) ? p.window : DEFAULT_W;
  ig.P = IP_P;
  if (ig.K > IP_KMAX || ig.K < 8) return IRS_ERR_ARG;
  ig.variant = p.kernel_variant;
  if (ig.variant < 0 || ig.variant >= IP_NVARIANT) return IRS_ERR_ARG;
  if (ig.W < 1) ig.W = 1;

  Fft2d& f = S->fft;
  f.num_sms = P->num_sms;
  // padded lengths >= 2n - 1 (linear convolution), of the form 2^a 3^b
  f.Nx = fft_good_size(2 * ncx - 1, &f.n3x, &f.n2x);
  f.Ny = fft_good_size(2 * ncy - 1, &f.n3y, &f.n2y);
  if (f.Nx < 0 || f.Ny < 0) return IRS_ERR_OVERFLOW;
  if (fft_setup_attributes() != cudaSuccess) return IRS_ERR_CUDA;
  if (fft_twiddles(f.Nx, &f.tw_x) != cudaSuccess) return IRS_ERR_OOM;
  if (fft_twiddles(f.Ny, &f.tw_y) != cudaSuccess) return IRS_ERR_OOM;

  const int64_t ncells = ncx * ncy, nrc = (int64_t)ig.nrcx * ig.nrcy;
  const int64_t G = (int64_t)f.Nx * f.Ny;
  size_t off = 0;
  auto take = [&](size_t b) {
    size_t o = off;
    off += (b + 255) & ~(size_t)255;
    return o;
  };
  const size_t o_cnt = take(sizeof(int32_t) * ncells), o_start = take(sizeof(int32_t) * (ncells + 1));
  const size_t o_cur = take(sizeof(int32_t) * ncells);
  const size_t o_sb = take(sizeof(int32_t) * ((ncells + SCAN_B - 1) / SCAN_B + 1));
  static_assert(IP_KD <= IP_PD && IP_KF - IP_KD <= IP_P - IP_PD, "local spectra overwrite multipole spectra");
  const size_t o_mpd = take(sizeof(float4) * IP_PD * ncells), o_mpf = take(sizeof(float2) * (IP_P - IP_PD) * ncells);
  const size_t o_cvd = take(sizeof(float4) * IP_KD * ncells), o_cvf = take(sizeof(float2) * (IP_KF - IP_KD) * ncells);
  const size_t o_spd = take(sizeof(float4) * IP_PD * G), o_spf = take(sizeof(float2) * (IP_P - IP_PD) * G);
  const size_t o_ksd = take(sizeof(float4) * IP_NKD * G), o_ksf = take(sizeof(float2) * (IP_P + IP_KF - 1) * G);
  const size_t o_rec = take(sizeof(CellRec) * nrc), o_coef = take(sizeof(float2) * ig.K * nrc);
  const bool rect = p.plane == IRS_PLANE_RECT;
  const size_t o_shd = take(rect ? sizeof(double2) * FIN_K64 * nrc : 0);
  const size_t o_shf = take(rect ? sizeof(float2) * (ig.K - FIN_K64) * nrc : 0);
  const size_t o_shn = take(rect ? sizeof(uint8_t) * nrc : 0);
  if (cudaMalloc(&S->ws, off) != cudaSuccess) {
    cudaGetLastError();
    S->ws = nullptr;
    return IRS_ERR_OOM;
  }
  S->ws_bytes = off;
  char* b = static_cast<char*>(S->ws);
  S->cell_count = reinterpret_cast<int32_t*>(b + o_cnt);
  P->d_zero = S->cell_count;
  P->n_zero = ncells;
  S->cell_start = reinterpret_cast<int32_t*>(b + o_start);
  S->cell_cursor = reinterpret_cast<int32_t*>(b + o_cur);
  S->scan_blocks = reinterpret_cast<int32_t*>(b + o_sb);
  S->mpole_d = reinterpret_cast<float4*>(b + o_mpd);
  S->mpole_f = reinterpret_cast<float2*>(b + o_mpf);
  S->conv_d = reinterpret_cast<float4*>(b + o_cvd);
  S->conv_f = reinterpret_cast<float2*>(b + o_cvf);
  S->spec_d = reinterpret_cast<float4*>(b + o_spd);
  S->spec_f = reinterpret_cast<float2*>(b + o_spf);
  S->kspec_d = reinterpret_cast<float4*>(b + o_ksd);
  S->kspec_f = reinterpret_cast<float2*>(b + o_ksf);
  S->recs = reinterpret_cast<CellRec*>(b + o_rec);
  S->coef = reinterpret_cast<float2*>(b + o_coef);
  S->sheet_d = rect ? reinterpret_cast<double2*>(b + o_shd) : nullptr;
  S->sheet_f = rect ? reinterpret_cast<float2*>(b + o_shf) : nullptr;
  S->sheet_near = rect ? reinterpret_cast<uint8_t*>(b + o_shn) : nullptr;
  irs_status st = alloc_lens_buffers(P, S, nstar + nstar / 4 + 256);
  if (st != IRS_OK) return st;
  // translation kernels and their spectra, once per plan
  const int nker = ig.P + IP_KF - 1;
  k_ip_kernel_grid<<<(unsigned)((G + 255) / 256), 256>>>(f.Nx, f.Ny, ig.W, nker, IP_NKD, S->kspec_d, S->kspec_f);
  if (cudaGetLastError() != cudaSuccess) return IRS_ERR_CUDA;
  if (fft2d_forward(S->kspec_d, S->kspec_d, IP_NKD, S->kspec_f, S->kspec_f, nker, f.Nx, f.Ny, G, f, 0) != cudaSuccess)
    return IRS_ERR_CUDA;
  if (rect && nrc > 0) {  // the sheet's corner series, once per plan
    k_ip_sheet_table<<<(unsigned)((nrc + 127) / 128), 128>>>(g, ig, S->sheet_d, S->sheet_f, S->sheet_near, nrc);
    if (cudaGetLastError() != cudaSuccess) return IRS_ERR_CUDA;
  }
  if (cudaDeviceSynchronize() != cudaSuccess) return IRS_ERR_CUDA;
  if (ip_ray_attributes(ig.variant) != cudaSuccess) return IRS_ERR_CUDA;
  if (p.method == IRS_MLP) {
    if (p.plane != IRS_PLANE_RECT) return IRS_ERR_UNSUPPORTED;
    irs_status st2 = mlp_plan(P, ig.gx0, ig.gy0, ig.h, ig.ncx, ig.ncy, ig.nrcx, ig.nrcy, ig.ox, ig.oy, 1 << 20);
    if (st2 != IRS_OK) return st2;
  }
  return IRS_OK;
}

double interp_cell_side(const irs_plan_t* P) { return S_(P) ? S_(P)->ig.h : 0.0; }
double interp_rule_rays(const irs_plan_t* P) { return S_(P) ? S_(P)->rule_rays : 0.0; }

void interp_fill_info(const irs_plan_t* P, irs_plan_info* info) {
  const InterpState* S = S_(P);
  if (!S) return;
  info->cell_x = info->cell_y = S->ig.h;
  info->ncell_x = S->ig.ncx;
  info->ncell_y = S->ig.ncy;
  info->rays_per_cell_x = info->rays_per_cell_y = (int32_t)S->ig.k;
  info->far_order = S->ig.K;
  info->window = S->ig.W;
}

int64_t interp_workspace_bytes(const irs_plan_t* P) {
  const InterpState* S = S_(P);
  return S ? (int64_t)(S->ws_bytes + S->lens_ws_bytes) : 0;
}

irs_status interp_run(irs_plan_t* P, const double* xy, const double* mass, int64_t n, int64_t row0,
                      int64_t row1, uint32_t* counts, cudaStream_t s) {
  InterpState* S = S_(P);
  mark(P, EV_PREP, s);
  // only the cell rows the band touches need their series
  const int64_t k = S->ig.k;
  const int64_t rc0 = row1 > row0 ? (row0 / k) * S->ig.nrcx : 0;
  const int64_t rc1 = row1 > row0 ? ((row1 + k - 1) / k) * S->ig.nrcx : 0;
  irs_status st = build_cells_and_far(P, xy, mass, n, s, rc0, rc1);
  if (st != IRS_OK) return st;
  mark(P, EV_RAY0, s);
  P->launches += far_launches(S, n) - (rc1 > rc0 ? 0 : 1) + (row1 > row0 ? 1 : 0);
  if (row1 > row0) {
    IpRayArgs a = ray_args(P);
    a.counts = counts;
    a.row0 = row0;
    a.row1 = row1;
    a.rc_base = rc0;
    a.nwork = rc1 - rc0;
    if (launch_ip_ray(P->num_sms, s, P->g, S->ig, a) != cudaSuccess) return IRS_ERR_CUDA;
  }
  mark(P, EV_RAY1, s);
  return IRS_OK;
}

irs_status interp_set_variant(irs_plan_t* P, int variant) {
  InterpState* S = S_(P);
  if (!S || variant < 0 || variant >= IP_NVARIANT) return IRS_ERR_ARG;
  if (ip_ray_attributes(variant) != cudaSuccess) return IRS_ERR_CUDA;
  S->ig.variant = variant;
  P->p.kernel_variant = variant;
  return IRS_OK;
}

irs_status interp_raypass_rows(irs_plan_t* P, int64_t row0, int64_t row1, uint32_t* counts, cudaStream_t s,
                               cudaEvent_t e0, cudaEvent_t e1) {
  InterpState* S = S_(P);
  if (!S || row0 < 0 || row1 <= row0 || row1 > P->g.nry) return IRS_ERR_ARG;
  const int64_t k = S->ig.k;
  const int64_t rc0 = (row0 / k) * S->ig.nrcx, rc1 = ((row1 + k - 1) / k) * S->ig.nrcx;
  IpRayArgs a = ray_args(P);
  a.counts = counts;
  a.row0 = row0;
  a.row1 = row1;
  a.rc_base = rc0;
  a.nwork = rc1 - rc0;
  if (cudaMemsetAsync(P->d_queue, 0, sizeof(unsigned long long), s) != cudaSuccess) return IRS_ERR_CUDA;
  if (cudaEventRecord(e0, s) != cudaSuccess) return IRS_ERR_CUDA;
  if (launch_ip_ray(P->num_sms, s, P->g, S->ig, a) != cudaSuccess) return IRS_ERR_CUDA;
  if (cudaEventRecord(e1, s) != cudaSuccess) return IRS_ERR_CUDA;
  return IRS_OK;
}

irs_status interp_shoot_rays(irs_plan_t* P, const double* xy, const double* mass, int64_t n,
                             const int64_t* idx, int64_t nidx, double* beta, int64_t* pix,
                             cudaStream_t s) {
  InterpState* S = S_(P);
  irs_status st = build_cells_and_far(P, xy, mass, n, s);
  if (st != IRS_OK) return st;
  IpRayArgs a = ray_args(P);
  a.idx = idx;
  a.beta_out = beta;
  a.pix_out = pix;
  a.nwork = nidx;
  return launch_ip_dump(s, P->g, S->ig, a) == cudaSuccess ? IRS_OK : IRS_ERR_CUDA;
}

irs_status interp_ensure_capacity(irs_plan_t* P, int64_t n) {
  InterpState* S = S_(P);
  if (n <= S->cap) return IRS_OK;
  if (cudaDeviceSynchronize() != cudaSuccess) return IRS_ERR_CUDA;
  return alloc_lens_buffers(P, S, n + n / 4);
}

irs_status interp_prepare(irs_plan_t* P, const double* xy, const double* mass, int64_t n,
                          cudaStream_t s) {
  return build_cells_and_far(P, xy, mass, n, s);
}

int interp_variant(const irs_plan_t* P) { return S_(P)->ig.variant; }
int interp_row_entries(const irs_plan_t* P) { return S_(P)->ig.nrow; }
int interp_near_cap(const irs_plan_t* P, int64_t n) { return ip_near_cap(S_(P)->ig, n); }
bool interp_small_ctas(const irs_plan_t* P, int64_t n) {
  const InterpState* S = S_(P);
  return ip_launch_shape(S->ig.variant, S->ig.nrow, ip_near_cap(S->ig, n), P->num_sms).threads == 128;
}
int interp_num_variants() { return IP_NVARIANT; }
bool interp_variant_distinct(int variant) { return ip_kernel_of(variant) == variant; }

size_t interp_desc_bytes(int nmaps) { return sizeof(MapDesc) * (size_t)(nmaps > 0 ? nmaps : 1); }

int64_t interp_fill_descs(irs_plan_t* const* plans, uint32_t* const* counts, int nmaps, int nrow, int near_cap,
                          void* host, bool* cut) {
  MapDesc* d = static_cast<MapDesc*>(host);
  int64_t items = 0, cells = 0;
  *cut = false;
  for (int k = 0; k < nmaps; ++k) cells += (int64_t)S_(plans[k])->ig.nrcx * S_(plans[k])->ig.nrcy;
  const int grid = nmaps > 0 ? ip_launch_shape(interp_variant(plans[0]), nrow, near_cap, plans[0]->num_sms).grid : 0;
  for (int k = 0; k < nmaps; ++k) {
    InterpState* S = S_(plans[k]);
    memset(&d[k], 0, sizeof(MapDesc));
    d[k].g = plans[k]->g;
    d[k].ig = S->ig;
    d[k].a = ray_args(plans[k]);
    d[k].a.counts = counts[k];
    d[k].a.row0 = 0;
    d[k].a.row1 = plans[k]->g.nry;
    d[k].a.rc_base = 0;
    d[k].a.nwork = (int64_t)S->ig.nrcx * S->ig.nrcy;
    d[k].a.parts = ip_parts(cells, S->ig.k, grid);  // as if the group were one map
    *cut = *cut || d[k].a.parts > 1;
    d[k].item0 = items;
    items += d[k].a.nwork * d[k].a.parts;
  }
  return items;
}

irs_status interp_batch_launch(int variant, const void* dev_descs, int nmaps, int64_t nitems, bool cut,
                               unsigned long long* queue, int num_sms, int nrow, int near_cap, cudaStream_t s) {
  if (nmaps <= 0 || nitems <= 0) return IRS_OK;
  const IpShape sh = ip_launch_shape(variant, nrow, near_cap, num_sms);
  if (cudaMemsetAsync(queue, 0, sizeof(unsigned long long), s) != cudaSuccess) return IRS_ERR_CUDA;
  return launch_ip_ray_batch(variant, sh, s, static_cast<const MapDesc*>(dev_descs), nmaps, nitems, cut, queue,
                             near_cap) == cudaSuccess
             ? IRS_OK
             : IRS_ERR_CUDA;
}

void interp_destroy(irs_plan_t* P) {
  mlp_destroy(P);
  InterpState* S = S_(P);
  if (!S) return;
  if (S->ws) cudaFree(S->ws);
  if (S->lens_ws) cudaFree(S->lens_ws);
  if (S->fft.tw_x) cudaFree(S->fft.tw_x);
  if (S->fft.tw_y) cudaFree(S->fft.tw_y);
  delete S;
  P->interp = nullptr;
}

}  // namespace irs
