// irs_fft.cu -- complex 2-D FFTs of length 2^a 3^b for the far-field
// convolution on the level-1 cell grid, in double-float arithmetic
// (irs_df.cuh: 48-bit significands on the FP32 pipes; float4 elements) or in
// FP32 (float2 elements).
//
// A CTA takes B lines of length L = 3^n3 2^n2 (B as large as keeps it within
// 74 KB of shared memory, at least one, fewer in small launches) with a twiddle table W_L^t (t < L/2;
// W_L^(t + L/2) = -W_L^t) beside them, and runs the butterfly stages in passes:
// up to three radix-2 or two radix-3 stages of a line's element group in
// registers, then an exchange through shared memory; the first pass reads
// memory, the last writes it.  Neither direction permutes: the forward
// transform runs decimation in frequency (n2 radix-2 then n3 radix-3 stages) on
// natural-order input and leaves X[k] at the mixed-radix digit reversal of k;
// the inverse runs decimation in time (n3 radix-3 then n2 radix-2 stages), which
// takes its input in exactly that order and returns natural order.  The
// convolution between them is pointwise, so the spectra never need sorting.
// Rows are contiguous lines; columns are strided lines, B adjacent columns at a
// time so that each row segment is one coalesced access.  Zero padding is
// implicit: input elements at or beyond `in_len` read as 0, and only the first
// `out_len` outputs of a line are written.
//
// The stages were one pass each (a round trip through shared memory and a
// barrier for every stage, with adjacent columns in the same bank): the eight
// launches of a paper-mid map took 1,332 us, 6.1 ms at the high-res map; four
// to six launches of fused passes 855 us and 5.1 ms, and without bank conflicts in
// the twiddles and with packed double-float sums 740 us and 4.2 ms.
#include <math.h>

#include <type_traits>
#include <vector>

#include "irs_common.cuh"
#include "irs_df.cuh"
#include "irs_fft.cuh"

namespace irs {

namespace {

constexpr int FFT_REGS = 80;  // per thread: 24 warps per SM

// Complex arithmetic of the two element types: float4 is double-float
// (re.hi, im.hi, re.lo, im.lo), float2 is FP32 (re, im).
__device__ __forceinline__ float4 c_add(float4 a, float4 b) { return dfc_add(a, b); }
__device__ __forceinline__ float4 c_sub(float4 a, float4 b) { return dfc_sub(a, b); }
__device__ __forceinline__ float4 c_mul(float4 a, float4 b) { return dfc_mul(a, b); }
__device__ __forceinline__ float4 c_neg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
__device__ __forceinline__ float4 c_conj(float4 a) { return make_float4(a.x, -a.y, a.z, -a.w); }
__device__ __forceinline__ float4 c_half(float4 a) { return make_float4(0.5f * a.x, 0.5f * a.y, 0.5f * a.z, 0.5f * a.w); }
__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 c_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 c_conj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 c_half(float2 a) { return make_float2(0.5f * a.x, 0.5f * a.y); }

template <class T> __device__ __forceinline__ T c_zero();
template <> __device__ __forceinline__ float4 c_zero<float4>() { return make_float4(0.f, 0.f, 0.f, 0.f); }
template <> __device__ __forceinline__ float2 c_zero<float2>() { return make_float2(0.f, 0.f); }

// twiddle table entry in the element type (the table holds double-float)
template <class T> __device__ __forceinline__ T tw_elem(float4 v);
template <> __device__ __forceinline__ float4 tw_elem<float4>(float4 v) { return v; }
template <> __device__ __forceinline__ float2 tw_elem<float2>(float4 v) { return dfc_hi(v); }

// Radix-3 butterfly on a and the twiddled p, q:
// x0 = a + t1, x1,2 = a - t1/2 -+ i s3 (p - q) with t1 = p + q and
// s3 = +-sqrt(3)/2 (the sign of the transform's exponent).
__device__ __forceinline__ void radix3(float4 a, float4 p, float4 q, bool inv, float4& x0, float4& x1,
                                       float4& x2) {
  const float2 s3 = inv ? make_float2(-8.660253882e-01f, -1.554362505e-08f)
                        : make_float2(8.660253882e-01f, 1.554362505e-08f);  // sqrt(3)/2 = hi + lo
  const float4 t1 = dfc_add(p, q);
  const float4 t2 = dfc_sub(a, c_half(t1));
  const float4 dd = dfc_sub(p, q);
  // (s3 Im(dd), -s3 Re(dd))
  const float4 uv = dfc_make(df_mul(s3, dfc_im(dd)), df_mul(df_neg(s3), dfc_re(dd)));
  x0 = dfc_add(a, t1);
  x1 = dfc_add(t2, uv);
  x2 = dfc_sub(t2, uv);
}
__device__ __forceinline__ void radix3(float2 a, float2 p, float2 q, bool inv, float2& x0, float2& x1,
                                       float2& x2) {
  const float s3 = inv ? -0.8660254038f : 0.8660254038f;
  const float2 t1 = c_add(p, q);
  const float2 t2 = c_sub(a, c_half(t1));
  const float2 dd = c_sub(p, q);
  const float u = s3 * dd.y, v = s3 * dd.x;
  x0 = c_add(a, t1);
  x1 = make_float2(t2.x + u, t2.y - v);
  x2 = make_float2(t2.x - u, t2.y + v);
}

// Quotient by a divisor d that is fixed for a loop: umulhi(x, ceil(2^32 / d))
// equals floor(x / d) whenever x d < 2^32 (here x < 2^15 and d < 2^14), with
// no division instruction sequence per element.
struct FastDiv {
  uint32_t d, m;
  __device__ explicit FastDiv(uint32_t dv) : d(dv), m(dv > 1u ? 0xFFFFFFFFu / dv + 1u : 0u) {}
  __device__ __forceinline__ uint32_t div(uint32_t x) const { return d > 1u ? __umulhi(x, m) : x; }
};

// Place of entry t of the twiddle table in shared memory: a gap after every 128
// bytes.  The later stages of a pass read every 4th, 8th or 16th entry, which
// without the gaps share one or two of the eight (sixteen) bank groups.
template <class T> __host__ __device__ __forceinline__ int tw_place(int t) { return t + (t >> (sizeof(T) == 16 ? 3 : 4)); }

// W_L^t for 0 <= t < L from the half table, conjugated for the inverse
template <bool INV, class T>
__device__ __forceinline__ T tw_at(const T* w, int t, int half) {
  T v = w[tw_place<T>(t < half ? t : t - half)];
  if (t >= half) v = c_neg(v);
  return INV ? c_conj(v) : v;
}

// One pass over a line takes several stages in registers.  F radix-2 stages:
// 2^F elements per work item, or F radix-3 stages: 3^F elements, `gap` apart;
// stride0 is the twiddle stride L / m of the widest stage (the decimation in
// frequency's first, the decimation in time's last).  Every butterfly is the one of a single stage,
// with the same twiddle, so how the stages are grouped does not change a bit.
template <bool INV, int F, class T>
__device__ __forceinline__ void fused2(T* v, const T* w, int j, int gap, int stride0, int half_L) {
#pragma unroll
  for (int f = 0; f < F; ++f) {
    // frequency: pairs 2^(F-1), ..., 2, 1 apart; time: 1, 2, ..., 2^(F-1)
    const int d = INV ? 1 << f : 1 << (F - 1 - f);
    const int stride = stride0 << (INV ? F - 1 - f : f);
#pragma unroll
    for (int q = 0; q < 1 << F; ++q) {
      if (q & d) continue;
      const T t = tw_at<INV>(w, (j + (q & (d - 1)) * gap) * stride, half_L);
      if (INV) {
        const T u = v[q], x = c_mul(v[q + d], t);
        v[q] = c_add(u, x);
        v[q + d] = c_sub(u, x);
      } else {
        const T u = v[q], x = v[q + d];
        v[q] = c_add(u, x);
        v[q + d] = c_mul(c_sub(u, x), t);
      }
    }
  }
}
template <bool INV, int F, class T>
__device__ __forceinline__ void fused3(T* v, const T* w, int j, int gap, int stride0, int half_L) {
  constexpr int N = F == 2 ? 9 : 3;
#pragma unroll
  for (int f = 0; f < F; ++f) {
    const int d = (INV ? f == 0 : f == F - 1) ? 1 : 3;
    const int stride = (INV ? F == 2 && f == 0 : f == 1) ? 3 * stride0 : stride0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (q / d % 3) continue;
      const int t = (j + (q % d) * gap) * stride;
      if (INV) {
        const T p = c_mul(v[q + d], tw_at<INV>(w, t, half_L));
        const T r = c_mul(v[q + 2 * d], tw_at<INV>(w, 2 * t, half_L));
        radix3(v[q], p, r, true, v[q], v[q + d], v[q + 2 * d]);
      } else {
        T y0, y1, y2;
        radix3(v[q], v[q + d], v[q + 2 * d], false, y0, y1, y2);
        v[q] = y0;
        v[q + d] = c_mul(y1, tw_at<INV>(w, t, half_L));
        v[q + 2 * d] = c_mul(y2, tw_at<INV>(w, 2 * t, half_L));
      }
    }
  }
}

// Sequence of passes of a line of 2^n2 3^n3: radix-2 stages by threes (a
// remainder of one or two, and 4 as 2 + 2), radix-3 stages by twos; in this
// order for the forward transform, reversed for the inverse.
__host__ __device__ __forceinline__ int fft_passes2(int n2) { return (n2 + 2) / 3; }
__host__ __device__ __forceinline__ int fft_pass2_stages(int n2, int p) {  // stages of pass p
  const int np = fft_passes2(n2);
  return n2 / np + (p < n2 % np ? 1 : 0);
}

// Lines of one CTA.  The first pass reads its elements from memory and the last
// writes them there; shared memory holds the line between passes, lines L + 1
// elements apart so that a warp's adjacent columns fall in distinct banks.
template <bool INV, class T>
__device__ __forceinline__ void fft_lines(const T* in, T* out, const FftLines& d, const float4* __restrict__ tw,
                                          int64_t block, float4* sm) {
  const int L = d.L, B = d.B, n3 = d.n3, n2 = d.n2, half_L = L / 2, LS = L + 1;
  T* x = reinterpret_cast<T*>(sm);      // [B][LS]
  T* w = x + (size_t)B * LS;            // [L/2] at tw_place
  const int64_t blocks_per_grid = (d.n_lines + B - 1) / B;
  const int64_t grid = block / blocks_per_grid, line0 = (block - grid * blocks_per_grid) * B;
  in += grid * d.in_grid_stride;
  out += grid * d.out_grid_stride;
  const int nthr = blockDim.x;
  for (int k = threadIdx.x; k < half_L; k += nthr) w[tw_place<T>(k)] = tw_elem<T>(tw[k]);
  int pow3 = 1;
  for (int i = 0; i < n3; ++i) pow3 *= 3;
  const int np2 = fft_passes2(n2), np3 = (n3 + 1) / 2, np = np2 + np3;
  after_wait();  // the twiddles are the plan's
  __syncthreads();
  int span = INV ? 1 : L;  // forward: widest span left; inverse: span done so far
  for (int p = 0; p < np; ++p) {
    const int pf = INV ? np - 1 - p : p;  // the forward transform's number of this pass
    const bool two = pf < np2;
    const int stages = two ? fft_pass2_stages(n2, pf) : (pf - np2 == np3 - 1 && (n3 & 1) ? 1 : 2);
    const int N = two ? 1 << stages : (stages == 2 ? 9 : 3);
    if (INV) span *= N;
    const int gap = span / N, items = L / N, stride0 = L / span;
    const bool first = p == 0, last = p == np - 1;
    // items dealt along the line, or across the lines where those are adjacent in memory
    const bool across = d.in_elem_stride != 1;
    const FastDiv fdB((uint32_t)B), fdI((uint32_t)items), fdg((uint32_t)gap);
    for (int t = threadIdx.x; t < B * items; t += nthr) {
      int b, k;
      if (across) {
        k = (int)fdB.div((uint32_t)t);
        b = t - k * B;
      } else {
        b = (int)fdI.div((uint32_t)t);
        k = t - b * items;
      }
      const int g = (int)fdg.div((uint32_t)k), j = k - g * gap, e0 = g * span + j;
      const int64_t line = line0 + b;
      const bool on = line < d.n_lines;
      T* xl = x + (size_t)b * LS;
      T v[9];
      auto load = [&](auto n) {
#pragma unroll
        for (int q = 0; q < decltype(n)::value; ++q) {
          const int e = e0 + q * gap;
          if (!first) v[q] = xl[e];
          else v[q] = on && e < d.in_len ? in[line * d.in_line_stride + (int64_t)e * d.in_elem_stride] : c_zero<T>();
        }
      };
      auto store = [&](auto n) {
#pragma unroll
        for (int q = 0; q < decltype(n)::value; ++q) {
          const int e = e0 + q * gap;
          if (!last) xl[e] = v[q];
          else if (on && e < d.out_len) out[line * d.out_line_stride + (int64_t)e * d.out_elem_stride] = v[q];
        }
      };
      if (two && stages == 3) {
        load(std::integral_constant<int, 8>{});
        fused2<INV, 3>(v, w, j, gap, stride0, half_L);
        store(std::integral_constant<int, 8>{});
      } else if (two && stages == 2) {
        load(std::integral_constant<int, 4>{});
        fused2<INV, 2>(v, w, j, gap, stride0, half_L);
        store(std::integral_constant<int, 4>{});
      } else if (two) {
        load(std::integral_constant<int, 2>{});
        fused2<INV, 1>(v, w, j, gap, stride0, half_L);
        store(std::integral_constant<int, 2>{});
      } else if (stages == 2) {
        load(std::integral_constant<int, 9>{});
        fused3<INV, 2>(v, w, j, gap, stride0, half_L);
        store(std::integral_constant<int, 9>{});
      } else {
        load(std::integral_constant<int, 3>{});
        fused3<INV, 1>(v, w, j, gap, stride0, half_L);
        store(std::integral_constant<int, 3>{});
      }
    }
    if (!INV) span = gap;
    if (!last) __syncthreads();
  }
}

// The double-float planes' lines, the FP32 planes', or both in one launch.
template <bool INV>
__global__ void __maxnreg__(FFT_REGS)
k_fft_lines(const float4* in4, float4* out4, FftLines d4, int64_t blocks4, const float2* in2, float2* out2,
            FftLines d2, const float4* __restrict__ tw) {
  extern __shared__ float4 sm_raw[];
  after_ready();
  if ((int64_t)blockIdx.x < blocks4) fft_lines<INV>(in4, out4, d4, tw, blockIdx.x, sm_raw);
  else fft_lines<INV>(in2, out2, d2, tw, (int64_t)blockIdx.x - blocks4, sm_raw);
}

}  // namespace

int fft_good_size(int64_t n_min, int* n3, int* n2) {
  int64_t best = -1;
  int b3 = 0, b2 = 0;
  int64_t p3 = 1;
  for (int i3 = 0; p3 <= FFT_MAX_LEN; ++i3, p3 *= 3) {
    int64_t v = p3 * 2;
    int i2 = 1;
    while (v < n_min) {
      v *= 2;
      ++i2;
    }
    if (v <= FFT_MAX_LEN && (best < 0 || v < best)) {
      best = v;
      b3 = i3;
      b2 = i2;
    }
  }
  if (best < 0) return -1;
  *n3 = b3;
  *n2 = b2;
  return (int)best;
}

cudaError_t fft_twiddles(int L, float4** d_tw) {
  std::vector<float4> h((size_t)(L / 2 > 0 ? L / 2 : 1));
  for (int k = 0; k < L / 2; ++k) {
    const double a = -2.0 * M_PI * (double)k / (double)L;
    h[k] = dfc_from_double(cos(a), sin(a));
  }
  cudaError_t e = cudaMalloc(d_tw, h.size() * sizeof(float4));
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*d_tw, h.data(), h.size() * sizeof(float4), cudaMemcpyHostToDevice);
}

cudaError_t fft_setup_attributes() {
  const int max_smem = (int)(((size_t)FFT_MAX_LEN + 1 + tw_place<float4>(FFT_MAX_LEN / 2)) * sizeof(float4));
  cudaError_t e = cudaFuncSetAttribute(k_fft_lines<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fft_lines<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  return e;
}

namespace {

// Lines per CTA for a line length L: as many as keep the CTA's lines and
// twiddle table within a third of the SM's shared memory (three CTAs of 256
// threads at 80 registers share an SM and hide each other's barriers), at
// least one; 8 double-float or 16 FP32 columns where they fit, a 128-byte
// segment of every row and a set of lines whose elements lie in distinct banks.
// Fewer while a launch would not give every SM three CTAs.
constexpr size_t FFT_CTA_BYTES = 74 * 1024;
size_t cta_bytes(int L, int B, size_t elem) {
  return ((size_t)B * (L + 1) + (elem == sizeof(float4) ? tw_place<float4>(L / 2) : tw_place<float2>(L / 2))) * elem;
}
int lines_per_cta(int L, size_t elem) {
  const int most = (int)(128 / elem);
  int B = 1;
  while (B < most && cta_bytes(L, B + 1, elem) <= FFT_CTA_BYTES) ++B;
  return B;
}
int64_t ctas(const FftLines& d, int B, int ngrids) { return (d.n_lines + B - 1) / B * ngrids; }

// Threads of a CTA with `smem` bytes: the SM's 24 warps over the CTAs that fit
int cta_threads(size_t smem) {
  const size_t fit = (size_t)228 * 1024 / (smem + 1024);
  return fit >= 3 ? 256 : fit == 2 ? 384 : 768;
}

// One pass (rows or columns) of both plane sets: in one launch while three CTAs
// of either kind share an SM (short lines, where launches and tails count),
// else each with the shared memory and threads of its own.
cudaError_t launch_lines(bool inverse, const float4* in4, float4* out4, FftLines d4, int ngrids4, const float2* in2,
                         float2* out2, FftLines d2, int ngrids2, const float4* tw, int num_sms, cudaStream_t s) {
  d4.B = lines_per_cta(d4.L, sizeof(float4));
  d2.B = lines_per_cta(d2.L, sizeof(float2));
  while (ctas(d4, d4.B, ngrids4) + ctas(d2, d2.B, ngrids2) < 3 * (int64_t)num_sms && d4.B > 1) {
    d4.B = (d4.B + 1) / 2;
    d2.B = (d2.B + 1) / 2;
  }
  const int64_t b4 = ctas(d4, d4.B, ngrids4), b2 = ctas(d2, d2.B, ngrids2);
  const size_t smem4 = cta_bytes(d4.L, d4.B, sizeof(float4)), smem2 = cta_bytes(d2.L, d2.B, sizeof(float2));
  auto launch = [&](int64_t n4, int64_t n2, size_t smem) {
    if (n4 + n2 <= 0) return cudaSuccess;
    const int threads = cta_threads(smem);
    return launch_after(inverse ? k_fft_lines<true> : k_fft_lines<false>, (unsigned)(n4 + n2), (unsigned)threads, smem,
                        s, in4, out4, d4, n4, in2, out2, d2, tw);
  };
  const size_t both = smem4 > smem2 ? smem4 : smem2;
  if (cta_threads(both) == 256) return launch(b4, b2, both);
  cudaError_t e = launch(b4, 0, smem4);
  return e == cudaSuccess ? launch(0, b2, smem2) : e;
}

FftLines row_lines(const Fft2d& f, int64_t ny) {
  FftLines r{};
  r.L = f.Nx; r.n3 = f.n3x; r.n2 = f.n2x;
  r.n_lines = ny;
  r.in_elem_stride = 1; r.out_elem_stride = 1;
  return r;
}

FftLines col_lines(const Fft2d& f) {
  FftLines c{};
  c.L = f.Ny; c.n3 = f.n3y; c.n2 = f.n2y;
  c.n_lines = f.Nx;
  c.in_line_stride = 1; c.in_elem_stride = f.Nx; c.out_line_stride = 1; c.out_elem_stride = f.Nx;
  c.in_grid_stride = (int64_t)f.Nx * f.Ny; c.out_grid_stride = (int64_t)f.Nx * f.Ny;
  return c;
}

}  // namespace

int fft2d_launches(const Fft2d& f) {
  int n = 0;
  for (int L : {f.Nx, f.Ny}) {
    const size_t s4 = cta_bytes(L, lines_per_cta(L, sizeof(float4)), sizeof(float4));
    n += cta_threads(s4) == 256 ? 1 : 2;
  }
  return n;
}

cudaError_t fft2d_forward(const float4* compact4, float4* spec4, int ngrids4, const float2* compact2, float2* spec2,
                          int ngrids2, int64_t nx, int64_t ny, int64_t in_grid_stride, const Fft2d& f,
                          cudaStream_t s) {
  // rows: compact rows [0, ny) -> spectrum rows, zero-padded to Nx
  FftLines r = row_lines(f, ny);
  r.in_len = (int)nx; r.out_len = f.Nx;
  r.in_line_stride = nx; r.out_line_stride = f.Nx;
  r.in_grid_stride = in_grid_stride; r.out_grid_stride = (int64_t)f.Nx * f.Ny;
  cudaError_t e = launch_lines(false, compact4, spec4, r, ngrids4, compact2, spec2, r, ngrids2, f.tw_x, f.num_sms, s);
  if (e != cudaSuccess) return e;
  // columns: all Nx, rows >= ny read as zero
  FftLines c = col_lines(f);
  c.in_len = (int)ny; c.out_len = f.Ny;
  return launch_lines(false, spec4, spec4, c, ngrids4, spec2, spec2, c, ngrids2, f.tw_y, f.num_sms, s);
}

cudaError_t fft2d_inverse(float4* spec4, float4* compact4, int ngrids4, float2* spec2, float2* compact2, int ngrids2,
                          const Fft2d& f, int64_t nx, int64_t ny, int64_t out_grid_stride, cudaStream_t s) {
  FftLines c = col_lines(f);
  c.in_len = f.Ny; c.out_len = (int)ny;
  cudaError_t e = launch_lines(true, spec4, spec4, c, ngrids4, spec2, spec2, c, ngrids2, f.tw_y, f.num_sms, s);
  if (e != cudaSuccess) return e;
  FftLines r = row_lines(f, ny);
  r.in_len = f.Nx; r.out_len = (int)nx;
  r.in_line_stride = f.Nx; r.out_line_stride = nx;
  r.in_grid_stride = (int64_t)f.Nx * f.Ny; r.out_grid_stride = out_grid_stride;
  return launch_lines(true, spec4, compact4, r, ngrids4, spec2, compact2, r, ngrids2, f.tw_x, f.num_sms, s);
}

}  // namespace irs
