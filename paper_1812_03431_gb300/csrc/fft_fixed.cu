// Longitude transforms of the FP64 form (paper Sec. 3) in block fixed point: the sums, packing and
// layouts of fft.cu, with 64-bit integers in place of binary64 inside the transform.
//
// A binary64 FFT is adds and multiply-adds on a unit that issues one warp instruction per 64
// cycles and scheduler on GB300 (0.99 and 1.11 ms at T341 with 16 states).  Here a row's data
// are integers below 2^58 with a common power of two; an add is two integer instructions, a
// product by a twiddle (two signed limbs of radix 2^30, 59 bits) three 32 x 32 -> 64 bit
// multiply-adds of 4 cycles.  Before each pass a row whose largest part has reached 2^58 is
// shifted down (rounding); its largest is found while the pass before writes, so a row keeps
// 57 bits below its own largest value throughout.  Rows are scaled and put into fixed point on
// the way in, and rounded to binary64 once on the way out.
//
// Measured on GB300 (forward, inverse; against the binary64 passes): T341 x 16 0.325, 0.315 / 0.992,
// 1.107 ms; T255 x 8 0.121, 0.115 / 0.318, 0.349; T63 x 1 0.010, 0.011 / 0.014, 0.015.  The integer
// pipe is 53 to 63 % busy (ncu, T255 x 8); latency between the passes' barriers takes the rest.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "fixed.h"
#include "rexi_internal.h"

namespace rexi {

using namespace fixed;

namespace {

typedef longlong2 I2;
constexpr int kTop = 58;  // a pass starts with parts below 2^58

struct FixedFft {
  const int4 *tw;  // n twiddles e^{-2 pi i k / n} as limbs {re hi, re lo, im hi, im lo}
  int n, h, nstages, N, nlat, ncol, np;  // h = n / 2 complex points per row; np rows per CTA
  int radix[24];
  uint32_t mag_nb[24], mag_ns[24], mag_h, mag_np;  // divisions by run-time sizes as multiply-highs
  int2 r2, c3, s3, c5a, s5a, c5b, s5b;  // 1/sqrt(2), cos/sin of 2pi/3, 2pi/5, 4pi/5 as limbs
};

// exact for 0 <= x < 2^16 and 1 <= d < 2^16
__device__ __forceinline__ int fdiv(int x, uint32_t mag, int d) { return d == 1 ? x : (int)__umulhi((uint32_t)x, mag); }

__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// acc (hi sums, rounded middle sums) += v t for a limb pair t, |v| < 2^61 (4 sqrt(2) 2^kTop in radix 8)
struct Acc {
  long long hh = 0, hl = 1 << 29;
  __device__ __forceinline__ void add(int2 v, int2 t) {
    mad_wide(hh, v.x, t.x);
    mad_wide(hl, v.x, t.y);
    mad_wide(hl, v.y, t.x);
  }
  __device__ __forceinline__ long long get() const { return hh + (hl >> 30); }
};
__device__ __forceinline__ int2 split(long long v) {
  return make_int2((int)((v + (1 << 29)) >> 30), (int)((unsigned)v << 2) >> 2);
}
__device__ __forceinline__ int2 neg(int2 t) { return make_int2(-t.x, -t.y); }
__device__ __forceinline__ long long scale(long long v, int2 t) {
  Acc a;
  a.add(split(v), t);
  return a.get();
}
__device__ __forceinline__ I2 cmul(I2 v, int4 t) {
  const int2 x = split(v.x), y = split(v.y), tr = make_int2(t.x, t.y), ti = make_int2(t.z, t.w);
  Acc re, im;
  re.add(x, tr);
  re.add(y, neg(ti));
  im.add(x, ti);
  im.add(y, tr);
  return I2{re.get(), im.get()};
}
__device__ __forceinline__ I2 add(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ I2 sub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ I2 mulmi(I2 a) { return I2{a.y, -a.x}; }  // -i a

// In-register DFT of R points (forward, e^{-2 pi i jk/R})
template <int R>
__device__ __forceinline__ void dft_small(I2 *v, const FixedFft &a) {
  if constexpr (R == 2) {
    const I2 t = v[0];
    v[0] = add(t, v[1]);
    v[1] = sub(t, v[1]);
  } else if constexpr (R == 4) {
    const I2 t0 = add(v[0], v[2]), t1 = sub(v[0], v[2]), t2 = add(v[1], v[3]), t3 = mulmi(sub(v[1], v[3]));
    v[0] = add(t0, t2);
    v[2] = sub(t0, t2);
    v[1] = add(t1, t3);
    v[3] = sub(t1, t3);
  } else if constexpr (R == 8) {
    const I2 a0 = add(v[0], v[4]), a1 = sub(v[0], v[4]), a2 = add(v[2], v[6]), a3 = mulmi(sub(v[2], v[6]));
    const I2 b0 = add(v[1], v[5]), b1 = sub(v[1], v[5]), b2 = add(v[3], v[7]), b3 = mulmi(sub(v[3], v[7]));
    const I2 e0 = add(a0, a2), e2 = sub(a0, a2), e1 = add(a1, a3), e3 = sub(a1, a3);
    const I2 o0 = add(b0, b2), o2 = sub(b0, b2), o1 = add(b1, b3), o3 = sub(b1, b3);
    // o1 (1 - i)/sqrt(2), o2 (-i), o3 (-1 - i)/sqrt(2)
    const I2 w1 = {scale(o1.x, a.r2) + scale(o1.y, a.r2), scale(o1.y, a.r2) - scale(o1.x, a.r2)};
    const I2 w2 = mulmi(o2);
    const long long p = scale(o3.x, a.r2), q = scale(o3.y, a.r2);
    const I2 w3 = {q - p, -p - q};
    v[0] = add(e0, o0);
    v[4] = sub(e0, o0);
    v[1] = add(e1, w1);
    v[5] = sub(e1, w1);
    v[2] = add(e2, w2);
    v[6] = sub(e2, w2);
    v[3] = add(e3, w3);
    v[7] = sub(e3, w3);
  } else if constexpr (R == 3) {
    const I2 s = add(v[1], v[2]), d = sub(v[1], v[2]);
    const I2 t = {v[0].x + scale(s.x, a.c3), v[0].y + scale(s.y, a.c3)};
    const I2 u = mulmi(I2{scale(d.x, a.s3), scale(d.y, a.s3)});
    v[0] = add(v[0], s);
    v[1] = add(t, u);
    v[2] = sub(t, u);
  } else {  // R == 5
    const I2 b1 = add(v[1], v[4]), b2 = add(v[2], v[3]), d1 = sub(v[1], v[4]), d2 = sub(v[2], v[3]);
    auto two = [](long long x, int2 s, long long y, int2 t) {
      Acc c;
      c.add(split(x), s);
      c.add(split(y), t);
      return c.get();
    };
    const I2 t1 = {v[0].x + two(b1.x, a.c5a, b2.x, a.c5b), v[0].y + two(b1.y, a.c5a, b2.y, a.c5b)};
    const I2 t2 = {v[0].x + two(b1.x, a.c5b, b2.x, a.c5a), v[0].y + two(b1.y, a.c5b, b2.y, a.c5a)};
    const I2 u1 = mulmi(I2{two(d1.x, a.s5a, d2.x, a.s5b), two(d1.y, a.s5a, d2.y, a.s5b)});
    const I2 u2 = mulmi(I2{two(d1.x, a.s5b, d2.x, neg(a.s5a)), two(d1.y, a.s5b, d2.y, neg(a.s5a))});
    v[0] = add(v[0], add(b1, b2));
    v[1] = add(t1, u1);
    v[4] = sub(t1, u1);
    v[2] = add(t2, u2);
    v[3] = sub(t2, u2);
  }
}

// bits 32 ... 62 of the larger part's magnitude (one's complement for negatives)
__device__ __forceinline__ int size_of(I2 v) {
  const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
  return max(x ^ (x >> 31), y ^ (y >> 31));
}
// how far a row whose largest is `top` (size_of) has to come down to be below 2^kTop
__device__ __forceinline__ int down(int top) { return max(0, 64 - kTop - __clz(top)); }
__device__ __forceinline__ long long shift(long long v, int s) { return (v + ((1ll << s) >> 1)) >> s; }

// atomicMax(p + q, v), one per warp where its threads share a row
__device__ __forceinline__ void row_max(int *p, int q, int v) {
  const unsigned mask = __activemask();
  const int first = __ffs(mask) - 1;
  if (__all_sync(mask, q == __shfl_sync(mask, q, first))) {
    v = (int)__reduce_max_sync(mask, (unsigned)v);
    if ((int)(threadIdx.x & 31) == first) atomicMax(p + q, v);
  } else {
    atomicMax(p + q, v);
  }
}

// One Stockham pass of radix R over np rows of n points: src -> dst.  top: the rows' largest
// on entry, next: those on exit (zero before), ex: the rows' exponents.
template <int R>
__device__ __forceinline__ void stockham_pass(const I2 *src, I2 *dst, int n, int Ns, uint32_t mnb, uint32_t mns,
                                              const int *top, int *next, int *ex, const FixedFft &a) {
  const int nb = n / R;
  const int tstep = 2 * (n / (Ns * R));  // twiddle e^{-2 pi i jm r / (Ns R)} = tw[r jm tstep]
  for (int t = threadIdx.x; t < a.np * nb; t += blockDim.x) {
    const int q = fdiv(t, mnb, nb), jb = t - q * nb;
    const I2 *in = src + q * n;
    I2 *out = dst + q * n;
    const int jd = fdiv(jb, mns, Ns), jm = jb - jd * Ns;
    const int s = down(top[q]);
    if (jb == 0) ex[q] += s;
    I2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = in[jb + r * nb];
      if (s) v[r] = I2{shift(v[r].x, s), shift(v[r].y, s)};
    }
    if (jm) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(a.tw + r * jm * tstep));
    }
    dft_small<R>(v, a);
    const int od = jd * Ns * R + jm;
    int big = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      out[od + r * Ns] = v[r];
      big = max(big, size_of(v[r]));
    }
    row_max(next, q, big);
  }
}

// In-shared-memory forward FFT of np rows of h points; returns the buffer holding the result
__device__ I2 *fft_smem(I2 *buf0, I2 *buf1, int *tops, int *ex, const FixedFft &a) {
  const int n = a.h;
  I2 *src = buf0, *dst = buf1;
  int Ns = 1;
  for (int s = 0; s < a.nstages; ++s) {
    const int R = a.radix[s];
    const uint32_t mnb = a.mag_nb[s], mns = a.mag_ns[s];
    const int *top = tops + s * a.np;
    int *next = tops + (s + 1) * a.np;
    switch (R) {  // uniform across the block
      case 8: stockham_pass<8>(src, dst, n, Ns, mnb, mns, top, next, ex, a); break;
      case 4: stockham_pass<4>(src, dst, n, Ns, mnb, mns, top, next, ex, a); break;
      case 2: stockham_pass<2>(src, dst, n, Ns, mnb, mns, top, next, ex, a); break;
      case 3: stockham_pass<3>(src, dst, n, Ns, mnb, mns, top, next, ex, a); break;
      default: stockham_pass<5>(src, dst, n, Ns, mnb, mns, top, next, ex, a); break;
    }
    __syncthreads();
    I2 *tmp = src;
    src = dst;
    dst = tmp;
    Ns *= R;
  }
  return src;
}

// Shared memory: two buffers of np x h, then per row: the largest part before each pass and
// after the last, the exponent, the binary64 exponent of the row's largest input.
struct Rows {
  I2 *buf0, *buf1;
  int *tops, *ex, *emax;
  __device__ Rows(unsigned char *sm, const FixedFft &a) {
    buf0 = reinterpret_cast<I2 *>(sm);
    buf1 = buf0 + a.np * a.h;
    tops = reinterpret_cast<int *>(buf1 + a.np * a.h);
    ex = tops + (a.nstages + 1) * a.np;
    emax = ex + a.np;
    for (int t = threadIdx.x; t < (a.nstages + 3) * a.np; t += blockDim.x) tops[t] = 0;
  }
  // row q's exponent once its largest input is known: parts below 2^kTop
  __device__ __forceinline__ void begin(int q) {
    ex[q] = emax[q] == 0x7ff ? kNotFinite : emax[q] - 1023 - (kTop - 1);
    tops[q] = (1 << (kTop - 32)) - 1;
  }
};

__device__ __forceinline__ int larger(double2 v) { return max(bexp(v.x), bexp(v.y)); }
// v as integers in units of 2^(E - 1023 - 57): 2^58 at most
__device__ __forceinline__ I2 to_int(double2 v, int E) {
  return I2{(to_fixed(v.x, E - bexp(v.x)) + 8) >> 4, (to_fixed(v.y, E - bexp(v.y)) + 8) >> 4};
}

__global__ void __launch_bounds__(256) fft_fixed_fwd_kernel(FixedFft a, const double *grid, double2 *four,
                                                            const double *in_scale, const double *m_scale) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Rows w(smraw, a);
  __syncthreads();
  const int h = a.h, j = blockIdx.y, c0 = blockIdx.x * a.np, total = a.np * h;
  const double2 *g2 = reinterpret_cast<const double2 *>(grid);
  double2 *raw = reinterpret_cast<double2 *>(w.buf1);
  constexpr int kLd = 8;  // loads of a chunk issued before any use
  for (int t0 = 0; t0 < total; t0 += kLd * blockDim.x) {
    double2 x[kLd];
    double sv[kLd];
    bool ok[kLd];
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      const int t = t0 + i * blockDim.x + threadIdx.x;
      const int q = fdiv(t, a.mag_h, h), k = t - q * h, c = c0 + q;
      ok[i] = t < total && c < a.ncol;
      x[i] = g2[ok[i] ? ((int64_t)c * a.nlat + j) * h + k : 0];
      sv[i] = in_scale[ok[i] ? (c % 3) * a.nlat + j : 0];
    }
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      const int t = t0 + i * blockDim.x + threadIdx.x;
      if (t >= total) break;
      const double2 v = ok[i] ? make_double2(sv[i] * x[i].x, sv[i] * x[i].y) : make_double2(0, 0);
      raw[t] = v;
      row_max(w.emax, fdiv(t, a.mag_h, h), larger(v));
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < a.np; q += blockDim.x) w.begin(q);
  for (int t = threadIdx.x; t < total; t += blockDim.x) w.buf0[t] = to_int(raw[t], w.emax[fdiv(t, a.mag_h, h)]);
  __syncthreads();
  const I2 *Z = fft_smem(w.buf0, w.buf1, w.tops, w.ex, a);
  const int M1 = a.N + 1;
  for (int t = threadIdx.x; t < a.np * M1; t += blockDim.x) {
    const int m = fdiv(t, a.mag_np, a.np), q = t - m * a.np, c = c0 + q;
    if (c >= a.ncol) continue;
    const int s = down(w.tops[a.nstages * a.np + q]);
    I2 zm = Z[q * h + m], zr = Z[q * h + (m == 0 ? 0 : h - m)];
    zm = I2{shift(zm.x, s), shift(zm.y, s)};
    zr = I2{shift(zr.x, s), shift(zr.y, s)};
    // 2 E = Z_m + conj Z_{h-m},  2 O = (Z_m - conj Z_{h-m}) / i
    const I2 E = {zm.x + zr.x, zm.y - zr.y}, O = {zm.y + zr.y, zr.x - zm.x};
    const I2 X = add(E, cmul(O, __ldg(a.tw + m)));
    const double sc = m_scale[m];
    const int e = w.ex[q] >= kNotFinite / 2 ? kNotFinite : w.ex[q] + s - 1;
    four[((int64_t)j * M1 + m) * a.ncol + c] = make_double2(sc * fixed_to_double(X.x, e), sc * fixed_to_double(X.y, e));
  }
}

__global__ void __launch_bounds__(256) fft_fixed_inv_kernel(FixedFft a, const double2 *four, double *grid,
                                                            const double *m_scale, const double *out_scale) {
  extern __shared__ __align__(16) unsigned char smraw[];
  Rows w(smraw, a);
  __syncthreads();
  const int h = a.h, j = blockIdx.y, c0 = blockIdx.x * a.np, N = a.N, M1 = N + 1, total = a.np * M1;
  double2 *raw = reinterpret_cast<double2 *>(w.buf1);  // [row][M1], M1 <= h
  constexpr int kLd = 4;
  // column index fastest, so that neighbouring threads read neighbouring Fourier columns
  for (int t0 = 0; t0 < total; t0 += kLd * blockDim.x) {
    double2 x[kLd];
    double sv[kLd];
    bool ok[kLd];
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      const int t = t0 + i * blockDim.x + threadIdx.x;
      const int m = fdiv(t, a.mag_np, a.np), c = c0 + t - m * a.np;
      ok[i] = t < total && c < a.ncol;
      x[i] = four[ok[i] ? ((int64_t)j * M1 + m) * a.ncol + c : 0];
      sv[i] = m_scale[ok[i] ? m : 0];
    }
#pragma unroll
    for (int i = 0; i < kLd; ++i) {
      const int t = t0 + i * blockDim.x + threadIdx.x;
      if (t >= total) break;
      const int m = fdiv(t, a.mag_np, a.np), q = t - m * a.np;
      // X_0 is real
      const double2 v = ok[i] ? make_double2(sv[i] * x[i].x, m == 0 ? 0.0 : sv[i] * x[i].y) : make_double2(0, 0);
      raw[q * M1 + m] = v;
      atomicMax(w.emax + q, larger(v));
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < a.np; q += blockDim.x) {
    w.begin(q);
    w.ex[q] += 2;  // the parts below are kept at a quarter: Z' has up to 2 + 2 sqrt(2) times the largest,
                   // 1.2 x 2^kTop, which the first pass has room for
  }
  for (int t = threadIdx.x; t < a.np * h; t += blockDim.x) {
    const int q = fdiv(t, a.mag_h, h), m = t - q * h, mr = h - m;  // partner X_{h-m}, present when h - m <= N
    const int E2 = w.emax[q];
    const I2 zero = {0, 0};
    const I2 A = m <= N ? to_int(raw[q * M1 + m], E2) : zero;
    I2 B = m > 0 && mr <= N ? to_int(raw[q * M1 + mr], E2) : zero;
    B.y = -B.y;  // conj(X_{h-m})
    const I2 A4 = {shift(A.x, 2), shift(A.y, 2)}, B4 = {shift(B.x, 2), shift(B.y, 2)};
    // E' = X_m + conj X_{h-m},  O' = (X_m - conj X_{h-m}) e^{+2 pi i m / n},  Z' = E' + i O'
    const int4 tw = __ldg(a.tw + m);
    const I2 E = add(A4, B4), O = cmul(sub(A4, B4), make_int4(tw.x, tw.y, -tw.z, -tw.w));
    w.buf0[t] = I2{E.x - O.y, -E.y - O.x};  // conj(Z') for the inverse by a forward FFT
  }
  __syncthreads();
  const I2 *r = fft_smem(w.buf0, w.buf1, w.tops, w.ex, a);
  double2 *g2 = reinterpret_cast<double2 *>(grid);
  for (int t = threadIdx.x; t < a.np * h; t += blockDim.x) {
    const int q = fdiv(t, a.mag_h, h), k = t - q * h, c = c0 + q;
    if (c >= a.ncol) continue;
    const double s = out_scale[(c % 3) * a.nlat + j];
    const I2 v = r[t];  // conj of z_k = x_{2k} + i x_{2k+1}
    const int e = w.ex[q] >= kNotFinite / 2 ? kNotFinite : w.ex[q];
    g2[((int64_t)c * a.nlat + j) * h + k] = make_double2(s * fixed_to_double(v.x, e), -s * fixed_to_double(v.y, e));
  }
}

int2 host_limbs(double t) {  // |t| <= 1 as x 2^-30 + y 2^-60
  const double x = std::nearbyint(std::ldexp(t, 30));
  return make_int2((int)x, (int)std::nearbyint(std::ldexp(t - std::ldexp(x, -30), 60)));
}

uint32_t magic(int d) { return d > 1 ? (uint32_t)((1ull << 32) / (unsigned)d + 1) : 0u; }

int rows_per_cta(const Plan &pl, int B) {
  // the plan's nsplit (its shared memory holds that many), spread evenly over the fewest CTAs
  // a latitude needs
  const int ncol = 3 * B, nblk = (ncol + pl.fft.nsplit - 1) / pl.fft.nsplit;
  return (ncol + nblk - 1) / nblk;
}

size_t smem_bytes(const Plan &pl, int np) {
  return (size_t)np * pl.fft.n * sizeof(I2) + (size_t)(pl.fft.nstages + 3) * np * sizeof(int);
}

FixedFft make_args(const Plan &pl, int B) {
  FixedFft a;
  a.tw = static_cast<const int4 *>(pl.fft.tw_dev);
  a.n = pl.fft.n;
  a.h = pl.fft.n / 2;
  a.nstages = pl.fft.nstages;
  a.N = pl.N;
  a.nlat = pl.nlat;
  a.ncol = 3 * B;
  a.np = rows_per_cta(pl, B);
  int Ns = 1;
  for (int s = 0; s < a.nstages; ++s) {
    a.radix[s] = pl.fft.radix[s];
    a.mag_nb[s] = magic(a.h / a.radix[s]);
    a.mag_ns[s] = magic(Ns);
    Ns *= a.radix[s];
  }
  a.mag_h = magic(a.h);
  a.mag_np = magic(a.np);
  a.r2 = host_limbs(std::sqrt(0.5));
  a.c3 = host_limbs(std::cos(2.0 * M_PI / 3.0));
  a.s3 = host_limbs(std::sin(2.0 * M_PI / 3.0));
  a.c5a = host_limbs(std::cos(2.0 * M_PI / 5.0));
  a.s5a = host_limbs(std::sin(2.0 * M_PI / 5.0));
  a.c5b = host_limbs(std::cos(4.0 * M_PI / 5.0));
  a.s5b = host_limbs(std::sin(4.0 * M_PI / 5.0));
  return a;
}

}  // namespace

// the twiddles as limbs
void fft_fixed_twiddles(const std::vector<double2> &tw, std::vector<int4> &limbs) {
  for (const double2 &t : tw) {
    const int2 re = host_limbs(t.x), im = host_limbs(t.y);
    limbs.push_back(make_int4(re.x, re.y, im.x, im.y));
  }
}

cudaError_t launch_fft_fixed_fwd(Plan &pl, const double *grid, double2 *four, int B, const double *in_scale,
                                 const double *m_scale, cudaStream_t st) {
  const FixedFft a = make_args(pl, B);
  const dim3 g((unsigned)((a.ncol + a.np - 1) / a.np), (unsigned)pl.nlat);
  fft_fixed_fwd_kernel<<<g, 256, smem_bytes(pl, a.np), st>>>(a, grid, four, in_scale, m_scale);
  return cudaGetLastError();
}

cudaError_t launch_fft_fixed_inv(Plan &pl, const double2 *four, double *grid, int B, const double *m_scale,
                                 const double *out_scale, cudaStream_t st) {
  const FixedFft a = make_args(pl, B);
  const dim3 g((unsigned)((a.ncol + a.np - 1) / a.np), (unsigned)pl.nlat);
  fft_fixed_inv_kernel<<<g, 256, smem_bytes(pl, a.np), st>>>(a, four, grid, m_scale, out_scale);
  return cudaGetLastError();
}

cudaError_t fft_fixed_configure(Plan &pl) {
  const int bytes = (int)smem_bytes(pl, pl.fft.nsplit);
  cudaError_t e = cudaFuncSetAttribute(fft_fixed_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fft_fixed_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace rexi
