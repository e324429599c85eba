// Device code of the fast cosine transforms behind the direct depth solve (spectral.cu) and the preconditioner of
// the weighted solves (poisson.cu); what it computes and why: spectral.cu.
#pragma once

#include "irtps_internal.h"

namespace irtps {
namespace spec {

constexpr int kSpecThreads = 256;

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cneg_i(float2 a) { return make_float2(a.y, -a.x); }  // -i a
__device__ __forceinline__ float2 cswap(float2 a) { return make_float2(a.y, a.x); }

// DFTs of R points (e^{-2 pi i / R}) in registers.
template <int R>
__device__ __forceinline__ void dft_small(float2 (&v)[R]);
template <>
__device__ __forceinline__ void dft_small<2>(float2 (&v)[2]) {
  const float2 a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}
__device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d) {
  const float2 t0 = cadd(a, c), t1 = csub(a, c), t2 = cadd(b, d), t3 = cneg_i(csub(b, d));
  a = cadd(t0, t2);
  b = cadd(t1, t3);
  c = csub(t0, t2);
  d = csub(t1, t3);
}
template <>
__device__ __forceinline__ void dft_small<4>(float2 (&v)[4]) { dft4(v[0], v[1], v[2], v[3]); }
template <>
__device__ __forceinline__ void dft_small<8>(float2 (&v)[8]) {
  float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  dft4(e[0], e[1], e[2], e[3]);
  dft4(o[0], o[1], o[2], o[3]);
  const float r = 0.70710678118654752440f;
  o[1] = make_float2(r * (o[1].x + o[1].y), r * (o[1].y - o[1].x));
  o[2] = cneg_i(o[2]);
  o[3] = make_float2(r * (o[3].y - o[3].x), -r * (o[3].x + o[3].y));
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = cadd(e[k], o[k]);
    v[k + 4] = csub(e[k], o[k]);
  }
}
// odd R: pairs v[m] +- v[R - m] against the cosines and sines of 2 pi k m / R (C[j], S[j], j = k m mod R)
template <int R>
__device__ __forceinline__ void dft_odd(float2 (&v)[R], const float (&C)[R], const float (&S)[R]) {
  constexpr int h = R / 2;
  float2 a[h], b[h];
#pragma unroll
  for (int m = 1; m <= h; ++m) {
    a[m - 1] = cadd(v[m], v[R - m]);
    b[m - 1] = csub(v[m], v[R - m]);
  }
  const float2 v0 = v[0];
#pragma unroll
  for (int m = 0; m < h; ++m) v[0] = cadd(v[0], a[m]);
#pragma unroll
  for (int k = 1; k <= h; ++k) {
    float2 p = v0, q = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int m = 1; m <= h; ++m) {
      const int j = (k * m) % R;
      p.x = fmaf(C[j], a[m - 1].x, p.x);
      p.y = fmaf(C[j], a[m - 1].y, p.y);
      q.x = fmaf(S[j], b[m - 1].x, q.x);
      q.y = fmaf(S[j], b[m - 1].y, q.y);
    }
    v[k] = cadd(p, cneg_i(q));
    v[R - k] = csub(p, cneg_i(q));
  }
}
template <>
__device__ __forceinline__ void dft_small<3>(float2 (&v)[3]) {
  constexpr float C[3] = {1.0f, -0.5f, -0.5f};
  constexpr float S[3] = {0.0f, 0.86602540378443864676f, -0.86602540378443864676f};
  dft_odd<3>(v, C, S);
}
template <>
__device__ __forceinline__ void dft_small<5>(float2 (&v)[5]) {
  constexpr float C[5] = {1.0f, 0.30901699437494742410f, -0.80901699437494742410f, -0.80901699437494742410f,
                          0.30901699437494742410f};
  constexpr float S[5] = {0.0f, 0.95105651629515357212f, 0.58778525229247312917f, -0.58778525229247312917f,
                          -0.95105651629515357212f};
  dft_odd<5>(v, C, S);
}
template <>
__device__ __forceinline__ void dft_small<7>(float2 (&v)[7]) {
  constexpr float C[7] = {1.0f,
                          0.62348980185873353053f,
                          -0.22252093395631440429f,
                          -0.90096886790241912624f,
                          -0.90096886790241912624f,
                          -0.22252093395631440429f,
                          0.62348980185873353053f};
  constexpr float S[7] = {0.0f,
                          0.78183148246802980871f,
                          0.97492791218182360702f,
                          0.43388373911755812048f,
                          -0.43388373911755812048f,
                          -0.97492791218182360702f,
                          -0.78183148246802980871f};
  dft_odd<7>(v, C, S);
}

// Line element i in shared memory: one pad element in 16, so that a radix-8 stage's stores (8 elements
// apart) meet at most two to a bank.
__device__ __forceinline__ int at(int i) { return i + (i >> 4); }
__host__ __device__ inline int line_stride(int m) { return m + (m >> 4) + 1; }

// One autosort stage of radix R over L lines of m points: sub-transforms of ns points become ns R.
template <int R>
__device__ __forceinline__ void fft_stage(const float2 *__restrict__ in, float2 *__restrict__ out, int m, int ns, int L,
                                          const float2 *__restrict__ tw) {
  const int nb = m / R, step = nb / ns, ls = line_stride(m);
  const float inv = 1.0f / (float)ns;
  for (int i = threadIdx.x; i < L * nb; i += blockDim.x) {
    int j = i, base = 0;
    while (j >= nb) {  // L is at most 4
      j -= nb;
      base += ls;
    }
    const int q = (int)(((float)j + 0.5f) * inv), k = j - q * ns;  // exact: j < 2^13
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = in[base + at(j + r * nb)];
    if (ns > 1) {  // one table load, the other powers by products (a few roundings more, against R - 1 scattered loads)
      float2 w[R];
      w[1] = __ldg(tw + k * step);
#pragma unroll
      for (int r = 2; r < R; ++r) w[r] = cmul(w[r / 2], w[r - r / 2]);
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], w[r]);
    }
    dft_small<R>(v);
    const int o = q * ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) out[base + at(o + r * ns)] = v[r];
  }
  __syncthreads();
}

// FFT (e^{-...}) of L lines of P.m points held in a; the result is in the returned buffer (a or b).
__device__ __forceinline__ float2 *fft_lines(const FftPlan &P, float2 *a, float2 *b, int L) {
  int ns = 1;
#pragma unroll 1
  for (int s = 0; s < P.stages; ++s) {
    const int R = P.radix[s];
    switch (R) {
      case 8: fft_stage<8>(a, b, P.m, ns, L, P.tw); break;
      case 7: fft_stage<7>(a, b, P.m, ns, L, P.tw); break;
      case 5: fft_stage<5>(a, b, P.m, ns, L, P.tw); break;
      case 4: fft_stage<4>(a, b, P.m, ns, L, P.tw); break;
      case 3: fft_stage<3>(a, b, P.m, ns, L, P.tw); break;
      default: fft_stage<2>(a, b, P.m, ns, L, P.tw); break;
    }
    ns *= R;
    float2 *t = a;
    a = b;
    b = t;
  }
  return a;
}

// DFT of L lines of P.n points in a (natural order, written by the block, not yet synchronised).
// Lengths whose prime factors exceed 7 go through Bluestein's chirp convolution of a length m >= 2n - 1.
__device__ __forceinline__ float2 *dft_lines(const FftPlan &P, float2 *a, float2 *b, int L) {
  __syncthreads();
  if (!P.chirp) return fft_lines(P, a, b, L);
  const int n = P.n, m = P.m, ls = line_stride(m);
  for (int l = 0; l < L; ++l)
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      float2 &v = a[l * ls + at(i)];
      v = i < n ? cmul(v, __ldg(P.chirp + i)) : make_float2(0.0f, 0.0f);
    }
  __syncthreads();
  float2 *x = fft_lines(P, a, b, L);
  float2 *y = x == a ? b : a;
  for (int l = 0; l < L; ++l)
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      float2 &v = x[l * ls + at(i)];
      v = cswap(cmul(v, __ldg(P.filter + i)));
    }
  __syncthreads();
  x = fft_lines(P, x, y, L);
  for (int l = 0; l < L; ++l)
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      float2 &v = x[l * ls + at(i)];
      v = cmul(cswap(v), __ldg(P.chirp + i));
    }
  __syncthreads();
  return x;
}

// Place of sample j of a line in its FFT: even samples ascending, then odd ones descending.
__device__ __forceinline__ int place(int j, int n) { return (j & 1) ? n - 1 - (j >> 1) : j >> 1; }

// Coefficients C[k] = sum_i x_i cos(pi k (2i+1) / 2n) of the two lines packed in Z, from Z[k] and Z[n-k].
__device__ __forceinline__ float2 dct_pair(float2 z, float2 zr, float2 w) {
  const float2 va = make_float2(0.5f * (z.x + zr.x), 0.5f * (z.y - zr.y));
  const float2 vb = make_float2(0.5f * (z.y + zr.y), 0.5f * (zr.x - z.x));
  return make_float2(w.x * va.x - w.y * va.y, w.x * vb.x - w.y * vb.y);
}
// The packed spectrum of two lines from their coefficients c = C[k], cr = C[n-k] (0 for k = 0), times `scale`
// and swapped (real <-> imaginary), so that a forward DFT gives the swapped inverse.
__device__ __forceinline__ float2 idct_pair(float2 c, float2 cr, float2 w, float scale) {
  // V = e^{i pi k / 2n} (C[k] - i C[n-k]) per line, w = e^{-i pi k / 2n}; Z = V_a + i V_b
  const float2 va = make_float2(w.x * c.x - w.y * cr.x, -w.x * cr.x - w.y * c.x);
  const float2 vb = make_float2(w.x * c.y - w.y * cr.y, -w.x * cr.y - w.y * c.y);
  return make_float2((va.y + vb.x) * scale, (va.x - vb.y) * scale);
}

// A sum of quotients a / b of FP32 numbers to about 48 bits, on the FP32 pipes: each is a FP32 quotient plus the
// quotient of its exact remainder; the quotients are added with an error-free two-sum.
struct QuotientSum {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float a, float b) {
    const float q = __fdiv_rn(a, b);
    const float e = __fdividef(__fmaf_rn(-q, b, a), b);
    const float s = __fadd_rn(hi, q), t = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(q, t)), e));
    hi = s;
  }
};

// Right-hand side b = D^T g of pixel (i, j): trapezoidal edge targets h (s_a + s_b) / 2, slopes -n_x / n_z, -n_y / n_z.
__device__ __forceinline__ double rhs_at(const SpecObj &o, int i, int j) {
  const float4 *n = o.nrm + (size_t)i * o.W + j;
  const bool l = j > 0, r = j < o.W - 1, u = i > 0, d = i < o.H - 1;
  QuotientSum v;
  auto add = [&](float c, const float4 &m) { v.add(c, fmaxf(m.z, o.nz_min)); };
  if (l) { const float4 m = __ldg(n - 1); add(-m.x, m); }
  if (r) { const float4 m = __ldg(n + 1); add(m.x, m); }
  if (u) { const float4 m = __ldg(n - o.W); add(-m.y, m); }
  if (d) { const float4 m = __ldg(n + o.W); add(m.y, m); }
  if (l != r || u != d) {  // on a border the pixel's own slope does not cancel
    const float4 m = __ldg(n);
    if (l != r) add(l ? -m.x : m.x, m);
    if (u != d) add(u ? -m.y : m.y, m);
  }
  return 0.5 * o.h * ((double)v.hi + (double)v.lo);
}

// r = b - A x of pixel (i, j) in FP64.
__device__ __forceinline__ double residual_at(const SpecObj &o, int i, int j) {
  const size_t p = (size_t)i * o.W + j;
  const double *x = o.x + p;
  if (j > 0 && j < o.W - 1 && i > 0 && i < o.H - 1)  // FP64 is what bounds this: five operations
    return fma(-4.0, x[0], (x[-1] + x[1]) + (x[-o.W] + x[o.W])) + o.b[p];
  double s = o.b[p];
  if (j > 0) s += x[-1] - x[0];
  if (j < o.W - 1) s += x[1] - x[0];
  if (i > 0) s += x[-o.W] - x[0];
  if (i < o.H - 1) s += x[o.W] - x[0];
  return s;
}

// Block sum in FP64; the result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double *sh) {
  for (int k = 16; k > 0; k >>= 1) v += __shfl_down_sync(0xffffffffu, v, k);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < blockDim.x / 32 ? sh[threadIdx.x] : 0.0;
    for (int k = 16; k > 0; k >>= 1) v += __shfl_down_sync(0xffffffffu, v, k);
  }
  return v;
}

extern __shared__ __align__(16) float2 spec_smem[];

// Rows forward: two rows per block, of b (from the normals, kept; |b|^2 partials), of the residual, or of the values
// load(p) of the pixels.
struct NoCall {
  __device__ float operator()(size_t, float = 0.0f) const { return 0.0f; }
};
enum : int { SRC_RHS = 0, SRC_RESIDUAL = 1, SRC_CALL = 2 };
template <int SRC, class F = NoCall>
__device__ __forceinline__ void rows_forward(const SpecObj &o, int blk, F load = F()) {
  const FftPlan &P = o.row;
  const int n = o.W, i0 = 2 * blk;
  const bool two = i0 + 1 < o.H;
  float2 *a = spec_smem, *b = a + line_stride(P.m);
  double bb = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    if (SRC == SRC_CALL) {
      const size_t p = (size_t)i0 * n + j;
      a[at(place(j, n))] = make_float2(load(p), two ? load(p + n) : 0.0f);
      continue;
    }
    double u, v = 0.0;
    if (SRC == SRC_RHS) {
      u = rhs_at(o, i0, j);
      o.b[(size_t)i0 * n + j] = u;
      if (two) {
        v = rhs_at(o, i0 + 1, j);
        o.b[(size_t)(i0 + 1) * n + j] = v;
      }
      bb += u * u + v * v;
    } else {
      u = residual_at(o, i0, j);
      if (two) v = residual_at(o, i0 + 1, j);
    }
    a[at(place(j, n))] = make_float2((float)u, (float)v);
  }
  if (SRC == SRC_RHS) {
    __shared__ double sh[32];
    bb = block_sum(bb, sh);
    if (threadIdx.x == 0) {
      o.part[blk] = bb;
      if (blk == 0) {  // barrier state of the last pass
        o.ctl->count = 0u;
        o.ctl->err = 0;
      }
    }
  }
  const float2 *z = dft_lines(P, a, b, 1);
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const float2 c = dct_pair(z[at(k)], z[at(k ? n - k : 0)], __ldg(P.half + k));
    o.t[(size_t)i0 * n + k] = c.x;
    if (two) o.t[(size_t)(i0 + 1) * n + k] = c.y;
  }
}

// Columns: 2 L columns per block, forward, divided by the eigenvalues, and back.
template <int L>
__device__ __forceinline__ void columns_of(const SpecObj &o, int blk) {
  constexpr int C = 2 * L;
  const FftPlan &P = o.col;
  const int n = o.H, W = o.W, c0 = blk * C;
  const int ls = line_stride(P.m);
  float2 *a = spec_smem, *b = a + L * ls;
#pragma unroll 4
  for (int e = threadIdx.x; e < n * C; e += blockDim.x) {
    const int i = e / C, cc = e - i * C;
    const float v = c0 + cc < W ? o.t[(size_t)i * W + c0 + cc] : 0.0f;
    reinterpret_cast<float *>(a + (cc >> 1) * ls + at(place(i, n)))[cc & 1] = v;
  }
  float2 *z = dft_lines(P, a, b, L);
  const float s0 = 1.0f / (float)n;
  const int nk = n / 2 + 1;
  for (int e = threadIdx.x; e < L * nk; e += blockDim.x) {
    const int k = e / L, l = e - k * L, kr = k ? n - k : 0;
    float2 *p = z + l * ls + at(k), *pr = z + l * ls + at(kr);
    const float2 zk = *p, zr = *pr;
    const float2 w = __ldg(P.half + k), wr = __ldg(P.half + kr);
    const float na = __ldg(o.nu + min(c0 + 2 * l, W - 1)), nb = __ldg(o.nu + min(c0 + 2 * l + 1, W - 1));
    const float mk = __ldg(o.mu + k), mr = __ldg(o.mu + kr);
    float2 c = dct_pair(zk, zr, w), cr = dct_pair(zr, zk, wr);
    c.x = mk + na > 0.0f ? c.x / (mk + na) : 0.0f;
    c.y = mk + nb > 0.0f ? c.y / (mk + nb) : 0.0f;
    cr.x = mr + na > 0.0f ? cr.x / (mr + na) : 0.0f;
    cr.y = mr + nb > 0.0f ? cr.y / (mr + nb) : 0.0f;
    const float2 zero = make_float2(0.0f, 0.0f);
    *p = idct_pair(c, k ? cr : zero, w, s0);
    if (k) *pr = idct_pair(cr, c, wr, s0);
  }
  float2 *y = z == a ? b : a;
  z = dft_lines(P, z, y, L);
#pragma unroll 4
  for (int e = threadIdx.x; e < n * C; e += blockDim.x) {
    const int i = e / C, cc = e - i * C;
    if (c0 + cc < W)  // swapped: the first line of a pair is in the imaginary part
      o.t[(size_t)i * W + c0 + cc] = reinterpret_cast<const float *>(z + (cc >> 1) * ls + at(place(i, n)))[1 - (cc & 1)];
  }
}

__device__ __forceinline__ void columns(const SpecObj &o, int blk, int L) {
  if (L == 4) columns_of<4>(o, blk);
  else if (L == 2) columns_of<2>(o, blk);
  else columns_of<1>(o, blk);
}

// Rows back: two rows per block, into the FP64 iterate (set, or added to; the last one's partial sums give the
// mean), or handed to store(p, value).
enum : int { DST_SET = 0, DST_ADD = 1, DST_ADD_LAST = 2, DST_CALL = 3 };
template <int DST, class F = NoCall>
__device__ __forceinline__ void rows_back(const SpecObj &o, int blk, F store = F()) {
  constexpr bool FIRST = DST == DST_SET, LAST = DST == DST_ADD_LAST;
  const FftPlan &P = o.row;
  const int n = o.W, i0 = 2 * blk;
  const bool two = i0 + 1 < o.H;
  float2 *a = spec_smem, *b = a + line_stride(P.m);
  const float *ta = o.t + (size_t)i0 * n, *tb = ta + (two ? n : 0);
  const float s0 = 1.0f / (float)n;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const float2 c = make_float2(ta[k], two ? tb[k] : 0.0f);
    const float2 cr = k ? make_float2(ta[n - k], two ? tb[n - k] : 0.0f) : make_float2(0.0f, 0.0f);
    a[at(k)] = idct_pair(c, cr, __ldg(P.half + k), s0);
  }
  const float2 *z = dft_lines(P, a, b, 1);
  double *xa = o.x + (size_t)i0 * n, *xb = xa + n;
  double sum = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const float2 v = z[at(place(j, n))];
    if (DST == DST_CALL) {
      const size_t p = (size_t)i0 * n + j;
      store(p, v.y);
      if (two) store(p + n, v.x);
      continue;
    }
    const double ua = FIRST ? (double)v.y : xa[j] + (double)v.y;
    xa[j] = ua;
    if (LAST) sum += ua;
    if (two) {
      const double ub = FIRST ? (double)v.x : xb[j] + (double)v.x;
      xb[j] = ub;
      if (LAST) sum += ub;
    }
  }
  if (LAST) {
    __shared__ double sh[32];
    sum = block_sum(sum, sh);
    if (threadIdx.x == 0) o.part[o.row_blocks + blk] = sum;
  }
}

}  // namespace spec
}  // namespace irtps
