// Direct depth solve by the cosine transform (option precond = 2).  With unit
// edge weights the normal equations of the integration are A x = b with A the
// graph Laplacian of the H x W grid (Neumann boundary), the sum of the path
// Laplacians of the rows and of the columns.  The DCT-II vectors cos(pi k (2i+1) / 2n)
// diagonalise a path Laplacian of n nodes, eigenvalue 4 sin^2(pi k / 2n).  So
//
//     x = DCT^-1 [ DCT(b) ./ (mu_l + nu_k) ],   the (0, 0) term dropped,
//
// is the mean-zero least-squares surface.
//
// Fast transforms in FP32, iterative refinement in FP64.  A transform of n points is a
// complex FFT of n points over two lines at once (one in the real, one in the imaginary
// part; even samples ascending, then odd ones descending), held in shared memory, so a
// solve is three passes over the grid: rows forward, columns forward - divided by the
// eigenvalues - and back, rows back.  One such solve has a relative residual of about
// 1e-3 at 2048 x 2048 (the rounding of x in FP32 against the second differences in b);
// the FP64 residual r = b - A x, solved for the same way and added to the FP64 iterate,
// lowers it by 1e-4 or more a step (a rough r needs little of x's range), so three solves
// end below 1e-10, where FP64 transforms end too, while GB300's FP64 pipe (2
// multiply-adds per clock and SM) does only the 13 operations of the residual per pixel.
// The slopes in b are quotients of FP32 numbers: FP32 quotient plus FP32 remainder
// quotient (48 bits) instead of FP64 divisions.
//
// Against the dense FP64 transforms this replaces up to 1024 on a side and the multigrid PCG
// beyond: see launch_spectral.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdint>
#include <cstring>
#include <vector>

#include "irtps_internal.h"

namespace irtps {

namespace {

constexpr int kSpecThreads = 256;
constexpr int kMaxSmem = 227 * 1024;

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
    if (ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(tw + r * k * step));
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

// n.x / nz as a FP32 quotient plus the quotient of its exact remainder (48 bits), in FP64.
__device__ __forceinline__ double quotient(float a, float b) {
  const float q = __fdiv_rn(a, b);
  return (double)q + (double)__fdividef(fmaf(-q, b, a), b);
}
__device__ __forceinline__ double slope_p(const float4 &n, float nz_min) { return -quotient(n.x, fmaxf(n.z, nz_min)); }
__device__ __forceinline__ double slope_q(const float4 &n, float nz_min) { return -quotient(n.y, fmaxf(n.z, nz_min)); }

// Right-hand side b = D^T g of pixel (i, j): trapezoidal edge targets h (s_a + s_b) / 2.
__device__ __forceinline__ double rhs_at(const SpecObj &o, int i, int j) {
  const float4 *n = o.nrm + (size_t)i * o.W + j;
  const bool l = j > 0, r = j < o.W - 1, u = i > 0, d = i < o.H - 1;
  double v = 0.0;
  if (l) v += slope_p(__ldg(n - 1), o.nz_min);
  if (r) v -= slope_p(__ldg(n + 1), o.nz_min);
  if (u) v += slope_q(__ldg(n - o.W), o.nz_min);
  if (d) v -= slope_q(__ldg(n + o.W), o.nz_min);
  if (l != r || u != d) {  // on a border the pixel's own slope does not cancel
    const float4 c = __ldg(n);
    if (l != r) v += l ? slope_p(c, o.nz_min) : -slope_p(c, o.nz_min);
    if (u != d) v += u ? slope_q(c, o.nz_min) : -slope_q(c, o.nz_min);
  }
  return 0.5 * o.h * v;
}

// r = b - A x of pixel (i, j) in FP64.
__device__ __forceinline__ double residual_at(const SpecObj &o, int i, int j) {
  const size_t p = (size_t)i * o.W + j;
  const double *x = o.x + p;
  double s = 0.0;
  int deg = 0;
  if (j > 0) { s += x[-1]; ++deg; }
  if (j < o.W - 1) { s += x[1]; ++deg; }
  if (i > 0) { s += x[-o.W]; ++deg; }
  if (i < o.H - 1) { s += x[o.W]; ++deg; }
  return o.b[p] - fma((double)deg, x[0], -s);
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

// Rows forward: two rows per block, of b (from the normals, kept; |b|^2 partials) or of the residual.
template <bool FIRST>
__device__ __forceinline__ void rows_forward(const SpecObj &o, int blk) {
  const FftPlan &P = o.row;
  const int n = o.W, i0 = 2 * blk;
  const bool two = i0 + 1 < o.H;
  float2 *a = spec_smem, *b = a + line_stride(P.m);
  double bb = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double u, v = 0.0;
    if (FIRST) {
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
  if (FIRST) {
    __shared__ double sh[32];
    bb = block_sum(bb, sh);
    if (threadIdx.x == 0) {
      o.part[blk] = bb;
      if (blk == 0) o.ctl->count = 0u;  // arrivals of the check pass
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
__device__ __forceinline__ void columns(const SpecObj &o, int blk) {
  const FftPlan &P = o.col;
  const int n = o.H, W = o.W, L = o.col_lines, C = 2 * L, c0 = blk * C;
  const int ls = line_stride(P.m);
  float2 *a = spec_smem, *b = a + L * ls;
  for (int e = threadIdx.x; e < n * C; e += blockDim.x) {
    const int i = e / C, cc = e - i * C;  // C is 2, 4 or 8
    const float v = c0 + cc < W ? o.t[(size_t)i * W + c0 + cc] : 0.0f;
    reinterpret_cast<float *>(a + (cc >> 1) * ls + at(place(i, n)))[cc & 1] = v;
  }
  float2 *z = dft_lines(P, a, b, L);
  const float s0 = 1.0f / (float)n;
  const int nk = n / 2 + 1;
  for (int e = threadIdx.x; e < L * nk; e += blockDim.x) {
    const int l = e / nk, k = e - l * nk, kr = k ? n - k : 0;
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
  for (int e = threadIdx.x; e < n * C; e += blockDim.x) {
    const int i = e / C, cc = e - i * C;
    if (c0 + cc < W)  // swapped: the first line of a pair is in the imaginary part
      o.t[(size_t)i * W + c0 + cc] = reinterpret_cast<const float *>(z + (cc >> 1) * ls + at(place(i, n)))[1 - (cc & 1)];
  }
}

// Rows back: two rows per block, into the FP64 iterate (set, or added to); the last one's partial sums give the mean.
template <bool FIRST, bool LAST>
__device__ __forceinline__ void rows_back(const SpecObj &o, int blk) {
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

// The FP64 residual against the tolerance, and the FP32 surface of mean zero (the (0, 0) term was dropped, but
// FP32 transforms leave a mean of their rounding, which no residual sees).
__device__ __forceinline__ void check(const SpecObj &o, int blk, int nblk) {
  __shared__ double sh[32];
  __shared__ double s_mean;
  __shared__ bool last;
  const int P = o.H * o.W;
  double rr = 0.0;
  for (int i = threadIdx.x; i < o.row_blocks; i += blockDim.x) rr += __ldcg(o.part + o.row_blocks + i);
  rr = block_sum(rr, sh);
  if (threadIdx.x == 0) s_mean = rr / (double)P;
  __syncthreads();
  const double mean = s_mean;
  rr = 0.0;
  for (int p = blk * blockDim.x + threadIdx.x; p < P; p += nblk * blockDim.x) {
    const int i = p / o.W;
    const double r = residual_at(o, i, p - i * o.W);
    rr += r * r;
    o.depth[p] = (float)(o.x[p] - mean);
  }
  rr = block_sum(rr, sh);
  double *part = o.part + 2 * o.row_blocks;
  if (threadIdx.x == 0) {
    part[blk] = rr;
    __threadfence();
    last = atomicAdd(&o.ctl->count, 1u) == (unsigned)nblk - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double bb = 0.0;
  rr = 0.0;
  for (int i = threadIdx.x; i < o.row_blocks; i += blockDim.x) bb += __ldcg(o.part + i);
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) rr += __ldcg(part + i);
  bb = block_sum(bb, sh);
  __syncthreads();
  rr = block_sum(rr, sh);
  if (threadIdx.x == 0) {
    CGCtl *ctl = o.ctl;
    ctl->count = 0u;
    ctl->bnorm = sqrt(bb);
    ctl->rel = bb > 0.0 ? sqrt(rr) / sqrt(bb) : 0.0;
    ctl->iters = 1;
    o.acc->iters += 1;
    o.acc->last_iters = 1;
    o.acc->rel_last = ctl->rel;
    if (!isfinite(bb) || !isfinite(ctl->rel) || ctl->rel > o.tol) o.acc->bad = 1;
  }
}

enum : int { SP_ROWS_FIRST = 0, SP_ROWS = 1, SP_COLS = 2, SP_BACK_FIRST = 3, SP_BACK = 4, SP_BACK_LAST = 5, SP_CHECK = 6 };
template <int PASS>
__device__ __forceinline__ void spec_pass(const SpecObj &o, int blk) {
  if (PASS == SP_ROWS_FIRST) rows_forward<true>(o, blk);
  if (PASS == SP_ROWS) rows_forward<false>(o, blk);
  if (PASS == SP_COLS) columns(o, blk);
  if (PASS == SP_BACK_FIRST) rows_back<true, false>(o, blk);
  if (PASS == SP_BACK) rows_back<false, false>(o, blk);
  if (PASS == SP_BACK_LAST) rows_back<false, true>(o, blk);
  if (PASS == SP_CHECK) check(o, blk, o.check_blocks);
}
template <int PASS>
__global__ void __launch_bounds__(kSpecThreads) k_spec(const __grid_constant__ SpecObj o) {
  spec_pass<PASS>(o, blockIdx.x);
}

// Batched: object i owns the blocks [blk[g] of i, blk[g] of i + 1) of a launch, g = 0 rows, 1 columns, 2 check.
template <int PASS>
__global__ void __launch_bounds__(kSpecThreads) k_spec_b(const SpecObj *__restrict__ objs, int n) {
  constexpr int g = PASS == SP_COLS ? 1 : (PASS == SP_CHECK ? 2 : 0);
  __shared__ int s_o;
  if (threadIdx.x == 0) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (objs[mid].blk[g] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    s_o = lo;
  }
  __syncthreads();
  const SpecObj &o = objs[s_o];
  spec_pass<PASS>(o, (int)blockIdx.x - o.blk[g]);
}

// ---- host: plans ----

using cd = std::complex<double>;
const double kPi = 3.14159265358979323846;

// Radices of a 7-smooth length (8 and 4 first), empty when it is not.
std::vector<int> radices(int m) {
  std::vector<int> r;
  for (int p : {8, 4, 2, 7, 5, 3})
    while (m % p == 0 && m > 1) {
      r.push_back(p);
      m /= p;
    }
  if (m != 1 || r.size() > (size_t)kMaxFftStages) return {};
  return r;
}

// Recursive DFT on the host (filters of Bluestein plans); w: the roots of unity of the whole length, m n of them.
void host_fft(cd *x, int n, const std::vector<cd> &w) {
  if (n == 1) return;
  int p = 2;
  while (n % p) ++p;
  const int m = n / p, stride = (int)w.size() / n;
  std::vector<cd> y(n);
  for (int r = 0; r < p; ++r) {
    for (int i = 0; i < m; ++i) y[(size_t)r * m + i] = x[i * p + r];
    host_fft(y.data() + (size_t)r * m, m, w);
  }
  for (int k = 0; k < n; ++k) {
    cd v = 0.0;
    for (int r = 0; r < p; ++r) v += w[(size_t)((long long)r * k % n) * stride] * y[(size_t)r * m + k % m];
    x[k] = v;
  }
}

// The tables of a plan, appended to `pool` (offsets in float2 for its device pointers).
struct PlanTables {
  FftPlan p{};
  size_t tw = 0, half = 0, chirp = 0, filter = 0;
  bool blue = false;
};
PlanTables make_plan(int n, std::vector<float2> &pool) {
  PlanTables t;
  t.p.n = n;
  std::vector<int> r = radices(n);
  int m = n;
  if (r.empty()) {  // Bluestein: the cheapest smooth length that holds the convolution
    t.blue = true;
    double best = 1e300;
    for (int c = 2 * n - 1; c <= 4 * n; ++c) {
      const std::vector<int> q = radices(c);
      if (q.empty()) continue;
      double cost = 0.0;
      for (int f : q) cost += (f == 8 ? 1.3 : f == 4 ? 1.0 : f == 2 ? 0.8 : f == 3 ? 1.2 : f == 5 ? 1.5 : 2.0);
      if (cost * c < best) {
        best = cost * c;
        m = c;
        r = q;
      }
    }
  }
  t.p.m = m;
  t.p.stages = (int)r.size();
  for (size_t i = 0; i < r.size(); ++i) t.p.radix[i] = r[i];
  auto put = [&](cd v) { pool.push_back(make_float2((float)v.real(), (float)v.imag())); };
  t.tw = pool.size();
  for (int i = 0; i < m; ++i) put(std::polar(1.0, -2.0 * kPi * i / m));
  t.half = pool.size();
  for (int k = 0; k < n; ++k) put(std::polar(1.0, -kPi * k / (2.0 * n)));
  if (t.blue) {
    std::vector<cd> c(n), f(m, cd(0.0));
    for (int i = 0; i < n; ++i) c[i] = std::polar(1.0, -kPi * (double)((long long)i * i % (2LL * n)) / n);
    for (int i = 0; i < n; ++i) f[i] = std::conj(c[i]);
    for (int i = 1; i < n; ++i) f[m - i] = std::conj(c[i]);
    std::vector<cd> w(m);
    for (int i = 0; i < m; ++i) w[i] = std::polar(1.0, -2.0 * kPi * i / m);
    host_fft(f.data(), m, w);
    t.chirp = pool.size();
    for (int i = 0; i < n; ++i) put(c[i]);
    t.filter = pool.size();
    for (int i = 0; i < m; ++i) put(f[i] / (double)m);
  }
  return t;
}

size_t row_smem(const SpecObj &o) { return sizeof(float2) * 2 * line_stride(o.row.m); }
size_t col_smem(const SpecObj &o) { return sizeof(float2) * 2 * o.col_lines * line_stride(o.col.m); }

// Solves after which the refinement ends: three pass the default tolerance (1e-9) with two orders of margin
// on every grid up to 4096 on a side; tighter tolerances get two more, down to the floor of FP64.
int refinements(double tol) { return tol >= 1e-10 ? 2 : 4; }

template <typename F>
cudaError_t allow_smem(F *k, size_t bytes) {
  return bytes > 48 * 1024 ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes)
                           : cudaSuccess;
}

}  // namespace

bool spectral_fits(int H, int W) { return H <= kSpectralMaxSide && W <= kSpectralMaxSide; }

cudaError_t spectral_setup(Ctx &c) {
  const int H = c.H, W = c.W;
  SpecObj &o = c.sp;
  std::vector<float2> pool;
  const PlanTables row = make_plan(W, pool), col = H == W ? row : make_plan(H, pool);
  std::vector<float> lam(H + W);
  for (int k = 0; k < H; ++k) lam[k] = (float)(4.0 * std::pow(std::sin(kPi * k / (2.0 * H)), 2));
  for (int k = 0; k < W; ++k) lam[H + k] = (float)(4.0 * std::pow(std::sin(kPi * k / (2.0 * W)), 2));
  o.H = H;
  o.W = W;
  o.row_blocks = (H + 1) / 2;
  o.check_blocks = std::min((H * W + kSpecThreads - 1) / kSpecThreads, 4 * (c.sms > 0 ? c.sms : 1));
  // column lines per block: the widest loads (8 columns, a 32-byte sector) that still give every SM a block
  o.col_lines = 1;
  for (int L : {4, 2})
    if (o.col_lines == 1 && (W + 2 * L - 1) / (2 * L) >= (c.sms > 0 ? c.sms : 1) &&
        sizeof(float2) * 2 * L * line_stride(col.p.m) <= (size_t)kMaxSmem)
      o.col_lines = L;
  o.col_blocks = (W + 2 * o.col_lines - 1) / (2 * o.col_lines);
  const size_t pb = sizeof(float2) * pool.size(), lb = (sizeof(float) * lam.size() + 15) / 16 * 16;
  const size_t qb = sizeof(double) * (2 * o.row_blocks + o.check_blocks);
  cudaError_t e = cudaMalloc(&c.sp_pool, pb + lb + qb);
  if (e == cudaSuccess) e = cudaMalloc((void **)&c.sp_t, sizeof(float) * (size_t)H * W);
  if (e != cudaSuccess) return e;
  char *d = (char *)c.sp_pool;
  if ((e = cudaMemcpy(d, pool.data(), pb, cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  if ((e = cudaMemcpy(d + pb, lam.data(), sizeof(float) * lam.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
  auto bind = [&](const PlanTables &t) {
    FftPlan p = t.p;
    const float2 *f = (const float2 *)d;
    p.tw = f + t.tw;
    p.half = f + t.half;
    p.chirp = t.blue ? f + t.chirp : nullptr;
    p.filter = t.blue ? f + t.filter : nullptr;
    return p;
  };
  o.row = bind(row);
  o.col = bind(col);
  o.mu = (const float *)(d + pb);
  o.nu = o.mu + H;
  o.part = (double *)(d + pb + lb);
  o.t = c.sp_t;
  return cudaSuccess;
}

// The descriptor of a context's direct solve, its statistics in `acc`.
static SpecObj spec_object(const Ctx &c, CGAcc *acc) {
  SpecObj o = c.sp;
  o.h = 1.0 / (double)c.W;
  o.nz_min = c.opt.nz_min;
  o.tol = c.opt.cg_tol;
  o.nrm = c.nrm;
  o.depth = c.depth;
  o.x = c.cg_x;
  o.b = c.cg_b;
  o.ctl = (CGCtl *)c.cg_ctl;
  o.acc = acc;
  return o;
}

cudaError_t launch_spectral(Ctx &c) {
  const SpecObj o = spec_object(c, &c.dstats->cg);
  const size_t rs = row_smem(o), cs = col_smem(o);
  cudaError_t e;
  if ((e = allow_smem(k_spec<SP_ROWS_FIRST>, rs)) != cudaSuccess || (e = allow_smem(k_spec<SP_ROWS>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec<SP_BACK_FIRST>, rs)) != cudaSuccess || (e = allow_smem(k_spec<SP_BACK>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec<SP_BACK_LAST>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec<SP_COLS>, cs)) != cudaSuccess)
    return e;
  cudaStream_t s = c.stream;
  k_spec<SP_ROWS_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  k_spec<SP_COLS><<<o.col_blocks, kSpecThreads, cs, s>>>(o);
  k_spec<SP_BACK_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  const int n = refinements(o.tol);
  for (int i = 0; i < n; ++i) {
    k_spec<SP_ROWS><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
    k_spec<SP_COLS><<<o.col_blocks, kSpecThreads, cs, s>>>(o);
    if (i + 1 < n)
      k_spec<SP_BACK><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
    else
      k_spec<SP_BACK_LAST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  }
  k_spec<SP_CHECK><<<o.check_blocks, kSpecThreads, 0, s>>>(o);
  c.stats.launches += 4 + 3 * n;
  return cudaGetLastError();
}

// Batched direct solves: one launch per pass over the objects whose unit-weight solves are direct.
cudaError_t spectral_batch_setup(const std::vector<Ctx *> &objs, DevStats *ds, SpectralBatch &sb) {
  sb.n = 0;
  std::vector<SpecObj> t;
  for (size_t i = 0; i < objs.size(); ++i) {
    const Ctx &c = *objs[i];
    if (!direct_solve(c)) continue;
    SpecObj o = spec_object(c, &ds[i].cg);
    o.blk[0] = sb.blocks[0];
    o.blk[1] = sb.blocks[1];
    o.blk[2] = sb.blocks[2];
    sb.blocks[0] += o.row_blocks;
    sb.blocks[1] += o.col_blocks;
    sb.blocks[2] += o.check_blocks;
    sb.row_smem = std::max(sb.row_smem, row_smem(o));
    sb.col_smem = std::max(sb.col_smem, col_smem(o));
    sb.refine = std::max(sb.refine, refinements(o.tol));
    t.push_back(o);
    ++sb.n;
  }
  if (sb.n == 0) return cudaSuccess;
  cudaError_t e = cudaMalloc(&sb.table, sizeof(SpecObj) * sb.n);
  if (e != cudaSuccess) return e;
  return cudaMemcpy(sb.table, t.data(), sizeof(SpecObj) * sb.n, cudaMemcpyHostToDevice);
}

int spectral_batch_kernels(const SpectralBatch &sb) { return sb.n > 0 ? 4 + 3 * sb.refine : 0; }

cudaError_t launch_spectral_batch(cudaStream_t s, const SpectralBatch &sb) {
  if (sb.n == 0) return cudaSuccess;
  const SpecObj *t = (const SpecObj *)sb.table;
  const int n = sb.n;
  const size_t rs = sb.row_smem, cs = sb.col_smem;
  cudaError_t e;
  if ((e = allow_smem(k_spec_b<SP_ROWS_FIRST>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec_b<SP_ROWS>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec_b<SP_BACK_FIRST>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec_b<SP_BACK>, rs)) != cudaSuccess ||
      (e = allow_smem(k_spec_b<SP_BACK_LAST>, rs)) != cudaSuccess || (e = allow_smem(k_spec_b<SP_COLS>, cs)) != cudaSuccess)
    return e;
  k_spec_b<SP_ROWS_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  k_spec_b<SP_COLS><<<sb.blocks[1], kSpecThreads, cs, s>>>(t, n);
  k_spec_b<SP_BACK_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  for (int i = 0; i < sb.refine; ++i) {
    k_spec_b<SP_ROWS><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
    k_spec_b<SP_COLS><<<sb.blocks[1], kSpecThreads, cs, s>>>(t, n);
    if (i + 1 < sb.refine)
      k_spec_b<SP_BACK><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
    else
      k_spec_b<SP_BACK_LAST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  }
  k_spec_b<SP_CHECK><<<sb.blocks[2], kSpecThreads, 0, s>>>(t, n);
  return cudaGetLastError();
}

}  // namespace irtps
