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
// The same three passes in FP32 precondition the weighted (IRLS) solves (poisson.cu).
//
// Whole calls against the dense FP64 transforms (to 1024 on a side) and the multigrid PCG (beyond) that it replaced:
// 512 x 512 684 -> 135 us, 637 x 899 1862 -> 283 us, classic PS and surface at 2048 x 2048 26.4 -> 1.19 ms.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdint>
#include <cstring>
#include <vector>

#include "irtps_internal.h"
#include "spectral.cuh"

namespace irtps {

namespace {

using namespace spec;

constexpr int kMaxSmem = 227 * 1024;

enum : int { SP_ROWS_FIRST = 0, SP_ROWS = 1, SP_COLS = 2, SP_BACK_FIRST = 3, SP_BACK = 4, SP_BACK_LAST = 5, SP_CHECK = 6 };
template <int PASS>
__device__ __forceinline__ void spec_pass(const SpecObj &o, int blk) {
  if (PASS == SP_ROWS_FIRST) rows_forward<SRC_RHS>(o, blk);
  if (PASS == SP_ROWS) rows_forward<SRC_RESIDUAL>(o, blk);
  if (PASS == SP_COLS) columns(o, blk, o.col_lines);
  if (PASS == SP_BACK_FIRST) rows_back<DST_SET>(o, blk);
  if (PASS == SP_BACK) rows_back<DST_ADD>(o, blk);
  if (PASS == SP_BACK_LAST) rows_back<DST_ADD_LAST>(o, blk);
  if (PASS == SP_CHECK) check(o, blk, o.check_blocks);
}
#ifndef IRTPS_COL_THREADS
#define IRTPS_COL_THREADS 512
#endif
constexpr int kColThreads = IRTPS_COL_THREADS;  // threads of a column block
template <int PASS>
__global__ void __launch_bounds__(PASS == SP_COLS ? kColThreads : kSpecThreads) k_spec(const __grid_constant__ SpecObj o) {
  spec_pass<PASS>(o, blockIdx.x);
}

// Batched: object i owns the blocks [blk[g] of i, blk[g] of i + 1) of a launch, g = 0 rows, 1 columns, 2 check.
template <int PASS>
__global__ void __launch_bounds__(PASS == SP_COLS ? kColThreads : kSpecThreads) k_spec_b(const SpecObj *__restrict__ objs, int n) {
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

// Refinement steps after the first solve: two pass the default tolerance (1e-9) with two orders of margin on
// every grid up to 4096 on a side, and one does up to 128 on a side (residual 5e-12 at 64, 3e-11 at 129); tighter
// tolerances get four, down to the floor of FP64.
int refinements(const SpecObj &o) { return o.tol < 1e-10 ? 4 : (std::max(o.H, o.W) <= 128 ? 1 : 2); }

}  // namespace

cudaError_t allow_max_smem(const void *kernel) {
  int dev = 0, most = 0;
  cudaFuncAttributes a;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
}

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
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)k_spec<SP_ROWS_FIRST>, (const void *)k_spec<SP_ROWS>, (const void *)k_spec<SP_COLS>,
                        (const void *)k_spec<SP_BACK_FIRST>, (const void *)k_spec<SP_BACK>,
                        (const void *)k_spec<SP_BACK_LAST>})
    if ((e = allow_max_smem(k)) != cudaSuccess) return e;
  if (c.opt.irls_iters > 0 && (e = cg_allow_smem()) != cudaSuccess) return e;
  e = cudaMalloc(&c.sp_pool, pb + lb + qb);
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
SpecObj spec_object(const Ctx &c, CGAcc *acc) {
  SpecObj o = c.sp;
  o.h = 1.0 / (double)c.W;
  o.inv_p = 1.0 / ((double)c.H * c.W);
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

size_t spec_line_smem(const Ctx &c) {
  return sizeof(float2) * 2 * (size_t)std::max(line_stride(c.sp.row.m), line_stride(c.sp.col.m));
}

cudaError_t launch_spectral(Ctx &c) {
  const SpecObj o = spec_object(c, &c.dstats->cg);
  const size_t rs = row_smem(o), cs = col_smem(o);
  cudaStream_t s = c.stream;
  k_spec<SP_ROWS_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  k_spec<SP_COLS><<<o.col_blocks, kColThreads, cs, s>>>(o);
  k_spec<SP_BACK_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  const int n = refinements(o);
  for (int i = 0; i < n; ++i) {
    k_spec<SP_ROWS><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
    k_spec<SP_COLS><<<o.col_blocks, kColThreads, cs, s>>>(o);
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
    sb.refine = std::max(sb.refine, refinements(o));
    t.push_back(o);
    ++sb.n;
  }
  if (sb.n == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)k_spec_b<SP_ROWS_FIRST>, (const void *)k_spec_b<SP_ROWS>,
                        (const void *)k_spec_b<SP_COLS>, (const void *)k_spec_b<SP_BACK_FIRST>,
                        (const void *)k_spec_b<SP_BACK>, (const void *)k_spec_b<SP_BACK_LAST>})
    if ((e = allow_max_smem(k)) != cudaSuccess) return e;
  e = cudaMalloc(&sb.table, sizeof(SpecObj) * sb.n);
  if (e != cudaSuccess) return e;
  return cudaMemcpy(sb.table, t.data(), sizeof(SpecObj) * sb.n, cudaMemcpyHostToDevice);
}

int spectral_batch_kernels(const SpectralBatch &sb) { return sb.n > 0 ? 4 + 3 * sb.refine : 0; }

cudaError_t launch_spectral_batch(cudaStream_t s, const SpectralBatch &sb) {
  if (sb.n == 0) return cudaSuccess;
  const SpecObj *t = (const SpecObj *)sb.table;
  const int n = sb.n;
  const size_t rs = sb.row_smem, cs = sb.col_smem;
  k_spec_b<SP_ROWS_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  k_spec_b<SP_COLS><<<sb.blocks[1], kColThreads, cs, s>>>(t, n);
  k_spec_b<SP_BACK_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  for (int i = 0; i < sb.refine; ++i) {
    k_spec_b<SP_ROWS><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
    k_spec_b<SP_COLS><<<sb.blocks[1], kColThreads, cs, s>>>(t, n);
    if (i + 1 < sb.refine)
      k_spec_b<SP_BACK><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
    else
      k_spec_b<SP_BACK_LAST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n);
  }
  k_spec_b<SP_CHECK><<<sb.blocks[2], kSpecThreads, 0, s>>>(t, n);
  return cudaGetLastError();
}

}  // namespace irtps
