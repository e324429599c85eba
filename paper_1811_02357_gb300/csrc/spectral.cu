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
// eigenvalues - and back, rows back.  One such solve leaves a relative residual that grows with
// the square of the longer side and with the smoothness of the slopes (the rounding of x in FP32
// against the second differences in b): 1e-3 with noise, 0.1 without for 2048 points.  The FP64
// residual r = b - A x, solved for the same way and added to the FP64 iterate, lowers it step by
// step (2048 x 2048, noise-free slopes of the lowest modes: 0.1, 3e-8, 4e-10, 9e-11; the last
// is the rounding of the FP64 residual), while GB300's FP64 pipe (2 multiply-adds per clock and SM)
// does only the 14 operations of the residual per pixel.  One or two steps are launched ahead; the last
// pass measures the residual and takes more where it is still above the tolerance (finish).
// The slopes in b are quotients of FP32 numbers: FP32 quotient plus FP32 remainder
// quotient (48 bits) instead of FP64 divisions.
//
// The same three passes in FP32 precondition the weighted (IRLS) solves (poisson.cu).
//
// Whole calls against the dense FP64 transforms (to 1024 on a side) and the multigrid PCG (beyond) that it replaced:
// 512 x 512 689 -> 135 us, 637 x 899 1864 -> 285 us, classic PS and surface at 2048 x 2048 26.7 -> 1.18 ms; noise-free
// slopes at 4096 x 4096, with a third refinement, 50.7 -> 3.5 ms.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdint>
#include <cstring>
#include <vector>

#include "irtps_internal.h"
#include "spectral.cuh"
#include "team.cuh"

namespace irtps {

namespace {

using namespace spec;

constexpr int kMaxSmem = 227 * 1024;

enum : int { SP_ROWS_FIRST = 0, SP_ROWS = 1, SP_COLS = 2, SP_BACK_FIRST = 3, SP_BACK = 4, SP_BACK_LAST = 5 };
template <int PASS>
__device__ __forceinline__ void spec_pass(const SpecObj &o, int blk) {
  if (PASS == SP_ROWS_FIRST) rows_forward<SRC_RHS>(o, blk);
  if (PASS == SP_ROWS) rows_forward<SRC_RESIDUAL>(o, blk);
  if (PASS == SP_COLS) columns(o, blk, o.col_lines);
  if (PASS == SP_BACK_FIRST) rows_back<DST_SET>(o, blk);
  if (PASS == SP_BACK) rows_back<DST_ADD>(o, blk);
  if (PASS == SP_BACK_LAST) rows_back<DST_ADD_LAST>(o, blk);
}
constexpr int kColThreads = 512;  // threads of a column block
template <int PASS>
__global__ void __launch_bounds__(PASS == SP_COLS ? kColThreads : kSpecThreads) k_spec(const __grid_constant__ SpecObj o) {
  spec_pass<PASS>(o, blockIdx.x);
}

// One more refinement step by the blocks of a cooperative launch (dynamic shared memory: one line pair).
__device__ __noinline__ void refine_again(const SpecObj &o, Team t) {
  CGCtl *ctl = o.ctl;
  for (int i = t.bid; i < o.row_blocks; i += t.nblk) {
    rows_forward<SRC_RESIDUAL>(o, i);
    __syncthreads();
  }
  grid_barrier(&ctl->count, &ctl->gen, &ctl->err, t.nblk);
  for (int i = t.bid; i < (o.W + 1) / 2; i += t.nblk) {
    columns(o, i, 1);
    __syncthreads();
  }
  grid_barrier(&ctl->count, &ctl->gen, &ctl->err, t.nblk);
  for (int i = t.bid; i < o.row_blocks; i += t.nblk) {
    rows_back<DST_ADD_LAST>(o, i);
    __syncthreads();
  }
  grid_barrier(&ctl->count, &ctl->gen, &ctl->err, t.nblk);
}

// Sum of n partials by one warp, valid in its first lane.  (A warp's FP64 instruction holds the SM's FP64 pipe for 16
// cycles: sums by one warp a block instead of all eight take 4 us off the last pass at 512 x 512.)
__device__ __forceinline__ double warp_total(const double *part, int n) {
  double v = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < n; i += 32) v += __ldcg(part + i);
  for (int k = 16; k > 0; k >>= 1) v += __shfl_down_sync(0xffffffffu, v, k);
  return v;
}

// The end of a solve (cooperative; 18 us at 512 x 512 and 25 at 637 x 899, where a plain launch whose last block
// checks took 18 and 23): the FP64 residual against the tolerance, and the FP32 surface of mean zero (the
// (0, 0) term was dropped, but FP32 transforms leave a mean of their rounding, which no residual sees).  While the
// residual is above the tolerance and a step at least halves it, further refinement steps follow (a step lowers it
// by orders of magnitude or has met the rounding of the FP64 residual).  Every block sums the same partials in the
// same order and so takes the same decisions.
constexpr int kMoreSteps = 8;
__device__ __forceinline__ void finish(const SpecObj &o, Team t) {
  __shared__ double s_sq[kSpecThreads], s_bb, s_mean, s_rel;
  const int P = o.H * o.W, warp = threadIdx.x >> 5;
  CGCtl *ctl = o.ctl;
  double *part = o.part + 2 * o.row_blocks;
  double rel, last = INFINITY;
  for (int more = 0;; ++more) {
    if (warp < 2) {
      const double v = warp_total(o.part + warp * o.row_blocks, o.row_blocks);
      if (threadIdx.x == 0) s_bb = v;
      if (threadIdx.x == 32) s_mean = v * o.inv_p;
    }
    __syncthreads();
    const double mean = s_mean;
    double rr = 0.0;
    for (int p = t.bid * blockDim.x + threadIdx.x; p < P; p += t.nblk * blockDim.x) {
      const int i = p / o.W;
      const double r = residual_at(o, i, p - i * o.W);
      rr = fma(r, r, rr);
      o.depth[p] = (float)(o.x[p] - mean);
    }
    s_sq[threadIdx.x] = rr;
    __syncthreads();
    if (warp == 0) {
      for (int k = 1; k < kSpecThreads / 32; ++k) rr += s_sq[threadIdx.x + 32 * k];
      for (int k = 16; k > 0; k >>= 1) rr += __shfl_down_sync(0xffffffffu, rr, k);
      if (threadIdx.x == 0) part[t.bid] = rr;
    }
    grid_barrier(&ctl->count, &ctl->gen, &ctl->err, t.nblk);
    if (warp == 0) {
      rr = warp_total(part, t.nblk);
      if (threadIdx.x == 0) s_rel = s_bb > 0.0 ? sqrt(rr / s_bb) : 0.0;
    }
    __syncthreads();
    rel = s_rel;
    if (!(rel > o.tol) || !(rel < 0.5 * last) || more == kMoreSteps || *(volatile int *)&ctl->err) break;
    last = rel;
    refine_again(o, t);
  }
  if (t.bid == 0 && threadIdx.x == 0) {
    ctl->rel = rel;
    ctl->iters = 1;
    o.acc->iters += 1;
    o.acc->last_iters = 1;
    o.acc->rel_last = rel;
    if (*(volatile int *)&ctl->err) o.acc->err = 1;
    if (!isfinite(s_bb) || !isfinite(rel) || rel > o.tol) o.acc->bad = 1;
  }
}

// The last pass, cooperative (registers for the four blocks an SM that the residual's loads want).
__global__ void __launch_bounds__(kSpecThreads, 4) k_spec_finish(const __grid_constant__ SpecObj o) {
  finish(o, Team{(int)blockIdx.x, (int)gridDim.x});
}

// Batched: object i owns the blocks [blk[g] of i, blk[g] of i + 1) of a launch, g = 0 rows, 1 columns, 2 last pass.
__device__ __forceinline__ int object_of(const SpecObj *__restrict__ objs, int n, int g) {
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
  return s_o;
}
// step: -1 for the first solve, then the refinement steps; an object takes as many as it does alone.
template <int PASS>
__global__ void __launch_bounds__(PASS == SP_COLS ? kColThreads : kSpecThreads)
    k_spec_b(const SpecObj *__restrict__ objs, int n, int step) {
  constexpr int g = PASS == SP_COLS ? 1 : 0;
  const SpecObj &o = objs[object_of(objs, n, g)];
  if (step >= o.refine) return;
  if (PASS == SP_BACK && step + 1 == o.refine)
    spec_pass<SP_BACK_LAST>(o, (int)blockIdx.x - o.blk[g]);
  else
    spec_pass<PASS>(o, (int)blockIdx.x - o.blk[g]);
}
__global__ void __launch_bounds__(kSpecThreads, 4) k_spec_finish_b(const SpecObj *__restrict__ objs, int n) {
  const SpecObj &o = objs[object_of(objs, n, 2)];
  finish(o, Team{(int)blockIdx.x - o.blk[2], o.check_blocks});
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

size_t line_smem(const FftPlan &row, const FftPlan &col) {
  return sizeof(float2) * 2 * (size_t)std::max(line_stride(row.m), line_stride(col.m));
}
// Co-resident blocks of the last pass (also raises its shared-memory limit); 0 on an error.
template <typename F>
int finish_blocks_most(F *k, size_t smem, int sms) {
  int per = 0;
  if (allow_max_smem((const void *)k) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kSpecThreads, smem) != cudaSuccess)
    return 0;
  return std::min(per, 4) * (sms > 0 ? sms : 1);
}

// Refinement steps launched ahead of the last pass, which adds those that are missing: one up to 128 on a side (residual 2e-10 or less at the default tolerance of 1e-9), two beyond
// (4e-10 or less to 2048; from there on smooth slopes take a third), four for tolerances near the floor of FP64.
int refinements(const Ctx &c) { return c.opt.cg_tol < 1e-10 ? 4 : (std::max(c.H, c.W) <= 128 ? 1 : 2); }

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
  // column lines per block: the widest loads (8 columns, a 32-byte sector) that still give every SM a block
  o.col_lines = 1;
  for (int L : {4, 2})
    if (o.col_lines == 1 && (W + 2 * L - 1) / (2 * L) >= (c.sms > 0 ? c.sms : 1) &&
        sizeof(float2) * 2 * L * line_stride(col.p.m) <= (size_t)kMaxSmem)
      o.col_lines = L;
  o.col_blocks = (W + 2 * o.col_lines - 1) / (2 * o.col_lines);
  const size_t pb = sizeof(float2) * pool.size(), lb = (sizeof(float) * lam.size() + 15) / 16 * 16;
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)k_spec<SP_ROWS_FIRST>, (const void *)k_spec<SP_ROWS>, (const void *)k_spec<SP_COLS>,
                        (const void *)k_spec<SP_BACK_FIRST>, (const void *)k_spec<SP_BACK>,
                        (const void *)k_spec<SP_BACK_LAST>})
    if ((e = allow_max_smem(k)) != cudaSuccess) return e;
  if (c.opt.irls_iters > 0 && (e = cg_allow_smem()) != cudaSuccess) return e;
  const int most = finish_blocks_most(k_spec_finish, line_smem(row.p, col.p), c.sms);
  if (most < 1) return cudaErrorInvalidConfiguration;
  o.check_blocks = std::min((H * W + kSpecThreads - 1) / kSpecThreads, most);
  const size_t qb = sizeof(double) * (2 * o.row_blocks + o.check_blocks);
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
  o.refine = refinements(c);
  o.nrm = c.nrm;
  o.depth = c.depth;
  o.x = c.cg_x;
  o.b = c.cg_b;
  o.ctl = (CGCtl *)c.cg_ctl;
  o.acc = acc;
  return o;
}

size_t spec_line_smem(const Ctx &c) { return line_smem(c.sp.row, c.sp.col); }

// Iterations after which a weighted solve on nblk blocks has taken as long with the spectral preconditioner as with the
// multigrid one from the start, from the measured times of an iteration (us):
//  - spectral: 12 for the barriers, and per line pair and block 2 + m / 100 a transform of m points (rows
//    twice, columns both ways): 27 at 128 x 128, 49 at 375 x 421, 90 at 1024 x 1024, 332 at 2048 x 2048, 45 at 24 x 24 and
//    150 at 2 x 1000, where the few blocks have many short lines each;
//  - multigrid: 60 up to 4096 points (one block), else 90 + 11 for every point a thread: 100 at 128 x 128, 240 at
//    1024 x 1024, 600 at 2048 x 2048; its iterations grow like 10 P^0.2 (50 at 64 x 64, 110 at 375 x 421, 210 at 2048 x
//    2048 with 5 % outliers and a threshold of 1e-3).
// So the limit is 54 at 24 x 24, 110 at 64 x 64, about 300 from 128 x 128 to 512 x 512, 390 at 2048 x 2048; below 24
// (17 at 2 x 1000) multigrid does the whole solve, which on such strips takes 20 iterations whatever the weights.
// Two reweightings with 5 % outliers at thresholds of 0.05, 1e-3 and 1e-4, ms: multigrid alone 17.1, 26.6, 30.1 at 256 x
// 200 and 27.7, 41.1, 47.0 at 375 x 421; spectral alone 5.3, 28.4, 72.7 and 9.0, 47.8, 121; with the limit 5.4, 21.4,
// 26.7 and 9.0, 29.6, 39.4.
int spectral_limit(const Ctx &c, int nblk) {
  const SpecObj &o = c.sp;
  auto rounds = [&](int lines) { return (double)((lines + nblk - 1) / nblk); };
  const double P = (double)c.H * c.W;
  const double spectral = 12.0 + 2.0 * rounds(o.row_blocks) * (2.0 + 0.01 * o.row.m) +
                          rounds((c.W + 1) / 2) * (2.0 + 0.02 * o.col.m);
  const double multigrid = P <= 4096.0 ? 60.0 : 90.0 + 11.0 * P / (256.0 * nblk);
  const int limit = (int)(10.0 * std::pow(P, 0.2) * multigrid / spectral);
  return limit < 24 ? 0 : limit;
}

cudaError_t launch_spectral(Ctx &c) {
  const SpecObj o = spec_object(c, &c.dstats->cg);
  const size_t rs = row_smem(o), cs = col_smem(o);
  cudaStream_t s = c.stream;
  k_spec<SP_ROWS_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  k_spec<SP_COLS><<<o.col_blocks, kColThreads, cs, s>>>(o);
  k_spec<SP_BACK_FIRST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  const int n = o.refine;
  for (int i = 0; i < n; ++i) {
    k_spec<SP_ROWS><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
    k_spec<SP_COLS><<<o.col_blocks, kColThreads, cs, s>>>(o);
    if (i + 1 < n)
      k_spec<SP_BACK><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
    else
      k_spec<SP_BACK_LAST><<<o.row_blocks, kSpecThreads, rs, s>>>(o);
  }
  void *args[] = {(void *)&o};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_spec_finish, dim3(o.check_blocks),
                                                    dim3(kSpecThreads), args, line_smem(o.row, o.col), s);
  if (e != cudaSuccess) return e;
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
    sb.blocks[0] += o.row_blocks;
    sb.blocks[1] += o.col_blocks;
    sb.row_smem = std::max(sb.row_smem, row_smem(o));
    sb.col_smem = std::max(sb.col_smem, col_smem(o));
    sb.line_smem = std::max(sb.line_smem, line_smem(o.row, o.col));
    sb.refine = std::max(sb.refine, o.refine);
    t.push_back(o);
    ++sb.n;
  }
  if (sb.n == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)k_spec_b<SP_ROWS_FIRST>, (const void *)k_spec_b<SP_ROWS>,
                        (const void *)k_spec_b<SP_COLS>, (const void *)k_spec_b<SP_BACK_FIRST>,
                        (const void *)k_spec_b<SP_BACK>})
    if ((e = allow_max_smem(k)) != cudaSuccess) return e;
  // last pass: the co-resident blocks shared in proportion to the pixel counts, at least one an object
  const int most = finish_blocks_most(k_spec_finish_b, sb.line_smem, objs[0]->sms);
  if (most < sb.n) return cudaErrorInvalidConfiguration;
  double pixels = 0.0;
  for (const SpecObj &o : t) pixels += (double)o.H * o.W;
  for (SpecObj &o : t) {
    const int share = 1 + (int)((double)(most - sb.n) * ((double)o.H * o.W) / pixels);
    o.check_blocks = std::min(o.check_blocks, share);
    o.blk[2] = sb.blocks[2];
    sb.blocks[2] += o.check_blocks;
  }
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
  k_spec_b<SP_ROWS_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n, -1);
  k_spec_b<SP_COLS><<<sb.blocks[1], kColThreads, cs, s>>>(t, n, -1);
  k_spec_b<SP_BACK_FIRST><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n, -1);
  for (int i = 0; i < sb.refine; ++i) {
    k_spec_b<SP_ROWS><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n, i);
    k_spec_b<SP_COLS><<<sb.blocks[1], kColThreads, cs, s>>>(t, n, i);
    k_spec_b<SP_BACK><<<sb.blocks[0], kSpecThreads, rs, s>>>(t, n, i);
  }
  void *args[] = {(void *)&t, (void *)&n};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_spec_finish_b, dim3(sb.blocks[2]),
                                                    dim3(kSpecThreads), args, sb.line_smem, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace irtps
