// Radial F_s: Kaiser-Bessel gridding NUFFT of the non-uniform DFT
//   y_m = N^{-1/2} sum_j v_j exp(-i k_m . (j - n/2)),  k in rad/pixel,
// the operator the paper takes as given for non-Cartesian data (Results,
// "2D synthetic radial sequences").  Steps (forward):
//   1. scale by 1/Phi(t) per axis (deapodisation, t = j - n/2) and 1/n, zero-pad
//      centred into a G x G grid (G = sigma n) with the image-side sign (-1)^g;
//   2. plain FFT along y then x (the k-side sign (-1)^g is applied at read time,
//      so the two signs make the centred DFT of the grid);
//   3. interpolate at kappa = k G / (2 pi) with the separable kernel
//      phi(u) = I0(beta sqrt(1 - (2u/W)^2)) / I0(beta) over the W grid points
//      floor(kappa) - W/2 + 1 ... floor(kappa) + W/2 (periodic), reading the
//      grid through shared-memory tiles (samples binned by first-tap tile).
// The adjoint runs the transposed steps: spread, inverse FFTs, crop with the
// sign and deapodisation (the zero-padding of step 1 and the crop are folded
// into the FFT pass along y).  Spreading is output-driven: each grid cell sums the
// samples whose W x W footprint covers it, found through a per-plan CSR of the
// samples by first-tap cell, so no cell is written twice and no atomics run.
// beta = pi sqrt((W/sigma)^2 (sigma - 1/2)^2 - 0.8) (Beatty et al. 2005);
// Phi(t) = W sinh(z) / (z I0(beta)), z = sqrt(beta^2 - (pi W t / G)^2).
// Grid positions, start taps and weights are computed once per plan in FP64.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mpi_internal.h"
#include "ptx.cuh"

namespace {

// I0(x) by its power series sum_k (x^2/4)^k / (k!)^2 (all terms positive).
__device__ double bessel_i0(double x) {
  const double q = 0.25 * x * x;
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 200; ++k) {
    term *= q / ((double)k * (double)k);
    sum += term;
    if (term < 1e-18 * sum) break;
  }
  return sum;
}

__global__ void k_nufft_setup(const float* __restrict__ traj, int M, int G, int W, double beta,
                              double kscale, int32_t* __restrict__ gstart, float* __restrict__ gw) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;  // (m, axis)
  if (e >= 2 * M) return;
  const double kap = (double)traj[e] * kscale;
  const double fl = floor(kap);
  const long start = (long)fl - W / 2 + 1;  // centred index of the first tap
  long g = (start + G / 2) % G;
  if (g < 0) g += G;
  gstart[e] = (int32_t)g;
  const double i0b = bessel_i0(beta);
  for (int a = 0; a < W; ++a) {
    const double u = kap - (double)(start + a);
    const double r = 1.0 - (2.0 * u / W) * (2.0 * u / W);
    gw[(size_t)e * W + a] = r >= 0.0 ? (float)(bessel_i0(beta * sqrt(r)) / i0b) : 0.f;
  }
}

__global__ void k_nufft_deap(int n, int G, int W, double beta, float* __restrict__ deap) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double t = (double)(j - n / 2);
  const double x = M_PI * W * t / G;
  const double z2 = beta * beta - x * x;
  double phi;
  if (z2 > 0) {
    const double z = sqrt(z2);
    phi = sinh(z) / z;
  } else if (z2 < 0) {
    const double z = sqrt(-z2);
    phi = sin(z) / z;
  } else {
    phi = 1.0;
  }
  phi = W * phi / bessel_i0(beta);
  deap[j] = (float)(1.0 / phi);
}

constexpr int kInterpTile = 32;    // first-tap tile of the shared-memory interpolation
constexpr int kInterpChunk = 256;  // samples per interpolation work item (one per thread)

// Interpolation through shared memory: CTA (item, group of `per` coils) takes
// a chunk of at most kInterpChunk of the samples whose first tap lies in one 32 x 32
// tile (the plan's tile-sorted list).  Each thread loads its sample's first tap
// and weights (before waiting on the kernel that writes the grid) and forms the
// addresses of its share of the grid cells that the chunk reads, (32 + W - 1)^2 from
// the tile's corner (periodic); then, coil by coil, the CTA copies those cells to
// shared memory, the next coil's loads in flight while each thread forms its
// sample's W x W sum there.  The set-up (divisions by the tile width, wraps,
// scattered weights) was most of the kernel when every CTA did one coil:
// 256^2, 12 coils, 64 spokes 26.2 -> 22.4 us.  With few items there are too few such
// CTAs, and started early they share a few SMs: a forward takes, with 1, 2 and 4 coils per
// CTA, 30, 33 and 43 us with 810 (item, coil) pairs (G = 96, W = 8, 30 coils), 28, 30 and
// 33 with 1,020, 34, 33 and 36 with 2,040, 45, 40 and 36 with 2,608, 54, 45 and 42 with
// 5,312.
int interp_coils(const mpi_ctx* ctx, int items, int C) {
  const long pairs = (long)items * C, sms = std::max(ctx->num_sms, 1);
  return pairs < 7 * sms ? 1 : (pairs < 16 * sms ? 2 : 4);
}

template <int W>
__global__ void __launch_bounds__(kInterpChunk) k_nufft_interp_tiled(const float2* __restrict__ grid, int C, int G,
                                                                     int M, const int32_t* __restrict__ gstart,
                                                                     const float* __restrict__ gw, float ksign,
                                                                     const int32_t* __restrict__ items,
                                                                     const int32_t* __restrict__ samples,
                                                                     float2* __restrict__ y, int per) {
  mpi_ptx::pdl_trigger();
  constexpr int TT = kInterpTile + W - 1;
  constexpr int PER = (TT * TT + kInterpChunk - 1) / kInterpChunk;  // cells per thread
  __shared__ float2 tile[TT * TT];
  const int it = blockIdx.x, c0 = blockIdx.y * per, c1 = min(c0 + per, C);
  const int t = items[3 * it], s0 = items[3 * it + 1], cnt = items[3 * it + 2];
  const int tpr = (G + kInterpTile - 1) / kInterpTile;
  const int oy = (t / tpr) * kInterpTile, ox = (t % tpr) * kInterpTile;
  const bool active = (int)threadIdx.x < cnt;
  const int m = samples[s0 + (active ? (int)threadIdx.x : 0)];
  const int sx = gstart[2 * m], sy = gstart[2 * m + 1];
  // weights with the k-side sign (-1)^(gx + gy) folded in: (-1)^b and the sample's own
  // parity along x, (-1)^a along y (G is even, so wrapping keeps the parity)
  const int odd = (sx + sy) & 1;
  float wx[W], wy[W];
#pragma unroll
  for (int a = 0; a < W; ++a) {
    wx[a] = gw[(size_t)(2 * m) * W + a];
    wy[a] = gw[(size_t)(2 * m + 1) * W + a];
    if ((a + odd) & 1) wx[a] = -wx[a];
    if (a & 1) wy[a] = -wy[a];
  }
  int off[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int e = threadIdx.x + kInterpChunk * j, r = e / TT, q = e - r * TT;
    off[j] = e < TT * TT ? ((oy + r) % G) * G + (ox + q) % G : 0;
  }
  mpi_ptx::pdl_wait();
  const float2* gc = grid + (size_t)c0 * G * G;
  float2 cell[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) cell[j] = gc[off[j]];
  const float2* tp = tile + (sy - oy) * TT + (sx - ox);
  for (int c = c0; c < c1; ++c) {
    if (c > c0) __syncthreads();  // the previous coil's tile has been read
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (threadIdx.x + kInterpChunk * j < TT * TT) tile[threadIdx.x + kInterpChunk * j] = cell[j];
    gc += (size_t)G * G;
    if (c + 1 < c1) {
#pragma unroll
      for (int j = 0; j < PER; ++j) cell[j] = gc[off[j]];
    }
    __syncthreads();
    if (!active) continue;
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < W; ++a) {
      float2 racc = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < W; ++b) {
        const float2 g = tp[a * TT + b];
        racc.x = fmaf(wx[b], g.x, racc.x);
        racc.y = fmaf(wx[b], g.y, racc.y);
      }
      acc.x = fmaf(wy[a], racc.x, acc.x);
      acc.y = fmaf(wy[a], racc.y, acc.y);
    }
    y[(size_t)c * M + m] = make_float2(acc.x * ksign, acc.y * ksign);
  }
}

constexpr int kSpreadCoils = 4;   // coils of a group; a spreading thread accumulates up to kSpreadGroups of them
constexpr int kSpreadGroups = 3;
constexpr int kSpreadDense = 24;  // cells with more samples in their window go to the warp kernel

// Groups per spreading thread (and per warp of a dense cell) for C coils: as many as
// leave 131,072 threads (some 860 per SM; a 192^2 grid with 5 coils is slower with two
// groups per thread, 11.5 against 9.3 us), at most kSpreadGroups, in as few passes over
// the samples as that allows and with at most a quarter more padded coils than single
// groups have (12 coils of 256^2 in two groups of eight: 91 against 81 us).  One group
// where the fullest cell is a large part of the work: a warp takes 12 ns per sample of it
// with three groups and 5 with one, the rest some 3e-6 us per sample, tap and coil and
// 5e-6 us per grid cell and coil.  Adjoint at G = 512, W = 6, 12 coils, 40,000 samples
// with 861, 3,028 and 10,913 in the fullest cell: three groups 72, 96 and 235 us, one group
// 94, 106 and 183.  A coil's values do not depend on it.
int spread_groups(const mpi_plan* plan, int C) {
  const int g = (C + kSpreadCoils - 1) / kSpreadCoils;
  const double cells = (double)plan->G * plan->G;
  if (plan->dense_max > (double)plan->M * plan->W * plan->W * C / 9260 + cells * C / 5555 + 360) return 1;
  for (int ng = std::min(kSpreadGroups, g); ng > 1; --ng) {
    const int z = (g + ng - 1) / ng, even = (g + z - 1) / z;
    if (cells * z >= 131072 && 4 * even * z <= 5 * g) return even;
  }
  return 1;
}
int spread_coils_padded(const mpi_plan* plan, int C) {
  const int per = kSpreadCoils * spread_groups(plan, C);
  return (C + per - 1) / per * per;
}

// ys[cell_rank[m]][c] = ksign * y[c][m] for c < C, zero for C <= c < Cp (C
// padded to whole spreading threads, see spread_groups): the samples in first-tap-cell order, the
// coils of one sample contiguous.  Reads follow y's layout; writes scatter.
__global__ void k_nufft_sort_y(const float2* __restrict__ y, int C, int Cp, int M,
                               const int32_t* __restrict__ cell_rank, float ksign, float2* __restrict__ ys) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)Cp * M) return;
  const int c = (int)(e / M), m = (int)(e % M);
  float2 v = make_float2(0.f, 0.f);
  if (c < C) {
    const float2 t = y[e];
    v = make_float2(t.x * ksign, t.y * ksign);
  }
  ys[(size_t)cell_rank[m] * Cp + c] = v;
}

// The samples that reach grid cell (gy, gx) from first-tap row sy = gy - a:
// first taps (sy, gx - b), b = 0 .. W-1, one CSR range [r[0], r[1]) and, when
// the window wraps past column 0 (G >= 2W: once at most), a second [r[2], r[3]).
template <int W>
__device__ __forceinline__ void spread_row_ranges(const int32_t* __restrict__ rp, int gx, int G, int r[4]) {
  const int lo = gx - (W - 1);
  r[1] = rp[gx + 1];
  if (lo >= 0) {
    r[0] = rp[lo];
    r[2] = r[3] = 0;
  } else {
    r[0] = rp[0];
    r[2] = rp[G + lo];
    r[3] = rp[G];
  }
}

// One sample's term: weight phi_x(b) phi_y(a) with b = gx - sx (mod G) read
// from the sample's own first tap, times the 4 NG coils of ys from yc.
template <int W, int NG>
__device__ __forceinline__ void spread_term(const float* __restrict__ cell_w, const int32_t* __restrict__ cell_sx,
                                            const float4* __restrict__ yc, int ystride, int k, int gx, int a,
                                            int G, float (&acc)[8 * NG]) {
  int b = gx - cell_sx[k];
  if (b < 0) b += G;
  const float w = cell_w[k * 2 * W + b] * cell_w[k * 2 * W + W + a];
#pragma unroll
  for (int g = 0; g < 2 * NG; ++g) {
    const float4 u = yc[(size_t)k * ystride + g];
    acc[4 * g + 0] = fmaf(w, u.x, acc[4 * g + 0]);
    acc[4 * g + 1] = fmaf(w, u.y, acc[4 * g + 1]);
    acc[4 * g + 2] = fmaf(w, u.z, acc[4 * g + 2]);
    acc[4 * g + 3] = fmaf(w, u.w, acc[4 * g + 3]);
  }
}

template <int NG>
__device__ __forceinline__ void spread_store(float2* __restrict__ grid, int C, int G, int c0, int gy, int gx,
                                             const float (&acc)[8 * NG]) {
  const float s = ((gx + gy) & 1) ? -1.f : 1.f;  // the k-side sign (-1)^(gx + gy)
#pragma unroll
  for (int j = 0; j < kSpreadCoils * NG; ++j)
    if (c0 + j < C) grid[((size_t)(c0 + j) * G + gy) * G + gx] = make_float2(s * acc[2 * j], s * acc[2 * j + 1]);
}

struct SpreadArgs {
  const float4* ys;
  int C, Cp, G;
  const int32_t* cell_ptr;
  const int32_t* cell_sx;
  const float* cell_w;
  const int32_t* dense;  // the plan's list of dense cells
  int n_dense;
  float2* grid;
};

// Output-driven spreading, sparse cells: thread (gy, gx, 4 NG coils) sums the
// samples whose W x W footprint covers its cell, i.e. whose first tap is
// (gy - a, gx - b) (mod G) for 0 <= a, b < W, and stores the cell once; no
// atomics.  A cell whose window holds more than kSpreadDense samples is left
// to spread_dense (its thread would hold the CTA up).  Finding a cell's
// samples (the CSR ranges of W rows) costs about as much as adding a few coils of
// them, so a thread takes up to three groups of four coils: at 256^2, 12 coils,
// 64 spokes 54 us (both kinds of cells) -> 40.
template <int W, int NG>
__device__ __forceinline__ void spread_sparse(const SpreadArgs& s, int gx, int gy, int c0) {
  const int C = s.C, Cp = s.Cp, G = s.G;
  const int32_t *cell_ptr = s.cell_ptr, *cell_sx = s.cell_sx;
  const float* cell_w = s.cell_w;
  if (gx >= G || gy >= G) return;
  // the plan's ranges do not depend on earlier work
  int lo[W], hi[W], n = 0;
#pragma unroll
  for (int a = 0; a < W; ++a) {
    int sy = gy - a;
    if (sy < 0) sy += G;
    int r[4];
    spread_row_ranges<W>(cell_ptr + sy * G, gx, G, r);
    lo[a] = r[0];
    hi[a] = r[1];
    n += r[1] - r[0] + r[3] - r[2];
  }
  if (n > kSpreadDense) return;
  mpi_ptx::pdl_wait();
  const int ystride = Cp / 2;
  const float4* yc = s.ys + c0 / 2;
  float acc[8 * NG] = {};
  if (n > 0) {
#pragma unroll
    for (int a = 0; a < W; ++a)
      for (int k = lo[a]; k < hi[a]; ++k) spread_term<W, NG>(cell_w, cell_sx, yc, ystride, k, gx, a, G, acc);
    if (gx < W - 1) {  // the window wraps past column 0: the rows' second ranges
      for (int a = 0; a < W; ++a) {
        int sy = gy - a;
        if (sy < 0) sy += G;
        int r[4];
        spread_row_ranges<W>(cell_ptr + sy * G, gx, G, r);
        for (int k = r[2]; k < r[3]; ++k) spread_term<W, NG>(cell_w, cell_sx, yc, ystride, k, gx, a, G, acc);
      }
    }
  }
  spread_store<NG>(s.grid, C, G, c0, gy, gx, acc);
}

// Output-driven spreading, dense cells (the plan's list of cells whose window
// holds more than kSpreadDense samples): warp (cell i, 4 NG coils), the lanes
// taking every 32nd sample of each row range, then a butterfly sum.  With one group the
// loads of four samples are in flight (a cell of thousands of samples is a chain of
// them: 40,000 samples towards the centre of a 96^2 grid 126 -> 76 us); with more, a
// sample's own loads are as many.
template <int W, int NG>
__device__ __forceinline__ void spread_dense(const SpreadArgs& s, int i, int c0) {
  const int C = s.C, Cp = s.Cp, G = s.G;
  const int32_t *cell_ptr = s.cell_ptr, *cell_sx = s.cell_sx;
  const float* cell_w = s.cell_w;
  const int lane = threadIdx.x & 31;
  mpi_ptx::pdl_wait();
  if (i >= s.n_dense) return;
  const int cell = s.dense[i], gy = cell / G, gx = cell % G;
  const int ystride = Cp / 2;
  const float4* yc = s.ys + c0 / 2;
  float acc[8 * NG] = {};
  constexpr int kUnroll = NG == 1 ? 4 : 1;
#pragma unroll
  for (int a = 0; a < W; ++a) {
    int sy = gy - a;
    if (sy < 0) sy += G;
    int r[4];
    spread_row_ranges<W>(cell_ptr + sy * G, gx, G, r);
#pragma unroll kUnroll
    for (int k = r[0] + lane; k < r[1]; k += 32) spread_term<W, NG>(cell_w, cell_sx, yc, ystride, k, gx, a, G, acc);
    for (int k = r[2] + lane; k < r[3]; k += 32) spread_term<W, NG>(cell_w, cell_sx, yc, ystride, k, gx, a, G, acc);
  }
#pragma unroll
  for (int j = 0; j < 8 * NG; ++j)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
  if (lane == 0) spread_store<NG>(s.grid, C, G, c0, gy, gx, acc);
}

// Both kinds of cells in one launch, the dense ones' CTAs (a warp per cell) first: a
// grid cell has one kind, so they need no order, and neither fills the chip by itself
// (the dense cells of a radial trajectory's centre are few and long, most sparse ones
// are empty).  One group: four CTAs per SM (G = 96 as above 96 -> 76 us).
template <int W, int NG>
__global__ void __launch_bounds__(256, NG == 1 ? 4 : 0) k_nufft_spread(SpreadArgs s, int dense_ctas) {
  mpi_ptx::pdl_trigger();
  const int c0 = blockIdx.y * kSpreadCoils * NG, warp = threadIdx.x >> 5;
  if ((int)blockIdx.x < dense_ctas) {
    spread_dense<W, NG>(s, blockIdx.x * 8 + warp, c0);
  } else {
    const int b = blockIdx.x - dense_ctas, tx = (s.G + 31) / 32;
    spread_sparse<W, NG>(s, b % tx * 32 + (threadIdx.x & 31), b / tx * 8 + warp, c0);
  }
}

float axis_sign(int n) { return ((n / 2) & 1) ? -1.f : 1.f; }

unsigned blocks_for(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// load_lo, load_hi: the elements of each line read (the rest taken as zero);
// keep_lo, keep_hi: the elements of each transformed line stored back (default: all)
mpi_status launch_fft_rows_inplace(mpi_ctx* ctx, float2* data, long n_rows, int L, bool inverse, int load_lo = 0,
                                   int load_hi = -1, int keep_lo = 0, int keep_hi = -1);

size_t nufft_grid_elems(const mpi_plan* plan, int C) {
  return (size_t)C * plan->G * plan->G + (size_t)spread_coils_padded(plan, C) * plan->M;
}

mpi_status nufft_plan_init(mpi_ctx* ctx, mpi_plan* plan, const float* traj_host) {
  const int M = plan->M, W = plan->W, G = plan->G, n = plan->nx;
  const double sigma = (double)G / n;
  const double beta = M_PI * sqrt((W / sigma) * (W / sigma) * (sigma - 0.5) * (sigma - 0.5) - 0.8);
  cudaError_t e = cudaMalloc(&plan->deap, (size_t)n * sizeof(float));
  if (e != cudaSuccess) return cuda_check(ctx, e, "nufft plan alloc");
  if (M > 0) {
    e = cudaMalloc(&plan->traj, (size_t)M * 2 * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&plan->gstart, (size_t)M * 2 * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc(&plan->gw, (size_t)M * 2 * W * sizeof(float));
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->traj, traj_host, (size_t)M * 2 * sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_check(ctx, e, "nufft plan alloc");
    const double kscale = (double)G / (2.0 * M_PI);
    MPI_PROF(ctx, KF_NUFFT);
    k_nufft_setup<<<blocks_for((size_t)2 * M, 256), 256, 0, ctx->stream>>>(plan->traj, M, G, W, beta, kscale,
                                                                          plan->gstart, plan->gw);
    MPI_LAUNCH_CHECK(ctx, "k_nufft_setup");
  }
  MPI_PROF(ctx, KF_NUFFT);
  k_nufft_deap<<<blocks_for(n, 256), 256, 0, ctx->stream>>>(n, G, W, beta, plan->deap);
  MPI_LAUNCH_CHECK(ctx, "k_nufft_deap");
  e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "nufft plan setup");
  // Spreading CSR, built from the device's own first taps and weights (so it
  // agrees with the interpolation bit for bit): a counting sort of the samples
  // by first-tap cell sy * G + sx, stable in the sample index.
  if (M > 0) {
    std::vector<int32_t> gs((size_t)2 * M);
    std::vector<float> w((size_t)2 * M * W);
    e = cudaMemcpy(gs.data(), plan->gstart, gs.size() * sizeof(int32_t), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(w.data(), plan->gw, w.size() * sizeof(float), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_check(ctx, e, "nufft spreading index");
    const size_t GG = (size_t)G * G;
    std::vector<int32_t> ptr(GG + 1, 0), samp(M), rank(M), sx(M), dense;
    std::vector<float> cw((size_t)2 * M * W);
    for (int m = 0; m < M; ++m) ++ptr[(size_t)gs[2 * m + 1] * G + gs[2 * m] + 1];
    for (size_t t = 0; t < GG; ++t) ptr[t + 1] += ptr[t];
    std::vector<int32_t> fill(ptr.begin(), ptr.end() - 1);
    for (int m = 0; m < M; ++m) {
      const int k = fill[(size_t)gs[2 * m + 1] * G + gs[2 * m]]++;
      samp[k] = m;
      rank[m] = k;
      sx[k] = gs[2 * m];
      std::copy(w.begin() + (size_t)2 * m * W, w.begin() + (size_t)(2 * m + 2) * W, cw.begin() + (size_t)2 * k * W);
    }
    // Cells whose W x W window of first taps holds more than kSpreadDense
    // samples (a radial trajectory's centre), counted the way the kernels do.
    for (int gy = 0; gy < G; ++gy)
      for (int gx = 0; gx < G; ++gx) {
        long cnt = 0;
        for (int a = 0; a < W; ++a) {
          const int sy = (gy - a + G) % G;
          for (int b = 0; b < W; ++b) {
            const size_t t = (size_t)sy * G + (gx - b + G) % G;
            cnt += ptr[t + 1] - ptr[t];
          }
        }
        if (cnt > kSpreadDense) dense.push_back(gy * G + gx);
        plan->dense_max = std::max(plan->dense_max, (int)cnt);
      }
    plan->n_dense = (int)dense.size();
    e = cudaMalloc(&plan->cell_ptr, ptr.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc(&plan->cell_rank, (size_t)M * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc(&plan->cell_sx, (size_t)M * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc(&plan->cell_w, cw.size() * sizeof(float));
    if (e == cudaSuccess && !dense.empty()) e = cudaMalloc(&plan->cell_dense, dense.size() * sizeof(int32_t));
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->cell_ptr, ptr.data(), ptr.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->cell_rank, rank.data(), (size_t)M * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(plan->cell_sx, sx.data(), (size_t)M * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(plan->cell_w, cw.data(), cw.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !dense.empty())
      e = cudaMemcpy(plan->cell_dense, dense.data(), dense.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    // Interpolation work list: a counting sort of the samples by the 32 x 32
    // tile of their first tap, then one item per chunk of a tile's samples.
    const int tpr = (G + kInterpTile - 1) / kInterpTile, n_tiles = tpr * tpr;
    std::vector<int32_t> tcount(n_tiles + 1, 0), tsorted(M), items;
    for (int m = 0; m < M; ++m)
      ++tcount[(gs[2 * m + 1] / kInterpTile) * tpr + gs[2 * m] / kInterpTile + 1];
    for (int t = 0; t < n_tiles; ++t) tcount[t + 1] += tcount[t];
    std::vector<int32_t> tfill(tcount.begin(), tcount.end() - 1);
    for (int m = 0; m < M; ++m) tsorted[tfill[(gs[2 * m + 1] / kInterpTile) * tpr + gs[2 * m] / kInterpTile]++] = m;
    for (int t = 0; t < n_tiles; ++t)
      for (int s0 = tcount[t]; s0 < tcount[t + 1]; s0 += kInterpChunk) {
        items.push_back(t);
        items.push_back(s0);
        items.push_back(std::min(kInterpChunk, tcount[t + 1] - s0));
      }
    plan->n_tile_items = (int)(items.size() / 3);
    if (e == cudaSuccess) e = cudaMalloc(&plan->tile_items, items.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMalloc(&plan->tile_samples, (size_t)M * sizeof(int32_t));
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->tile_items, items.data(), items.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = cudaMemcpy(plan->tile_samples, tsorted.data(), (size_t)M * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_check(ctx, e, "nufft spreading index");
  }
  return MPI_OK;
}

mpi_status nufft_forward(mpi_ctx* ctx, const mpi_plan* plan, const float2* v, int C, float2* y, float2* grid) {
  const int n = plan->nx, G = plan->G, M = plan->M;
  // zero-pad with deapodisation and sign, folded into the pass along y
  mpi_status st = launch_fft_cols_window(ctx, grid, C, G, v, nullptr, plan->deap, n, false);
  if (st) return st;
  // the pass along y wrote only the window's columns; the rest are zero
  const int o = G / 2 - n / 2;
  st = launch_fft_rows_inplace(ctx, grid, (long)C * G, G, false, o, o + n);
  if (st) return st;
  if (M == 0) return MPI_OK;
  const float ks = axis_sign(G) * axis_sign(G);
  const int per = interp_coils(ctx, plan->n_tile_items, C);
  const dim3 igrid((unsigned)plan->n_tile_items, (unsigned)((C + per - 1) / per));
  MPI_PROF(ctx, KF_NUFFT);
  switch (plan->W) {
#define MPI_W_CASE(w)                                                                                \
  case w:                                                                                            \
    launch_pdl(ctx, k_nufft_interp_tiled<w>, igrid, dim3(kInterpChunk), 0,                                         \
               grid, C, G, M, plan->gstart, plan->gw, ks, plan->tile_items, plan->tile_samples, y, per);    \
    break;
    MPI_W_CASE(2) MPI_W_CASE(3) MPI_W_CASE(4) MPI_W_CASE(5) MPI_W_CASE(6) MPI_W_CASE(7) MPI_W_CASE(8)
#undef MPI_W_CASE
    default:
      return set_err(ctx, MPI_ERR_ARG, "kernel width");
  }
  MPI_LAUNCH_CHECK(ctx, "k_nufft_interp");
  return MPI_OK;
}

mpi_status nufft_adjoint(mpi_ctx* ctx, const mpi_plan* plan, const float2* y, int C, float2* out, float2* grid) {
  const int n = plan->nx, G = plan->G, M = plan->M;
  const size_t total = (size_t)C * G * G;
  if (M == 0) {
    cudaError_t e = cudaMemsetAsync(grid, 0, total * sizeof(float2), ctx->stream);
    if (e != cudaSuccess) return cuda_check(ctx, e, "grid clear");
  } else {
    const float ks = axis_sign(G) * axis_sign(G);
    const int Cp = spread_coils_padded(plan, C);
    float2* ys = grid + total;  // nufft_grid_elems reserves the sorted copy after the grid
    MPI_PROF(ctx, KF_NUFFT);
    launch_pdl(ctx, k_nufft_sort_y, dim3(blocks_for((size_t)M * Cp, 256)), dim3(256), 0, y, C, Cp, M,
               plan->cell_rank, ks, ys);
    MPI_LAUNCH_CHECK(ctx, "k_nufft_sort_y");
    const int ng = spread_groups(plan, C);
    const unsigned groups = (unsigned)(Cp / (kSpreadCoils * ng));
    const int dense_ctas = (plan->n_dense + 7) / 8;
    const dim3 sgrid((unsigned)(dense_ctas + (G + 31) / 32 * ((G + 7) / 8)), groups);
    const SpreadArgs sa{(const float4*)ys, C, Cp, G, plan->cell_ptr, plan->cell_sx, plan->cell_w, plan->cell_dense,
                        plan->n_dense, grid};
    // crowded cells (G = 32, W = 8, 9 coils, 40,000 samples: adjoint 122 us started early, 74
    // after the sort; small work gains 2-3 us by an early start)
    const NoEarlyStart late(ctx, plan->dense_max >= 1024 && (long)sgrid.x * sgrid.y <= 4L * std::max(ctx->num_sms, 1));
    MPI_PROF(ctx, KF_NUFFT);
#define MPI_SPREAD(w, g) \
  if (plan->W == w && ng == g) launch_pdl(ctx, k_nufft_spread<w, g>, sgrid, dim3(256), 0, sa, dense_ctas);
#define MPI_W_CASE(w) MPI_SPREAD(w, 1) MPI_SPREAD(w, 2) MPI_SPREAD(w, 3)
    MPI_W_CASE(2) MPI_W_CASE(3) MPI_W_CASE(4) MPI_W_CASE(5) MPI_W_CASE(6) MPI_W_CASE(7) MPI_W_CASE(8)
#undef MPI_W_CASE
#undef MPI_SPREAD
    if (plan->W < 2 || plan->W > 8) return set_err(ctx, MPI_ERR_ARG, "kernel width");
    MPI_LAUNCH_CHECK(ctx, "k_nufft_spread");
  }
  // only the columns of the centred window reach the cropping pass along y
  const int o = G / 2 - n / 2;
  mpi_status st = launch_fft_rows_inplace(ctx, grid, (long)C * G, G, true, 0, G, o, o + n);
  if (st) return st;
  // the inverse pass along y stores only the centred window, with deapodisation and sign
  return launch_fft_cols_window(ctx, grid, C, G, nullptr, out, plan->deap, n, true);
}
