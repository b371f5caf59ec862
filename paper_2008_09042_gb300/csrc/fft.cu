// Cartesian F_s (Eq. 1): centred unitary DFT per coil followed by selection of
// the sampled points, as shared-memory FFT passes.
//
// The centred DFT along an axis of even length n is
//   F_c = (-1)^(n/2) D F D / sqrt(n),  D = diag((-1)^j),
// with F the plain DFT.  The image-side sign D and the 1/sqrt(N) scale are
// applied by the expansion kernels; these passes do the plain FFTs, the
// k-side sign and the gather / zero-fill of the sampled points.
// The line FFTs themselves are in fft_tile.cuh (Stockham, shared memory) and
// dft_reg.cuh (registers).
#include <stdio.h>

#include <cuda.h>

#include <algorithm>
#include <vector>

#include "dft_reg.cuh"
#include "fft_rows.cuh"
#include "fft_tile.cuh"
#include "mpi_internal.h"
#include "ptx.cuh"

namespace {

using namespace mpi_fft;

// Rows along x of a Cartesian plan.  A warp takes R of a coil's k-space rows with
// samples (row_list; null: every row) through the register FFT of fft_rows.cuh,
// the warps striding over all of them (the grid is capped at a few CTAs per SM:
// volumes have hundreds of thousands of rows, and one CTA each would make the pass
// bound by CTA launches).  256^2, 16 coils, warm L2: 7 us with a Stockham line per
// warp, 5 this way; 288 coils of 320^2 in one launch 131 -> 85 us (gather), 118 -> 85
// (scatter), of which the 236 MB they read or write take 35 at HBM's rate.
//
// Forward: FFT along x, k-side centring sign, gather the row's samples (contiguous
// in the sorted list); rows without samples are not touched.
// TAB (a batch's group of slices): coil c has its own sampling and data block, tab[c].
struct RowsArgs {
  int C, n_rows, ny, M;
  int n_list;  // rows with samples (TAB: the most that any coil has)
  const int32_t* row_list;
  const int32_t* idx;
  const int32_t* row_ptr;
  float ksign;
  const float2* tw;
  const CoilSamples* tab;
};

template <int NX, bool TAB = false>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows_fwd_gather(const float2* __restrict__ data,
                                                                    float2* __restrict__ y, RowsArgs a) {
  using F = Rows<NX>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* b = buf[warp];
  const int per = (a.n_list + F::R - 1) / F::R, total = a.C * per;
  for (int gi = blockIdx.x * kRowWarps + warp; gi < total; gi += gridDim.x * kRowWarps) {
    // a group's data may exceed L2: last coil first, so that this pass and the one along
    // y meet at the coils that are still there
    const int gq = TAB ? total - 1 - gi : gi;
    const int c = gq / per, j0 = (gq - c * per) * F::R;
    const int n_list = TAB ? a.tab[c].n_list : a.n_list;
    const int32_t* list = TAB ? a.tab[c].row_list : a.row_list;
    const int32_t* idx = TAB ? a.tab[c].idx : a.idx;
    const int32_t* row_ptr = TAB ? a.tab[c].row_ptr : a.row_ptr;
    float2* yc = TAB ? a.tab[c].y : y + (size_t)c * a.M;
    if (j0 >= n_list) continue;  // warp-uniform
    // the group's rows, their (kz + ky) parities and the range of their samples
    int row[F::R], rpar[F::R], m0 = 0, m1 = 0;
#pragma unroll
    for (int r = 0; r < F::R; ++r) {
      const bool in = j0 + r < n_list;
      row[r] = in ? (list ? list[j0 + r] : j0 + r) : 0x7fffffff;
      rpar[r] = in ? (row[r] / a.ny + row[r] % a.ny) & 1 : 0;
    }
    m0 = row_ptr[row[0]];
    m1 = row_ptr[(list ? list[min(j0 + F::R, n_list) - 1] : min(j0 + F::R, n_list) - 1) + 1];
    float2 v[F::T1][F::A];
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int j = j0 + (lane + 32 * i) / F::P;
      if (j < n_list) {
        const float2* src = data + ((size_t)c * a.n_rows + (list ? list[j] : j)) * NX + lane % F::P;
#pragma unroll
        for (int e = 0; e < F::A; ++e) v[i][e] = src[F::P * e];
      }
    }
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int r = (lane + 32 * i) / F::P;
      if (j0 + r < n_list) F::template step1<false>(v[i], r, lane % F::P, b, a.tw);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int t = lane + 32 * i, r = t / F::A, k1 = t % F::A;
      if (r < F::R && j0 + r < n_list) {
        float2 u[F::P];
        F::template step2<false>(u, r, k1, b);
#pragma unroll
        for (int k = 0; k < F::P; ++k) b[r * F::S + k1 * (F::P + 1) + k] = u[k];
      }
    }
    __syncwarp();
    F::samples(row, m0, m1, lane, [&](int m) { return idx[m]; }, [](int) { return 0; },
               [&](int m, int r, int kx, int) {
      const float sg = ((kx + rpar[r]) & 1) ? -a.ksign : a.ksign;
      const float2 t = b[F::out_at(r, kx)];
      yc[m] = make_float2(t.x * sg, t.y * sg);
    });
    __syncwarp();  // the buffer is refilled for the next rows
  }
}

// Adjoint: zero-fill the row from its samples (with the k-side sign), inverse
// FFT.  Rows without samples are not written: the pass along y that follows
// reads them as zeros.
template <int NX, bool TAB = false>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows_scatter_inv(const float2* __restrict__ y,
                                                                     float2* __restrict__ data, RowsArgs a) {
  using F = Rows<NX>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* b = buf[warp];
  const int per = (a.n_list + F::R - 1) / F::R, total = a.C * per;
  for (int gi = blockIdx.x * kRowWarps + warp; gi < total; gi += gridDim.x * kRowWarps) {
    // a group's data may exceed L2: last coil first, so that this pass and the one along
    // y meet at the coils that are still there
    const int gq = TAB ? total - 1 - gi : gi;
    const int c = gq / per, j0 = (gq - c * per) * F::R;
    const int n_list = TAB ? a.tab[c].n_list : a.n_list;
    const int32_t* list = TAB ? a.tab[c].row_list : a.row_list;
    const int32_t* idx = TAB ? a.tab[c].idx : a.idx;
    const int32_t* row_ptr = TAB ? a.tab[c].row_ptr : a.row_ptr;
    const float2* yc = TAB ? a.tab[c].y : y + (size_t)c * a.M;
    if (j0 >= n_list) continue;  // warp-uniform
    // the group's rows, their (kz + ky) parities and the range of their samples
    int row[F::R], rpar[F::R], m0 = 0, m1 = 0;
#pragma unroll
    for (int r = 0; r < F::R; ++r) {
      const bool in = j0 + r < n_list;
      row[r] = in ? (list ? list[j0 + r] : j0 + r) : 0x7fffffff;
      rpar[r] = in ? (row[r] / a.ny + row[r] % a.ny) & 1 : 0;
    }
    m0 = row_ptr[row[0]];
    m1 = row_ptr[(list ? list[min(j0 + F::R, n_list) - 1] : min(j0 + F::R, n_list) - 1) + 1];
    for (int i = lane; i < F::kSmem; i += 32) b[i] = make_float2(0.f, 0.f);
    __syncwarp();
    F::samples(row, m0, m1, lane, [&](int m) { return idx[m]; }, [&](int m) { return yc[m]; },
               [&](int, int r, int kx, float2 t) {
      const float sg = ((kx + rpar[r]) & 1) ? -a.ksign : a.ksign;
      b[F::in_at(r, kx)] = make_float2(t.x * sg, t.y * sg);
    });
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {  // a lane's task reads and writes the same places
      const int r = (lane + 32 * i) / F::P, p = lane % F::P;
      float2 v[F::A];
#pragma unroll
      for (int e = 0; e < F::A; ++e) v[e] = b[r * F::S + e * (F::P + 1) + p];
      F::template step1<true>(v, r, p, b, a.tw);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int t = lane + 32 * i, r = t / F::A, k1 = t % F::A;
      if (r < F::R && j0 + r < n_list) {
        float2 u[F::P];
        F::template step2<true>(u, r, k1, b);
        float2* dst = data + ((size_t)c * a.n_rows + (list ? list[j0 + r] : j0 + r)) * NX + k1;
#pragma unroll
        for (int k = 0; k < F::P; ++k) dst[F::A * k] = u[k];
      }
    }
    __syncwarp();
  }
}

// In-place FFT of lines of length L with element stride `stride`.  A CTA takes
// TILE lines that are adjacent in memory (consecutive x): it loads them as
// TILE-element row segments (64, 128 or 256 bytes), transposes into shared
// memory (one contiguous padded line each), transforms them (TILE / 8 lines
// per warp) and writes back.  Wide tiles make long DRAM bursts for passes over
// volumes that do not fit in L2; narrow ones give more CTAs for small grids.
// Tiles are enumerated as (slab, x-tile) with slab base offset
// (slab / inner) * outer_stride + (slab % inner) * inner_stride.
template <int L, bool INV, int TILE>
__global__ void __launch_bounds__(kLineWarps * 32, (L * TILE <= 2048) ? 4 : (L * TILE >= 4096 ? 2 : 3)) k_fft_lines(float2* __restrict__ data, int nx,
                                                              long stride, int n_slabs, int inner,
                                                              long outer_stride, long inner_stride,
                                                              const float2* __restrict__ tw_g,
                                                              const uint8_t* __restrict__ rmask, int mask_nz) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  constexpr int S = col_stride(L, TILE);
  constexpr int T = kLineWarps * 32;         // threads
  constexpr int RSTEP = T / TILE;            // rows covered per pass of the CTA
  constexpr int PER = (L + RSTEP - 1) / RSTEP;  // elements per thread
  __shared__ float2 tw[L];
  __shared__ float2 buf[TILE * S];
  const int tid = threadIdx.x;
  for (int i = tid; i < L; i += T) tw[i] = tw_g[i];
  const int x_tiles = (nx + TILE - 1) / TILE;
  const int tile = (int)blockIdx.x;
  const int slab = tile / x_tiles;
  const int x0 = (tile - slab * x_tiles) * TILE;
  if (slab >= n_slabs) return;
  const size_t base = (size_t)(slab / inner) * outer_stride + (size_t)(slab % inner) * inner_stride + x0;
  // thread -> (column cx, rows r0 + RSTEP u): all PER loads are issued before any is used
  const int cx = tid % TILE, r0 = tid / TILE;
  const bool ok = x0 + cx < nx;
  const float2* src = data + base + cx;
  // With a row mask (rmask[z * L + r], z = slab % mask_nz: 1 where k-space row r
  // of this slab has samples): inverse, the rows without samples are taken as
  // zeros without being read, whatever the buffer holds there (the adjoint's
  // row pass does not write them); forward, only the rows with samples are
  // stored (the row pass that follows reads no other row).
  const uint8_t* rm = rmask ? rmask + (size_t)(slab % mask_nz) * L : nullptr;
  float2 v[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int r = r0 + RSTEP * u;
    if (ok && r < L) v[u] = (INV && rm && !rm[r]) ? make_float2(0.f, 0.f) : src[(size_t)r * stride];
  }
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (ok && r0 + RSTEP * u < L) buf[cx * S + pad8(r0 + RSTEP * u)] = v[u];
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  fft_tile_lines<L, INV, TILE, S>(buf, tw, warp, lane);
  __syncthreads();
  float2* dst = data + base + cx;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int r = r0 + RSTEP * u;
    if (ok && r < L && (INV || !rm || rm[r])) dst[(size_t)r * stride] = buf[cx * S + pad8(r)];
  }
}

template <int L, bool INV, int TILE>
void lines_launch(mpi_ctx* ctx, long blocks, float2* data, int nx, long stride, int n_slabs, int inner,
                  long outer_stride, long inner_stride, const float2* tw, const uint8_t* rmask, int mask_nz) {
  launch_pdl(ctx, k_fft_lines<L, INV, TILE>, dim3((unsigned)blocks), dim3(kLineWarps * 32), 0, data, nx, stride,
             n_slabs, inner, outer_stride, inner_stride, tw, rmask, mask_nz);
}

// Tile width: the widest (longest row segments) that keeps at most 16 elements
// per thread in the copy phases and still gives every SM four or more CTAs.
int lines_tile(const mpi_ctx* ctx, int L, int nx, int n_slabs) {
  const long want = 4L * std::max(ctx->num_sms, 1);
  const int tiles[3] = {32, 16, 8};
  for (int t : tiles) {
    if (L * t / (kLineWarps * 32) > 16) continue;
    if (t == 8 || (long)n_slabs * ((nx + t - 1) / t) >= want) return t;
  }
  return 8;
}

// The pass along y as a two-step FFT in registers: L = R1 R2 points per
// column, y = r + R2 m.  A CTA takes TILE adjacent columns (32: a warp per r; 16: half
// a warp) of one (coil, z) plane.  Step 1: for each r, the R1 values y = r + R2 m are
// loaded (row segments of TILE columns: coalesced), transformed (R1-point DFT in
// registers) and twiddled by w_L^(r k1) into shared memory [k1][r][column].  Step 2:
// for each k1, the R2 values are read back, transformed (R2-point DFT) and stored to
// rows k = k1 + R1 k2.  One shared-memory write and read per element (the
// Stockham passes take one per radix stage plus two transposes).  The inverse
// is the forward of the conjugated data, conjugated back.  Row mask as in
// k_fft_lines: inverse, rows without samples are read as zeros; forward, only
// rows with samples are stored.  32 columns make longer bursts for volumes that do
// not fit in L2; 16 make twice the CTAs, each with half the work: 16 coils of
// 256^2, 128 CTAs of 32 columns on 152 SMs 7.0 us, 256 of 16 columns 4.9.  The width does
// not change a column's arithmetic.
template <int R1, int R2, bool INV, int TILE>
__global__ void __launch_bounds__(256, 2) k_fft_cols_reg(float2* __restrict__ data, int nx, int n_slabs, long plane,
                                                      const float2* __restrict__ tw_g,
                                                      const uint8_t* __restrict__ rmask, int mask_nz) {
  constexpr int L = R1 * R2, GROUPS = 256 / TILE;
  __shared__ float2 sY[L * TILE];  // [k1][r][column]
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int tid = threadIdx.x, col_i = tid % TILE, w = tid / TILE;
  const int x_tiles = (nx + TILE - 1) / TILE;
  const int slab = (int)blockIdx.x / x_tiles, x0 = ((int)blockIdx.x - slab * x_tiles) * TILE;
  const bool ok = x0 + col_i < nx;
  float2* col = data + (size_t)slab * plane + x0 + col_i;
  const uint8_t* rm = rmask ? rmask + (size_t)(slab % mask_nz) * L : nullptr;
#pragma unroll
  for (int it = 0; it < (R2 + GROUPS - 1) / GROUPS; ++it) {
    const int r = w + GROUPS * it;
    if (r >= R2) break;
    float2 v[R1];
    uint8_t keep[R1];  // the mask's loads in flight together, then the values'
#pragma unroll
    for (int m = 0; m < R1; ++m) keep[m] = INV && rm ? rm[r + R2 * m] : 1;
#pragma unroll
    for (int m = 0; m < R1; ++m) {
      const int y = r + R2 * m;
      float2 t = make_float2(0.f, 0.f);
      if (ok && keep[m]) t = col[(size_t)y * nx];
      v[m] = INV ? make_float2(t.x, -t.y) : t;
    }
    float2 tw[R1];
#pragma unroll
    for (int k1 = 1; k1 < R1; ++k1) tw[k1] = __ldg(tw_g + r * k1);
    mpi_dft::dft_r<R1>(v);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) sY[(k1 * R2 + r) * TILE + col_i] = k1 ? mpi_dft::cmulf(v[k1], tw[k1]) : v[0];
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < (R1 + GROUPS - 1) / GROUPS; ++it) {
    const int k1 = w + GROUPS * it;
    if (k1 >= R1) break;
    float2 u[R2];
#pragma unroll
    for (int r = 0; r < R2; ++r) u[r] = sY[(k1 * R2 + r) * TILE + col_i];
    mpi_dft::dft_r<R2>(u);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      const int k = k1 + R1 * k2;
      if (ok && (INV || !rm || rm[k])) col[(size_t)k * nx] = INV ? make_float2(u[k2].x, -u[k2].y) : u[k2];
    }
  }
}

// Line kernels by choice: 8, 16, 32 lines per CTA (Stockham), or the register pass
// along y with 32 (-1) or 16 (-16) columns per CTA.
constexpr int kRegCols32 = -1, kRegCols16 = -16;
int kernel_cols(int choice) { return choice == kRegCols32 ? 32 : (choice == kRegCols16 ? 16 : choice); }

// Whether lines of length L with this geometry have a register pass.
bool cols_reg_has(int L, int nx, long stride, int inner) {
  return stride == nx && inner == 1 && (L == 64 || L == 96 || L == 128 || L == 192 || L == 256 || L == 320);
}

// Passes along y over at most this many bytes take 16 register columns untimed.  Over
// 1 to 32 coils of 64^2 to 320^2 (26 MB), masked and not, they were the fastest of the
// five candidates or within the timer's 0.7 us of it (32 coils of 256^2: 8-line Stockham
// 11.1 us, 32 columns 8.4, 16 columns 7.7), while timing all five cost a plan's first call
// 0.2 ms and let noise choose.  Beyond half of L2 a pass runs at HBM's rate and is timed.
constexpr size_t kRegCols16Bytes = 64u << 20;

// Launch of the register pass along y for length L; false where L has no
// (R1, R2) split or the geometry is not a y pass (lines of stride nx in
// planes of `outer_stride`).
template <bool INV>
bool cols_reg_launch(mpi_ctx* ctx, int choice, int L, float2* data, int nx, long stride, int n_slabs, int inner,
                     long outer_stride, const float2* tw, const uint8_t* rmask, int mask_nz) {
  if (stride != nx || inner != 1) return false;
  const int cols = kernel_cols(choice);
  const long blocks = (long)n_slabs * ((nx + cols - 1) / cols);
  if (blocks == 0 || blocks > 0x7fffffffL) return false;
#define MPI_CREG(n, r1, r2)                                                                                   \
  case n:                                                                                                    \
    if (cols == 32)                                                                                          \
      launch_pdl(ctx, k_fft_cols_reg<r1, r2, INV, 32>, dim3((unsigned)blocks), dim3(256), 0, data, nx, n_slabs, \
                 outer_stride, tw, rmask, mask_nz);                                                          \
    else                                                                                                     \
      launch_pdl(ctx, k_fft_cols_reg<r1, r2, INV, 16>, dim3((unsigned)blocks), dim3(256), 0, data, nx, n_slabs, \
                 outer_stride, tw, rmask, mask_nz);                                                          \
    return true;
  switch (L) {
    MPI_CREG(64, 8, 8)
    MPI_CREG(96, 8, 12)
    MPI_CREG(128, 8, 16)
    MPI_CREG(192, 16, 12)
    MPI_CREG(256, 16, 16)
    MPI_CREG(320, 16, 20)
    default:
      return false;
  }
#undef MPI_CREG
}

// Launch of one line pass with kernel `tile` (8, 16 or 32 lines, or a register
// pass along y); false when the length / tile pair is not
// compiled.
template <bool INV>
bool lines_launch_tile(mpi_ctx* ctx, int tile, int L, long blocks, float2* data, int nx, long stride, int n_slabs,
                       int inner, long outer_stride, long inner_stride, const float2* tw, const uint8_t* rmask,
                       int mask_nz) {
  if (tile < 0) return cols_reg_launch<INV>(ctx, tile, L, data, nx, stride, n_slabs, inner, outer_stride, tw, rmask, mask_nz);
#define MPI_LINES_CASE(n)                                                                                     \
  case n:                                                                                                     \
    if (tile == 32 && n <= 128)                                                                               \
      lines_launch<n, INV, (n <= 128 ? 32 : 8)>(ctx, blocks, data, nx, stride, n_slabs, inner, outer_stride,   \
                                                inner_stride, tw, rmask, mask_nz);                           \
    else if (tile == 16 && n <= 256)                                                                          \
      lines_launch<n, INV, (n <= 256 ? 16 : 8)>(ctx, blocks, data, nx, stride, n_slabs, inner, outer_stride,   \
                                                inner_stride, tw, rmask, mask_nz);                           \
    else if (tile == 8)                                                                                       \
      lines_launch<n, INV, 8>(ctx, blocks, data, nx, stride, n_slabs, inner, outer_stride, inner_stride, tw,    \
                              rmask, mask_nz);                                                               \
    else                                                                                                      \
      return false;                                                                                           \
    return true;
  switch (L) {
    MPI_LINES_CASE(16)
    MPI_LINES_CASE(32)
    MPI_LINES_CASE(48)
    MPI_LINES_CASE(64)
    MPI_LINES_CASE(96)
    MPI_LINES_CASE(128)
    MPI_LINES_CASE(192)
    MPI_LINES_CASE(256)
    MPI_LINES_CASE(320)
    MPI_LINES_CASE(512)
    default:
      return false;
  }
#undef MPI_LINES_CASE
}

// Autotuner of the line passes' tile width.  A pass shape is tuned once per
// context: each candidate width (at most 16 elements per thread in the copy
// phases) is launched once to warm up and then three times between two CUDA
// events on the context's stream, on the tuning scratch buffer (the pass's
// timing does not depend on the values it transforms); the fastest is kept.
// Returns 0 when this call cannot tune (no scratch, capture in progress,
// tuning off).
template <bool INV>
int lines_autotune(mpi_ctx* ctx, const long (&key)[10], int L, float2* data, int nx, long stride, int n_slabs,
                   int inner, long outer_stride, long inner_stride, const float2* tw, const uint8_t* rmask,
                   int mask_nz) {
  if (!ctx->autotune || !ctx->tune_scratch) return 0;
  // the elements the pass touches, from `data`: every slab base plus a full line set
  const long last_slab = n_slabs - 1;
  const size_t extent = (size_t)(last_slab / inner) * outer_stride + (size_t)(last_slab % inner) * inner_stride +
                        (size_t)(L - 1) * stride + nx;
  if (extent * sizeof(float2) > ctx->tune_scratch_bytes) return 0;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cap != cudaStreamCaptureStatusNone) return 0;
  float2* scratch = (float2*)ctx->tune_scratch;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaGetLastError();
    cudaEventDestroy(e0);
    return 0;
  }
  mpi_ctx::TuneRecord rec;
  for (int i = 0; i < 10; ++i) rec.key[i] = key[i];
  rec.n = 0;
  rec.choice = 0;
  float best = 1e30f;
  const int cands[5] = {8, 16, 32, kRegCols32, kRegCols16};
  for (int tile : cands) {
    if (tile > 0 && (long)L * tile / (kLineWarps * 32) > 16) continue;
    const int cols = kernel_cols(tile);  // columns per CTA
    const long blocks = (long)n_slabs * ((nx + cols - 1) / cols);
    if (blocks > 0x7fffffffL) continue;
    if (!lines_launch_tile<INV>(ctx, tile, L, blocks, scratch, nx, stride, n_slabs, inner, outer_stride,
                                inner_stride, tw, rmask, mask_nz))
      continue;
    cudaEventRecord(e0, ctx->stream);
    for (int r = 0; r < 3; ++r)
      lines_launch_tile<INV>(ctx, tile, L, blocks, scratch, nx, stride, n_slabs, inner, outer_stride, inner_stride,
                             tw, rmask, mask_nz);
    cudaEventRecord(e1, ctx->stream);
    float ms = 0.f;
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    const float us = 1e3f * ms / 3.f;
    rec.cand[rec.n] = tile;
    rec.us[rec.n] = us;
    rec.n++;
    if (us < best) {
      best = us;
      rec.choice = tile;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!rec.choice || cudaGetLastError() != cudaSuccess) return 0;
  char buf[320];
  auto tname = [](int t, char* b, size_t n) {
    if (t < 0) snprintf(b, n, "register two-step, %d columns", kernel_cols(t));
    else snprintf(b, n, "%d lines", t);
  };
  char tn[48];
  tname(rec.choice, tn, sizeof tn);
  int len = snprintf(buf, sizeof buf, "FFT line pass L=%d %s stride=%ld lines=%ld%s: %s (", L, INV ? "inverse" : "forward",
                     stride, (long)n_slabs * nx, rmask ? " row-masked" : "", tn);
  for (int i = 0; i < rec.n && len < (int)sizeof buf; ++i) {
    tname(rec.cand[i], tn, sizeof tn);
    len += snprintf(buf + len, sizeof buf - len, "%s%s: %.1f us", i ? ", " : "", tn, rec.us[i]);
  }
  if (len < (int)sizeof buf) snprintf(buf + len, sizeof buf - len, ")");
  rec.what = buf;
  ctx->tuned.push_back(rec);
  return rec.choice;
}

// The tile width of a line pass: the caller's fixed choice where it applies,
// else the tuned one (tuning it now if this call can), else 0.
template <bool INV>
int lines_choose(mpi_ctx* ctx, float2* data, int L, int nx, long stride, int n_slabs, int inner, long outer_stride,
                 long inner_stride, const float2* tw, const uint8_t* rmask, int mask_nz) {
  const long key[10] = {L, INV ? 1 : 0, nx, stride, n_slabs, inner, outer_stride, inner_stride, rmask ? 1 : 0,
                        mask_nz};
  int tile = 0;
  // a caller's fixed choice (mpi_ctx_set_line_kernel), where this pass has it
  if (ctx->line_kernel) {
    const int t = ctx->line_kernel;
    const bool ok = t == -1 ? cols_reg_has(L, nx, stride, inner)
                            : (t == 8 || (t == 16 && L <= 256) || (t == 32 && L <= 128));
    if (ok) tile = t;
  }
  if (!tile && cols_reg_has(L, nx, stride, inner) && (size_t)n_slabs * L * nx * sizeof(float2) <= kRegCols16Bytes)
    tile = kRegCols16;
  for (const auto& r : ctx->tuned) {
    if (tile) break;
    if (std::equal(r.key, r.key + 10, key)) tile = r.choice;
  }
  if (!tile)
    tile = lines_autotune<INV>(ctx, key, L, data, nx, stride, n_slabs, inner, outer_stride, inner_stride, tw, rmask,
                               mask_nz);
  return tile;
}

template <bool INV>
mpi_status lines_dispatch(mpi_ctx* ctx, const char* name, float2* data, int L, int nx, long stride, int n_slabs,
                          int inner, long outer_stride, long inner_stride, const uint8_t* rmask = nullptr,
                          int mask_nz = 1) {
  const float2* tw = twiddle_table(ctx, L);
  if (!tw) return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  if ((long)n_slabs * nx == 0) return MPI_OK;
  int tile = lines_choose<INV>(ctx, data, L, nx, stride, n_slabs, inner, outer_stride, inner_stride, tw, rmask,
                               mask_nz);
  if (!tile) tile = lines_tile(ctx, L, nx, n_slabs);
  const int tw_cols = kernel_cols(tile);
  const int x_tiles = (nx + tw_cols - 1) / tw_cols;
  const long blocks = (long)n_slabs * x_tiles;
  if (blocks > 0x7fffffffL) return set_err(ctx, MPI_ERR_SHAPE, "too many FFT tiles");
  MPI_PROF(ctx, KF_FFT_LINES);
  if (!lines_launch_tile<INV>(ctx, tile, L, blocks, data, nx, stride, n_slabs, inner, outer_stride, inner_stride, tw,
                              rmask, mask_nz))
    return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  MPI_LAUNCH_CHECK(ctx, name);
  return MPI_OK;
}

// Line pass along y over the oversampled radial grid [C][G][G] (L = G) with the
// centred n x n window folded in, in place of separate zero-pad and crop
// passes.  Each grid cell of the window (gy, gx) = (o + y, o + x) carries the
// factor deap[y] deap[x] / n (-1)^(gx + gy).  Forward (src set): the column is
// formed on the fly from the image [C][n][n] (zero outside the window) and its
// transform written to the grid.  Inverse (dst set): the grid column's
// transform is stored only inside the window, scaled, into the image
// [C][n][n]; the grid is not written back.  Tiles of 8 columns; a tile wholly
// outside the window does nothing: forward, those grid columns are zero and
// the row pass that follows reads them as zeros without loading them.
struct LineWin {
  const float2* src;
  float2* dst;
  const float* deap;
  int n, o;
};

template <int L, bool INV>
__global__ void __launch_bounds__(kLineWarps * 32, (L * 8 <= 2048) ? 4 : (L * 8 >= 4096 ? 2 : 3))
    k_fft_lines_win(float2* __restrict__ grid, int C, LineWin win, const float2* __restrict__ tw_g) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  constexpr int TILE = 8;
  constexpr int S = col_stride(L, TILE);
  constexpr int T = kLineWarps * 32;
  constexpr int RSTEP = T / TILE;
  constexpr int PER = (L + RSTEP - 1) / RSTEP;
  __shared__ float2 tw[L];
  __shared__ float2 buf[TILE * S];
  constexpr int x_tiles = L / TILE;
  const int c = (int)blockIdx.x / x_tiles, x0 = ((int)blockIdx.x % x_tiles) * TILE;
  if (c >= C) return;
  const bool tile_in = x0 < win.o + win.n && x0 + TILE > win.o;  // CTA-uniform
  const int tid = threadIdx.x, cx = tid % TILE, r0 = tid / TILE;
  const int gx = x0 + cx, xi = gx - win.o;
  const bool colin = xi >= 0 && xi < win.n;
  float2* gcol = grid + (size_t)c * L * L + gx;
  if (!tile_in) return;  // forward: those columns are zero, and the row pass reads them as such
  for (int i = tid; i < L; i += T) tw[i] = tw_g[i];
  float2 v[PER];
  if (!INV) {
    const float2* src = win.src + (size_t)c * win.n * win.n + xi;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int r = r0 + RSTEP * u, yi = r - win.o;
      v[u] = make_float2(0.f, 0.f);
      if (r < L && colin && yi >= 0 && yi < win.n) {
        const float2 val = src[(size_t)yi * win.n];
        float f = win.deap[yi] * win.deap[xi] / (float)win.n;
        if ((gx + r) & 1) f = -f;
        v[u] = make_float2(val.x * f, val.y * f);
      }
    }
  } else {
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (r0 + RSTEP * u < L) v[u] = gcol[(size_t)(r0 + RSTEP * u) * L];
  }
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (r0 + RSTEP * u < L) buf[cx * S + pad8(r0 + RSTEP * u)] = v[u];
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  fft_tile_lines<L, INV, TILE, S>(buf, tw, warp, lane);
  __syncthreads();
  if (!INV) {
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (r0 + RSTEP * u < L) gcol[(size_t)(r0 + RSTEP * u) * L] = buf[cx * S + pad8(r0 + RSTEP * u)];
  } else {
    float2* dst = win.dst + (size_t)c * win.n * win.n + xi;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int r = r0 + RSTEP * u, yi = r - win.o;
      if (r < L && colin && yi >= 0 && yi < win.n) {
        const float2 t = buf[cx * S + pad8(r)];
        float f = win.deap[yi] * win.deap[xi] / (float)win.n;
        if ((gx + r) & 1) f = -f;
        dst[(size_t)yi * win.n] = make_float2(t.x * f, t.y * f);
      }
    }
  }
}

// The windowed pass along y as a two-step register FFT (G = R1 R2, see
// k_fft_cols_reg), 16 adjacent columns per CTA (two rows per warp step): one write
// and read of shared memory per element instead of one per radix stage and two
// transposes, and the padded rows are never loaded.  Tiles wholly outside the window are
// not launched.  256^2, 12 coils, G = 512: 17.6 -> 12.4 us; small grids and few coils have
// too few of these CTAs, of too much work each (see kWinReg).
template <int R1, int R2, bool INV>
__global__ void __launch_bounds__(256) k_fft_cols_win(float2* __restrict__ grid, int C, LineWin win, int x_first,
                                                      int x_tiles, const float2* __restrict__ tw_g) {
  constexpr int L = R1 * R2, TILE = 16;
  extern __shared__ float2 sY[];  // [k1][r][column]
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int tid = threadIdx.x, col = tid % TILE, s0 = tid / TILE;
  const int c = (int)blockIdx.x / x_tiles, gx = x_first + ((int)blockIdx.x - c * x_tiles) * TILE + col;
  const int xi = gx - win.o;
  const bool colin = gx < L && xi >= 0 && xi < win.n;  // else a column of zeros: nothing reads or keeps it
  float2* gcol = grid + (size_t)c * L * L + gx;
  const float fx = colin ? win.deap[xi] / (float)win.n : 0.f;
#pragma unroll
  for (int it = 0; it < (R2 + 15) / 16; ++it) {
    const int r = s0 + 16 * it;
    if (r >= R2) break;
    float2 v[R1];
    if (!INV) {
      const float2* src = win.src + (size_t)c * win.n * win.n + xi;
      float f[R1];
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const int yi = r + R2 * m - win.o;
        const bool in = colin && yi >= 0 && yi < win.n;
        v[m] = in ? src[(size_t)yi * win.n] : make_float2(0.f, 0.f);
        f[m] = in ? win.deap[yi] * fx : 0.f;
      }
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const float g = ((gx + r + R2 * m) & 1) ? -f[m] : f[m];
        v[m] = make_float2(v[m].x * g, v[m].y * g);
      }
    } else {
#pragma unroll
      for (int m = 0; m < R1; ++m) {
        const float2 e = colin ? gcol[(size_t)(r + R2 * m) * L] : make_float2(0.f, 0.f);
        v[m] = make_float2(e.x, -e.y);  // the inverse on conjugated values
      }
    }
    float2 w[R1];
#pragma unroll
    for (int k1 = 1; k1 < R1; ++k1) w[k1] = __ldg(tw_g + r * k1);
    mpi_dft::dft_r<R1>(v);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) sY[(k1 * R2 + r) * TILE + col] = k1 ? mpi_dft::cmulf(v[k1], w[k1]) : v[0];
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < (R1 + 15) / 16; ++it) {
    const int k1 = s0 + 16 * it;
    if (k1 >= R1 || !colin) break;
    float2 u[R2];
#pragma unroll
    for (int r = 0; r < R2; ++r) u[r] = sY[(k1 * R2 + r) * TILE + col];
    mpi_dft::dft_r<R2>(u);
    if (!INV) {
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) gcol[(size_t)(k1 + R1 * k2) * L] = u[k2];
    } else {
      float2* dst = win.dst + (size_t)c * win.n * win.n + xi;
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) {
        const int gy = k1 + R1 * k2, yi = gy - win.o;
        if (yi >= 0 && yi < win.n) {
          float f = win.deap[yi] * fx;
          if ((gx + gy) & 1) f = -f;
          dst[(size_t)yi * win.n] = make_float2(u[k2].x * f, -u[k2].y * f);
        }
      }
    }
  }
}

float axis_sign(int n) { return ((n / 2) & 1) ? -1.f : 1.f; }

// The passes along y and x of one (coil, kz) plane of a 3D volume in one CTA,
// the plane held in shared memory S [NY][NX] (NY x NX x 8 bytes, at most 128 KB).
// NX / 8 warps: four per 32-column group.
//  forward: the DFT along y as a register two-step (NY = 8 R2; y = r + R2 m):
//    DFT8 over m straight from the coalesced rows of global memory, twiddle
//    w_NY^(r k1), into S rows r + R2 k1; then for each k1 the R2 rows R2 k1 + r
//    are read back, transformed (R2-point DFT) and written in place, so that
//    row R2 (ky % 8) + ky / 8 holds k-space row ky.  Then each k-space row with
//    samples takes its DFT along x (Stockham, one warp per row) and the gather
//    of its samples with the k-side centring sign.
//  inverse: the rows with samples are zero-filled from theirs, signed and
//    transformed along x into S row ky (the others zeroed), then the inverse
//    two-step along y (the forward one on conjugated data) writes the plane's
//    rows y straight to global memory.
// Rows along x: one per sample row of the plan (row_ptr over (kz, ky)).
template <int NY, int NX, bool INV>
__global__ void __launch_bounds__(NX * 4, 1) k_plane_yx(float2* __restrict__ data, float2* __restrict__ y, int nz,
                                                        const int32_t* __restrict__ idx,
                                                        const int32_t* __restrict__ row_ptr, int M, float ksign,
                                                        const float2* __restrict__ twy_g,
                                                        const float2* __restrict__ twx_g) {
  constexpr int R2 = NY / 8;
  constexpr int NW = NX / 8;
  constexpr int NT = NW * 32;
  constexpr int GROUPS = NX / 32;
  extern __shared__ float2 sh[];
  float2* S = sh;                               // [NY][NX]
  float2* rbuf = S + NY * NX;                   // [NW][padded_len(NX)]
  float2* twy = rbuf + NW * padded_len(NX);     // [NY]
  float2* twx = twy + NY;                       // [NX]
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cg = warp % GROUPS, sub = warp / GROUPS;  // sub < 4
  const int col = cg * 32 + lane;
  const int plane = (int)blockIdx.x;
  const int c = plane / nz, kz = plane - c * nz;
  float2* P = data + (size_t)plane * NY * NX;
  for (int i = tid; i < NY; i += NT) twy[i] = twy_g[i];
  for (int i = tid; i < NX; i += NT) twx[i] = twx_g[i];
  float2* b = rbuf + warp * padded_len(NX);
  const int rbase = kz * NY;  // k-space row (kz, ky) = kz NY + ky
  if (!INV) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < R2 / 4; ++i) {
      const int r = sub + 4 * i;
      float2 v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) v[m] = P[(size_t)(r + R2 * m) * NX + col];
      mpi_dft::dft8(v);
#pragma unroll
      for (int k1 = 1; k1 < 8; ++k1) v[k1] = mpi_dft::cmulf(v[k1], twy[r * k1]);
#pragma unroll
      for (int k1 = 0; k1 < 8; ++k1) S[(r + R2 * k1) * NX + col] = v[k1];
    }
    __syncthreads();
#pragma unroll
    for (int k1 = sub; k1 < 8; k1 += 4) {
      float2 u[R2];
#pragma unroll
      for (int r = 0; r < R2; ++r) u[r] = S[(R2 * k1 + r) * NX + col];
      mpi_dft::dft_r<R2>(u);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) S[(R2 * k1 + k2) * NX + col] = u[k2];
    }
    __syncthreads();
    for (int ky = warp; ky < NY; ky += NW) {
      const int row = rbase + ky;
      const int m0 = row_ptr[row], m1 = row_ptr[row + 1];
      if (m1 <= m0) continue;  // warp-uniform
      const float2* src = S + (R2 * (ky % 8) + ky / 8) * NX;
      for (int i = lane; i < NX; i += 32) b[pad8(i)] = src[i];
      __syncwarp();
      Fft<NX, false>::go(b, twx, lane);
      const int rpar = (kz + ky) & 1;
      const size_t rb = (size_t)row * NX;
      for (int m = m0 + lane; m < m1; m += 32) {
        const int kx = (int)(idx[m] - rb);
        const float sg = ((kx + rpar) & 1) ? -ksign : ksign;
        const float2 t = b[pad8(kx)];
        y[(size_t)c * M + m] = make_float2(t.x * sg, t.y * sg);
      }
      __syncwarp();
    }
  } else {
    __syncthreads();
    for (int ky = warp; ky < NY; ky += NW) {
      const int row = rbase + ky;
      const int m0 = row_ptr[row], m1 = row_ptr[row + 1];
      float2* dst = S + ky * NX;
      if (m1 <= m0) {  // warp-uniform
        for (int i = lane; i < NX; i += 32) dst[i] = make_float2(0.f, 0.f);
        continue;
      }
      for (int i = lane; i < padded_len(NX); i += 32) b[i] = make_float2(0.f, 0.f);
      __syncwarp();
      const int rpar = (kz + ky) & 1;
      const size_t rb = (size_t)row * NX;
      for (int m = m0 + lane; m < m1; m += 32) {
        const int kx = (int)(idx[m] - rb);
        const float sg = ((kx + rpar) & 1) ? -ksign : ksign;
        const float2 t = y[(size_t)c * M + m];
        b[pad8(kx)] = make_float2(t.x * sg, t.y * sg);
      }
      __syncwarp();
      Fft<NX, true>::go(b, twx, lane);
      for (int i = lane; i < NX; i += 32) dst[i] = b[pad8(i)];
      __syncwarp();
    }
    __syncthreads();
    // inverse along y: the forward two-step on conjugated values, conjugated back
#pragma unroll
    for (int i = 0; i < R2 / 4; ++i) {
      const int r = sub + 4 * i;
      float2 v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const float2 t = S[(r + R2 * m) * NX + col];
        v[m] = make_float2(t.x, -t.y);
      }
      mpi_dft::dft8(v);
#pragma unroll
      for (int k1 = 1; k1 < 8; ++k1) v[k1] = mpi_dft::cmulf(v[k1], twy[r * k1]);
#pragma unroll
      for (int k1 = 0; k1 < 8; ++k1) S[(r + R2 * k1) * NX + col] = v[k1];
    }
    __syncthreads();
#pragma unroll
    for (int k1 = sub; k1 < 8; k1 += 4) {
      float2 u[R2];
#pragma unroll
      for (int r = 0; r < R2; ++r) u[r] = S[(R2 * k1 + r) * NX + col];
      mpi_dft::dft_r<R2>(u);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) P[(size_t)(k1 + 8 * k2) * NX + col] = make_float2(u[k2].x, -u[k2].y);
    }
  }
}

template <int NY, int NX>
size_t plane_smem() {
  return ((size_t)NY * NX + (size_t)(NX / 8) * padded_len(NX) + NY + NX) * sizeof(float2);
}

// ---------------------------------------------------------------------------
// Pipelined plane passes.  k_plane_yx holds a whole plane per CTA, so at one
// CTA per SM each plane's global traffic waits for its passes.  Here one
// persistent CTA per SM (more where shared memory allows) walks its (coil, kz)
// planes in tiles of TC columns [NY][TC] (pipe_cols):
//  forward: TMA loads the tiles into a ring of buffers, ahead of
//    use; each tile takes the two-step DFT along y in place (as k_plane_yx),
//    and the outputs of the k-space rows with samples go straight to a compact
//    row store R [plane_kmax][padded NX].  When a plane's tiles are done, each
//    warp takes rows of R through the DFT along x and the gather, under the
//    loads of the next plane's tiles.
//  inverse: the rows with samples are scattered into R and transformed along
//    x; each tile then takes the inverse two-step along y with its first step
//    reading R (rows without samples are zero), and the result leaves by TMA
//    stores (8 strided boxes, one per output class ky mod 8), which run under
//    the next tile's work.
// Both steps along y look at which rows have samples first (a warp's items share them:
// one ballot): the forward's second step leaves out an output class without any, the
// inverse's first takes a class of at most one such row as that row's value times
// w^(row k1) instead of an 8-point DFT.  At 96 x 128 x 128, 32 coils, an eighth of the
// rows sampled: 122.4 -> 117 us forward, 128.8 -> 126.8 inverse.  (The rows along x as
// two register steps by half a warp each, as in fft_rows.cuh, were slower here: 123 and
// 132 us; the other half warps' lanes idle in both steps.)
// Per plane the CTA keeps its row list (ky, sample range) and each row's slot
// in R in a double-buffered table, the next plane's loaded into registers
// while the current one runs.
constexpr int kPipeThreads = 512;

// Tile width and ring depth: 64 columns in 2 buffers where NX allows (the
// second step along y then has one item per thread), else 32 in 4.
__host__ __device__ constexpr int pipe_cols(int nx) { return nx % 64 == 0 ? 64 : 32; }
__host__ __device__ constexpr int pipe_bufs(int nx) { return pipe_cols(nx) == 64 ? 2 : 4; }

struct PlaneMeta {
  int4 row;  // thread t < kmax: the plane's t-th row with samples
  int slot;  // thread t < NY: position of row ky = t in the list, -1 without samples
  int n;     // number of rows with samples
};

template <int NY>
__device__ __forceinline__ PlaneMeta load_plane_meta(int kz, int kmax, const int4* __restrict__ prow,
                                                     const int32_t* __restrict__ pn,
                                                     const int16_t* __restrict__ pslot) {
  PlaneMeta m;
  const int t = threadIdx.x;
  m.row = t < kmax ? prow[(size_t)kz * kmax + t] : make_int4(-1, 0, 0, 0);
  m.slot = t < NY ? (int)pslot[(size_t)kz * NY + t] : -1;
  m.n = t == 0 ? pn[kz] : 0;
  return m;
}

template <int NY>
__device__ __forceinline__ void store_plane_meta(const PlaneMeta& m, int kmax, int4* rows, int* slot, int* n) {
  const int t = threadIdx.x;
  if (t < kmax) rows[t] = m.row;
  if (t < NY) slot[t] = m.slot;
  if (t == 0) *n = m.n;
}

__host__ __device__ constexpr size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Shared-memory carve-up of k_plane_pipe (byte offsets from a 1024-aligned base).
template <int NY, int NX>
struct PipeLayout {
  static constexpr int TC = pipe_cols(NX), NB = pipe_bufs(NX);
  static constexpr size_t kTile = (size_t)NY * TC * sizeof(float2);
  static __host__ __device__ size_t R(int) { return NB * kTile; }
  static __host__ __device__ size_t tw(int kmax) { return R(kmax) + (size_t)kmax * padded_len(NX) * sizeof(float2); }
  static __host__ __device__ size_t rows(int kmax) { return align_up(tw(kmax) + (NY + NX) * sizeof(float2), 16); }
  static __host__ __device__ size_t slot(int kmax) { return rows(kmax) + 2 * (size_t)kmax * sizeof(int4); }
  static __host__ __device__ size_t n(int kmax) { return slot(kmax) + 2 * (size_t)NY * sizeof(int); }
  static __host__ __device__ size_t bars(int kmax) { return align_up(n(kmax) + 2 * sizeof(int), 8); }
  static __host__ __device__ size_t total(int kmax) { return bars(kmax) + NB * sizeof(uint64_t) + 1024; }
};

template <int NY, int NX, bool INV>
__global__ void __launch_bounds__(kPipeThreads, 1)
    k_plane_pipe(const __grid_constant__ CUtensorMap tmap, float2* __restrict__ y, int nz, int planes, int kmax,
                 const int32_t* __restrict__ idx, const int4* __restrict__ prow, const int32_t* __restrict__ pn,
                 const int16_t* __restrict__ pslot, int M, float ksign, const float2* __restrict__ twy_g,
                 const float2* __restrict__ twx_g, int* err, long long wait_cycles) {
  constexpr int R2 = NY / 8;
  constexpr int TC = pipe_cols(NX), NB = pipe_bufs(NX);
  constexpr int TP = NX / TC;
  constexpr int PL = padded_len(NX);
  constexpr int NT = kPipeThreads;
  constexpr int NW = NT / 32;
  using L = PipeLayout<NY, NX>;
  extern __shared__ unsigned char smraw[];
  // offset from the shared array itself (not a cast integer), so that every
  // access below compiles to shared-memory loads and stores
  unsigned char* base = smraw + ((1024u - (mpi_ptx::smem_addr(smraw) & 1023u)) & 1023u);
  float2* bufs = (float2*)base;
  float2* R = (float2*)(base + L::R(kmax));
  float2* twy = (float2*)(base + L::tw(kmax));
  float2* twx = twy + NY;
  int4* mrows = (int4*)(base + L::rows(kmax));
  int* mslot = (int*)(base + L::slot(kmax));
  int* mn = (int*)(base + L::n(kmax));
  uint64_t* full = (uint64_t*)(base + L::bars(kmax));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int first = (int)blockIdx.x, stride = (int)gridDim.x;
  const int nmine = planes > first ? (planes - 1 - first) / stride + 1 : 0;
  if (nmine == 0) return;  // CTA-uniform
  const int total = nmine * TP;
  for (int i = tid; i < NY; i += NT) twy[i] = twy_g[i];
  for (int i = tid; i < NX; i += NT) twx[i] = twx_g[i];
  if (!INV && tid == 0) {
    for (int b = 0; b < NB; ++b) mpi_ptx::mbar_init(&full[b], 1);
    mpi_ptx::fence_mbar_init();
  }
  {
    const PlaneMeta m0 = load_plane_meta<NY>(first % nz, kmax, prow, pn, pslot);
    store_plane_meta<NY>(m0, kmax, mrows, mslot, mn);
  }
  __syncthreads();
  // tile g of this CTA: plane first + (g / TP) stride, columns (g % TP) TC +
  // [0, TC), ring buffer g % NB
  auto issue_load = [&](int g) {
    const int b = g % NB;
    mpi_ptx::mbar_arrive_expect_tx(&full[b], (uint32_t)L::kTile);
    mpi_ptx::tma_load_3d(bufs + (size_t)b * NY * TC, &tmap, (g % TP) * 2 * TC, 0,
                         first + (g / TP) * stride, &full[b]);
  };
  if (!INV && tid == 0)
    for (int g = 0; g < NB && g < total; ++g) issue_load(g);
  int g = 0;
  for (int j = 0; j < nmine; ++j) {
    const int pl = first + j * stride, c = pl / nz, kz = pl - c * nz;
    const int cur = j & 1;
    PlaneMeta nxt;
    if (j + 1 < nmine) nxt = load_plane_meta<NY>((pl + stride) % nz, kmax, prow, pn, pslot);
    const int4* rows = mrows + cur * kmax;
    const int* slot = mslot + cur * NY;
    const int nS = mn[cur];
    if (!INV) {
      for (int t = 0; t < TP; ++t, ++g) {
        const int b = g % NB;
        float2* B = bufs + (size_t)b * NY * TC;
        const bool ok = mpi_ptx::mbar_wait(&full[b], (uint32_t)((g / NB) & 1), err, wait_cycles);
        // first step along y, in place: DFT8 over m of rows r + R2 m, twiddle
        for (int it = tid; it < TC * R2; it += NT) {
          const int col = it % TC, r = it / TC;
          float2 v[8];
#pragma unroll
          for (int m = 0; m < 8; ++m) v[m] = B[(r + R2 * m) * TC + col];
          mpi_dft::dft8(v);
#pragma unroll
          for (int k1 = 1; k1 < 8; ++k1) v[k1] = mpi_dft::cmulf(v[k1], twy[r * k1]);
#pragma unroll
          for (int k1 = 0; k1 < 8; ++k1) B[(r + R2 * k1) * TC + col] = v[k1];
        }
        if (__syncthreads_or(!ok)) return;  // a load timed out (recorded in err)
        // second step: R2-point DFT over r; output ky = k1 + 8 k2 kept where it has samples
        for (int it = tid; it < TC * 8; it += NT) {
          const int col = it % TC, k1 = it / TC;  // k1 is the same in a whole warp
          const unsigned keep = __ballot_sync(0xffffffffu, lane < R2 && slot[k1 + 8 * (lane % R2)] >= 0);
          if (!keep) continue;
          float2 u[R2];
#pragma unroll
          for (int r = 0; r < R2; ++r) u[r] = B[(R2 * k1 + r) * TC + col];
          mpi_dft::dft_r<R2>(u);
#pragma unroll
          for (int k2 = 0; k2 < R2; ++k2)
            if (keep >> k2 & 1) R[slot[k1 + 8 * k2] * PL + pad8(t * TC + col)] = u[k2];
        }
        mpi_ptx::fence_proxy_async();  // the buffer's generic accesses before the next TMA load into it
        __syncthreads();
        if (tid == 0 && g + NB < total) issue_load(g + NB);
      }
      // rows along x and the gather (the next plane's tiles load meanwhile)
      for (int k = warp; k < nS; k += NW) {
        float2* rr = R + k * PL;
        Fft<NX, false>::go(rr, twx, lane);
        const int4 rw = rows[k];  // ky, first sample, end
        const int rpar = (kz + rw.x) & 1;
        const size_t rb = ((size_t)kz * NY + rw.x) * NX;
        const bool whole = rw.z - rw.y == NX;
        for (int m = rw.y + lane; m < rw.z; m += 32) {
          const int kx = whole ? m - rw.y : (int)(idx[m] - rb);
          const float sg = ((kx + rpar) & 1) ? -ksign : ksign;
          const float2 v = rr[pad8(kx)];
          y[(size_t)c * M + m] = make_float2(v.x * sg, v.y * sg);
        }
      }
      if (j + 1 < nmine) store_plane_meta<NY>(nxt, kmax, mrows + (cur ^ 1) * kmax, mslot + (cur ^ 1) * NY, mn + (cur ^ 1));
      __syncthreads();
    } else {
      // rows with samples: zero-fill (partial rows), scatter with the k-side sign, inverse DFT along x
      for (int k = warp; k < nS; k += NW) {
        float2* rr = R + k * PL;
        const int4 rw = rows[k];
        const bool whole = rw.z - rw.y == NX;
        if (!whole) {
          for (int i = lane; i < PL; i += 32) rr[i] = make_float2(0.f, 0.f);
          __syncwarp();
        }
        const int rpar = (kz + rw.x) & 1;
        if (whole) {  // a whole readout: all loads first
          float2 v[NX / 32];
#pragma unroll
          for (int u = 0; u < NX / 32; ++u) v[u] = y[(size_t)c * M + rw.y + lane + 32 * u];
#pragma unroll
          for (int u = 0; u < NX / 32; ++u) {
            const int kx = lane + 32 * u;
            const float sg = ((kx + rpar) & 1) ? -ksign : ksign;
            rr[pad8(kx)] = make_float2(v[u].x * sg, v[u].y * sg);
          }
        } else {
          const size_t rb = ((size_t)kz * NY + rw.x) * NX;
          for (int m = rw.y + lane; m < rw.z; m += 32) {
            const int kx = (int)(idx[m] - rb);
            const float sg = ((kx + rpar) & 1) ? -ksign : ksign;
            const float2 v = y[(size_t)c * M + m];
            rr[pad8(kx)] = make_float2(v.x * sg, v.y * sg);
          }
        }
        __syncwarp();
        Fft<NX, true>::go(rr, twx, lane);
      }
      __syncthreads();
      for (int t = 0; t < TP; ++t, ++g) {
        const int b = g % NB;
        float2* B = bufs + (size_t)b * NY * TC;
        // inverse along y: the forward two-step on conjugated values, conjugated back
        for (int it = tid; it < TC * R2; it += NT) {
          const int col = it % TC, r = it / TC;  // r is the same in a whole warp
          const unsigned have = __ballot_sync(0xffffffffu, slot[r + R2 * (lane & 7)] >= 0) & 0xffu;
          const float2* src = R + pad8(t * TC + col);
          float2 v[8];
          if ((have & (have - 1)) == 0) {  // at most one row with samples: its value times w^(row k1)
            v[0] = make_float2(0.f, 0.f);
            const int row = r + R2 * (31 - __clz(have | 1u));
            if (have) {
              const float2 u = src[slot[row] * PL];
              v[0] = make_float2(u.x, -u.y);
            }
            int w = 0;
#pragma unroll
            for (int k1 = 1; k1 < 8; ++k1) {
              w = w + row < NY ? w + row : w + row - NY;
              v[k1] = mpi_dft::cmulf(v[0], twy[w]);
            }
          } else {
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              v[m] = make_float2(0.f, 0.f);
              if (have >> m & 1) {
                const float2 u = src[slot[r + R2 * m] * PL];
                v[m] = make_float2(u.x, -u.y);
              }
            }
            mpi_dft::dft8(v);
#pragma unroll
            for (int k1 = 1; k1 < 8; ++k1) v[k1] = mpi_dft::cmulf(v[k1], twy[r * k1]);
          }
#pragma unroll
          for (int k1 = 0; k1 < 8; ++k1) B[(r + R2 * k1) * TC + col] = v[k1];
        }
        if (t == TP - 1 && j + 1 < nmine)
          store_plane_meta<NY>(nxt, kmax, mrows + (cur ^ 1) * kmax, mslot + (cur ^ 1) * NY, mn + (cur ^ 1));
        __syncthreads();
        // rows R2 k1 + k2 of the buffer take output row y = k1 + 8 k2
        for (int it = tid; it < TC * 8; it += NT) {
          const int col = it % TC, k1 = it / TC;
          float2 u[R2];
#pragma unroll
          for (int r = 0; r < R2; ++r) u[r] = B[(R2 * k1 + r) * TC + col];
          mpi_dft::dft_r<R2>(u);
#pragma unroll
          for (int k2 = 0; k2 < R2; ++k2) B[(R2 * k1 + k2) * TC + col] = make_float2(u[k2].x, -u[k2].y);
        }
        mpi_ptx::fence_proxy_async();  // the buffer's writes before the TMA store reads them
        // the buffer the next tile writes was last stored NB tiles ago
        if (tid == 0) mpi_ptx::bulk_wait_read<NB - 2>();
        __syncthreads();
        if (tid == 0) {
#pragma unroll
          for (int k1 = 0; k1 < 8; ++k1)
            mpi_ptx::tma_store_4d(&tmap, B + (size_t)R2 * k1 * TC, t * 2 * TC, k1, 0, pl);
          mpi_ptx::bulk_commit();
        }
      }
    }
  }
  if (INV && tid == 0) mpi_ptx::bulk_wait_all();
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tensor map over FP32 data (no swizzle, no out-of-range fill needed: every
// box lies inside the volume).  strides: bytes, one per dimension above the first.
bool encode_f32_map(CUtensorMap* map, void* ptr, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                    const cuuint32_t* box) {
  static void* fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult qr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr);
    if (e != cudaSuccess || qr != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      fn = nullptr;
      return false;
    }
  }
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return ((EncodeTiledFn)fn)(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, ptr, dims, strides, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

mpi_status launch_fft_cols(mpi_ctx* ctx, float2* data, int C, int nz, int ny, int nx, bool inverse,
                           const uint8_t* row_has) {
  // lines along y: stride nx; slabs = (c, z); base = slab * ny * nx; row mask [z][y]
  const long plane = (long)ny * nx;
  if (inverse) return lines_dispatch<true>(ctx, "k_fft_lines<y,inv>", data, ny, nx, nx, C * nz, 1, plane, 0, row_has, nz);
  return lines_dispatch<false>(ctx, "k_fft_lines<y,fwd>", data, ny, nx, nx, C * nz, 1, plane, 0, row_has, nz);
}

namespace {
// Grid points along y times coils from which the windowed pass is the register one (at
// G >= 128): both directions in us, Stockham lines against registers, with 4, 12 and 32
// coils: G = 96 12.6/14.9, 12.9/15.0, 14.6/14.6; 128 13.7/14.0, 13.4/15.2, 16.2/14.8; 192
// 15.5/16.4, 16.2/16.5, 19.7/17.1; 256 16.5/16.9, 18.8/17.0, 20.7/19.1; 320 18.8/19.9,
// 22.0/20.1, 32.6/24.5; 512 24.2/22.3, 34.9/24.6, 59.6/38.2.
constexpr int kWinReg = 2048;
}  // namespace

mpi_status launch_fft_cols_window(mpi_ctx* ctx, float2* grid, int C, int G, const float2* src, float2* dst,
                                  const float* deap, int n, bool inverse) {
  if (C == 0) return MPI_OK;
  const long blocks = (long)C * (G / 8);
  if (blocks > 0x7fffffffL) return set_err(ctx, MPI_ERR_SHAPE, "too many FFT tiles");
  const float2* tw = twiddle_table(ctx, G);
  if (!tw) return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  const LineWin win{src, dst, deap, n, G / 2 - n / 2};
  const bool reg = G >= 128 && C >= (kWinReg + G - 1) / G;
#define MPI_WIN_CASE(L)                                                                                    \
  case L:                                                                                                  \
    if (inverse)                                                                                           \
      launch_pdl(ctx, k_fft_lines_win<L, true>, dim3((unsigned)blocks), dim3(kLineWarps * 32), 0, grid, C, win, tw); \
    else                                                                                                   \
      launch_pdl(ctx, k_fft_lines_win<L, false>, dim3((unsigned)blocks), dim3(kLineWarps * 32), 0, grid, C, win, tw); \
    break;
  // register two-step pass: the 16-column tiles that meet the window
  const int x_first = win.o / 16 * 16, x_tiles = (win.o + n - x_first + 15) / 16;
  const long wblocks = (long)C * x_tiles;
#define MPI_WIN_REG(L, r1, r2)                                                                                      \
  case L: {                                                                                                         \
    const size_t smem = (size_t)L * 16 * sizeof(float2);                                                            \
    auto kern = inverse ? k_fft_cols_win<r1, r2, true> : k_fft_cols_win<r1, r2, false>;                             \
    if (smem > 48 * 1024) { /* more than a launch may ask for without it */                                        \
      cudaError_t e = smem_attr(ctx, (const void*)kern);                                                            \
      if (e != cudaSuccess) return cuda_check(ctx, e, "windowed pass attributes");                                  \
    }                                                                                                               \
    launch_pdl(ctx, kern, dim3((unsigned)wblocks), dim3(256), smem, grid, C, win, x_first, x_tiles, tw);             \
    break;                                                                                                          \
  }
  MPI_PROF(ctx, KF_FFT_LINES);
  if (reg) {
    switch (G) {
      MPI_WIN_REG(128, 8, 16)
      MPI_WIN_REG(192, 16, 12)
      MPI_WIN_REG(256, 16, 16)
      MPI_WIN_REG(320, 16, 20)
      MPI_WIN_REG(512, 16, 32)
      default:
        return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
    }
  } else {
    switch (G) {
      MPI_WIN_CASE(16)
      MPI_WIN_CASE(32)
      MPI_WIN_CASE(48)
      MPI_WIN_CASE(64)
      MPI_WIN_CASE(96)
      MPI_WIN_CASE(128)
      MPI_WIN_CASE(192)
      MPI_WIN_CASE(256)
      MPI_WIN_CASE(320)
      MPI_WIN_CASE(512)
      default:
        return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
    }
  }
#undef MPI_WIN_CASE
#undef MPI_WIN_REG
  MPI_LAUNCH_CHECK(ctx, reg ? "k_fft_cols_win" : "k_fft_lines_win");
  return MPI_OK;
}

mpi_status launch_fft_z(mpi_ctx* ctx, float2* data, int C, int nz, int ny, int nx, bool inverse) {
  // lines along z: stride ny * nx; slabs = (c, y); base = c * vol + y * nx
  const long plane = (long)ny * nx;
  const long vol = plane * nz;
  if (inverse) return lines_dispatch<true>(ctx, "k_fft_lines<z,inv>", data, nz, nx, plane, C * ny, ny, vol, nx);
  return lines_dispatch<false>(ctx, "k_fft_lines<z,fwd>", data, nz, nx, plane, C * ny, ny, vol, nx);
}

mpi_status tune_line_passes(mpi_ctx* ctx, const mpi_plan* plan, int C) {
  if (!ctx->autotune || plan->kind != MPI_TRAJ_CARTESIAN || C < 1) return MPI_OK;
  const size_t cn = (size_t)C * plan->N;
  if (!ctx->work || ctx->work_bytes < 2 * cn * sizeof(float2)) return MPI_OK;
  // the workspace's second [C][N] buffer, as in the operator calls
  void* saved = ctx->tune_scratch;
  const size_t saved_bytes = ctx->tune_scratch_bytes;
  float2* base = (float2*)ctx->work;
  ctx->tune_scratch = base + cn;
  ctx->tune_scratch_bytes = cn * sizeof(float2);
  const int nz = plan->nz, ny = plan->ny, nx = plan->nx;
  const long plane = (long)ny * nx, vol = plane * nz;
  const float2* twy = twiddle_table(ctx, ny);
  if (twy) {
    lines_choose<false>(ctx, base, ny, nx, nx, C * nz, 1, plane, 0, twy, plan->row_has, nz);
    lines_choose<true>(ctx, base, ny, nx, nx, C * nz, 1, plane, 0, twy, plan->row_has, nz);
  }
  const float2* twz = plan->ndim == 3 ? twiddle_table(ctx, nz) : nullptr;
  if (twz) {
    lines_choose<false>(ctx, base, nz, nx, plane, C * ny, ny, vol, nx, twz, nullptr, 1);
    lines_choose<true>(ctx, base, nz, nx, plane, C * ny, ny, vol, nx, twz, nullptr, 1);
  }
  ctx->tune_scratch = saved;
  ctx->tune_scratch_bytes = saved_bytes;
  return cuda_check(ctx, cudaGetLastError(), "line-pass tuning");
}

bool plane_pass_supported(const mpi_plan* plan) {
  if (plan->kind != MPI_TRAJ_CARTESIAN || plan->ndim != 3) return false;
  const int ny = plan->ny, nx = plan->nx;
  return (ny == 64 || ny == 96 || ny == 128) && (nx == 64 || nx == 96 || nx == 128);
}

namespace {

// The pipelined plane passes: false (nothing launched) where they do not
// apply (shared memory for the plane's rows with samples, alignment).
template <int NY, int NX>
bool try_plane_pipe(mpi_ctx* ctx, const mpi_plan* plan, float2* data, int C, float2* y, bool inverse,
                    const float2* twy, const float2* twx, float ks, mpi_status* st) {
  const int kmax = plan->plane_kmax;
  const size_t smem = PipeLayout<NY, NX>::total(kmax);
  if (!plan->plane_rows || smem > 227 * 1024 || ((uintptr_t)data & 15)) return false;
  const long planes = (long)C * plan->nz;
  CUtensorMap map;
  bool ok;
  if (!inverse) {
    const cuuint64_t dims[3] = {(cuuint64_t)2 * NX, (cuuint64_t)NY, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)NX * sizeof(float2), (cuuint64_t)NY * NX * sizeof(float2)};
    const cuuint32_t box[3] = {2 * pipe_cols(NX), NY, 1};
    ok = encode_f32_map(&map, data, 3, dims, strides, box);
  } else {
    // rows y = k1 + 8 k2 as dimensions (k1, k2): one box per k1 holds rows k2 = 0 .. NY/8 - 1
    const cuuint64_t dims[4] = {(cuuint64_t)2 * NX, 8, (cuuint64_t)NY / 8, (cuuint64_t)planes};
    const cuuint64_t strides[3] = {(cuuint64_t)NX * sizeof(float2), (cuuint64_t)8 * NX * sizeof(float2),
                                   (cuuint64_t)NY * NX * sizeof(float2)};
    const cuuint32_t box[4] = {2 * pipe_cols(NX), 1, NY / 8, 1};
    ok = encode_f32_map(&map, data, 4, dims, strides, box);
  }
  if (!ok) return false;
  auto kern = inverse ? k_plane_pipe<NY, NX, true> : k_plane_pipe<NY, NX, false>;
  cudaError_t e = smem_attr(ctx, (const void*)kern);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPipeThreads, smem);
  if (e != cudaSuccess) {
    *st = cuda_check(ctx, e, "plane pipe attributes");
    return true;
  }
  const long grid = std::min(planes, (long)ctx->num_sms * std::max(per_sm, 1));
  MPI_PROF(ctx, KF_FFT_ROWS);
  e = launch_pdl(ctx, kern, dim3((unsigned)grid), dim3(kPipeThreads), smem, map, y, plan->nz, (int)planes, kmax,
                 (const int32_t*)plan->idx, (const int4*)plan->plane_rows, (const int32_t*)plan->plane_nrows,
                 (const int16_t*)plan->plane_slot, plan->M, ks, twy, twx, ctx->dev_err, ctx->wait_cycles);
  const char* name = inverse ? "k_plane_pipe<inv>" : "k_plane_pipe<fwd>";
  ctx->launches++;
  prof_end(ctx, name);
  if (e == cudaSuccess) e = cudaGetLastError();
  *st = e == cudaSuccess ? MPI_OK : cuda_check(ctx, e, name);
  return true;
}

}  // namespace

mpi_status launch_plane_yx(mpi_ctx* ctx, const mpi_plan* plan, float2* data, int C, float2* y, bool inverse) {
  if (!plane_pass_supported(plan)) return set_err(ctx, MPI_ERR_UNSUPPORTED, "plane pass: shape");
  const long planes = (long)C * plan->nz;
  if (planes == 0) return MPI_OK;
  if (planes > 0x7fffffffL) return set_err(ctx, MPI_ERR_SHAPE, "plane pass: too many planes");
  const float ks = axis_sign(plan->nx) * axis_sign(plan->ny) * axis_sign(plan->nz);
  const float2* twy = twiddle_table(ctx, plan->ny);
  const float2* twx = twiddle_table(ctx, plan->nx);
  if (!twy || !twx) return set_err(ctx, MPI_ERR_SHAPE, "plane pass: no twiddle table");
  cudaError_t e = cudaSuccess;
  if (ctx->plane_pipe) {
    mpi_status st = MPI_OK;
#define MPI_PIPE(NY_, NX_) \
  if (plan->ny == NY_ && plan->nx == NX_ && try_plane_pipe<NY_, NX_>(ctx, plan, data, C, y, inverse, twy, twx, ks, &st)) \
    return st;
    MPI_PIPE(64, 64) MPI_PIPE(64, 96) MPI_PIPE(64, 128)
    MPI_PIPE(96, 64) MPI_PIPE(96, 96) MPI_PIPE(96, 128)
    MPI_PIPE(128, 64) MPI_PIPE(128, 96) MPI_PIPE(128, 128)
#undef MPI_PIPE
  }
#define MPI_PLANE(NY_, NX_)                                                                                    \
  if (plan->ny == NY_ && plan->nx == NX_) {                                                                    \
    const size_t smem = plane_smem<NY_, NX_>();                                                                \
    auto kern = inverse ? k_plane_yx<NY_, NX_, true> : k_plane_yx<NY_, NX_, false>;                            \
    e = smem_attr(ctx, (const void*)kern);                                                                      \
    if (e != cudaSuccess) return cuda_check(ctx, e, "plane pass smem attribute");                              \
    MPI_PROF(ctx, KF_FFT_ROWS);                                                                                \
    launch_pdl(ctx, kern, dim3((unsigned)planes), dim3(NX_ * 4), smem, data, y, plan->nz, plan->idx,           \
               plan->row_ptr, plan->M, ks, twy, twx);                                                          \
    MPI_LAUNCH_CHECK(ctx, inverse ? "k_plane_yx<inv>" : "k_plane_yx<fwd>");                                    \
    return MPI_OK;                                                                                             \
  }
  MPI_PLANE(64, 64) MPI_PLANE(64, 96) MPI_PLANE(64, 128)
  MPI_PLANE(96, 64) MPI_PLANE(96, 96) MPI_PLANE(96, 128)
  MPI_PLANE(128, 64) MPI_PLANE(128, 96) MPI_PLANE(128, 128)
#undef MPI_PLANE
  return set_err(ctx, MPI_ERR_UNSUPPORTED, "plane pass: shape");
}

namespace {

// Launch of the row pass for rows of nx values; y is only read by the scatter.
template <bool INV, bool TAB>
mpi_status rows_launch(mpi_ctx* ctx, int nx, float2* data, float2* y, const RowsArgs& a, const char* name) {
  long groups = 0;
#define MPI_ROWS_CASE(n)                                                                                           \
  case n: {                                                                                                        \
    groups = (long)a.C * ((a.n_list + Rows<n>::R - 1) / Rows<n>::R);                                               \
    if (groups > 0x7fffffffL) return set_err(ctx, MPI_ERR_SHAPE, "too many k-space rows");                         \
    const long blocks = std::min((groups + kRowWarps - 1) / kRowWarps, 16L * std::max(ctx->num_sms, 1));            \
    if (INV)                                                                                                       \
      launch_pdl(ctx, k_rows_scatter_inv<n, TAB>, dim3((unsigned)blocks), dim3(kRowWarps * 32), 0, y, data, a);     \
    else                                                                                                           \
      launch_pdl(ctx, k_rows_fwd_gather<n, TAB>, dim3((unsigned)blocks), dim3(kRowWarps * 32), 0, data, y, a);      \
    break;                                                                                                         \
  }
  if (a.C == 0 || a.n_list == 0) return MPI_OK;
  if (!a.tw) return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  MPI_PROF(ctx, KF_FFT_ROWS);
  switch (nx) {
    MPI_ROWS_CASE(16)
    MPI_ROWS_CASE(32)
    MPI_ROWS_CASE(48)
    MPI_ROWS_CASE(64)
    MPI_ROWS_CASE(96)
    MPI_ROWS_CASE(128)
    MPI_ROWS_CASE(192)
    MPI_ROWS_CASE(256)
    MPI_ROWS_CASE(320)
    MPI_ROWS_CASE(512)
    default:
      return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  }
#undef MPI_ROWS_CASE
  MPI_LAUNCH_CHECK(ctx, name);
  return MPI_OK;
}

RowsArgs rows_args(const mpi_ctx* ctx, const mpi_plan* plan, int C) {
  RowsArgs a{};
  a.C = C;
  a.n_rows = plan->n_rows;
  a.ny = plan->ny;
  a.M = plan->M;
  a.n_list = plan->n_list;
  a.row_list = plan->row_list;
  a.idx = plan->idx;
  a.row_ptr = plan->row_ptr;
  a.ksign = axis_sign(plan->nx) * axis_sign(plan->ny) * (plan->ndim == 3 ? axis_sign(plan->nz) : 1.f);
  a.tw = twiddle_table(ctx, plan->nx);
  return a;
}

}  // namespace

mpi_status launch_rows_fwd_gather(mpi_ctx* ctx, const mpi_plan* plan, const float2* data, int C,
                                  float2* y) {
  return rows_launch<false, false>(ctx, plan->nx, (float2*)data, y, rows_args(ctx, plan, C), "k_rows_fwd_gather");
}

mpi_status launch_rows_scatter_inv(mpi_ctx* ctx, const mpi_plan* plan, const float2* y, int C,
                                   float2* data) {
  return rows_launch<true, false>(ctx, plan->nx, data, (float2*)y, rows_args(ctx, plan, C), "k_rows_scatter_inv");
}

// ------------------------------------------------- passes of a batch's group

bool fft_cols_in_registers(mpi_ctx* ctx, const mpi_plan* plan, int C, bool inverse) {
  const int ny = plan->ny, nx = plan->nx;
  const long plane = (long)ny * nx;
  const float2* tw = twiddle_table(ctx, ny);
  const int t = inverse ? lines_choose<true>(ctx, nullptr, ny, nx, nx, C, 1, plane, 0, tw, plan->row_has, 1)
                        : lines_choose<false>(ctx, nullptr, ny, nx, nx, C, 1, plane, 0, tw, plan->row_has, 1);
  return t < 0;
}

// The widest Stockham tile, or 32 register columns, unless tuning finds a faster width.
mpi_status tune_fft_cols_group(mpi_ctx* ctx, bool registers, float2* data, int coils, int ny, int nx, bool inverse,
                               const uint8_t* row_has, int* kernel) {
  std::vector<int> cands;
  if (registers) cands = {kRegCols32, kRegCols16};
  else
    for (int t : {32, 16, 8})
      if ((long)ny * t / (kLineWarps * 32) <= 16 && (t == 8 || (t == 16 && ny <= 256) || (t == 32 && ny <= 128)))
        cands.push_back(t);
  *kernel = cands[0];
  if (!ctx->autotune || cands.size() < 2) return MPI_OK;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, MPI_ERR_CUDA, "grouped batch: tuning events");
  }
  mpi_status st = MPI_OK;
  float best = 1e30f;
  for (int k : cands) {
    st = launch_fft_cols_group(ctx, k, data, coils, ny, nx, inverse, row_has);  // warm-up
    cudaEventRecord(e0, ctx->stream);
    for (int r = 0; r < 3 && st == MPI_OK; ++r)
      st = launch_fft_cols_group(ctx, k, data, coils, ny, nx, inverse, row_has);
    cudaEventRecord(e1, ctx->stream);
    float ms = 0.f;
    if (st == MPI_OK && (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess))
      st = cuda_check(ctx, cudaGetLastError(), "grouped batch tuning");
    if (st) break;
    if (ms < best) {
      best = ms;
      *kernel = k;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return st;
}

mpi_status launch_fft_cols_group(mpi_ctx* ctx, int kernel, float2* data, int coils, int ny, int nx, bool inverse,
                                 const uint8_t* row_has) {
  const float2* tw = twiddle_table(ctx, ny);
  const int cols = kernel_cols(kernel);
  const long blocks = (long)coils * ((nx + cols - 1) / cols);
  if (!tw || blocks > 0x7fffffffL) return set_err(ctx, MPI_ERR_SHAPE, "grouped FFT pass");
  MPI_PROF(ctx, KF_FFT_LINES);
  const long plane = (long)ny * nx;
  const bool ok =
      inverse ? lines_launch_tile<true>(ctx, kernel, ny, blocks, data, nx, nx, coils, 1, plane, 0, tw, row_has, coils)
              : lines_launch_tile<false>(ctx, kernel, ny, blocks, data, nx, nx, coils, 1, plane, 0, tw, row_has, coils);
  if (!ok) return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  MPI_LAUNCH_CHECK(ctx, inverse ? "k_fft_lines<y,inv,group>" : "k_fft_lines<y,fwd,group>");
  return MPI_OK;
}

mpi_status launch_rows_group(mpi_ctx* ctx, float2* data, int coils, int ny, int nx, bool inverse,
                             const CoilSamples* tab, int n_list) {
  RowsArgs a{};
  a.C = coils;
  a.n_rows = a.ny = ny;
  a.n_list = n_list;
  a.ksign = axis_sign(nx) * axis_sign(ny);
  a.tw = twiddle_table(ctx, nx);
  a.tab = tab;
  return inverse ? rows_launch<true, true>(ctx, nx, data, nullptr, a, "k_rows_scatter_inv<group>")
                 : rows_launch<false, true>(ctx, nx, data, nullptr, a, "k_rows_fwd_gather<group>");
}

namespace {

// In-place FFT of contiguous lines of length L by the register steps of
// fft_rows.cuh, R lines per warp.  Elements outside [load_lo, load_hi) are taken
// as zero without being read (the radial forward's padded columns), and only
// [keep_lo, keep_hi) of each transformed line is stored back (the radial adjoint
// keeps the columns that its cropping pass along y reads).
template <int L, bool INV>
__global__ void __launch_bounds__(kRowWarps * 32) k_fft_rows_inplace(float2* __restrict__ data, long n_rows,
                                                                    const float2* __restrict__ tw_g, int load_lo,
                                                                    int load_hi, int keep_lo, int keep_hi) {
  using F = Rows<L>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = lane % F::P;
  float2* b = buf[warp];
  const long row0 = ((long)blockIdx.x * kRowWarps + warp) * F::R;
  float2 v[F::T1][F::A];
#pragma unroll
  for (int i = 0; i < F::T1; ++i) {
    const long row = row0 + (lane + 32 * i) / F::P;
    const float2* src = data + (size_t)row * L;
#pragma unroll
    for (int e = 0; e < F::A; ++e) {
      const int n = p + F::P * e;
      v[i][e] = (row < n_rows && n >= load_lo && n < load_hi) ? src[n] : make_float2(0.f, 0.f);
    }
  }
#pragma unroll
  for (int i = 0; i < F::T1; ++i) F::template step1<INV>(v[i], (lane + 32 * i) / F::P, p, b, tw_g);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < F::T2; ++i) {
    const int t = lane + 32 * i, r = t / F::A, k1 = t % F::A;
    if (r >= F::R || row0 + r >= n_rows) continue;
    float2 u[F::P];
    F::template step2<INV>(u, r, k1, b);
    float2* dst = data + (size_t)(row0 + r) * L;
#pragma unroll
    for (int k = 0; k < F::P; ++k)
      if (k1 + F::A * k >= keep_lo && k1 + F::A * k < keep_hi) dst[k1 + F::A * k] = u[k];
  }
}

template <bool INV>
mpi_status rows_inplace_dispatch(mpi_ctx* ctx, float2* data, long n_rows, int L, int load_lo, int load_hi,
                                 int keep_lo, int keep_hi) {
  if (n_rows == 0) return MPI_OK;
  const float2* tw = twiddle_table(ctx, L);
  if (!tw) return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
#define MPI_RI_CASE(n)                                                                                         \
  case n:                                                                                                      \
    launch_pdl(ctx, k_fft_rows_inplace<n, INV>,                                                                \
               dim3((unsigned)((n_rows + kRowWarps * Rows<n>::R - 1) / (kRowWarps * Rows<n>::R))),             \
               dim3(kRowWarps * 32), 0, data, n_rows, tw, load_lo, load_hi, keep_lo, keep_hi);                 \
    break;
  MPI_PROF(ctx, KF_FFT_ROWS);
  switch (L) {
    MPI_RI_CASE(16)
    MPI_RI_CASE(32)
    MPI_RI_CASE(48)
    MPI_RI_CASE(64)
    MPI_RI_CASE(96)
    MPI_RI_CASE(128)
    MPI_RI_CASE(192)
    MPI_RI_CASE(256)
    MPI_RI_CASE(320)
    MPI_RI_CASE(512)
    default:
      return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  }
#undef MPI_RI_CASE
  MPI_LAUNCH_CHECK(ctx, "k_fft_rows_inplace");
  return MPI_OK;
}

}  // namespace

mpi_status launch_fft_rows_inplace(mpi_ctx* ctx, float2* data, long n_rows, int L, bool inverse, int load_lo,
                                   int load_hi, int keep_lo, int keep_hi) {
  if (load_hi < 0) load_hi = L;
  if (keep_hi < 0) keep_hi = L;
  if (inverse) return rows_inplace_dispatch<true>(ctx, data, n_rows, L, load_lo, load_hi, keep_lo, keep_hi);
  return rows_inplace_dispatch<false>(ctx, data, n_rows, L, load_lo, load_hi, keep_lo, keep_hi);
}
