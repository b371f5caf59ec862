// MPI-L (scaled ADMM, Eqs. 8-11) on 2D Cartesian grids with a dense basis, one
// slice or several frames that share the maps: the solve's passes fused.
//
// The coefficients alpha are fixed for a solve, so its maps s_k = U alpha_k are
// expanded once, by the same expansion the operator calls run, and every operator
// of the solve multiplies by them: C N complex values (8.4 MB at 256^2 and 16
// coils, which stay in L2) instead of the basis (67 MB) per application.  What is
// left of an operator are FFT passes over C N values, a few microseconds each, so
// the point-wise steps and the sums live in those passes:
//   k_maps_cols<fwd>    v = s p (sign, scale) formed on load, DFT along y; in the
//                       CG the new direction d = r + beta d is formed there too
//   k_rows_normal       DFT along x, sampling mask, inverse DFT along x (the
//                       normal operator never leaves k-space rows); not run where
//                       every row is sampled whole or not at all, since it is
//                       then a multiplication by nx
//   k_maps_cols<inv>    inverse DFT along y, times conj(s) on store
//   k_coil_sum          sum over coils, + d, and the CG's <d, A d>
//   k_cg_update         x, r, |r|^2
// and an outer step adds the norms of the ball projection (k_ball_norm), the
// projection inside the scatter of the k-space rows (k_rows_scatter_ball), the dual
// update of the data blocks and their residual norms inside the gather
// (k_rows_gather_dual) and the image's dual update with the choice of rho
// (k_admm_dual).
//   The CG starts from the previous p, whose F_s S p is at hand (Apk), so its first
// residual is one adjoint:  r = S^H F_s^H (z_k - u_k - F_s S p) + z_0 - u_0 - p.
//   rho's rescaling of the scaled duals is applied where they are read (ufac).
//   Reductions: partial sums per CTA, added in a fixed order by the kernels that use
// them, so results do not depend on the order the CTAs run in.
// At 256^2, 16 coils, q = 128 an outer step (5 CG, 10 TV iterations) went from 725
// to 195 us, in 33 launches instead of 124.
#include <math.h>

#include <algorithm>
#include <vector>

#include "admm.h"
#include "dft_reg.cuh"
#include "fft_rows.cuh"
#include "fft_tile.cuh"
#include "ptx.cuh"

namespace {

using namespace mpi_fft;

constexpr int kThreads = 256;      // column and reduction kernels
constexpr int kElemThreads = 256;  // element-wise kernels
constexpr int kMaxElemBlocks = 512;  // also the partial sums that a consumer adds
constexpr int kBallBlocks = 8;     // CTAs per coil of the ball norms

// device scalars
enum { S_RHO = 0, S_UFAC, S_NUM };

// ------------------------------------------------------------- reductions
//
// Sums are software floats of 58-bit mantissas with exponents of their own (Sum: v 2^e),
// from the threads to the partial sums.  They are no less accurate than the FP64 sums of
// the solve on the operator calls (errors of random dot products, and of sums of squared
// differences of two and three terms, 0.06 to 0.6 of FP64's), and their range has no end,
// where squares of FP32 values leave FP32's long before the values do: maps of magnitude
// s make <d, A d> grow as s^4.  FP64 itself runs at two operations per clock and SM here:
// an outer step at 256^2 and 16 coils took 290 us with it, 219 with pairs of FP32 values
// (48 bits, FP32's range) and 225 this way (all with passes started early, see
// admm_maps_record).

struct alignas(16) Sum {
  long long v;  // |v| < 2^58
  int e;
};
constexpr int kEmpty = -(1 << 22), kNotFinite = 1 << 24;  // exponents of zero, and of an infinity or NaN

__device__ __forceinline__ Sum sum_zero() { return Sum{0, kEmpty}; }
__device__ __forceinline__ bool not_finite(Sum s) { return s.e >= kNotFinite / 2; }

// |x| = m 2^e with m's leading bit at bit 23 (zero: m = 0)
__device__ __forceinline__ void float_parts(float x, unsigned& m, int& e) {
  const unsigned b = __float_as_uint(x) & 0x7fffffffu;
  m = (b & 0x7fffffu) | 0x800000u;
  e = (int)(b >> 23) - 150;
  if (b - 0x00800000u >= 0x7f000000u) {  // zero, subnormal, infinite or NaN
    const int n = __clz(b) - 8;
    m = b >= 0x7f800000u ? 0x800000u : (b ? b << n : 0u);
    e = b >= 0x7f800000u ? kNotFinite : (b ? -149 - n : kEmpty);
  }
}
// v with the sign of x y
__device__ __forceinline__ long long signed_by(long long v, float x, float y = 0.f) {
  return (int)(__float_as_uint(x) ^ __float_as_uint(y)) < 0 ? -v : v;
}
__device__ __forceinline__ long long shift_down(long long v, int n) { return v >> min(n, 63); }

__device__ __forceinline__ Sum sum_add(Sum a, Sum b) {
  const int e = max(a.e, b.e);
  const long long v = shift_down(a.v, e - a.e) + shift_down(b.v, e - b.e);
  const int over = (int)((unsigned long long)(v + (1LL << 58)) >> 59) & 1;  // |v| reached 2^58
  return Sum{v >> over, e + over};
}

// Re(conj(a) b); the products' leading bit is bit 55 or 56
__device__ __forceinline__ Sum sum_dot(float2 a, float2 b) {
  unsigned m[4];
  int e[4];
  float_parts(a.x, m[0], e[0]);
  float_parts(b.x, m[1], e[1]);
  float_parts(a.y, m[2], e[2]);
  float_parts(b.y, m[3], e[3]);
  const long long px = signed_by((long long)((unsigned long long)m[0] * m[1] << 9), a.x, b.x);
  const long long py = signed_by((long long)((unsigned long long)m[2] * m[3] << 9), a.y, b.y);
  const int ex = e[0] + e[1] - 9, ey = e[2] + e[3] - 9, ec = max(ex, ey);
  return Sum{shift_down(px, ec - ex) + shift_down(py, ec - ey), ec};
}

// d + e = a - b exactly (no overflow)
__device__ __forceinline__ float diff_exact(float a, float b, float& e) {
  const float d = a - b, t = d - a;
  e = (a - (d - t)) - (b + t);
  return d;
}

// (d + c + b)^2, |c| and |b| at most about half a unit in the last place of d
__device__ __forceinline__ Sum sum_sq(float d, float c, float b = 0.f) {
  unsigned md, m;
  int ed, e;
  float_parts(d, md, ed);
  long long v = signed_by((long long)md << 34, d);
  if (c != 0.f) {  // mostly not: differences of values within a factor of two are exact
    float_parts(c, m, e);
    v += signed_by(shift_down((long long)m << 34, ed - e), c);
  }
  if (b != 0.f) {
    float_parts(b, m, e);
    v += signed_by(shift_down((long long)m << 34, ed - e), b);
  }
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v) << 5;  // leading bit 61 to 63
  return Sum{(long long)(__umul64hi(u, u) >> 5), 2 * (ed - 39) + 69};
}

// |a - b|^2
__device__ __forceinline__ Sum sum_diff_sq(float2 a, float2 b) {
  float cx, cy;
  const float dx = diff_exact(a.x, b.x, cx), dy = diff_exact(a.y, b.y, cy);
  return sum_add(sum_sq(dx, cx), sum_sq(dy, cy));
}

// (a + b - c)^2
__device__ __forceinline__ Sum sum_diff3_sq(float a, float b, float c) {
  float c1, c2, c3;
  float d = diff_exact(a, -b, c1);
  d = diff_exact(d, c, c2);
  d = diff_exact(d, -c1, c3);  // d + c3 + c2; where the second difference cancels, c2 = 0
  return sum_sq(d, c3, c2);
}

// Sum of v over a warp, |v| < 2^58 (the same value in every lane).
__device__ __forceinline__ long long warp_add(long long v) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x7ffffffu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 27) & 0x7ffffffu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 54));
  return ((long long)hi << 54) + ((long long)mid << 27) + lo;
}
__device__ __forceinline__ Sum warp_sum(Sum s) {
  const int e = __reduce_max_sync(0xffffffffu, s.e);
  const long long v = warp_add(shift_down(s.v, e - s.e));  // below 2^63
  const unsigned long long u = v < 0 ? -(unsigned long long)v : (unsigned long long)v;
  const int n = max(6 - __clzll(u), 0);
  return Sum{v >> n, e + n};
}

// out[j] = the sum of v[j] over the CTA's NT threads, by lane 0 of warp j; sh holds
// NV x NT / 32 values.
template <int NV, int NT>
__device__ __forceinline__ void block_sums(const Sum (&v)[NV], Sum* sh, Sum* out) {
  constexpr int NW = NT / 32;
  static_assert(NV <= NW && NW <= 32, "a warp per sum");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    const Sum w = warp_sum(v[j]);
    if (lane == 0) sh[j * NW + warp] = w;
  }
  __syncthreads();
  if (warp < NV) {
    const Sum w = warp_sum(lane < NW ? sh[warp * NW + lane] : sum_zero());
    if (lane == 0) out[warp] = w;
  }
}

// The sum of n <= kMaxElemBlocks partial sums, by one warp in a fixed order (valid in
// every lane; |v| < 2^63): the kernels that use a reduction's result add its CTAs'
// partial sums themselves, which is faster than having the last CTA of the reduction do
// it (its fence, counter and second round trip were 3 us at the end of every such kernel).
__device__ __forceinline__ Sum partial_sum(const Sum* __restrict__ part, int n) {
  constexpr int PER = kMaxElemBlocks / 32;
  static_assert(PER <= 16, "four bits of headroom in a lane");
  Sum s[PER];
  int e = kEmpty;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = (threadIdx.x & 31) + 32 * j;
    s[j] = i < n ? part[i] : sum_zero();
    e = max(e, s[j].e);
  }
  e = __reduce_max_sync(0xffffffffu, e) + 4;
  long long v = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) v += shift_down(s[j].v, e - s[j].e);
  return Sum{warp_add(v), e};
}

// 2^e, e within FP64's normal range
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + min(max(e, -1022), 1023)) << 20, 0); }
__device__ __forceinline__ double to_double(Sum s) {
  if (not_finite(s)) return __longlong_as_double(0x7ff8000000000000LL);
  return (double)s.v * pow2(s.e);  // sums of squares of FP32 values: within FP64's range
}

// a / b, 0 unless b > 0
__device__ __forceinline__ float sum_ratio(Sum a, Sum b) {
  if (b.v <= 0 || not_finite(b)) return 0.f;
  return (float)(to_double(a) / to_double(b));
}

// ------------------------------------------------------------ column passes

struct MapsCols {
  float2* W;            // [T][C][N]
  const float2* S;      // maps [C][N]
  const float2* v;      // forward: image [T][N], or the CG's old direction
  const float2* r;      // forward, next CG direction d = r + beta d_old (null: v itself)
  float2* dnew;         // where that direction goes
  const Sum *rr, *rr_old;  // partial sums of |r|^2, now and before the last update: beta = rr / rr_old
  int n_part;
  int C, nx;
  size_t N;
  float scale;
  const uint8_t* rmask;  // [T][ny]: 1 where the k-space row has samples
  const float2* tw;
};

template <int L>
struct RegSplit {
  static constexpr int R1 = 0, R2 = 0;
};
template <> struct RegSplit<64> { static constexpr int R1 = 8, R2 = 8; };
template <> struct RegSplit<96> { static constexpr int R1 = 8, R2 = 12; };
template <> struct RegSplit<128> { static constexpr int R1 = 8, R2 = 16; };
template <> struct RegSplit<192> { static constexpr int R1 = 16, R2 = 12; };
template <> struct RegSplit<256> { static constexpr int R1 = 16, R2 = 16; };
template <> struct RegSplit<320> { static constexpr int R1 = 16, R2 = 20; };

constexpr int maps_cols_tile(int L) {
  return (L == 64 || L == 96 || L == 128 || L == 192 || L == 256 || L == 320) ? 16 : 8;
}

// R values of one thread: rows y0 + step m of column x, formed from the image and
// the map (forward) or read from the rows with samples (inverse).  All loads are
// issued before the first use or store: a CTA has 8 warps and there are only
// T C nx / 16 of them, so what a thread has in flight sets the time (the loads in
// turn, with the store of the new direction between them: 30 us per pass at
// 256^2 and 16 coils; batched: see the file header).
template <int R, bool INV>
__device__ __forceinline__ void maps_load(const MapsCols& a, float beta, int t, int c, int tc, int y0, int step,
                                          int x, int L, float2 (&u)[R]) {
  const size_t n0 = (size_t)y0 * a.nx + x, ns = (size_t)step * a.nx;
  if (INV) {
    const float2* W = a.W + (size_t)tc * a.N + n0;
    const uint8_t* rm = a.rmask + (size_t)t * L + y0;
    uint8_t keep[R];
#pragma unroll
    for (int m = 0; m < R; ++m) keep[m] = rm[step * m];
#pragma unroll
    for (int m = 0; m < R; ++m) u[m] = keep[m] ? W[ns * m] : make_float2(0.f, 0.f);
    return;
  }
  const float2* S = a.S + (size_t)c * a.N + n0;
  const float2* v = a.v + (size_t)t * a.N + n0;
  float2 s[R];
#pragma unroll
  for (int m = 0; m < R; ++m) u[m] = v[ns * m];
#pragma unroll
  for (int m = 0; m < R; ++m) s[m] = S[ns * m];
  if (a.r) {  // the CG's next direction, kept by the first coil's CTAs
    const float2* r = a.r + (size_t)t * a.N + n0;
    float2 rv[R];
#pragma unroll
    for (int m = 0; m < R; ++m) rv[m] = r[ns * m];
#pragma unroll
    for (int m = 0; m < R; ++m) u[m] = make_float2(fmaf(beta, u[m].x, rv[m].x), fmaf(beta, u[m].y, rv[m].y));
    if (c == 0) {
      float2* d = a.dnew + (size_t)t * a.N + n0;
#pragma unroll
      for (int m = 0; m < R; ++m) d[ns * m] = u[m];
    }
  }
#pragma unroll
  for (int m = 0; m < R; ++m) {
    const float2 e = cmul(s[m], u[m]);
    const float sg = ((x + y0 + step * m) & 1) ? -a.scale : a.scale;
    u[m] = make_float2(e.x * sg, e.y * sg);
  }
}

// The R transformed values of rows y0 + step m: forward, to the rows with samples;
// inverse, times conj(s) (the maps `s` loaded ahead by the caller).
template <int R, bool INV>
__device__ __forceinline__ void maps_store(const MapsCols& a, int t, int tc, int y0, int step, int x, int L,
                                           const float2 (&u)[R], const float2 (&s)[R]) {
  float2* W = a.W + (size_t)tc * a.N + (size_t)y0 * a.nx + x;
  const size_t ns = (size_t)step * a.nx;
  const uint8_t* rm = a.rmask + (size_t)t * L + y0;
#pragma unroll
  for (int m = 0; m < R; ++m) {
    if (INV)
      W[ns * m] = make_float2(s[m].x * u[m].x + s[m].y * u[m].y, s[m].x * u[m].y - s[m].y * u[m].x);
    else if (rm[step * m])
      W[ns * m] = u[m];
  }
}

template <int R>
__device__ __forceinline__ void maps_prefetch(const MapsCols& a, int c, int y0, int step, int x, float2 (&s)[R]) {
  const float2* S = a.S + (size_t)c * a.N + (size_t)y0 * a.nx + x;
  const size_t ns = (size_t)step * a.nx;
#pragma unroll
  for (int m = 0; m < R; ++m) s[m] = S[ns * m];
}

// The pass along y of one (frame, coil) and a tile of adjacent columns, with the
// products by the maps: the register two-step FFT (see k_fft_cols_reg) for lengths
// that have a split, else Stockham lines in shared memory.
template <int L, bool INV>
__global__ void __launch_bounds__(kThreads) k_maps_cols(MapsCols a) {
  constexpr int R1 = RegSplit<L>::R1, R2 = RegSplit<L>::R2;
  constexpr int TILE = maps_cols_tile(L);
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int x_tiles = (a.nx + TILE - 1) / TILE;
  const int tc = (int)blockIdx.x / x_tiles, x0 = ((int)blockIdx.x - tc * x_tiles) * TILE;
  const int t = tc / a.C, c = tc - t * a.C;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float beta = 0.f;
  if (!INV && a.r) {  // a warp each for the two sums (both by one: 2 us more per outer step)
    __shared__ Sum s_rr[2];
    __shared__ float s_beta;
    if (w < 2) {
      const Sum sum = partial_sum(w ? a.rr_old : a.rr, a.n_part);
      if (lane == 0) s_rr[w] = sum;
    }
    __syncthreads();
    if (tid == 0) s_beta = sum_ratio(s_rr[0], s_rr[1]);
    __syncthreads();
    beta = s_beta;
  }
  if constexpr (R1 > 0) {
    constexpr int G = kThreads / TILE;  // rows r (step 1) or k1 (step 2) at a time
    __shared__ float2 sY[L * TILE];     // [k1][r][column]
    const int ci = tid % TILE, g = tid / TILE, x = x0 + ci;
    const bool ok = x < a.nx;
    float2 u1[(R2 + G - 1) / G][R1];
#pragma unroll
    for (int it = 0; it < (R2 + G - 1) / G; ++it) {
      const int q = g + G * it;
      if (ok && q < R2) maps_load<R1, INV>(a, beta, t, c, tc, q, R2, x, L, u1[it]);
    }
#pragma unroll
    for (int it = 0; it < (R2 + G - 1) / G; ++it) {
      const int q = g + G * it;
      if (q >= R2) break;
      float2 (&u)[R1] = u1[it];
      float2 tw[R1];
#pragma unroll
      for (int k1 = 1; k1 < R1; ++k1) tw[k1] = __ldg(a.tw + q * k1);
      if (INV)  // the inverse on conjugated values
#pragma unroll
        for (int m = 0; m < R1; ++m) u[m].y = -u[m].y;
      mpi_dft::dft_r<R1>(u);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) sY[(k1 * R2 + q) * TILE + ci] = k1 ? mpi_dft::cmulf(u[k1], tw[k1]) : u[0];
    }
    float2 s[(R1 + G - 1) / G][R2];
    if (INV)
#pragma unroll
      for (int it = 0; it < (R1 + G - 1) / G; ++it)
        if (ok && g + G * it < R1) maps_prefetch<R2>(a, c, g + G * it, R1, x, s[it]);
    __syncthreads();
#pragma unroll
    for (int it = 0; it < (R1 + G - 1) / G; ++it) {
      const int k1 = g + G * it;
      if (k1 >= R1) break;
      float2 u[R2];
#pragma unroll
      for (int q = 0; q < R2; ++q) u[q] = sY[(k1 * R2 + q) * TILE + ci];
      mpi_dft::dft_r<R2>(u);
      if (INV)
#pragma unroll
        for (int q = 0; q < R2; ++q) u[q].y = -u[q].y;
      if (ok) maps_store<R2, INV>(a, t, tc, k1, R1, x, L, u, s[it]);
    }
  } else {
    constexpr int ST = col_stride(L, TILE);
    constexpr int RSTEP = kThreads / TILE;
    constexpr int PER = (L + RSTEP - 1) / RSTEP;  // rows r0 + RSTEP u of the thread's column
    constexpr int LAST = L - RSTEP * (PER - 1);   // threads with r0 below this have a last row
    __shared__ float2 tw[L];
    __shared__ float2 buf[TILE * ST];
    for (int i = tid; i < L; i += kThreads) tw[i] = a.tw[i];
    const int cx = tid % TILE, r0 = tid / TILE, x = x0 + cx;
    const bool ok = x < a.nx, all = r0 < LAST;
    float2 v[PER], e[1];
    if (ok) {
      if constexpr (PER > 1) {
        float2 (&v1)[PER - 1] = reinterpret_cast<float2 (&)[PER - 1]>(v);
        maps_load<PER - 1, INV>(a, beta, t, c, tc, r0, RSTEP, x, L, v1);
      }
      if (all) {
        maps_load<1, INV>(a, beta, t, c, tc, r0 + RSTEP * (PER - 1), RSTEP, x, L, e);
        v[PER - 1] = e[0];
      }
    }
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (r0 + RSTEP * u < L) buf[cx * ST + pad8(r0 + RSTEP * u)] = ok ? v[u] : make_float2(0.f, 0.f);
    __syncthreads();
    fft_tile_lines<L, INV, TILE, ST>(buf, tw, w, lane);
    __syncthreads();
    if (!ok) return;
    float2 s[PER];
    if (INV)
#pragma unroll
      for (int u = 0; u < PER; ++u)
        if (r0 + RSTEP * u < L) s[u] = a.S[(size_t)c * a.N + (size_t)(r0 + RSTEP * u) * a.nx + x];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      if (r0 + RSTEP * u >= L) continue;
      const float2 o[1] = {buf[cx * ST + pad8(r0 + RSTEP * u)]}, so[1] = {s[u]};
      maps_store<1, INV>(a, t, tc, r0 + RSTEP * u, RSTEP, x, L, o, so);
    }
  }
}

// --------------------------------------------------------------- row passes

struct MapsRows {
  float2* W;                 // [T][C][ny][NX]
  int TC, C, ny, M;
  const int32_t* row_list;   // [T][ny] rows with samples
  const int32_t* n_list;     // [T] their number
  int n_list_max;
  const uint8_t* mask;       // [T][ny][NX]
  const int32_t* idx;        // [T][M]
  const int32_t* row_ptr;    // [T][ny + 1]
  const float2* tw;
  float ksign;
  const float2* y;           // data [T][C][M]
  float2 *ap, *uk, *zk;      // F_s S p, the scaled duals, the projections [T][C][M]
  const Sum* ball;           // partial sums of the ball norms [T][C][kBallBlocks]
  const double* eps;         // ball radii [T][C]
  const double* sc;
  Sum* partials;
};

// One sample's F_s S p, scaled dual and datum or projection.
struct Sample {
  float2 ap, uk, yz;
};

// The normal operator in k-space: F_x, mask, F_x^H of every row with samples.
template <int NX>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows_normal(MapsRows a) {
  using F = Rows<NX>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = lane % F::P;
  float2* b = buf[warp];
  const int per = (a.n_list_max + F::R - 1) / F::R, total = a.TC * per;
  for (int gi = blockIdx.x * kRowWarps + warp; gi < total; gi += gridDim.x * kRowWarps) {
    const int tc = gi / per, j0 = (gi - tc * per) * F::R, t = tc / a.C;
    const int n_list = a.n_list[t];
    if (j0 >= n_list) continue;  // warp-uniform
    const int32_t* list = a.row_list + (size_t)t * a.ny;
    float2* W = a.W + (size_t)tc * a.ny * NX;
    float2 v[F::T1][F::A];
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int j = j0 + (lane + 32 * i) / F::P;
      if (j < n_list) {
        const float2* src = W + (size_t)list[j] * NX + p;
#pragma unroll
        for (int e = 0; e < F::A; ++e) v[i][e] = src[F::P * e];
      }
    }
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int r = (lane + 32 * i) / F::P;
      if (j0 + r < n_list) F::template step1<false>(v[i], r, p, b, a.tw);
    }
    __syncwarp();
    float2 u[F::T2][F::P];
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int q = lane + 32 * i, r = q / F::A, k1 = q % F::A;
      if (r < F::R && j0 + r < n_list) {
        const uint8_t* mk = a.mask + ((size_t)t * a.ny + list[j0 + r]) * NX + k1;
        uint8_t keep[F::P];
#pragma unroll
        for (int k = 0; k < F::P; ++k) keep[k] = mk[F::A * k];
        F::template step2<false>(u[i], r, k1, b);
#pragma unroll
        for (int k = 0; k < F::P; ++k)
          if (!keep[k]) u[i][k] = make_float2(0.f, 0.f);
      }
    }
    __syncwarp();  // every output is out of the exchange: back in as the inverse's input
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int q = lane + 32 * i, r = q / F::A, k1 = q % F::A;
      if (r < F::R && j0 + r < n_list) {
#pragma unroll
        for (int k = 0; k < F::P; ++k) b[F::in_at(r, k1 + F::A * k)] = u[i][k];
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int r = (lane + 32 * i) / F::P;
      if (j0 + r < n_list) {
#pragma unroll
        for (int e = 0; e < F::A; ++e) v[i][e] = b[r * F::S + e * (F::P + 1) + p];
        F::template step1<true>(v[i], r, p, b, a.tw);
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int q = lane + 32 * i, r = q / F::A, k1 = q % F::A;
      if (r < F::R && j0 + r < n_list) {
        F::template step2<true>(u[i], r, k1, b);
        float2* dst = W + (size_t)list[j0 + r] * NX + k1;
#pragma unroll
        for (int k = 0; k < F::P; ++k) dst[F::A * k] = u[i][k];
      }
    }
    __syncwarp();  // the buffer is refilled for the next rows
  }
}

// z_k = y + f_k (F_s S p + u_k - y), the l2-ball projection, and the zero-filled
// rows of z_k - u_k - F_s S p through the inverse DFT along x.
template <int NX>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows_scatter_ball(MapsRows a) {
  using F = Rows<NX>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  __shared__ float s_f[kRowWarps];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = lane % F::P;
  const float fu = (float)a.sc[S_UFAC];
  float2* b = buf[warp];
  const int per = (a.n_list_max + F::R - 1) / F::R, total = a.TC * per;
  for (int g0 = blockIdx.x * kRowWarps; g0 < total; g0 += gridDim.x * kRowWarps) {
    // f = eps / max(|.|, eps) of the warps' coils by one warp, a lane each: an FP64 root
    // and division by every warp would take the pass longer than its rows
    if (warp == 0 && lane < kRowWarps && g0 + lane < total) {
      const int tc = (g0 + lane) / per;
      Sum sq = sum_zero();
#pragma unroll
      for (int i = 0; i < kBallBlocks; ++i) sq = sum_add(sq, a.ball[(size_t)tc * kBallBlocks + i]);
      const double nrm = sqrt(to_double(sq)), eps = a.eps[tc];
      s_f[lane] = nrm > eps ? (float)(eps / nrm) : 1.f;
    }
    __syncthreads();
    const float fc = s_f[warp];
    __syncthreads();
    const int gi = g0 + warp;
    if (gi >= total) continue;  // warp-uniform, as below; every warp of the CTA runs all rounds
    const int tc = gi / per, j0 = (gi - tc * per) * F::R, t = tc / a.C;
    const int n_list = a.n_list[t];
    if (j0 >= n_list) continue;
    const int32_t* list = a.row_list + (size_t)t * a.ny;
    for (int i = lane; i < F::kSmem; i += 32) b[i] = make_float2(0.f, 0.f);
    __syncwarp();
    int row[F::R];  // the group's rows and the range of their samples
#pragma unroll
    for (int r = 0; r < F::R; ++r) row[r] = j0 + r < n_list ? list[j0 + r] : 0x7fffffff;
    const int32_t* rp = a.row_ptr + (size_t)t * (a.ny + 1);
    const int m0 = rp[row[0]], m1 = rp[list[min(j0 + F::R, n_list) - 1] + 1];
    const int32_t* idx = a.idx + (size_t)t * a.M;
    const size_t i0 = (size_t)tc * a.M;
    F::samples(
        row, m0, m1, lane, [&](int m) { return idx[m]; },
        [&](int m) { return Sample{a.ap[i0 + m], a.uk[i0 + m], a.y[i0 + m]}; },
        [&](int m, int r, int kx, const Sample& d) {
          const float sg = ((kx + row[r]) & 1) ? -a.ksign : a.ksign;
          const float2 u = make_float2(fu * d.uk.x, fu * d.uk.y);
          const float2 z = make_float2(d.yz.x + fc * (d.ap.x + u.x - d.yz.x), d.yz.y + fc * (d.ap.y + u.y - d.yz.y));
          a.zk[i0 + m] = z;
          b[F::in_at(r, kx)] = make_float2((z.x - u.x - d.ap.x) * sg, (z.y - u.y - d.ap.y) * sg);
        });
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int r = (lane + 32 * i) / F::P;
      float2 v[F::A];
#pragma unroll
      for (int e = 0; e < F::A; ++e) v[e] = b[r * F::S + e * (F::P + 1) + p];
      F::template step1<true>(v, r, p, b, a.tw);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int q = lane + 32 * i, r = q / F::A, k1 = q % F::A;
      if (r < F::R && j0 + r < n_list) {
        float2 u[F::P];
        F::template step2<true>(u, r, k1, b);
        float2* dst = a.W + ((size_t)tc * a.ny + list[j0 + r]) * NX + k1;
#pragma unroll
        for (int k = 0; k < F::P; ++k) dst[F::A * k] = u[k];
      }
    }
    __syncwarp();
  }
}

// F_s S p of every row (DFT along x, gather) with the data blocks' dual update
// u_k += F_s S p - z_k; per CTA the sums |F_s S p - z_k|^2 and |F_s S (p - p_prev)|^2.
template <int NX>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows_gather_dual(MapsRows a) {
  using F = Rows<NX>;
  __shared__ float2 buf[kRowWarps][F::kSmem];
  __shared__ Sum sh[2 * kRowWarps];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, p = lane % F::P;
  const float fu = (float)a.sc[S_UFAC];
  float2* b = buf[warp];
  Sum sums[2] = {sum_zero(), sum_zero()};
  const int per = (a.n_list_max + F::R - 1) / F::R, total = a.TC * per;
  for (int gi = blockIdx.x * kRowWarps + warp; gi < total; gi += gridDim.x * kRowWarps) {
    const int tc = gi / per, j0 = (gi - tc * per) * F::R, t = tc / a.C;
    const int n_list = a.n_list[t];
    if (j0 >= n_list) continue;  // warp-uniform
    const int32_t* list = a.row_list + (size_t)t * a.ny;
    const float2* W = a.W + (size_t)tc * a.ny * NX;
    float2 v[F::T1][F::A];
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int j = j0 + (lane + 32 * i) / F::P;
      if (j < n_list) {
        const float2* src = W + (size_t)list[j] * NX + p;
#pragma unroll
        for (int e = 0; e < F::A; ++e) v[i][e] = src[F::P * e];
      }
    }
#pragma unroll
    for (int i = 0; i < F::T1; ++i) {
      const int r = (lane + 32 * i) / F::P;
      if (j0 + r < n_list) F::template step1<false>(v[i], r, p, b, a.tw);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < F::T2; ++i) {
      const int q = lane + 32 * i, r = q / F::A, k1 = q % F::A;
      if (r < F::R && j0 + r < n_list) {
        float2 u[F::P];
        F::template step2<false>(u, r, k1, b);
#pragma unroll
        for (int k = 0; k < F::P; ++k) b[r * F::S + k1 * (F::P + 1) + k] = u[k];
      }
    }
    __syncwarp();
    int row[F::R];  // the group's rows and the range of their samples
#pragma unroll
    for (int r = 0; r < F::R; ++r) row[r] = j0 + r < n_list ? list[j0 + r] : 0x7fffffff;
    const int32_t* rp = a.row_ptr + (size_t)t * (a.ny + 1);
    const int m0 = rp[row[0]], m1 = rp[list[min(j0 + F::R, n_list) - 1] + 1];
    const int32_t* idx = a.idx + (size_t)t * a.M;
    const size_t i0 = (size_t)tc * a.M;
    F::samples(
        row, m0, m1, lane, [&](int m) { return idx[m]; },
        [&](int m) { return Sample{a.ap[i0 + m], a.uk[i0 + m], a.zk[i0 + m]}; },
        [&](int m, int r, int kx, const Sample& d) {
          const float sg = ((kx + row[r]) & 1) ? -a.ksign : a.ksign;
          const float2 e = b[F::out_at(r, kx)];
          const float2 ap = make_float2(e.x * sg, e.y * sg);
          a.ap[i0 + m] = ap;
          a.uk[i0 + m] = make_float2(fu * d.uk.x + ap.x - d.yz.x, fu * d.uk.y + ap.y - d.yz.y);
          sums[0] = sum_add(sums[0], sum_diff_sq(ap, d.yz));
          sums[1] = sum_add(sums[1], sum_diff_sq(ap, d.ap));
        });
    __syncwarp();
  }
  block_sums<2, kRowWarps * 32>(sums, sh, a.partials + 2 * (size_t)blockIdx.x);
}

// ------------------------------------------------------- element-wise passes

struct CoilSum {
  const float2* W;  // conj(s_k) w_k [T][C][N]
  int C, nx;
  size_t N, total;  // total = T N
  float scale;
  float2 *d, *Ad;                        // normal: A d = sum + d
  const float2 *z0, *u0, *p;             // residual: sum + z0 - ufac u0 - p
  float2 *r, *p_prev;                    //   into r and d; p kept as p_prev
  const double* sc;
  Sum* partials;  // per CTA: normal, <d, A d>; residual, |r|^2
};

// sum over coils of conj(s_k) w_k with sign and scale.  NORMAL: A d and <d, A d>;
// else the CG's first residual and |r|^2.
template <bool NORMAL>
__global__ void __launch_bounds__(kElemThreads) k_coil_sum(CoilSum a) {
  __shared__ Sum sh[kElemThreads / 32];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const float fu = NORMAL ? 1.f : (float)a.sc[S_UFAC];
  Sum s[1] = {sum_zero()};
  for (size_t i = (size_t)blockIdx.x * kElemThreads + threadIdx.x; i < a.total; i += (size_t)gridDim.x * kElemThreads) {
    const size_t t = i / a.N, n = i - t * a.N;
    const float2* w = a.W + t * a.C * a.N + n;
    float2 acc = make_float2(0.f, 0.f);
    int c = 0;
    for (; c + 8 <= a.C; c += 8) {
      float2 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = w[(size_t)(c + j) * a.N];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        acc.x += v[j].x;
        acc.y += v[j].y;
      }
    }
    for (; c < a.C; ++c) {
      const float2 v = w[(size_t)c * a.N];
      acc.x += v.x;
      acc.y += v.y;
    }
    const int y = (int)(n / a.nx), x = (int)(n - (size_t)y * a.nx);
    const float sg = ((x + y) & 1) ? -a.scale : a.scale;
    float2 o = make_float2(acc.x * sg, acc.y * sg);
    if (NORMAL) {
      const float2 d = a.d[i];
      o = make_float2(o.x + d.x, o.y + d.y);
      a.Ad[i] = o;
      s[0] = sum_add(s[0], sum_dot(d, o));
    } else {
      const float2 z = a.z0[i], u = a.u0[i], p = a.p[i];
      o = make_float2(o.x + z.x - fu * u.x - p.x, o.y + z.y - fu * u.y - p.y);
      a.r[i] = o;
      a.d[i] = o;
      a.p_prev[i] = p;
      s[0] = sum_add(s[0], sum_dot(o, o));
    }
  }
  block_sums<1, kElemThreads>(s, sh, a.partials + blockIdx.x);
}

// x += a d, r -= a A d with a = |r|^2 / <d, A d>, and the new |r|^2 (partial sums in
// and out; rr and rr_new are different buffers).
__global__ void __launch_bounds__(kElemThreads) k_cg_update(float2* __restrict__ x, float2* __restrict__ r,
                                                            const float2* __restrict__ d,
                                                            const float2* __restrict__ Ad, size_t n,
                                                            const Sum* __restrict__ rr,
                                                            const Sum* __restrict__ dad, int n_part,
                                                            Sum* __restrict__ rr_new) {
  __shared__ Sum sh[kElemThreads / 32];
  __shared__ float s_a;
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  if (threadIdx.x < 32) {  // (a warp per sum and a second barrier: slower by 1.5 us beside its neighbours)
    const Sum num = partial_sum(rr, n_part), den = partial_sum(dad, n_part);
    if (threadIdx.x == 0) s_a = sum_ratio(num, den);
  }
  const size_t i0 = (size_t)blockIdx.x * kElemThreads + threadIdx.x, step = (size_t)gridDim.x * kElemThreads;
  float2 dv, av, xv, rv;  // the first element's loads while the step size is formed
  if (i0 < n) {
    dv = d[i0];
    av = Ad[i0];
    xv = x[i0];
    rv = r[i0];
  }
  __syncthreads();
  const float a = s_a;
  Sum s[1] = {sum_zero()};
  for (size_t i = i0; i < n; i += step) {
    if (i != i0) {
      dv = d[i];
      av = Ad[i];
      xv = x[i];
      rv = r[i];
    }
    xv.x = fmaf(a, dv.x, xv.x);
    xv.y = fmaf(a, dv.y, xv.y);
    rv.x = fmaf(-a, av.x, rv.x);
    rv.y = fmaf(-a, av.y, rv.y);
    x[i] = xv;
    r[i] = rv;
    s[0] = sum_add(s[0], sum_dot(rv, rv));
  }
  block_sums<1, kElemThreads>(s, sh, rr_new + blockIdx.x);
}

// |F_s S p + u_k - y|^2 of every (frame, coil): kBallBlocks partial sums each.
__global__ void __launch_bounds__(kThreads) k_ball_norm(const float2* __restrict__ ap, const float2* __restrict__ uk,
                                                        const float2* __restrict__ y, int M,
                                                        const double* __restrict__ sc, Sum* __restrict__ partials) {
  __shared__ Sum sh[kThreads / 32];
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const int c = blockIdx.y;
  const float fu = (float)sc[S_UFAC];
  Sum s[1] = {sum_zero()};
  for (int m = blockIdx.x * kThreads + threadIdx.x; m < M; m += gridDim.x * kThreads) {
    const size_t i = (size_t)c * M + m;
    const float2 av = ap[i], uv = uk[i], yv = y[i];
    s[0] = sum_add(s[0], sum_add(sum_diff3_sq(av.x, __fmul_rn(fu, uv.x), yv.x), sum_diff3_sq(av.y, __fmul_rn(fu, uv.y), yv.y)));
  }
  block_sums<1, kThreads>(s, sh, partials + (size_t)c * kBallBlocks + blockIdx.x);
}

// u_0 += p - z_0; the residual norms of both blocks (row_part: the data blocks'
// sums per CTA) and the balancing of rho (He et al. 2000), by the last CTA to
// arrive at `counter` (zero before and after), which adds the partial sums in order.
__global__ void __launch_bounds__(kElemThreads) k_admm_dual(float2* __restrict__ u0, const float2* __restrict__ p,
                                                            const float2* __restrict__ z0,
                                                            const float2* __restrict__ p_prev, size_t n, double* sc,
                                                            Sum* partials, unsigned* counter,
                                                            const Sum* __restrict__ row_part, int n_row, double mu,
                                                            double tau, double* __restrict__ hist) {
  __shared__ Sum sh[2 * kElemThreads / 32], sums[2];
  __shared__ int last;
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const float fu = (float)sc[S_UFAC];
  Sum s[2] = {sum_zero(), sum_zero()};
  for (size_t i = (size_t)blockIdx.x * kElemThreads + threadIdx.x; i < n; i += (size_t)gridDim.x * kElemThreads) {
    const float2 pv = p[i], zv = z0[i], qv = p_prev[i];
    const float2 uv = u0[i];
    u0[i] = make_float2(fu * uv.x + pv.x - zv.x, fu * uv.y + pv.y - zv.y);
    s[0] = sum_add(s[0], sum_diff_sq(pv, zv));
    s[1] = sum_add(s[1], sum_diff_sq(pv, qv));
  }
  block_sums<2, kElemThreads>(s, sh, partials + 2 * (size_t)blockIdx.x);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  s[0] = s[1] = sum_zero();
  for (unsigned i = threadIdx.x; i < gridDim.x + n_row; i += kElemThreads) {
    const Sum* q = i < gridDim.x ? partials + 2 * (size_t)i : row_part + 2 * (size_t)(i - gridDim.x);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int4 w = __ldcg(reinterpret_cast<const int4*>(q + j));
      s[j] = sum_add(s[j], Sum{(long long)((unsigned long long)(unsigned)w.y << 32 | (unsigned)w.x), w.z});
    }
  }
  block_sums<2, kElemThreads>(s, sh, sums);
  __syncthreads();
  if (threadIdx.x) return;
  const double prim = sqrt(to_double(sums[0])), rho = sc[S_RHO], dual = rho * sqrt(to_double(sums[1]));
  hist[0] = prim;
  hist[1] = dual;
  hist[2] = rho;
  double f = 1.0;
  if (prim > mu * dual) {
    sc[S_RHO] = rho * tau;
    f = 1.0 / tau;
  } else if (dual > mu * prim) {
    sc[S_RHO] = rho / tau;
    f = tau;
  }
  sc[S_UFAC] = f;
}

__global__ void k_admm_start(double* sc, double rho0) {
  sc[S_RHO] = rho0;
  sc[S_UFAC] = 1.0;
}

// mask[t][idx[t][m]] = 1
__global__ void k_sample_mask(const int32_t* __restrict__ idx, int M, size_t N, uint8_t* __restrict__ mask) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < M) mask[(size_t)blockIdx.y * N + idx[(size_t)blockIdx.y * M + m]] = 1;
}

// --------------------------------------------------------------- launchers

template <bool INV>
mpi_status launch_maps_cols(mpi_ctx* ctx, int L, const MapsCols& a, int TC) {
  const int tile = maps_cols_tile(L);
  const unsigned blocks = (unsigned)((size_t)TC * ((a.nx + tile - 1) / tile));
  MPI_PROF(ctx, KF_FFT_LINES);
  switch (L) {
#define MPI_COLS(n)                                                                              \
  case n:                                                                                        \
    launch_pdl(ctx, k_maps_cols<n, INV>, dim3(blocks), dim3(kThreads), 0, a);                    \
    break;
    MPI_COLS(16) MPI_COLS(32) MPI_COLS(48) MPI_COLS(64) MPI_COLS(96) MPI_COLS(128) MPI_COLS(192) MPI_COLS(256)
    MPI_COLS(320) MPI_COLS(512)
#undef MPI_COLS
    default:
      return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  }
  MPI_LAUNCH_CHECK(ctx, INV ? "k_maps_cols<inv>" : "k_maps_cols<fwd>");
  return MPI_OK;
}

enum RowPass { ROWS_NORMAL, ROWS_SCATTER, ROWS_GATHER };

mpi_status launch_maps_rows(mpi_ctx* ctx, int nx, RowPass pass, const MapsRows& a, unsigned blocks) {
  MPI_PROF(ctx, KF_FFT_ROWS);
  switch (nx) {
#define MPI_ROWS(n)                                                                                             \
  case n:                                                                                                       \
    if (pass == ROWS_NORMAL) launch_pdl(ctx, k_rows_normal<n>, dim3(blocks), dim3(kRowWarps * 32), 0, a);       \
    else if (pass == ROWS_SCATTER)                                                                              \
      launch_pdl(ctx, k_rows_scatter_ball<n>, dim3(blocks), dim3(kRowWarps * 32), 0, a);                        \
    else launch_pdl(ctx, k_rows_gather_dual<n>, dim3(blocks), dim3(kRowWarps * 32), 0, a);                      \
    break;
    MPI_ROWS(16) MPI_ROWS(32) MPI_ROWS(48) MPI_ROWS(64) MPI_ROWS(96) MPI_ROWS(128) MPI_ROWS(192) MPI_ROWS(256)
    MPI_ROWS(320) MPI_ROWS(512)
#undef MPI_ROWS
    default:
      return set_err(ctx, MPI_ERR_SHAPE, "unsupported FFT length");
  }
  MPI_LAUNCH_CHECK(ctx, pass == ROWS_NORMAL ? "k_rows_normal"
                                            : (pass == ROWS_SCATTER ? "k_rows_scatter_ball" : "k_rows_gather_dual"));
  return MPI_OK;
}

float axis_sign(int n) { return ((n / 2) & 1) ? -1.f : 1.f; }

unsigned elem_blocks(size_t n) {
  return (unsigned)std::min<size_t>((n + kElemThreads - 1) / kElemThreads, kMaxElemBlocks);
}

// CTAs of a row pass over TC coils with at most n_list rows each, R rows per warp
unsigned row_blocks(const mpi_ctx* ctx, size_t TC, int n_list, int nx) {
  int R = 1;
#define MPI_ROWS(n) \
  if (nx == n) R = Rows<n>::R;
  MPI_ROWS(16) MPI_ROWS(32) MPI_ROWS(48) MPI_ROWS(64) MPI_ROWS(96) MPI_ROWS(128) MPI_ROWS(192) MPI_ROWS(256)
  MPI_ROWS(320) MPI_ROWS(512)
#undef MPI_ROWS
  const size_t groups = TC * (size_t)((n_list + R - 1) / R);
  return (unsigned)std::min<size_t>((groups + kRowWarps - 1) / kRowWarps, 16 * (size_t)std::max(ctx->num_sms, 1));
}

#define TRY(x)                       \
  do {                               \
    mpi_status st__ = (x);           \
    if (st__ != MPI_OK) return st__; \
  } while (0)

}  // namespace

bool admm_maps_supported(const mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                         mpi_precision prec) {
  if (ctx->line_kernel || basis->ctx != ctx || basis->tucker || basis->N != plans[0]->N || plans[0]->M < 1)
    return false;
  const bool bf = prec == MPI_PREC_BF16 || prec == MPI_PREC_MIXED;
  if (!bf && prec != MPI_PREC_FP32 && prec != MPI_PREC_FP32_SIMT) return false;
  if (bf && (!basis->Ubf || C > 128)) return false;
  for (int t = 0; t < T; ++t)
    if (plans[t]->ctx != ctx || plans[t]->kind != MPI_TRAJ_CARTESIAN || plans[t]->ndim != 2) return false;
  const size_t rows = (size_t)T * C * plans[0]->ny;
  return rows < 0x7fffffffu && (size_t)T * C <= 65535 && T <= 65535;
}

size_t admm_maps_layout(const mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                        const mpi_admm_params* prm, mpi_precision prec, void* mem, AdmmMaps* m) {
  const size_t N = plans[0]->N, M = plans[0]->M, TN = (size_t)T * N, CM = (size_t)T * C * M;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = (char*)mem + off;
    off += (bytes + 255) & ~(size_t)255;
    return p;
  };
  auto cplx = [&](size_t n) { return (float2*)take(n * sizeof(float2)); };
  m->in_y = cplx(CM);
  m->in_alpha = cplx((size_t)C * basis->q);
  m->in_eps = (double*)take((size_t)T * C * sizeof(double));
  m->hist = (double*)take(3 * (size_t)std::max(prm->n_outer, 1) * sizeof(double));
  m->S = cplx(C * N);
  m->S_cg = prec == MPI_PREC_MIXED ? cplx(C * N) : m->S;
  m->W = cplx((size_t)T * C * N);
  m->zero_begin = (char*)mem + off;  // cleared when a solve starts
  m->p = cplx(TN);
  m->u0 = cplx(TN);
  m->ap = cplx(CM);
  m->uk = cplx(CM);
  m->counter = (unsigned*)take(sizeof(unsigned));
  m->zero_bytes = (char*)mem + off - m->zero_begin;
  m->zk = cplx(CM);
  float2** img[] = {&m->z0, &m->r, &m->d[0], &m->d[1], &m->Ad, &m->p_prev};
  for (float2** b : img) *b = cplx(TN);
  m->tv = cplx(tv_scratch_elems(T > 1 ? 3 : 2, (long)TN, prm->n_tv));
  m->sc = (double*)take(S_NUM * sizeof(double));
  m->ball = take((size_t)T * C * kBallBlocks * sizeof(Sum));
  m->part = take(5 * (size_t)kMaxElemBlocks * sizeof(Sum));  // |r|^2 twice, <d, A d>, the dual's two
  int n_list = 0;
  for (int t = 0; t < T; ++t) n_list = std::max(n_list, plans[t]->n_list);
  m->row_part = take(2 * (size_t)row_blocks(ctx, (size_t)T * C, n_list, plans[0]->nx) * sizeof(Sum));
  m->idx = (int32_t*)take((size_t)T * M * sizeof(int32_t));
  m->row_ptr = (int32_t*)take((size_t)T * (plans[0]->ny + 1) * sizeof(int32_t));
  m->row_list = (int32_t*)take((size_t)T * plans[0]->ny * sizeof(int32_t));
  m->n_list = (int32_t*)take((size_t)T * sizeof(int32_t));
  m->rmask = (uint8_t*)take((size_t)T * plans[0]->ny);
  m->mask = (uint8_t*)take(TN);
  return off;
}

mpi_status admm_maps_tables(mpi_ctx* ctx, const mpi_plan* const* plans, int T, AdmmMaps* m) {
  const int ny = plans[0]->ny, nx = plans[0]->nx, M = plans[0]->M;
  const size_t N = plans[0]->N;
  std::vector<int32_t> rp((size_t)T * (ny + 1));
  std::vector<uint8_t> has((size_t)T * ny);
  std::vector<int32_t> list((size_t)T * ny, 0), count(T, 0);
  cudaError_t e = cudaMemsetAsync(m->mask, 0, (size_t)T * N, ctx->stream);
  for (int t = 0; t < T && e == cudaSuccess; ++t) {
    e = cudaMemcpyAsync(m->idx + (size_t)t * M, plans[t]->idx, (size_t)M * sizeof(int32_t), cudaMemcpyDeviceToDevice,
                        ctx->stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(rp.data() + (size_t)t * (ny + 1), plans[t]->row_ptr, (size_t)(ny + 1) * sizeof(int32_t),
                          cudaMemcpyDeviceToHost, ctx->stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "image solver tables");
  m->whole_rows = true;
  for (int t = 0; t < T; ++t)
    for (int r = 0; r < ny; ++r) {
      const int n = rp[(size_t)t * (ny + 1) + r + 1] - rp[(size_t)t * (ny + 1) + r];
      has[(size_t)t * ny + r] = n > 0;
      if (n > 0) list[(size_t)t * ny + count[t]++] = r;
      m->whole_rows &= n == 0 || n == nx;
    }
  e = cudaMemcpyAsync(m->row_ptr, rp.data(), rp.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(m->row_list, list.data(), list.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(m->n_list, count.data(), count.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->rmask, has.data(), has.size(), cudaMemcpyHostToDevice, ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "image solver tables");
  MPI_PROF(ctx, KF_SOLVER);
  k_sample_mask<<<dim3((unsigned)((M + 255) / 256), (unsigned)T), 256, 0, ctx->stream>>>(m->idx, M, N, m->mask);
  MPI_LAUNCH_CHECK(ctx, "k_sample_mask");
  return cuda_check(ctx, cudaStreamSynchronize(ctx->stream), "image solver tables");  // the host tables are read until here
}

mpi_status admm_maps_record(mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                            const mpi_admm_params* prm, mpi_precision prec, const AdmmMaps& m) {
  // In the graph a kernel's start costs little, and started early the passes' CTAs, some 120
  // to 500 that fit the chip at once, pile up on the SMs that the pass before has left: 256^2
  // and 16 coils 225 us per outer step started early, 195 not (rows alone not 211), 4 frames
  // of 128^2 91 and 68, 192^2 and 10 coils 195 and 146.
  const NoEarlyStart late(ctx, true);
  const int ny = plans[0]->ny, nx = plans[0]->nx, M = plans[0]->M, TC = T * C;
  const size_t N = plans[0]->N, TN = (size_t)T * N;
  const float scale = 1.0f / sqrtf((float)N);
  int n_list = 0;
  for (int t = 0; t < T; ++t) n_list = std::max(n_list, plans[t]->n_list);
  const unsigned eblk = elem_blocks(TN), rblk = row_blocks(ctx, TC, n_list, nx);
  Sum* part = (Sum*)m.part;
  Sum *rr[2] = {part, part + kMaxElemBlocks}, *dad = part + 2 * kMaxElemBlocks;
  TRY(cuda_check(ctx, cudaMemsetAsync(m.zero_begin, 0, m.zero_bytes, ctx->stream), "image solver start"));
  MPI_PROF(ctx, KF_SOLVER);
  k_admm_start<<<1, 1, 0, ctx->stream>>>(m.sc, prm->rho0);
  MPI_LAUNCH_CHECK(ctx, "k_admm_start");
  // MIXED: BF16 maps in the CG iterations; FP32 ones for the constraint-side
  // products and the CG's first residual
  TRY(mpi_basis_expand(ctx, basis, (const mpi_c32*)m.in_alpha, C, (mpi_c32*)m.S,
                       prec == MPI_PREC_MIXED ? MPI_PREC_FP32 : prec));
  if (m.S_cg != m.S) TRY(mpi_basis_expand(ctx, basis, (const mpi_c32*)m.in_alpha, C, (mpi_c32*)m.S_cg, MPI_PREC_BF16));

  MapsCols cols{};
  cols.W = m.W;
  cols.n_part = (int)eblk;
  cols.C = C;
  cols.nx = nx;
  cols.N = N;
  cols.scale = scale;
  cols.rmask = m.rmask;
  cols.tw = twiddle_table(ctx, ny);
  int par = 0;  // which of rr holds |r|^2
  auto cols_fwd = [&](const float2* S, const float2* v, const float2* r, float2* dnew) {
    MapsCols a = cols;
    a.S = S;
    a.v = v;
    a.r = r;
    a.dnew = dnew;
    a.rr = rr[par];
    a.rr_old = rr[par ^ 1];
    return launch_maps_cols<false>(ctx, ny, a, TC);
  };
  auto cols_inv = [&](const float2* S) {
    MapsCols a = cols;
    a.S = S;
    a.v = m.p;  // not read
    return launch_maps_cols<true>(ctx, ny, a, TC);
  };
  MapsRows rows{};
  rows.W = m.W;
  rows.TC = TC;
  rows.C = C;
  rows.ny = ny;
  rows.M = M;
  rows.row_list = m.row_list;
  rows.n_list = m.n_list;
  rows.n_list_max = n_list;
  rows.mask = m.mask;
  rows.idx = m.idx;
  rows.row_ptr = m.row_ptr;
  rows.tw = twiddle_table(ctx, nx);
  rows.ksign = axis_sign(nx) * axis_sign(ny);
  rows.y = m.in_y;
  rows.ap = m.ap;
  rows.uk = m.uk;
  rows.zk = m.zk;
  rows.ball = (const Sum*)m.ball;
  rows.eps = m.in_eps;
  rows.sc = m.sc;
  rows.partials = (Sum*)m.row_part;
  CoilSum sum{};
  sum.W = m.W;
  sum.C = C;
  sum.nx = nx;
  sum.N = N;
  sum.total = TN;
  sum.Ad = m.Ad;
  sum.z0 = m.z0;
  sum.u0 = m.u0;
  sum.p = m.p;
  sum.r = m.r;
  sum.p_prev = m.p_prev;
  sum.sc = m.sc;

  for (int it = 0; it < prm->n_outer; ++it) {
    // z_0 = prox_{TV/rho}(p + u_0), z_k = Pi(F_s S p + u_k)
    TRY(launch_tv_prox(ctx, T > 1 ? T : 1, ny, nx, T > 1 ? 3 : 2, m.p, m.u0, m.sc + S_UFAC, m.sc + S_RHO, 0.f,
                       prm->n_tv, m.tv, m.z0));
    MPI_PROF(ctx, KF_SOLVER);
    launch_pdl(ctx, k_ball_norm, dim3(kBallBlocks, (unsigned)TC), dim3(kThreads), 0, m.ap, m.uk, m.in_y, M,
               m.sc, (Sum*)m.ball);
    MPI_LAUNCH_CHECK(ctx, "k_ball_norm");
    TRY(launch_maps_rows(ctx, nx, ROWS_SCATTER, rows, rblk));
    // r = S^H F_s^H (z_k - u_k - F_s S p) + z_0 - u_0 - p
    TRY(cols_inv(m.S));
    int cur = 0;
    sum.scale = scale;
    sum.d = m.d[cur];
    sum.partials = rr[par];
    MPI_PROF(ctx, KF_SOLVER);
    launch_pdl(ctx, k_coil_sum<false>, dim3(eblk), dim3(kElemThreads), 0, sum);
    MPI_LAUNCH_CHECK(ctx, "k_coil_sum<residual>");
    for (int k = 0; k < prm->n_cg; ++k) {
      if (k) {
        TRY(cols_fwd(m.S_cg, m.d[cur], m.r, m.d[cur ^ 1]));
        cur ^= 1;
      } else {
        TRY(cols_fwd(m.S_cg, m.d[cur], nullptr, nullptr));
      }
      if (!m.whole_rows) TRY(launch_maps_rows(ctx, nx, ROWS_NORMAL, rows, rblk));
      TRY(cols_inv(m.S_cg));
      sum.scale = m.whole_rows ? scale * (float)nx : scale;  // F_x^H F_x = nx on whole rows
      sum.d = m.d[cur];
      sum.partials = dad;
      MPI_PROF(ctx, KF_SOLVER);
      launch_pdl(ctx, k_coil_sum<true>, dim3(eblk), dim3(kElemThreads), 0, sum);
      MPI_LAUNCH_CHECK(ctx, "k_coil_sum<normal>");
      MPI_PROF(ctx, KF_SOLVER);
      launch_pdl(ctx, k_cg_update, dim3(eblk), dim3(kElemThreads), 0, m.p, m.r, m.d[cur], m.Ad, TN, rr[par], dad,
                 (int)eblk, rr[par ^ 1]);
      MPI_LAUNCH_CHECK(ctx, "k_cg_update");
      par ^= 1;
    }
    // u += A p - z, the residuals, rho
    TRY(cols_fwd(m.S, m.p, nullptr, nullptr));
    TRY(launch_maps_rows(ctx, nx, ROWS_GATHER, rows, rblk));
    MPI_PROF(ctx, KF_SOLVER);
    launch_pdl(ctx, k_admm_dual, dim3(eblk), dim3(kElemThreads), 0, m.u0, m.p, m.z0, m.p_prev, TN, m.sc,
               part + 3 * kMaxElemBlocks, m.counter, (const Sum*)m.row_part, (int)rblk, prm->mu, prm->tau,
               m.hist + 3 * (size_t)it);
    MPI_LAUNCH_CHECK(ctx, "k_admm_dual");
  }
  return MPI_OK;
}
