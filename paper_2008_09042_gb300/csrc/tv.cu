// Total-variation prox of the image solver (the z_0 update of Eq. 11):
// argmin_x 1/2 ||x - b||^2 + lam TV(x), isotropic TV of a complex image with
// forward differences and a zero difference at the last sample, by FGP
// iterations on the dual (Beck & Teboulle 2009):
//   x  = b - lam D^H R,   Pn = proj(R + D x / (L lam)),   R = Pn + c (Pn - P),
// L = 4 nd, and x = b - lam D^H P at the end.
//
// An iteration touches 40 bytes per pixel and does some 60 operations on them,
// far too little for a launch: with two kernels per iteration and two fills, the
// ten iterations on a 256 x 256 image were 23 launches of 3-10 us each.
//  - 2D (k_tv_tile): a CTA keeps a tile of the image and its halo in shared
//    memory and runs up to kTileIters iterations there, the valid region
//    shrinking by one pixel per iteration (each iteration reads a neighbourhood
//    of radius one), so ten iterations are one launch.  The halo is recomputed
//    by its neighbours: at 32 x 32 outputs and ten iterations a CTA works on
//    about 42 x 42 pixels on average (1.7 times its own).
//  - 3D: the halo of several iterations would be most of the work.  Up to
//    kFusedBytes of P and two R (k_tv_step) an iteration is one launch, both updates
//    fused: each thread forms x at its pixel and at its forward neighbours from R.
//    Beyond, where the third array leaves L2, x is formed first (k_tv_out) and P and R
//    are updated in place (k_tv_dual).  An iteration takes, fused and not, 8.7 and 15 us
//    at 16 x 32 x 32, 15 and 27 at 64^3, 40 and 54 at 96^3 (64 MB), 134 and 80 at
//    96 x 96 x 128 (85 MB), 235 and 174 at 96 x 128 x 128.
#include <math.h>

#include <algorithm>

#include "mpi_internal.h"
#include "ptx.cuh"

namespace {

constexpr int kTvThreads = 512;
constexpr int kTileIters = 10;
constexpr size_t kFusedBytes = (size_t)64 << 20;

// lam = 1 / rho and the dual step rho / L, L = 4 nd, formed by one thread (an FP64
// division per thread costs more than the pixel's arithmetic at this GPU's FP64 rate).
struct TvScalars {
  float lam, step, fu;
};

struct TvIn {
  const float2* p;     // b = p (+ ufac u)
  const float2* u;     // may be null
  const double* ufac;  // device factor of u (null: 1)
  const double* rho;   // lam = 1 / rho (null: lam)
  float lam;
};

__device__ __forceinline__ float2 tv_input(const TvIn& in, float fu, size_t i) {
  float2 b = in.p[i];
  if (in.u) {
    const float2 u = in.u[i];
    b.x += fu * u.x;
    b.y += fu * u.y;
  }
  return b;
}

__device__ __forceinline__ TvScalars tv_scalars(const TvIn& in, int nd) {
  __shared__ TvScalars sh;
  if (threadIdx.x == 0) {
    const double L = 4.0 * nd;
    sh.lam = in.rho ? (float)(1.0 / *in.rho) : in.lam;
    sh.step = in.rho ? (float)(*in.rho / L) : 1.0f / ((float)L * in.lam);
    sh.fu = in.ufac ? (float)*in.ufac : 1.0f;
  }
  __syncthreads();
  return sh;
}

struct TvTile {
  int ny, nx, oy, ox;   // image and output tile
  int iters, first, last;  // iterations of this launch; first: P = R = 0; last: write x, else P and R
  float c[kTileIters];  // momentum of each iteration
};

// Shared memory: b, x, P (y and x components) and R over a region of
// (oy + 2 iters + last) x (ox + 2 iters + last) pixels that starts iters + last
// before the tile.  Threads walk the region linearly.
__global__ void __launch_bounds__(kTvThreads) k_tv_tile(TvIn in, TvTile t, const float2* __restrict__ Pin,
                                                        const float2* __restrict__ Rin, float2* __restrict__ Pout,
                                                        float2* __restrict__ Rout, float2* __restrict__ out) {
  extern __shared__ float2 sm[];
  const int lo = t.iters + t.last;
  const int W = t.ox + t.iters + lo, H = t.oy + t.iters + lo, A = W * H;
  float2 *sb = sm, *sx = sb + A, *P0 = sx + A, *P1 = P0 + A, *R0 = P1 + A, *R1 = R0 + A;  // component 0: x, 1: y
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const TvScalars sc = tv_scalars(in, 2);
  const float lam = sc.lam, step = sc.step, fu = sc.fu;
  const int x0 = (int)blockIdx.x * t.ox - lo, y0 = (int)blockIdx.y * t.oy - lo;  // image position of the region
  const size_t N = (size_t)t.ny * t.nx;
  const int sx0 = threadIdx.x % W, sy0 = threadIdx.x / W;
  const int dx = kTvThreads % W, dy = kTvThreads / W;
  // region point of linear index i: advanced without divisions
#define TV_WALK(body)                                                  \
  for (int i = threadIdx.x, rx = sx0, ry = sy0; i < A; i += kTvThreads) { \
    const int gx = x0 + rx, gy = y0 + ry;                               \
    body;                                                               \
    rx += dx;                                                           \
    ry += dy;                                                           \
    if (rx >= W) {                                                      \
      rx -= W;                                                          \
      ++ry;                                                             \
    }                                                                   \
  }
  TV_WALK({
    if (gx >= 0 && gx < t.nx && gy >= 0 && gy < t.ny) {
      const size_t n = (size_t)gy * t.nx + gx;
      sb[i] = tv_input(in, fu, n);
      const float2 zero = make_float2(0.f, 0.f);
      P0[i] = t.first ? zero : Pin[n];
      P1[i] = t.first ? zero : Pin[N + n];
      R0[i] = t.first ? zero : Rin[n];
      R1[i] = t.first ? zero : Rin[N + n];
    }
  })
  __syncthreads();
  // b - lam D^H (F0, F1) at region point i, image position (gx, gy); the
  // neighbours it reads lie inside the image
  auto primal = [&](const float2* F0, const float2* F1, int i, int gx, int gy) {
    float2 dh = make_float2(0.f, 0.f);
    if (gx >= 1) {
      const float2 v = F0[i - 1];
      dh.x += v.x;
      dh.y += v.y;
    }
    if (gx <= t.nx - 2) {
      const float2 v = F0[i];
      dh.x -= v.x;
      dh.y -= v.y;
    }
    if (gy >= 1) {
      const float2 v = F1[i - W];
      dh.x += v.x;
      dh.y += v.y;
    }
    if (gy <= t.ny - 2) {
      const float2 v = F1[i];
      dh.x -= v.x;
      dh.y -= v.y;
    }
    const float2 b = sb[i];
    return make_float2(b.x - lam * dh.x, b.y - lam * dh.y);
  };
  for (int k = 1; k <= t.iters; ++k) {
    // P_k is needed m pixels around the tile (and one more before it for the last primal)
    const int m = t.iters - k, a = lo - m - t.last, ex = lo + t.ox + m, ey = lo + t.oy + m;
    TV_WALK({
      if (rx >= a && rx <= ex && ry >= a && ry <= ey && rx < W && ry < H && gx >= 0 && gx < t.nx && gy >= 0 &&
          gy < t.ny)
        sx[i] = primal(R0, R1, i, gx, gy);
    })
    __syncthreads();
    const float c = t.c[k - 1];
    TV_WALK({
      if (rx >= a && rx < ex && ry >= a && ry < ey && gx >= 0 && gx < t.nx && gy >= 0 && gy < t.ny) {
        const float2 xi = sx[i];
        float2 g0 = make_float2(0.f, 0.f);
        float2 g1 = make_float2(0.f, 0.f);
        if (gx <= t.nx - 2) g0 = make_float2(sx[i + 1].x - xi.x, sx[i + 1].y - xi.y);
        if (gy <= t.ny - 2) g1 = make_float2(sx[i + W].x - xi.x, sx[i + W].y - xi.y);
        const float2 r0 = R0[i];
        const float2 r1 = R1[i];
        const float2 q0 = make_float2(fmaf(step, g0.x, r0.x), fmaf(step, g0.y, r0.y));
        const float2 q1 = make_float2(fmaf(step, g1.x, r1.x), fmaf(step, g1.y, r1.y));
        const float inv = 1.0f / fmaxf(1.0f, sqrtf(q0.x * q0.x + q0.y * q0.y + q1.x * q1.x + q1.y * q1.y));
        const float2 o0 = P0[i];
        const float2 o1 = P1[i];
        const float2 n0 = make_float2(q0.x * inv, q0.y * inv);
        const float2 n1 = make_float2(q1.x * inv, q1.y * inv);
        P0[i] = n0;
        P1[i] = n1;
        R0[i] = make_float2(n0.x + c * (n0.x - o0.x), n0.y + c * (n0.y - o0.y));
        R1[i] = make_float2(n1.x + c * (n1.x - o1.x), n1.y + c * (n1.y - o1.y));
      }
    })
    __syncthreads();
  }
  TV_WALK({
    if (rx >= lo && rx < lo + t.ox && ry >= lo && ry < lo + t.oy && gx < t.nx && gy < t.ny) {
      const size_t n = (size_t)gy * t.nx + gx;
      if (t.last) {
        out[n] = primal(P0, P1, i, gx, gy);
      } else {
        Pout[n] = P0[i];
        Pout[N + n] = P1[i];
        Rout[n] = R0[i];
        Rout[N + n] = R1[i];
      }
    }
  })
#undef TV_WALK
}

struct TvGrid {
  int n[3];  // x, y, z
};

// b - lam D^H F at voxel i (position pos), F [3][N] (null: zero)
__device__ __forceinline__ float2 tv_primal3(const TvIn& in, float fu, float lam, const float2* __restrict__ F,
                                             const TvGrid& g, size_t N, size_t i, const int pos[3]) {
  const size_t stride[3] = {1, (size_t)g.n[0], (size_t)g.n[0] * g.n[1]};
  float2 dh = make_float2(0.f, 0.f);
  if (F) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (pos[d] >= 1) {
        const float2 v = F[d * N + i - stride[d]];
        dh.x += v.x;
        dh.y += v.y;
      }
      if (pos[d] <= g.n[d] - 2) {
        const float2 v = F[d * N + i];
        dh.x -= v.x;
        dh.y -= v.y;
      }
    }
  }
  const float2 b = tv_input(in, fu, i);
  return make_float2(b.x - lam * dh.x, b.y - lam * dh.y);
}

// One FGP iteration of a 3D grid: P updated in place, R read from Rin (null: P =
// R = 0) and written to Rout.
__global__ void __launch_bounds__(256) k_tv_step(TvIn in, TvGrid g, size_t N, const float2* __restrict__ Rin,
                                                 float2* __restrict__ P, float2* __restrict__ Rout, float c) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const TvScalars sc = tv_scalars(in, 3);
  const float lam = sc.lam, stp = sc.step, fu = sc.fu;
  const size_t stride[3] = {1, (size_t)g.n[0], (size_t)g.n[0] * g.n[1]};
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const unsigned j = (unsigned)i, r = j / (unsigned)g.n[0], z = r / (unsigned)g.n[1];  // N < 2^31
    const int pos[3] = {(int)(j - r * g.n[0]), (int)(r - z * g.n[1]), (int)z};
    const float2 xi = tv_primal3(in, fu, lam, Rin, g, N, i, pos);
    float2 q[3];
    float mag2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float2 gd = make_float2(0.f, 0.f);
      if (pos[d] <= g.n[d] - 2) {
        const int pn[3] = {pos[0] + (d == 0), pos[1] + (d == 1), pos[2] + (d == 2)};
        const float2 xn = tv_primal3(in, fu, lam, Rin, g, N, i + stride[d], pn);
        gd = make_float2(xn.x - xi.x, xn.y - xi.y);
      }
      const float2 rv = Rin ? Rin[d * N + i] : make_float2(0.f, 0.f);
      q[d] = make_float2(fmaf(stp, gd.x, rv.x), fmaf(stp, gd.y, rv.y));
      mag2 += q[d].x * q[d].x + q[d].y * q[d].y;
    }
    const float inv = 1.0f / fmaxf(1.0f, sqrtf(mag2));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float2 o = Rin ? P[d * N + i] : make_float2(0.f, 0.f);
      const float2 nv = make_float2(q[d].x * inv, q[d].y * inv);
      P[d * N + i] = nv;
      Rout[d * N + i] = make_float2(nv.x + c * (nv.x - o.x), nv.y + c * (nv.y - o.y));
    }
  }
}

// P and R of one FGP iteration from x, in place (first: P = R = 0).
__global__ void __launch_bounds__(256) k_tv_dual(TvIn in, TvGrid g, size_t N, const float2* __restrict__ x,
                                                 float2* __restrict__ P, float2* __restrict__ R, int first, float c) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const float stp = tv_scalars(in, 3).step;
  const size_t stride[3] = {1, (size_t)g.n[0], (size_t)g.n[0] * g.n[1]};
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const unsigned j = (unsigned)i, r = j / (unsigned)g.n[0], z = r / (unsigned)g.n[1];  // N < 2^31
    const int pos[3] = {(int)(j - r * g.n[0]), (int)(r - z * g.n[1]), (int)z};
    const float2 xi = x[i];
    float2 q[3];
    float mag2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float2 gd = make_float2(0.f, 0.f);
      if (pos[d] <= g.n[d] - 2) {
        const float2 xn = x[i + stride[d]];
        gd = make_float2(xn.x - xi.x, xn.y - xi.y);
      }
      const float2 rv = first ? make_float2(0.f, 0.f) : R[d * N + i];
      q[d] = make_float2(fmaf(stp, gd.x, rv.x), fmaf(stp, gd.y, rv.y));
      mag2 += q[d].x * q[d].x + q[d].y * q[d].y;
    }
    const float inv = 1.0f / fmaxf(1.0f, sqrtf(mag2));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float2 o = first ? make_float2(0.f, 0.f) : P[d * N + i];
      const float2 nv = make_float2(q[d].x * inv, q[d].y * inv);
      P[d * N + i] = nv;
      R[d * N + i] = make_float2(nv.x + c * (nv.x - o.x), nv.y + c * (nv.y - o.y));
    }
  }
}

__global__ void __launch_bounds__(256) k_tv_out(TvIn in, TvGrid g, size_t N, const float2* __restrict__ P,
                                                float2* __restrict__ out) {
  mpi_ptx::pdl_trigger();
  mpi_ptx::pdl_wait();
  const TvScalars sc = tv_scalars(in, 3);
  const float lam = sc.lam, fu = sc.fu;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const unsigned j = (unsigned)i, r = j / (unsigned)g.n[0], z = r / (unsigned)g.n[1];  // N < 2^31
    const int pos[3] = {(int)(j - r * g.n[0]), (int)(r - z * g.n[1]), (int)z};
    out[i] = tv_primal3(in, fu, lam, P, g, N, i, pos);
  }
}

}  // namespace

namespace {
bool tv_fused(size_t N) { return 9 * N * sizeof(float2) <= kFusedBytes; }
}  // namespace

size_t tv_scratch_elems(int nd, long N, int n_iter) {
  if (nd == 3) return (size_t)N * (tv_fused((size_t)N) ? 9 : 6);
  return (size_t)N * 4 * std::clamp((n_iter + kTileIters - 1) / kTileIters - 1, 0, 2);  // P and R between launches
}

mpi_status launch_tv_prox(mpi_ctx* ctx, int nz, int ny, int nx, int nd, const float2* p, const float2* u,
                          const double* ufac, const double* rho, float lam, int n_iter, float2* scratch, float2* out) {
  const TvIn in{p, u, ufac, rho, lam};
  const size_t N = (size_t)nz * ny * nx;
  double tk = 1.0;
  auto momentum = [&]() {
    const double tn = 0.5 * (1.0 + sqrt(1.0 + 4.0 * tk * tk));
    const float c = (float)((tk - 1.0) / tn);
    tk = tn;
    return c;
  };
  if (nd == 3) {
    const TvGrid g{{nx, ny, nz}};
    const unsigned blocks = (unsigned)std::min<size_t>((N + 255) / 256, 16 * (size_t)std::max(ctx->num_sms, 1));
    const bool fused = tv_fused(N);
    float2 *P = scratch, *R[2] = {P + 3 * N, fused ? P + 6 * N : nullptr};
    for (int it = 0; it < n_iter; ++it) {
      const float c = momentum();
      MPI_PROF(ctx, KF_SOLVER);
      if (!fused) {
        launch_pdl(ctx, k_tv_out, dim3(blocks), dim3(256), 0, in, g, N, it ? R[0] : nullptr, out);
        MPI_LAUNCH_CHECK(ctx, "k_tv_out");
        MPI_PROF(ctx, KF_SOLVER);
        launch_pdl(ctx, k_tv_dual, dim3(blocks), dim3(256), 0, in, g, N, out, P, R[0], it == 0, c);
        MPI_LAUNCH_CHECK(ctx, "k_tv_dual");
        continue;
      }
      launch_pdl(ctx, k_tv_step, dim3(blocks), dim3(256), 0, in, g, N, it ? R[(it - 1) & 1] : nullptr, P, R[it & 1], c);
      MPI_LAUNCH_CHECK(ctx, "k_tv_step");
    }
    MPI_PROF(ctx, KF_SOLVER);
    launch_pdl(ctx, k_tv_out, dim3(blocks), dim3(256), 0, in, g, N, n_iter ? P : nullptr, out);
    MPI_LAUNCH_CHECK(ctx, "k_tv_out");
    return MPI_OK;
  }
  // 2D: launches of up to kTileIters iterations.  Output tile: 16 x 16 where that
  // is fewer pixels (halo included) for the busiest SM, else 32 x 32: at ten
  // iterations 37^2 against 53^2 pixels per tile.
  float2 *P[2] = {scratch, scratch + 4 * N}, *R[2] = {P[0] + 2 * N, P[1] + 2 * N};  // as many as there are launches to come
  int done = 0, launch = 0;
  do {
    TvTile t;
    t.ny = ny;
    t.nx = nx;
    t.iters = std::min(kTileIters, n_iter - done);
    t.first = launch == 0;
    t.last = done + t.iters == n_iter;
    for (int k = 0; k < t.iters; ++k) t.c[k] = momentum();
    long best = 0;
    for (int o : {16, 32}) {
      const long side = o + 2 * t.iters + t.last;
      const long tiles = (long)((ny + o - 1) / o) * ((nx + o - 1) / o), sms = std::max(ctx->num_sms, 1);
      const long cost = (tiles + sms - 1) / sms * side * side;
      if (!best || cost < best) {
        best = cost;
        t.oy = t.ox = o;
      }
    }
    const size_t side = t.ox + 2 * t.iters + t.last, smem = 6 * side * side * sizeof(float2);
    cudaError_t e = smem_attr(ctx, (const void*)k_tv_tile);
    if (e != cudaSuccess) return cuda_check(ctx, e, "TV tile attributes");
    const dim3 grid((unsigned)((nx + t.ox - 1) / t.ox), (unsigned)((ny + t.oy - 1) / t.oy));
    const int cur = launch & 1;
    MPI_PROF(ctx, KF_SOLVER);
    launch_pdl(ctx, k_tv_tile, grid, dim3(kTvThreads), smem, in, t, P[cur ^ 1], R[cur ^ 1], P[cur], R[cur], out);
    MPI_LAUNCH_CHECK(ctx, "k_tv_tile");
    done += t.iters;
    ++launch;
  } while (done < n_iter);
  return MPI_OK;
}
