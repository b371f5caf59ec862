// FFTs of contiguous rows in two register steps.  N = A P, P a power of two; row
// element n = p + P a.  Step 1: one lane per (row, p) takes the A-point DFT over a
// in registers and multiplies by w_N^(p k1); step 2: one lane per (row, k1) takes
// the P-point DFT over p; output k = k1 + A k2.  Between them one exchange through
// shared memory, so an element is written and read once there (a Stockham line
// takes that per radix stage) and the work per element is about a third: a
// 320-point row took some 1,150 warp instructions as 8 x 8 x 5 stages, most of them
// twiddle powers and index arithmetic, and the passes were bound by issuing them.
// The inverse is the forward of the conjugated data, conjugated back.
//
// A warp works on R rows at a time, R the fewest that give every lane a task of step
// 1 (more rows per warp mean fewer warps: at 320 points, four rows instead of two made
// a 16-coil slice's passes slower for all their shared second step saved).  Exchange layout of row r: value (k1, p) at r S + k1 (P + 1) + p, which
// keeps both steps' accesses free of bank conflicts (S = P mod 16 for P < 16); the
// outputs (k1, k2) go back to the same places.
#pragma once

#include "dft_reg.cuh"

namespace mpi_fft {

template <int N> struct RowSplit;
#define MPI_ROW_SPLIT(n, p, r)                      \
  template <> struct RowSplit<n> {                  \
    static constexpr int P = p, A = n / p, R = r;   \
  };
MPI_ROW_SPLIT(16, 4, 8)
MPI_ROW_SPLIT(32, 4, 8)
MPI_ROW_SPLIT(48, 4, 8)
MPI_ROW_SPLIT(64, 8, 4)
MPI_ROW_SPLIT(96, 8, 4)
MPI_ROW_SPLIT(128, 8, 4)
MPI_ROW_SPLIT(192, 16, 2)
MPI_ROW_SPLIT(256, 16, 2)
MPI_ROW_SPLIT(320, 16, 2)
MPI_ROW_SPLIT(512, 16, 2)
#undef MPI_ROW_SPLIT

template <int N>
struct Rows {
  static constexpr int P = RowSplit<N>::P, A = RowSplit<N>::A, R = RowSplit<N>::R;
  static constexpr int S = P < 16 ? A * (P + 1) + ((P - A * (P + 1)) % 16 + 16) % 16 : A * (P + 1);
  static constexpr int T1 = R * P / 32;             // step 1 tasks per lane
  static constexpr int T2 = (R * A + 31) / 32;      // step 2 tasks per lane (the last may be partial)
  static_assert(R * P % 32 == 0, "whole warps in step 1");
  static constexpr int kSmem = R * S;               // values per warp

  // place of input element n and of output element k of row r in the exchange
  static __device__ __forceinline__ int in_at(int r, int n) { return r * S + n / P * (P + 1) + n % P; }
  static __device__ __forceinline__ int out_at(int r, int k) { return r * S + k % A * (P + 1) + k / A; }

  // The samples of R rows with samples that follow one another in a coil's sorted list
  // are contiguous there.  use(m, r, kx, load(m)) for samples [m0, m1) of the rows
  // row[0 .. R) (ascending; unused ones past the last), spread over the lanes, four
  // per lane whose loads are all issued before the first use: the rows' own loops, one
  // after the other, would each wait for their loads in turn.
  template <class Idx, class Load, class Use>
  static __device__ __forceinline__ void samples(const int (&row)[R], int m0, int m1, int lane, Idx idx, Load load,
                                                 Use use) {
    for (int m = m0 + lane; m < m1; m += 128) {
      int k[4];
      decltype(load(0)) v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (m + 32 * j < m1) {
          k[j] = idx(m + 32 * j);
          v[j] = load(m + 32 * j);
        }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (m + 32 * j < m1) {
          const int y = k[j] / N;
          int r = 0;
#pragma unroll
          for (int i = 1; i < R; ++i) r += y >= row[i];
          use(m + 32 * j, r, k[j] - y * N, v[j]);
        }
    }
  }

  // Step 1 of the lane's task (row r, p): v[a] = element p + P a.
  template <bool INV>
  static __device__ __forceinline__ void step1(float2 (&v)[A], int r, int p, float2* b, const float2* __restrict__ tw) {
    float2 w[A];
#pragma unroll
    for (int k = 1; k < A; ++k) w[k] = __ldg(tw + p * k);
    if (INV)
#pragma unroll
      for (int a = 0; a < A; ++a) v[a].y = -v[a].y;
    mpi_dft::dft_r<A>(v);
#pragma unroll
    for (int k = 0; k < A; ++k) b[r * S + k * (P + 1) + p] = k ? mpi_dft::cmulf(v[k], w[k]) : v[0];
  }

  // Step 2 of the lane's task (row r, k1): u[k2] = output k1 + A k2.
  template <bool INV>
  static __device__ __forceinline__ void step2(float2 (&u)[P], int r, int k1, const float2* b) {
#pragma unroll
    for (int p = 0; p < P; ++p) u[p] = b[r * S + k1 * (P + 1) + p];
    mpi_dft::dft_r<P>(u);
    if (INV)
#pragma unroll
      for (int k = 0; k < P; ++k) u[k].y = -u[k].y;
  }
};

}  // namespace mpi_fft
