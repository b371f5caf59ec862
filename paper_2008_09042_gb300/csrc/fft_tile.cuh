// Shared-memory FFTs of whole lines (mixed-radix Stockham stages, one warp or
// half a warp per line) and the transposed tile they are run in, used by the
// Cartesian and radial passes and by the image solver's fused ones.
//
// Every line (one row, or one column of a tile) is transformed by one warp in
// shared memory (padded by one element per 8, see pad8) with a mixed-radix
// (2, 3, 4, 5, 8) Stockham auto-sort FFT: for
// a stage of radix R after Ns points have been combined, butterfly j reads
// x[j + r N/R], r < R, multiplies input r by w^(r (j mod Ns)) with w =
// exp(-+2 pi i / (Ns R)), takes an R-point DFT and writes output r to
// (j div Ns) Ns R + (j mod Ns) + r Ns.  Each lane keeps its butterflies in
// registers across a __syncwarp, so the stage runs in place.
#pragma once

#include <cuda_runtime.h>

namespace mpi_fft {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// multiply by -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 rot90(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// R-point DFT in registers, y[a] = sum_r x[r] exp(-+2 pi i a r / R).
template <int R, bool INV>
struct Dft;

template <bool INV>
struct Dft<2, INV> {
  static __device__ __forceinline__ void go(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <bool INV>
struct Dft<4, INV> {
  static __device__ __forceinline__ void go(float2* v) {
    const float2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
    const float2 s13 = cadd(v[1], v[3]), d13 = rot90<INV>(csub(v[1], v[3]));
    v[0] = cadd(s02, s13);
    v[2] = csub(s02, s13);
    v[1] = cadd(d02, d13);
    v[3] = csub(d02, d13);
  }
};

template <bool INV>
struct Dft<8, INV> {
  static __device__ __forceinline__ void go(float2* v) {
    // two 4-point DFTs on the even and odd inputs, then the radix-2 combine
    // with twiddles exp(-+2 pi i m / 8), m = 0..3.
    float2 e[4] = {v[0], v[2], v[4], v[6]};
    float2 o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4, INV>::go(e);
    Dft<4, INV>::go(o);
    const float h = 0.70710678118654752f;  // 1/sqrt(2)
    // o[1] *= exp(-+i pi/4), o[2] *= -+i, o[3] *= exp(-+3 i pi/4)
    const float2 o1 = INV ? make_float2(h * (o[1].x - o[1].y), h * (o[1].x + o[1].y))
                          : make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
    const float2 o2 = rot90<INV>(o[2]);
    const float2 o3 = INV ? make_float2(-h * (o[3].x + o[3].y), h * (o[3].x - o[3].y))
                          : make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[5] = csub(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cadd(e[3], o3);
    v[7] = csub(e[3], o3);
  }
};

template <bool INV>
struct Dft<3, INV> {
  static __device__ __forceinline__ void go(float2* v) {
    // c = cos(2 pi / 3) = -1/2, s = sin(2 pi / 3) = sqrt(3)/2
    const float s = INV ? -0.86602540378443865f : 0.86602540378443865f;
    const float2 t = cadd(v[1], v[2]);
    const float2 d = csub(v[1], v[2]);
    const float2 m = make_float2(v[0].x - 0.5f * t.x, v[0].y - 0.5f * t.y);
    // -+ i s d
    const float2 isd = make_float2(s * d.y, -s * d.x);
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, isd);
    v[2] = csub(m, isd);
  }
};

template <bool INV>
struct Dft<5, INV> {
  static __device__ __forceinline__ void go(float2* v) {
    // c1 = cos(2 pi/5) = (sqrt 5 - 1)/4, c2 = cos(4 pi/5) = -(sqrt 5 + 1)/4,
    // s1 = sin(2 pi/5), s2 = sin(4 pi/5)
    const float c1 = 0.30901699437494742f, c2 = -0.80901699437494742f;
    const float s1 = INV ? -0.95105651629515357f : 0.95105651629515357f;
    const float s2 = INV ? -0.58778525229247313f : 0.58778525229247313f;
    const float2 a1 = cadd(v[1], v[4]), b1 = csub(v[1], v[4]);
    const float2 a2 = cadd(v[2], v[3]), b2 = csub(v[2], v[3]);
    const float2 x0 = v[0];
    const float2 r1 = make_float2(x0.x + c1 * a1.x + c2 * a2.x, x0.y + c1 * a1.y + c2 * a2.y);
    const float2 r2 = make_float2(x0.x + c2 * a1.x + c1 * a2.x, x0.y + c2 * a1.y + c1 * a2.y);
    // forward: y1 = r1 - i (s1 b1 + s2 b2), y2 = r2 - i (s2 b1 - s1 b2)
    const float2 i1 = make_float2(s1 * b1.x + s2 * b2.x, s1 * b1.y + s2 * b2.y);
    const float2 i2 = make_float2(s2 * b1.x - s1 * b2.x, s2 * b1.y - s1 * b2.y);
    v[0] = make_float2(x0.x + a1.x + a2.x, x0.y + a1.y + a2.y);
    v[1] = make_float2(r1.x + i1.y, r1.y - i1.x);
    v[4] = make_float2(r1.x - i1.y, r1.y + i1.x);
    v[2] = make_float2(r2.x + i2.y, r2.y - i2.x);
    v[3] = make_float2(r2.x - i2.y, r2.y + i2.x);
  }
};

// Shared-memory index of element i of a line: one float2 of padding per 8,
// which leaves every Stockham stage's strided loads and stores at most
// two-way bank conflicted for the supported lengths.
__host__ __device__ __forceinline__ constexpr int pad8(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int padded_len(int n) { return n + n / 8; }

// One radix-R Stockham stage of an N-point line held in shared memory, its
// N / R butterflies spread over LANES lanes (a warp, or half a warp for short
// lines, two lines per warp).
template <int N, int R, int NS, bool INV, int LANES>
__device__ __forceinline__ void fft_stage(float2* buf, const float2* tw, int lane) {
  constexpr int NB = N / R;
  constexpr int PER = (NB + LANES - 1) / LANES;
  float2 v[PER][R];
#pragma unroll
  for (int b = 0; b < PER; ++b) {
    const int j = lane + LANES * b;
    if (j < NB) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = buf[pad8(j + r * NB)];
    }
  }
  __syncwarp();
#pragma unroll
  for (int b = 0; b < PER; ++b) {
    const int j = lane + LANES * b;
    if (j < NB) {
      const int k = j % NS;
      if (NS > 1) {
        // w^r for r = 1 .. R-1 from one table read: w^r = w^(r/2) w^(r - r/2),
        // so each power is at most three products deep (a few ulp)
        float2 w[R];
        w[1] = tw[k * (N / (NS * R))];
        if (INV) w[1].y = -w[1].y;
#pragma unroll
        for (int r = 2; r < R; ++r) w[r] = cmul(w[r / 2], w[r - r / 2]);
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], w[r]);
      }
      Dft<R, INV>::go(v[b]);
      const int base = (j / NS) * NS * R + k;
#pragma unroll
      for (int r = 0; r < R; ++r) buf[pad8(base + r * NS)] = v[b][r];
    }
  }
  __syncwarp();
}

template <int N, bool INV, int LANES, int NS, int R, int... Rest>
struct Run {
  static __device__ __forceinline__ void go(float2* b, const float2* tw, int lane) {
    fft_stage<N, R, NS, INV, LANES>(b, tw, lane);
    Run<N, INV, LANES, NS * R, Rest...>::go(b, tw, lane);
  }
};
template <int N, bool INV, int LANES, int NS, int R>
struct Run<N, INV, LANES, NS, R> {
  static __device__ __forceinline__ void go(float2* b, const float2* tw, int lane) {
    fft_stage<N, R, NS, INV, LANES>(b, tw, lane);
  }
};

template <int N, bool INV>
struct Fft;
#define MPI_FFT_PLAN(n, ...)                                                    \
  template <bool INV>                                                           \
  struct Fft<n, INV> {                                                          \
    template <int LANES = 32>                                                   \
    static __device__ __forceinline__ void go(float2* b, const float2* tw, int lane) { \
      Run<n, INV, LANES, 1, __VA_ARGS__>::go(b, tw, lane);                      \
    }                                                                           \
  };
MPI_FFT_PLAN(16, 4, 4)
MPI_FFT_PLAN(32, 8, 4)
MPI_FFT_PLAN(48, 4, 4, 3)
MPI_FFT_PLAN(64, 8, 8)
MPI_FFT_PLAN(96, 8, 4, 3)
MPI_FFT_PLAN(128, 8, 4, 4)
MPI_FFT_PLAN(192, 8, 8, 3)
MPI_FFT_PLAN(256, 8, 8, 4)
MPI_FFT_PLAN(320, 8, 8, 5)
MPI_FFT_PLAN(512, 8, 8, 8)
#undef MPI_FFT_PLAN

constexpr int kRowWarps = 4;   // warps per CTA of the row passes
constexpr int kLineWarps = 8;  // warps per CTA of the line pass

// The FFTs of a line pass's TILE lines, in shared memory at buf + line * S.
// Lines of up to 128 points take half a warp each (no stage of theirs has more
// than 16 butterflies), two lines per warp; every line of the tile is
// transformed, whether or not it is stored, so both halves of a warp run the
// same stages.
template <int L, bool INV, int TILE, int S>
__device__ __forceinline__ void fft_tile_lines(float2* buf, const float2* tw, int warp, int lane) {
  if constexpr (L <= 128) {
    for (int line = 2 * warp + (lane >> 4); line < TILE; line += 2 * kLineWarps)
      Fft<L, INV>::template go<16>(buf + line * S, tw, lane & 15);
  } else {
    for (int line = warp; line < TILE; line += kLineWarps) Fft<L, INV>::go(buf + line * S, tw, lane);
  }
}

// Column stride of the transposed tile: the padded line length rounded to
// 2 mod 16 float2 for TILE <= 16 (a warp's transposing accesses then cover 8
// or 16 lines x 4 or 2 rows) and to 1 mod 16 for TILE = 32 (32 lines of one
// row); either way they take the minimum two shared-memory wavefronts.
__host__ __device__ constexpr int col_stride(int L, int TILE) {
  return padded_len(L) + (((TILE == 32 ? 1 : 2) - padded_len(L)) % 16 + 16) % 16;
}


}  // namespace mpi_fft
