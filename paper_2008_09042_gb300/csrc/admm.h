// The image solver with its maps kept for the solve (admm.cu), used by
// mpi_image_solve and mpi_image_solve_dynamic for 2D Cartesian plans with a dense
// basis; every other combination runs on the operator calls (solvers.cu).
#pragma once

#include "mpi_internal.h"

// Buffers of one recorded solve over T frames: its inputs and outputs, the maps,
// the state and the frames' sampling tables, all in one allocation.
struct AdmmMaps {
  float2 *in_y, *in_alpha;
  double *in_eps, *hist;
  float2 *S, *S_cg;  // maps of the outer products and of the CG (the same unless MIXED)
  float2* W;         // [T][C][N]
  float2 *p, *u0, *ap, *uk, *zk;
  float2 *z0, *r, *d[2], *Ad, *p_prev, *tv;
  unsigned* counter;  // the dual's arrivals
  char* zero_begin;
  size_t zero_bytes;
  double* sc;
  void *ball, *part, *row_part;  // partial sums (admm.cu)
  int32_t *idx, *row_ptr, *row_list, *n_list;
  uint8_t *rmask, *mask;
  bool whole_rows;  // every k-space row of every frame is sampled whole or not at all
};

bool admm_maps_supported(const mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                         mpi_precision prec);
// Carves `mem` (may be null: only the size is wanted); returns the bytes needed.
size_t admm_maps_layout(const mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                        const mpi_admm_params* prm, mpi_precision prec, void* mem, AdmmMaps* m);
// Fills the sampling tables (synchronises; before the capture).
mpi_status admm_maps_tables(mpi_ctx* ctx, const mpi_plan* const* plans, int T, AdmmMaps* m);
// Enqueues the solve on the context's stream; the image is left in m.p.
mpi_status admm_maps_record(mpi_ctx* ctx, const mpi_plan* const* plans, int T, const mpi_basis* basis, int C,
                            const mpi_admm_params* prm, mpi_precision prec, const AdmmMaps& m);
