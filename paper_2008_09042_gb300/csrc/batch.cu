// Batched operator application over many slices of uneven grid size and coil
// count, replayed as one CUDA graph.
//
// mpi_batch_create orders the slices by basis (slices of the same grid share
// one Maxwell basis), sizes the context workspace for the largest slice, and
// records every kernel of every slice's operator calls into one graph by stream
// capture on a private stream.  mpi_batch_run launches that graph on the
// context's stream.  The captured pointers are the caller's buffers, which must
// stay valid for the life of the batch.
//
// Grouped expansion: consecutive slices on Cartesian plans of one grid that share a
// dense basis (FP32 or BF16, every slice's coils within one tensor-core pass) form a
// group.  The group's basis expansion is one launch over its slices (device tables give
// each CTA its slices' coefficients, images, per-coil data and outputs); the CTAs stream
// the same basis tiles in step, so the basis is read from DRAM about once per group
// instead of once per slice, and slices of few coils are bundled, their coefficients
// stacked into one operand, so that one CTA reads a tile for all.  Each slice's per-coil
// images live in a batch-owned buffer between the expansion and the FFT passes.  From
// kGroupedPasses 2D slices on, the FFT passes take all coils of a group's slices in one
// launch too (per run of slices whose pass along y is of the same kind, register or
// Stockham, so that a slice's values stay those of its own call; its width is timed for
// the group), with a table of every coil's sampling.  How the slices are bundled and how
// many CTAs each bundle gets is chosen at creation by timing the candidates (an
// autotuner decision the context records).
#include <algorithm>
#include <cstdio>
#include <numeric>
#include <string>
#include <vector>

#include "mpi_internal.h"

struct mpi_batch {
  mpi_ctx* ctx = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int n = 0;
  int64_t kernels = 0;  // kernels per replay
  void* work = nullptr;  // the context's workspace block that the recorded kernels use
  void* buf = nullptr;   // per-coil images of one group [sum C][N]
  void* ctas = nullptr;  // CTA and slice tables of every group's expansions (device)
  void* tabs = nullptr;  // sampling tables and row masks of the grouped passes (device)
  int groups = 0;        // grouped launches per direction
};

namespace {

mpi_status record_slice(mpi_ctx* ctx, const mpi_batch_slice& s, int kind, mpi_precision prec) {
  mpi_status st = MPI_OK;
  if (kind & MPI_BATCH_FORWARD)
    st = mpi_forward(ctx, s.plan, s.basis, s.alpha, s.C, s.p, s.y, prec);
  if (st == MPI_OK && (kind & MPI_BATCH_ADJOINT))
    st = mpi_adjoint(ctx, s.plan, s.basis, s.alpha, s.C, s.y, s.x, prec);
  return st;
}

// Slices a group needs for its FFT passes to be grouped.  A launch of its own costs a
// slice 5-14 us per pass (8-32 coils of 128^2 to 320^2), much of it fixed: 16 slices
// of 128^2 took 90 us in 16 row passes and 22 in one, of 320^2 219 and 131.  Two or
// three slices save a few microseconds at most and keep the passes of their own calls.
constexpr int kGroupedPasses = 4;

struct Group {
  std::vector<int> idx;  // slices, in recording order
  int Cmax = 0;
  long sumC = 0;
  // grouped expansions: the launches' CTA and slice tables (device), their CTAs and
  // the coils of the largest bundle
  ExpandRow *fwd_ctas = nullptr, *adj_ctas = nullptr;
  ExpandSeg *fwd_segs = nullptr, *adj_segs = nullptr;
  int n_ctas = 0, coils = 0;
  // grouped passes: runs of slices (first, count in coils) per direction and kernel
  struct Run {
    bool registers;
    int first, coils, kernel;
  };
  std::vector<Run> fwd, inv;  // empty: the passes run slice by slice
  const CoilSamples* tab = nullptr;
  const uint8_t* row_has = nullptr;
  int n_list = 0;  // the most rows with samples that any slice has
};

bool groupable(const mpi_batch_slice& s, mpi_precision prec) {
  return s.plan->kind == MPI_TRAJ_CARTESIAN && !s.basis->tucker && rows_supported(s.basis, s.C, prec);
}

// Whether two plans have the same grid: slices of equal N and nx may still be a 2D
// slice and a volume, or volumes split differently into y and z, whose centring signs
// and passes differ.
bool same_grid(const mpi_plan* a, const mpi_plan* b) {
  return a->ndim == b->ndim && a->nz == b->nz && a->ny == b->ny && a->nx == b->nx;
}

// The group's forward and adjoint expansions, and its slices' FFT passes.
mpi_status record_group(mpi_ctx* ctx, const mpi_batch_slice* sl, const Group& g, int kind, mpi_precision prec, float2* buf) {
  const mpi_batch_slice& s0 = sl[g.idx[0]];
  const long N = s0.plan->N;
  const int nr = (int)g.idx.size(), ny = s0.plan->ny, nx = s0.plan->nx;
  mpi_status st = MPI_OK;
  if (kind & MPI_BATCH_FORWARD) {
    st = expand_rows(ctx, s0.plan, s0.basis, EX_FWD, g.fwd_ctas, g.n_ctas, g.coils, prec);
    for (const Group::Run& r : g.fwd)
      if (st == MPI_OK)
        st = launch_fft_cols_group(ctx, r.kernel, buf + r.first * N, r.coils, ny, nx, false,
                                   g.row_has ? g.row_has + (size_t)r.first * ny : nullptr);
    if (st == MPI_OK && !g.fwd.empty()) st = launch_rows_group(ctx, buf, (int)g.sumC, ny, nx, false, g.tab, g.n_list);
    long off = 0;
    for (int i = 0; i < nr && st == MPI_OK && g.fwd.empty(); ++i) {
      const mpi_batch_slice& s = sl[g.idx[i]];
      st = plan_image_to_kspace(ctx, s.plan, buf + off * N, s.C, (float2*)s.y);
      off += s.C;
    }
  }
  if (st == MPI_OK && (kind & MPI_BATCH_ADJOINT)) {
    if (!g.inv.empty()) st = launch_rows_group(ctx, buf, (int)g.sumC, ny, nx, true, g.tab, g.n_list);
    for (const Group::Run& r : g.inv)
      if (st == MPI_OK)
        st = launch_fft_cols_group(ctx, r.kernel, buf + r.first * N, r.coils, ny, nx, true,
                                   g.row_has ? g.row_has + (size_t)r.first * ny : nullptr);
    long off = 0;
    for (int i = 0; i < nr && st == MPI_OK && g.inv.empty(); ++i) {
      const mpi_batch_slice& s = sl[g.idx[i]];
      st = plan_kspace_to_image(ctx, s.plan, (const float2*)s.y, s.C, buf + off * N);
      off += s.C;
    }
    if (st == MPI_OK) st = expand_rows(ctx, s0.plan, s0.basis, EX_ADJ, g.adj_ctas, g.n_ctas, g.coils, prec);
  }
  return st;
}

// Runs of the group's slices (already in an order that keeps equal kinds together)
// whose pass along y is of the same kind.
std::vector<Group::Run> pass_runs(mpi_ctx* ctx, const mpi_batch_slice* sl, const Group& g, bool inverse) {
  std::vector<Group::Run> runs;
  int off = 0;
  for (int i : g.idx) {
    const bool k = fft_cols_in_registers(ctx, sl[i].plan, sl[i].C, inverse);
    if (runs.empty() || runs.back().registers != k) runs.push_back({k, off, 0, 0});
    runs.back().coils += sl[i].C;
    off += sl[i].C;
  }
  return runs;
}

// The grouped passes' tables: every coil's sampling (idx, row_ptr, its samples) and,
// where some slice has rows without samples, every coil's row mask.
mpi_status group_tables(mpi_ctx* ctx, const mpi_batch_slice* sl, std::vector<Group>& groups, void** out) {
  std::vector<size_t> tab_off, mask_off;
  size_t bytes = 0;
  for (const Group& g : groups) {
    if (g.fwd.empty()) continue;
    tab_off.push_back(bytes);
    bytes += ((size_t)g.sumC * sizeof(CoilSamples) + 255) & ~(size_t)255;
    mask_off.push_back(bytes);
    bytes += ((size_t)g.sumC * sl[g.idx[0]].plan->ny + 255) & ~(size_t)255;
  }
  if (!bytes) return MPI_OK;
  cudaError_t e = cudaMalloc(out, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, MPI_ERR_OOM, "batch: group tables");
  }
  std::vector<unsigned char> host(bytes, 1);
  size_t k = 0;
  for (Group& g : groups) {
    if (g.fwd.empty()) continue;
    CoilSamples* tab = (CoilSamples*)(host.data() + tab_off[k]);
    const int ny = sl[g.idx[0]].plan->ny;
    long off = 0;
    bool masked = false;
    for (int i : g.idx) {
      const mpi_batch_slice& s = sl[i];
      unsigned char* m = host.data() + mask_off[k] + (size_t)off * ny;
      if (s.plan->row_has) {
        masked = true;
        e = cudaMemcpy(m, s.plan->row_has, ny, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_check(ctx, e, "batch: group tables");
        for (int c = 1; c < s.C; ++c) std::copy(m, m + ny, m + (size_t)c * ny);
      }
      for (int c = 0; c < s.C; ++c)
        tab[off + c] = CoilSamples{s.plan->idx,      s.plan->row_ptr, s.plan->row_list,
                                   s.plan->n_list, (float2*)s.y + (size_t)c * s.plan->M};
      g.n_list = std::max(g.n_list, s.plan->n_list);
      off += s.C;
    }
    g.tab = (const CoilSamples*)((char*)*out + tab_off[k]);
    g.row_has = masked ? (const uint8_t*)*out + mask_off[k] : nullptr;
    ++k;
  }
  return cuda_check(ctx, cudaMemcpy(*out, host.data(), bytes, cudaMemcpyHostToDevice), "batch: group tables");
}

// How a group's expansions are laid out: bundles of slices up to `chunks` x 8 coils
// (0: every slice alone), `total` CTAs shared out over them with `skew`.
struct Layout {
  int chunks, total;
  float skew;
};

int slice_chunks(const mpi_batch_slice& s) { return (s.C + 7) / 8; }

// The launches' tables.  Slices are bundled (largest first, each into the first bundle
// with room), since a bundle's CTAs load and split each tile of the basis once for all
// of its slices; more columns leave less room for the ring beside the coefficients.
// The CTAs, `total` of them (one per bundle at least), are shared out in proportion to
// 1 + skew x (a bundle's columns / 64).  A slice's values do not depend on either.
void layout_tables(const mpi_batch_slice* sl, Group& g, const Layout& lay, float2* buf, int n_tiles,
                   std::vector<ExpandRow> (&ctas)[2], std::vector<ExpandSeg> (&segs)[2]) {
  const int n = (int)g.idx.size();
  const long N = sl[g.idx[0]].plan->N;
  std::vector<long> off(n);
  std::vector<int> order(n);
  long sum = 0;
  for (int i = 0; i < n; ++i) {
    off[i] = sum;
    order[i] = i;
    sum += sl[g.idx[i]].C;
  }
  std::stable_sort(order.begin(), order.end(),
                   [&](int a, int b) { return slice_chunks(sl[g.idx[a]]) > slice_chunks(sl[g.idx[b]]); });
  struct Bundle {
    std::vector<int> slices;
    int chunks;
  };
  std::vector<Bundle> bundles;
  for (int i : order) {
    const int ch = slice_chunks(sl[g.idx[i]]);
    size_t b = 0;
    while (b < bundles.size() && bundles[b].chunks + ch > lay.chunks) ++b;
    if (b == bundles.size()) bundles.push_back({{}, 0});
    bundles[b].slices.push_back(i);
    bundles[b].chunks += ch;
  }
  const int nb = (int)bundles.size();
  std::vector<float> w(nb);
  std::vector<int> share(nb, 1);
  for (int b = 0; b < nb; ++b) w[b] = 1.f + lay.skew * (float)bundles[b].chunks / 4.f;
  for (int used = nb; used < lay.total; ++used) {
    int most = -1;
    for (int b = 0; b < nb; ++b)
      if (share[b] < n_tiles && (most < 0 || w[b] * share[most] > w[most] * share[b])) most = b;
    if (most < 0) break;
    ++share[most];
  }
  g.coils = 0;
  for (int d = 0; d < 2; ++d) {
    ctas[d].clear();
    segs[d].clear();
  }
  for (int b = 0; b < nb; ++b) {
    const size_t first = segs[0].size();
    int chunk = 0;
    for (int i : bundles[b].slices) {
      const mpi_batch_slice& s = sl[g.idx[i]];
      float2* W = buf + off[i] * N;
      segs[0].push_back(ExpandSeg{(const float2*)s.alpha, (const float2*)s.p, nullptr, W, s.C, chunk});
      segs[1].push_back(ExpandSeg{(const float2*)s.alpha, nullptr, W, (float2*)s.x, s.C, chunk});
      chunk += slice_chunks(s);
    }
    g.coils = std::max(g.coils, 8 * chunk);
    const int ns = (int)bundles[b].slices.size();
    for (int k = 0; k < share[b]; ++k) {
      ctas[0].push_back(ExpandRow{g.fwd_segs + first, ns, chunk, k, share[b]});
      ctas[1].push_back(ExpandRow{g.adj_segs + first, ns, chunk, k, share[b]});
    }
  }
  g.n_ctas = (int)ctas[0].size();
}

// The most CTAs a group's launch may have.
int most_ctas(const mpi_ctx* ctx, const Group& g) { return std::max(2 * std::max(ctx->num_sms, 1), (int)g.idx.size()); }

// Layout of a group's expansions: every candidate timed over three launches of the
// group's forward expansion (between events on the context's stream, after one
// warm-up launch), the fastest kept.  FP32 CTAs fill an SM each, BF16 ones half.
mpi_status tune_group(mpi_ctx* ctx, const mpi_batch_slice* sl, Group& g, mpi_precision prec, float2* buf) {
  const mpi_batch_slice& s0 = sl[g.idx[0]];
  const int nr = (int)g.idx.size(), n_tiles = (int)((s0.plan->N + 127) / 128);
  const int fill = std::max(ctx->num_sms, 1) * (prec == MPI_PREC_BF16 ? 2 : 1);
  const int most = (g.Cmax + 7) / 8;
  // An FP32 tile's time hardly depends on its coils: streaming and splitting U for every
  // slice is most of it.  16 slices of 320^2, q = 160, with 8, 16 and 32 coils: 331 us with
  // every slice in the largest one's operand, 296 alone in its own, 223 in bundles of 32
  // coils; of 192^2, q = 96, 81 alone and 88 in bundles.  BF16 tiles are bound by their
  // epilogues, which bundles do not share (120 us against 90): shares by coils instead.
  std::vector<Layout> cands = {{0, fill, 0.f}, {0, fill, 1.f}};
  if (prec == MPI_PREC_BF16) {
    cands.push_back({0, fill, 3.f});
  } else {
    cands.push_back({most, fill, 0.f});
    if (most < 4 && rows_supported(s0.basis, 32, prec)) cands.push_back({4, fill, 0.f});
  }
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    cudaGetLastError();
    return set_err(ctx, MPI_ERR_CUDA, "grouped batch: tuning events");
  }
  std::string rec = std::string("grouped expansion (") + std::to_string(nr) + " slices, N=" +
                    std::to_string(s0.plan->N) + ", q=" + std::to_string(s0.basis->q) + ", sumC=" +
                    std::to_string(g.sumC) + ", " + (prec == MPI_PREC_BF16 ? "bf16" : "fp32") + "):";
  float best = 1e30f;
  int pick = 0;
  mpi_status st = MPI_OK;
  std::vector<ExpandRow> ctas[2];
  std::vector<ExpandSeg> segs[2];
  auto upload = [&](const Layout& lay) {
    layout_tables(sl, g, lay, buf, n_tiles, ctas, segs);
    cudaError_t e = cudaStreamSynchronize(ctx->stream);  // the launches that read the last tables
    for (int d = 0; d < 2 && e == cudaSuccess; ++d) {
      e = cudaMemcpy(d ? g.adj_ctas : g.fwd_ctas, ctas[d].data(), ctas[d].size() * sizeof(ExpandRow),
                     cudaMemcpyHostToDevice);
      if (e == cudaSuccess)
        e = cudaMemcpy(d ? g.adj_segs : g.fwd_segs, segs[d].data(), segs[d].size() * sizeof(ExpandSeg),
                       cudaMemcpyHostToDevice);
    }
    return cuda_check(ctx, e, "batch: expansion tables");
  };
  for (int k = 0; k < (int)cands.size(); ++k) {
    st = upload(cands[k]);
    if (st == MPI_OK) st = expand_rows(ctx, s0.plan, s0.basis, EX_FWD, g.fwd_ctas, g.n_ctas, g.coils, prec);
    if (st) break;
    cudaEventRecord(e0, ctx->stream);
    for (int r = 0; r < 3 && st == MPI_OK; ++r)
      st = expand_rows(ctx, s0.plan, s0.basis, EX_FWD, g.fwd_ctas, g.n_ctas, g.coils, prec);
    cudaEventRecord(e1, ctx->stream);
    if (st) break;
    if (cudaEventSynchronize(e1) != cudaSuccess) {
      st = cuda_check(ctx, cudaGetLastError(), "grouped batch tuning");
      break;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    char line[96];
    snprintf(line, sizeof(line), " %d CTAs, bundles of %d, skew %g: %.2f us;", g.n_ctas, 8 * cands[k].chunks,
             cands[k].skew, ms / 3 * 1e3);
    rec += line;
    if (ms < best) {
      best = ms;
      pick = k;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st == MPI_OK) st = upload(cands[pick]);
  if (st) return st;
  mpi_ctx::TuneRecord tr{};
  tr.key[0] = -1;  // not a line-pass record
  tr.choice = g.n_ctas;
  char line[96];
  snprintf(line, sizeof(line), " chose %d, bundles of %d, skew %g (%.2f us)", g.n_ctas, 8 * cands[pick].chunks,
           cands[pick].skew, best / 3 * 1e3);
  tr.what = rec + line;
  ctx->tuned.push_back(tr);
  return MPI_OK;
}

}  // namespace

extern "C" mpi_status mpi_batch_create(mpi_ctx* ctx, const mpi_batch_slice* slices, int n, int kind,
                                       mpi_precision prec, mpi_batch** out) {
  if (!ctx) return MPI_ERR_ARG;
  if (!slices || n < 1 || !out || kind < 1 || kind > 3) return set_err(ctx, MPI_ERR_ARG, "batch: bad argument");
  *out = nullptr;
  cudaSetDevice(ctx->device);
  for (int i = 0; i < n; ++i) {
    const mpi_batch_slice& s = slices[i];
    if (!s.plan || !s.basis || !s.alpha || s.C < 1 || !s.p || !s.x || (s.plan->M > 0 && !s.y))
      return set_err(ctx, MPI_ERR_ARG, "batch: incomplete slice " + std::to_string(i));
    // reserve the workspace outside the capture (no allocation may happen inside it)
    mpi_status st = mpi_ctx_reserve(ctx, s.plan, s.basis, s.C);
    if (st) return st;
  }
  // tune the slices' FFT line passes now: no tuning happens inside the capture
  for (int i = 0; i < n; ++i) {
    mpi_status st = mpi_ctx_reserve(ctx, slices[i].plan, slices[i].basis, slices[i].C);
    if (st == MPI_OK) st = tune_line_passes(ctx, slices[i].plan, slices[i].C);
    if (st) return st;
  }
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(),
                   [&](int a, int b) { return slices[a].basis < slices[b].basis; });

  // groups: runs of groupable slices on one basis (and one grid); the rest alone
  std::vector<Group> groups;
  std::vector<int> solo;
  std::vector<std::pair<int, int>> seq;  // recording order: (0, group) or (1, slice)
  for (int i = 0; i < n;) {
    int j = i;
    const mpi_batch_slice& a = slices[order[i]];
    while (j < n && slices[order[j]].basis == a.basis && groupable(slices[order[j]], prec) && groupable(a, prec) &&
           same_grid(slices[order[j]].plan, a.plan))
      ++j;
    if (j - i >= 2) {
      Group g;
      for (int k = i; k < j; ++k) {
        g.idx.push_back(order[k]);
        g.Cmax = std::max(g.Cmax, slices[order[k]].C);
        g.sumC += slices[order[k]].C;
      }
      if (rows_supported(a.basis, g.Cmax, prec)) {
        seq.push_back({0, (int)groups.size()});
        groups.push_back(g);
        i = j;
        continue;
      }
    }
    seq.push_back({1, order[i]});
    ++i;
  }

  // grouped passes (2D; volumes keep the passes of their own calls): slices in the order
  // of the kinds of their passes along y
  for (Group& g : groups) {
    if ((int)g.idx.size() < kGroupedPasses || ctx->line_kernel || slices[g.idx[0]].plan->ndim != 2) continue;
    std::stable_sort(g.idx.begin(), g.idx.end(), [&](int a, int b) {
      const mpi_batch_slice &x = slices[a], &y = slices[b];
      const bool fa = fft_cols_in_registers(ctx, x.plan, x.C, false), fb = fft_cols_in_registers(ctx, y.plan, y.C, false);
      if (fa != fb) return fa < fb;
      return fft_cols_in_registers(ctx, x.plan, x.C, true) < fft_cols_in_registers(ctx, y.plan, y.C, true);
    });
    g.fwd = pass_runs(ctx, slices, g, false);
    g.inv = pass_runs(ctx, slices, g, true);
  }

  mpi_batch* bt = new mpi_batch();
  bt->ctx = ctx;
  bt->n = n;
  bt->groups = (int)groups.size();
  // the group buffer and the CTA tables
  size_t buf_elems = 0, n_ctas = 0, n_segs = 0;
  for (Group& g : groups) {
    buf_elems = std::max(buf_elems, (size_t)g.sumC * slices[g.idx[0]].plan->N);
    n_ctas += 2 * (size_t)most_ctas(ctx, g);
    n_segs += 2 * g.idx.size();
  }
  cudaError_t e = cudaSuccess;
  if (!groups.empty()) {
    e = cudaMalloc(&bt->buf, buf_elems * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc(&bt->ctas, n_ctas * sizeof(ExpandRow) + n_segs * sizeof(ExpandSeg));
    if (e != cudaSuccess) {
      cudaGetLastError();
      mpi_batch_destroy(bt);
      return set_err(ctx, MPI_ERR_OOM, "batch: group buffers");
    }
    ExpandRow* ctas = (ExpandRow*)bt->ctas;
    ExpandSeg* segs = (ExpandSeg*)(ctas + n_ctas);
    for (Group& g : groups) {
      g.fwd_ctas = ctas;
      g.adj_ctas = ctas + most_ctas(ctx, g);
      ctas += 2 * most_ctas(ctx, g);
      g.fwd_segs = segs;
      g.adj_segs = segs + g.idx.size();
      segs += 2 * g.idx.size();
    }
    mpi_status st = group_tables(ctx, slices, groups, &bt->tabs);
    if (st) {
      mpi_batch_destroy(bt);
      return st;
    }
    for (Group& g : groups) {
      mpi_status st = tune_group(ctx, slices, g, prec, (float2*)bt->buf);
      const mpi_plan* pl = slices[g.idx[0]].plan;
      for (int dir = 0; dir < 2; ++dir)
        for (Group::Run& r : dir ? g.inv : g.fwd)
          if (st == MPI_OK)
            st = tune_fft_cols_group(ctx, r.registers, (float2*)bt->buf + (size_t)r.first * pl->N, r.coils, pl->ny,
                                     pl->nx, dir == 1, g.row_has ? g.row_has + (size_t)r.first * pl->ny : nullptr,
                                     &r.kernel);
      if (st) {
        mpi_batch_destroy(bt);
        return st;
      }
    }
  }

  cudaStream_t cap = nullptr, user = ctx->stream;
  e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    mpi_batch_destroy(bt);
    return cuda_check(ctx, e, "batch stream");
  }
  // the capture must not wait on work still queued on the user's stream
  e = cudaStreamSynchronize(user);
  const bool prof = ctx->profiling;
  ctx->profiling = false;
  ctx->stream = cap;
  const int64_t l0 = ctx->launches;
  mpi_status st = MPI_OK;
  if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed);
  if (e == cudaSuccess) {
    for (size_t i = 0; i < seq.size() && st == MPI_OK; ++i) {
      if (seq[i].first == 0)
        st = record_group(ctx, slices, groups[seq[i].second], kind, prec, (float2*)bt->buf);
      else
        st = record_slice(ctx, slices[seq[i].second], kind, prec);
    }
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cap, &g);
    if (st == MPI_OK && e2 == cudaSuccess) {
      bt->graph = g;
      e2 = cudaGraphInstantiate(&bt->exec, g, 0);
    } else if (g) {
      cudaGraphDestroy(g);
    }
    if (st == MPI_OK && e2 != cudaSuccess) st = cuda_check(ctx, e2, "batch graph capture");
  } else {
    st = cuda_check(ctx, e, "batch capture begin");
  }
  bt->kernels = ctx->launches - l0;
  ctx->launches = l0;
  ctx->stream = user;
  ctx->profiling = prof;
  cudaStreamDestroy(cap);
  if (st != MPI_OK) {
    mpi_batch_destroy(bt);
    return st;
  }
  ctx_adopt(ctx, &bt->ctx);
  if (ctx->work) {
    bt->work = ctx->work;
    ctx->work_users.push_back(bt->work);
  }
  *out = bt;
  return MPI_OK;
}

extern "C" mpi_status mpi_batch_run(mpi_ctx* ctx, mpi_batch* bt) {
  if (!ctx) return MPI_ERR_ARG;
  if (!bt || bt->ctx != ctx || !bt->exec) return set_err(ctx, MPI_ERR_ARG, "batch: bad handle");
  cudaSetDevice(ctx->device);
  cudaError_t e = cudaGraphLaunch(bt->exec, ctx->stream);
  if (e != cudaSuccess) return cuda_check(ctx, e, "batch graph launch");
  ctx->launches += bt->kernels;
  return MPI_OK;
}

extern "C" int64_t mpi_batch_kernel_count(const mpi_batch* bt) { return bt ? bt->kernels : -1; }

extern "C" int mpi_batch_group_count(const mpi_batch* bt) { return bt ? bt->groups : -1; }

extern "C" mpi_status mpi_batch_destroy(mpi_batch* bt) {
  if (!bt) return MPI_ERR_ARG;
  if (bt->ctx && (bt->buf || bt->ctas || bt->tabs)) cudaStreamSynchronize(bt->ctx->stream);  // a replay may still run
  if (bt->ctx && bt->work) work_release(bt->ctx, bt->work);
  ctx_release(&bt->ctx);
  if (bt->exec) cudaGraphExecDestroy(bt->exec);
  if (bt->graph) cudaGraphDestroy(bt->graph);
  if (bt->buf) cudaFree(bt->buf);
  if (bt->ctas) cudaFree(bt->ctas);
  if (bt->tabs) cudaFree(bt->tabs);
  delete bt;
  return MPI_OK;
}
