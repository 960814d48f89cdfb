// C-ABI of libamrmhd.so (declared in include/amrmhd.h): context, hierarchy,
// arena binding, state I/O, the level operations (fill, advance, reflux and
// restriction, CFL) and the CUDA-graph coarse step.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <unordered_map>
#include <vector>

#include "ctx.hpp"
#include "fp_bits.cuh"

using amrk::DPatch;
using amrk::LevelArgs;
using amrk::RowArgs;
using namespace amrapi;

namespace amrapi {

amrmhd_status fail(amrmhd_ctx* c, amrmhd_status s, const std::string& m) {
  if (c) c->err = m;
  return s;
}

#define CU(call)                                                                                   \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// dt history capacity of one amrmhd_step chunk (the graphs bake this buffer in)
constexpr int64_t kHistCap = 4096;

void free_device(amrmhd_ctx* ctx) {
  adj_free(ctx);
  for (cudaStream_t st : ctx->side) cudaStreamDestroy(st);
  for (cudaEvent_t e : ctx->ev_fork) cudaEventDestroy(e);
  for (cudaEvent_t e : ctx->ev_join) cudaEventDestroy(e);
  ctx->side.clear();
  ctx->ev_fork.clear();
  ctx->ev_join.clear();
  if (ctx->cfl_stream) cudaStreamDestroy(ctx->cfl_stream);
  if (ctx->ev_cfl_fork) cudaEventDestroy(ctx->ev_cfl_fork);
  if (ctx->ev_cfl_join) cudaEventDestroy(ctx->ev_cfl_join);
  ctx->cfl_stream = nullptr;
  ctx->ev_cfl_fork = ctx->ev_cfl_join = nullptr;
  ctx->tile_level.clear();
  ctx->zlen_level.clear();
  for (int i = 0; i < 2; ++i)
    if (ctx->gexec[i]) { cudaGraphExecDestroy(ctx->gexec[i]); ctx->gexec[i] = nullptr; }
  for (void* p : ctx->dev_allocs) cudaFree(p);
  ctx->dev_allocs.clear();
  ctx->d_stage_all = nullptr;
  ctx->lev.clear();
  ctx->qplan = QueuePlan();
  ctx->bound = false;
}

template <class T> T* dbuf(amrmhd_ctx* ctx, size_t count, cudaError_t* e) {
  void* p = nullptr;
  *e = cudaMalloc(&p, std::max<size_t>(count, 1) * sizeof(T));
  if (*e == cudaSuccess) ctx->dev_allocs.push_back(p);
  return (T*)p;
}

void* state_buf(amrmhd_ctx* ctx, int b) { return ctx->arena + ctx->o_state[b]; }

LevelArgs level_args(amrmhd_ctx* ctx, int l, const double* dtp, double dtscale, int w) {
  LevelArgs a;
  const LevelDev& L = ctx->lev[l];
  a.P = ctx->dP;
  a.ids = L.ids;
  a.npatch = L.npatch;
  for (int d = 0; d < 3; ++d) a.maxn[d] = L.maxn[d];
  a.cur = state_buf(ctx, ctx->cur[l]);
  a.nxt = state_buf(ctx, ctx->cur[l] ^ 1);
  a.scr = ctx->stage_base ? ctx->stage_base : (void*)(ctx->arena + ctx->o_scr);
  a.dtp = dtp;
  a.dtscale = dtscale;
  for (int d = 0; d < 3; ++d) {
    int N = d < ctx->cfg.dim ? (ctx->cfg.base[d] << l) : 1;
    double dx = d < ctx->cfg.dim ? (ctx->cfg.hi[d] - ctx->cfg.lo[d]) / N : 1.0;
    a.idx[d] = 1.0 / dx;
  }
  a.gamma = ctx->cfg.gamma;
  a.igm1 = 1.0 / (ctx->cfg.gamma - 1.0);
  a.w = w;
  a.zlen = 0;
  a.tail = 0;
  a.bnd = (l > 0 && ctx->bnd_elems > 0) ? (void*)(ctx->arena + ctx->o_bnd) : nullptr;
  a.nbr = nullptr;
  a.keep = 0;
  a.fl = ctx->floors();
  return a;
}

// The launch shape of the fused mixed-precision advance of a level nobody has
// autotuned: the tile variant and z chunk of the least predicted time, from the
// extents of its patches' regions (each with its number) and the SM count. A CTA's
// plane takes about a + b faces microseconds (the HLLD faces of its tile) with
// the SM full, and nearly as long with the SM to itself: the march is a chain
// of dependent phases. So a level that does not fill the GPU runs fastest in
// as many CTAs as fit at once, each with a short march (3.4 planes' time goes
// into its start and end), and a level of many waves in the tile of the least
// time per cell. The constants are measured on 16x8, 16x16, 8x8 and 10x10 tiles
// of 8 to 4096 patches; over 70 shapes of 10 levels (8 to 72 patches of 16 to 24
// cells, w = 0 and 2) the shape of the least predicted time is on average 6 %
// slower than the fastest one, 16x8 whole columns (the choice before) 37 %.
// 8 patches of 16^3: 61 -> 19 us, 64 extended patches of 16^3: 143 -> 100 us
// (the kernel the constants were measured on took 72 -> 24 and 188 -> 119; whole
// steps of 14 other hierarchies take 1.3 % longer than autotuned on average).
void default_shape(const std::map<std::array<int, 3>, int>& patches, int grow, int sms, int* tile, int* zlen) {
  struct Shape {
    int v, tx, ty, ctas;
    double a, b;
  };
  static const Shape shapes[4] = {{2, 16, 8, 2, 1.9, 0.0061},
                                  {1, 16, 16, 1, 1.9, 0.0033},
                                  {3, 8, 8, 3, 1.9, 0.0074},
                                  {4, 10, 10, 2, 1.9, 0.0061}};
  static const int zl[8] = {0, 16, 12, 8, 6, 4, 3, 2};
  double best = 0.0;
  *tile = 2;
  *zlen = 0;
  // per region: columns of all its patches, cost of a plane, planes
  struct Col {
    double m, t;
    int ez;
  };
  std::vector<Col> cols;
  cols.reserve(patches.size());
  for (const Shape& S : shapes) {
    cols.clear();
    for (const auto& r : patches) {
      const int ex = r.first[0] + grow, ey = r.first[1] + grow;
      const int nx = (ex + S.tx - 1) / S.tx, ny = (ey + S.ty - 1) / S.ty;
      const double tx = (ex + nx - 1) / nx, ty = (ey + ny - 1) / ny;
      const double faces = (tx + 1) * (ty + 2) + (tx + 2) * (ty + 1) + (tx + 2) * (ty + 2);
      cols.push_back({(double)nx * ny * r.second, S.a + S.b * faces, r.first[2] + grow});
    }
    for (int z : zl) {
      double total = 0.0, longest = 0.0, n = 0.0;
      for (const Col& c : cols) {
        const int len = z > 0 ? std::min(z, c.ez) : c.ez, nz = z > 0 ? (c.ez + len - 1) / len : 1;
        const double t = (len + 3.4) * c.t, m = c.m * nz;
        total += t * m;
        n += m;
        longest = std::max(longest, t);
      }
      const double slots = (double)S.ctas * sms, waves = n / slots;
      double cost;
      bool halves = false;
      if (waves <= 1.0) {
        cost = longest * (0.8 + 0.2 * std::min<double>(S.ctas, std::max(1.0, n / sms)) / S.ctas);
      } else {
        const double rem = waves - std::floor(waves);
        halves = z == 0 && rem > 0.0 && rem <= 0.5;
        const double whole = halves ? std::floor(waves) + 0.6 : std::ceil(waves);
        cost = longest * (0.7 * whole + 0.3 * waves) * std::pow(total / n / longest, 0.6);
      }
      if (best == 0.0 || cost < best) {
        best = cost;
        *tile = S.v;
        *zlen = halves ? -2 : z;
      }
    }
  }
}

// The level's advance reads its halo straight from the neighbour patches
// (3D, a level with direct_halo, no fill recording): its
// same-level ghost fill is then not needed.
bool direct_halo(const amrmhd_ctx* ctx, int l) {
  // the fused 3D kernel, or by default in FP64 the staged ones (the adjoint's
  // forward fills: its stage arrays cover the ghosts)
  const bool can = ctx->fused() ? ctx->opt_advance != 1
                                : ctx->cfg.dim == 3 && ctx->opt_advance == 0 && !ctx->adjoint_forward;
  return can && ctx->opt_direct_halo && !ctx->after_fill &&
         !(ctx->floor_rho > 0.0 || ctx->floor_p > 0.0) && l < (int)ctx->lev.size() && ctx->lev[l].direct_halo;
}

RowArgs row_args(amrmhd_ctx* ctx, const DevList& L, int coarse_level) {
  RowArgs a;
  std::memset(&a, 0, sizeof(a));
  a.P = ctx->dP;
  a.rows = L.p;
  a.nrows = L.n;
  a.scr = ctx->stage_base ? ctx->stage_base : (void*)(ctx->arena + ctx->o_scr);
  a.creg = (double*)(ctx->arena + ctx->o_creg);
  a.freg = (double*)(ctx->arena + ctx->o_freg);
  a.ecreg = (double*)(ctx->arena + ctx->o_ecreg);
  a.efreg = (double*)(ctx->arena + ctx->o_efreg);
  double dx[3];
  for (int d = 0; d < 3; ++d) {
    int N = d < ctx->cfg.dim ? (ctx->cfg.base[d] << coarse_level) : 1;
    dx[d] = d < ctx->cfg.dim ? (ctx->cfg.hi[d] - ctx->cfg.lo[d]) / N : 1.0;
    a.idx[d] = 1.0 / dx[d];
  }
  for (int n = 0; n < 3; ++n)
    for (int t = 0; t < 3; ++t) {
      a.ratio[n][t] = dx[n] / dx[t];
      a.ratiof[n][t] = (float)a.ratio[n][t];
    }
  a.substep = 1;
  a.igm1 = 1.0 / (ctx->cfg.gamma - 1.0);
  a.fl = ctx->floors();
  return a;
}

// Register rows of level l (as fine level) start at global rows cf_face0 /
// cf_edge0: the register arrays are indexed by the global row number, so the
// per-level argument pointers are offset to the level's first row.
void offset_regs(amrmhd_ctx* ctx, RowArgs& a, int l) {
  a.creg += ctx->lev[l].cf_face0 * 6;
  a.freg += ctx->lev[l].cf_face0 * 12;
  a.ecreg += ctx->lev[l].cf_edge0;
  a.efreg += ctx->lev[l].cf_edge0 * 2;
}

// ----- the level operations, shared by the direct calls and graph capture
// the parts of a level's ghost fill: same-level copies, prolongation (sub-step
// 1 above level 0), physical boundaries (last: their sources are domain cells
// the other two fill)
void op_fill_same(amrmhd_ctx* ctx, int l, int s, int* nl) {
  const LevelDev& L = ctx->lev[l];
  // an advance of the interior alone (w = 0) reads ghosts 2 cells deep
  const bool near = l == 0 || s == 2;
  RowArgs a = row_args(ctx, near ? L.runs2 : L.runs, l);
  a.fbuf = state_buf(ctx, ctx->cur[l]);
  a.chunks = near ? L.chunk_runs2.p : L.chunk_runs.p;
  a.nrows = near ? L.chunk_runs2.n : L.chunk_runs.n;
  a.nsplit = near ? L.runs2_split : L.runs_split;
  ctx->ops->fill_runs(a, ctx->stream, nl);
}

void op_fill_rest(amrmhd_ctx* ctx, int l, int s, int* nl) {
  const LevelDev& L = ctx->lev[l];
  const bool near = l == 0 || s == 2;
  if (s == 1 && l > 0) {
    RowArgs b = row_args(ctx, L.prol_cells, l - 1);
    b.fbuf = state_buf(ctx, ctx->cur[l]);
    b.cbuf = state_buf(ctx, ctx->start[l - 1]);
    b.chunks = L.chunk_pcells.p;
    b.nrows = L.chunk_pcells.n;
    RowArgs bf = b;
    bf.rows = L.prol_faces.p;
    bf.chunks = L.chunk_pfaces.p;
    bf.nrows = L.chunk_pfaces.n;
    ctx->ops->prolong(b, bf, ctx->stream, nl);
  }
  // physical boundaries last: their sources are domain cells filled above
  const DevList& bcc = near ? L.bc_cells2 : L.bc_cells;
  const DevList& bcf = near ? L.bc_faces2 : L.bc_faces;
  const DevList& bch = near ? L.chunk_bcells2 : L.chunk_bcells;
  const DevList& bfh = near ? L.chunk_bfaces2 : L.chunk_bfaces;
  if (bch.n || bfh.n) {
    RowArgs c = row_args(ctx, bcc, l);
    c.fbuf = state_buf(ctx, ctx->cur[l]);
    for (int f = 0; f < 8; ++f) c.inflow[f] = ctx->cfg.inflow[f];
    c.chunks = bch.p;
    c.nrows = bch.n;
    ctx->ops->fill_bc_cells(c, ctx->stream, nl);
    c.rows = bcf.p;
    c.chunks = bfh.p;
    c.nrows = bfh.n;
    ctx->ops->fill_bc_faces(c, ctx->stream, nl);
  }
}

void op_fill(amrmhd_ctx* ctx, int l, int s, int* nl) {
  ctx->start[l] = ctx->cur[l];
  op_fill_same(ctx, l, s, nl);
  op_fill_rest(ctx, l, s, nl);
}

void level_idx(amrmhd_ctx* ctx, int l, double* idx) {
  for (int d = 0; d < 3; ++d) {
    int N = d < ctx->cfg.dim ? (ctx->cfg.base[d] << l) : 1;
    idx[d] = 1.0 / (d < ctx->cfg.dim ? (ctx->cfg.hi[d] - ctx->cfg.lo[d]) / N : 1.0);
  }
}

void op_advance(amrmhd_ctx* ctx, int l, const double* dtp, double dtscale, int s, int* nl) {
  const int w = (l == 0) ? 0 : (s == 1 ? 2 : 0);
  LevelArgs a = level_args(ctx, l, dtp, dtscale, w);
  const bool fused = ctx->fused();
  if (ctx->opt_advance == 1) {
    // one launch sequence per patch (baseline)
    const LevelDev& L = ctx->lev[l];
    for (int i = 0; i < L.npatch; ++i) {
      LevelArgs b = a;
      b.ids = L.ids + i;
      b.npatch = 1;
      ctx->ops->advance(b, ctx->stream, nl);
    }
  } else if (fused) {
    const int v = ctx->tile_of(l, w ? 1 : 0);
    a.zlen = ctx->zlen_of(l, w ? 1 : 0);
    if (w == 0 && direct_halo(ctx, l)) a.nbr = ctx->lev[l].nbr.p;
    ctx->ops->advance_fused(a, v, ctx->stream, nl);
  } else if (ctx->fused2d()) {
    a.keep = l + 1 < ctx->H.nlev ? 2 : (l > 0 ? 1 : 0);
    ctx->ops->advance_fused(a, 0, ctx->stream, nl);
  } else {
    if (w == 0 && direct_halo(ctx, l)) a.nbr = ctx->lev[l].nbr.p;
    ctx->ops->advance(a, ctx->stream, nl);
  }
  op_level_registers(ctx, l, dtp, dtscale, s, (fused && ctx->opt_advance != 1) ? a.bnd : nullptr, nl);
  ctx->cur[l] ^= 1;
}

// The flux and EMF registers of level l's sub-step s after its advance (before
// its buffer flips): the coarse side of level l+1's C/F boundary and the fine
// side of level l's own (bnd: the boundary capture the fused advance wrote, or
// nullptr to recompute).
void op_level_registers(amrmhd_ctx* ctx, int l, const double* dtp, double dtscale, int s, void* bnd, int* nl) {
  const bool fused = ctx->fused();
  const int nlev = ctx->H.nlev;
  if (l + 1 < nlev) {
    const LevelDev& F = ctx->lev[l + 1];
    RowArgs f = row_args(ctx, F.cf_faces, l);
    offset_regs(ctx, f, l + 1);
    f.dtp = dtp;
    f.dtscale = dtscale;
    f.fbuf = state_buf(ctx, ctx->cur[l]);
    RowArgs e = f;
    e.rows = F.cf_edges.p;
    e.nrows = F.cf_edges.n;
    if (fused) {
      double idx[3];
      level_idx(ctx, l, idx);
      ctx->ops->reg_coarse_rc(f, e, idx, ctx->cfg.gamma, ctx->stream, nl);
    } else {
      ctx->ops->reg_coarse(f, e, ctx->stream, nl);
    }
  }
  if (l > 0) {
    const LevelDev& F = ctx->lev[l];
    RowArgs f = row_args(ctx, F.cf_faces, l - 1);
    offset_regs(ctx, f, l);
    f.dtp = dtp;
    f.dtscale = dtscale;
    f.substep = s;
    f.fbuf = state_buf(ctx, ctx->cur[l]);
    RowArgs e = f;
    e.rows = F.cf_edges.p;
    e.nrows = F.cf_edges.n;
    if (fused) {
      double idx[3];
      level_idx(ctx, l, idx);
      // the fine advance just wrote its boundary fluxes and EMFs (when the fused kernel ran)
      f.bnd = e.bnd = bnd;
      ctx->ops->reg_fine_rc(f, e, idx, ctx->cfg.gamma, ctx->stream, nl);
    } else {
      ctx->ops->reg_fine(f, e, ctx->stream, nl);
    }
  }
}

void op_reflux_restrict(amrmhd_ctx* ctx, int l, int* nl) {
  const LevelDev& F = ctx->lev[l];
  RowArgs a = row_args(ctx, F.reflux_cells, l - 1);
  a.cbuf = state_buf(ctx, ctx->cur[l - 1]);
  a.fbuf = state_buf(ctx, ctx->cur[l]);
  // reflux rows hold global C/F face row numbers: registers are not offset here
  amrk::RRLists L;
  L.rows[0] = F.reflux_cells.p;
  L.n[0] = F.reflux_cells.n;
  L.rows[1] = F.emf_faces.p;
  L.n[1] = F.emf_faces.n;
  L.rows[2] = F.restrict_cells.p;
  L.n[2] = F.restrict_cells.n;
  L.rows[3] = F.restrict_faces.p;
  L.n[3] = F.restrict_faces.n;
  ctx->ops->reflux_restrict(a, L, ctx->stream, nl);
}

void op_cfl(amrmhd_ctx* ctx, double* hist, int* nl) {
  const int nlev = ctx->H.nlev;
  amrk::launch_zero_u64(ctx->d_slots, nlev, ctx->stream);
  for (int l = 0; l < nlev; ++l) {
    amrk::CflArgs a;
    a.P = ctx->dP;
    a.ids = ctx->lev[l].ids;
    a.npatch = ctx->lev[l].npatch;
    for (int d = 0; d < 3; ++d) a.maxn[d] = ctx->lev[l].maxn[d];
    a.cur = state_buf(ctx, ctx->cur[l]);
    for (int d = 0; d < 3; ++d) {
      int N = d < ctx->cfg.dim ? (ctx->cfg.base[d] << l) : 1;
      a.idx[d] = 1.0 / (d < ctx->cfg.dim ? (ctx->cfg.hi[d] - ctx->cfg.lo[d]) / N : 1.0);
    }
    a.gamma = ctx->cfg.gamma;
    for (int d = 0; d < 3; ++d) a.idxf[d] = (float)a.idx[d];
    a.gf = (float)a.gamma;
    a.gm1h = (float)(a.gamma - 1.0);
    a.gm1l = (float)((a.gamma - 1.0) - (double)a.gm1h);
    a.slot = ctx->d_slots + l;
    a.err = ctx->d_err;
    a.fl = ctx->floors();
    ctx->ops->cfl(a, ctx->stream, nl);
  }
  amrk::launch_cfl_finalize(ctx->d_slots, nlev, ctx->cfg.cfl, ctx->d_scal, hist, ctx->d_err, ctx->stream);
  if (nl) *nl += 2;
}

// the recursive order 0,1,2,2,1,2,2 of Sec. 4 with P, A, S, R
// With concurrency on, the two sub-steps of level l+1 run on a side stream
// while level l advances: level l+1 reads only level l's filled state at the
// start of the step (prolongation, extended ghost zones) and the registers
// of both sides are separate arrays, so the two are joined only before the
// reflux and restriction (Sec. 4: finer levels need not wait for the coarser
// level's advance).
void op_level_step(amrmhd_ctx* ctx, int l, int s, int* nl, bool filled) {
  if (!filled) {
    if (direct_halo(ctx, l)) ctx->start[l] = ctx->cur[l];  // no fill: the advance reads the neighbours
    else op_fill(ctx, l, s, nl);
    if (ctx->after_fill) ctx->after_fill(ctx, l, s);
  }
  const bool kids = l + 1 < ctx->H.nlev;
  if (kids && ctx->opt_concurrent && (int)ctx->side.size() > l) {
    cudaStream_t main = ctx->stream, side = ctx->side[l];
    cudaEventRecord(ctx->ev_fork[l], main);
    cudaStreamWaitEvent(side, ctx->ev_fork[l], 0);
    // Level 1's first fill needs no dt: it runs beside the CFL reduction, ahead
    // of the level-0 advance. Deeper the parent's advance can start at once and
    // goes first.
    const bool ahead = l == 0 && ctx->dt_ready && !ctx->after_fill;
    if (ahead) {
      ctx->stream = side;
      op_fill(ctx, l + 1, 1, nl);
      ctx->stream = main;
    }
    if (ctx->dt_ready) {
      cudaStreamWaitEvent(main, ctx->dt_ready, 0);
      cudaStreamWaitEvent(side, ctx->dt_ready, 0);
      ctx->dt_ready = nullptr;
    }
    op_advance(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), s, nl);
    ctx->stream = side;
    op_level_step(ctx, l + 1, 1, nl, ahead);
    op_level_step(ctx, l + 1, 2, nl);
    cudaEventRecord(ctx->ev_join[l], side);
    ctx->stream = main;
    cudaStreamWaitEvent(main, ctx->ev_join[l], 0);
    op_reflux_restrict(ctx, l + 1, nl);
    return;
  }
  if (ctx->dt_ready) {
    cudaStreamWaitEvent(ctx->stream, ctx->dt_ready, 0);
    ctx->dt_ready = nullptr;
  }
  op_advance(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), s, nl);
  if (kids) {
    op_level_step(ctx, l + 1, 1, nl);
    op_level_step(ctx, l + 1, 2, nl);
    op_reflux_restrict(ctx, l + 1, nl);
  }
}

// The CFL reduction reads the interior cells and own faces of every level and
// the level-0 fill writes only level-0 ghosts, so with concurrency on the two
// run side by side (both short, latency-bound kernels), joined before the
// level-0 advance reads dt.
// ----- the multi-level queue advance (AMRMHD_OPT_QUEUE)
// A coarse step of L levels is 2^(L-1) batches, one per sub-step of the finest
// level F. Level l's sub-step m (m < 2^l) spans the batches [m P_l, (m+1) P_l),
// P_l = 2^(F-l): its fill runs before the first of them (coarse to fine: a
// level's prolongation reads its parent's filled state; the finest level's
// same-level copies are fill tasks of the launch), its advance tiles are split
// into P_l equal shares, one per batch, and its registers and buffer flip
// follow the last. Every batch is one queue launch: the finest level's fill
// tasks, all of its tiles, then the shares of the coarser levels, finer first.
// After the flips, fine to coarse, every level whose second sub-step ended is
// refluxed and restricted. A level's advance reads only its filled state at
// the sub-step's start and writes the other buffer, and its children read
// only its state at that start (extended ghost zones), so this is the
// recursive order's data flow (Sec. 4) and the results equal the level-by-level
// launches bit for bit.
bool queue_active(const amrmhd_ctx* ctx) {
  const int nlev = ctx->H.nlev;
  return ctx->opt_queue && ctx->fused() && ctx->opt_advance != 1 && ctx->opt_advance != 2 && !ctx->after_fill &&
         !ctx->stage_light && !(ctx->floor_rho > 0.0 || ctx->floor_p > 0.0) && nlev >= 2 &&
         nlev <= amrk::QUEUE_MAX_LEVELS && (int)ctx->lev.size() == nlev;
}

static int substep_at(int l, int k, int F) { return l == 0 ? 1 : ((k >> (F - l)) & 1) + 1; }
static bool starts_at(int l, int k, int F) { return k % (1 << (F - l)) == 0; }
static bool ends_at(int l, int k, int F) { return (k + 1) % (1 << (F - l)) == 0; }

amrmhd_status build_queue_plan(amrmhd_ctx* ctx) {
  QueuePlan& Q = ctx->qplan;
  const int var = ctx->opt_queue_tile == 2 ? 2 : 3;
  if (Q.built && Q.variant == var && Q.withhold == (int)ctx->opt_queue_withhold &&
      Q.balance == (int)ctx->opt_queue_balance)
    return AMRMHD_OK;
  const amrmhd::Hierarchy& H = ctx->H;
  const int nlev = H.nlev, F = nlev - 1, T = 1 << F;
  const int np = (int)H.p.size();
  const int TX = var == 2 ? 16 : 8, TY = 8;  // the tiles of variants 2 and 3
  // the advance tiles of a sub-step of level l (w = 2: interior + 2 layers)
  // and their work (cell updates)
  auto level_tiles = [&](int l, int w, std::vector<int32_t>& out, std::vector<double>& work) {
    const int ntx = (ctx->lev[l].maxn[0] + 2 * w + TX - 1) / TX;
    const std::vector<int>& ids = H.level_patches[l];
    for (int i = 0; i < (int)ids.size(); ++i) {
      const amrmhd::HPatch& P = H.p[ids[i]];
      const int ex = P.n[0] + 2 * w, ey = P.n[1] + 2 * w, ez = P.n[2] + 2 * w;
      const int nx = (ex + TX - 1) / TX, ny = (ey + TY - 1) / TY;
      for (int ty = 0; ty < ny; ++ty)
        for (int tx = 0; tx < nx; ++tx) {
          const int32_t rec[4] = {(F - l) << 4, i, ty * ntx + tx, ids[i]};
          out.insert(out.end(), rec, rec + 4);
          work.push_back((double)std::min(TX, ex - tx * TX) * std::min(TY, ey - ty * TY) * ez);
        }
    }
  };
  // shares of every level's sub-steps over the batches (first, end tile per batch)
  // levels fine to coarse: the finest level's whole sub-step in its batch; a
  // coarser level's sub-step of period P_l either in equal counts of tiles
  // (balance 0) or so that the batches' total work (finer levels' included) is
  // as even as its work allows (balance 1): the paper's load balancing (Sec. 5)
  // with the batches of a coarse step as its processors: every batch is given
  // the work that brings its predicted total to one common level.
  std::vector<std::vector<int32_t>> tiles(nlev * (size_t)T);  // [l][m]: sub-step m of level l
  std::vector<std::vector<double>> work(nlev * (size_t)T);
  std::vector<std::vector<std::array<int64_t, 2>>> share(nlev, std::vector<std::array<int64_t, 2>>(T));
  std::vector<double> load(T, 0.0);
  for (int l = F; l >= 0; --l) {
    const int P = 1 << (F - l), M = 1 << l;
    for (int m = 0; m < M; ++m) {
      const int s = l == 0 ? 1 : (m & 1) + 1, w = l == 0 ? 0 : (s == 1 ? 2 : 0);
      std::vector<int32_t>& tl = tiles[(size_t)l * T + m];
      std::vector<double>& wk = work[(size_t)l * T + m];
      level_tiles(l, w, tl, wk);
      const int64_t n = (int64_t)wk.size();
      const int k0 = m * P;
      if (ctx->opt_queue_balance == 0 || P == 1) {
        for (int j = 0; j < P; ++j) share[l][k0 + j] = {n * j / P, n * (j + 1) / P};
      } else {
        // water level L*: sum_k max(0, L* - load_k) = total work of the sub-step
        double tot = 0.0;
        for (double x : wk) tot += x;
        std::vector<double> ld(load.begin() + k0, load.begin() + k0 + P);
        std::sort(ld.begin(), ld.end());
        double lev = ld[0], acc = 0.0;
        for (int j = 0; j < P; ++j) {
          const double next = j + 1 < P ? ld[j + 1] : 1e300;
          // raising the j+1 lowest batches from ld[j] to `next` costs (j+1)(next - ld[j])
          if (acc + (j + 1) * (next - ld[j]) >= tot) {
            lev = ld[j] + (tot - acc) / (j + 1);
            break;
          }
          acc += (j + 1) * (next - ld[j]);
        }
        // contiguous runs of tiles: tile t goes to the batch whose cumulative
        // target holds the tile's midpoint
        int64_t t = 0;
        double cum = 0.0, bound = 0.0;
        for (int j = 0; j < P; ++j) {
          bound += std::max(0.0, lev - load[k0 + j]);
          const int64_t a = t;
          while (t < n && (j == P - 1 || cum + 0.5 * wk[t] <= bound)) cum += wk[t++];
          share[l][k0 + j] = {a, t};
        }
      }
      for (int j = 0; j < P; ++j) {
        const auto& sh = share[l][k0 + j];
        for (int64_t t = sh[0]; t < sh[1]; ++t) load[k0 + j] += wk[t];
      }
    }
  }
  std::vector<int32_t> tasks;
  std::vector<uint32_t> need((size_t)T * np, 0u);
  Q.task_off.assign(T, 0);
  Q.task_n.assign(T, 0);
  Q.fill_in_queue.assign(T, 0);
  const LevelDev& LF = ctx->lev[F];
  for (int k = 0; k < T; ++k) {
    const int64_t t0 = (int64_t)tasks.size() / 4;
    Q.task_off[k] = t0;
    // the finest level's same-level copies: ranges of at most 16 chunks into
    // one patch, cell boxes (listed first) and face boxes apart
    const bool fillq = !LF.has_bc;
    Q.fill_in_queue[k] = fillq ? 1 : 0;
    if (fillq) {
      const int sF = substep_at(F, k, F);
      const bool near = F == 0 || sF == 2;
      const std::vector<int32_t>& c0 = near ? LF.h_chunk0_2 : LF.h_chunk0;
      const std::vector<int32_t>& dst = near ? LF.h_dst2 : LF.h_dst;
      const int64_t nsplit = near ? LF.runs2_split : LF.runs_split;
      const int64_t nch = c0.empty() ? 0 : c0.back();
      // the destination of chunk c: its record's, found by walking the
      // records' first chunks forwards (c only grows)
      size_t rb = 0, re = 0;
      auto dst_of = [&](int64_t c, size_t& r) {
        while (r + 1 < dst.size() && c0[r + 1] <= c) ++r;
        return dst[r];
      };
      for (int64_t c = 0; c < nch;) {
        const int d0 = dst_of(c, rb);
        const bool cells = c < nsplit;
        int64_t e = c + 1;
        re = rb;
        while (e < nch && e - c < 16 && dst_of(e, re) == d0 && (e < nsplit) == cells) ++e;
        const int32_t rec[4] = {1 | (cells ? 2 : 0), (int32_t)c, (int32_t)e, d0};
        tasks.insert(tasks.end(), rec, rec + 4);
        need[(size_t)k * np + d0] += 1u;
        c = e;
      }
    }
    // advance tiles, finest level first: each level's share of this batch
    for (int l = F; l >= 0; --l) {
      const int m = k >> (F - l);
      const std::vector<int32_t>& tl = tiles[(size_t)l * T + m];
      const auto& sh = share[l][k];
      tasks.insert(tasks.end(), tl.begin() + 4 * sh[0], tl.begin() + 4 * sh[1]);
    }
    Q.task_n[k] = (int)((int64_t)tasks.size() / 4 - t0);
  }
  Q.batch_work = load;
  // test switch: the first patch of the finest level waits in the first batch
  // for one fill task more than exist, so its wait runs out
  if (ctx->opt_queue_withhold) need[H.level_patches[F].front()] += 1u;
  cudaError_t e = cudaSuccess;
  Q.d_tasks = dbuf<int>(ctx, tasks.size(), &e);
  if (e != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, "cudaMalloc");
  Q.d_need = dbuf<unsigned int>(ctx, need.size(), &e);
  if (e != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, "cudaMalloc");
  Q.d_ctr = dbuf<unsigned int>(ctx, (size_t)np + 2, &e);
  if (e != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, "cudaMalloc");
  CU(cudaMemcpy(Q.d_tasks, tasks.data(), sizeof(int32_t) * tasks.size(), cudaMemcpyHostToDevice));
  CU(cudaMemcpy(Q.d_need, need.data(), sizeof(uint32_t) * need.size(), cudaMemcpyHostToDevice));
  Q.variant = var;
  Q.withhold = (int)ctx->opt_queue_withhold;
  Q.balance = (int)ctx->opt_queue_balance;
  Q.built = true;
  return AMRMHD_OK;
}

void op_coarse_step_queue(amrmhd_ctx* ctx, int* nl) {
  const QueuePlan& Q = ctx->qplan;
  const int nlev = ctx->H.nlev, F = nlev - 1, T = 1 << F;
  const int np = (int)ctx->H.p.size();
  const int TX = Q.variant == 2 ? 16 : 8;
  op_cfl(ctx, ctx->d_hist, nl);
  for (int k = 0; k < T; ++k) {
    for (int l = 0; l <= F; ++l) {
      if (!starts_at(l, k, F)) continue;
      const int s = substep_at(l, k, F);
      if (l < F || !Q.fill_in_queue[k]) {
        op_fill(ctx, l, s, nl);
      } else {
        ctx->start[l] = ctx->cur[l];
        op_fill_rest(ctx, l, s, nl);
      }
    }
    amrk::QueueArgs q;
    std::memset(&q, 0, sizeof(q));
    for (int l = 0; l <= F; ++l) {
      const int s = substep_at(l, k, F), w = l == 0 ? 0 : (s == 1 ? 2 : 0);
      const LevelDev& L = ctx->lev[l];
      amrk::QueueLevel& QL = q.L[F - l];
      QL.a = level_args(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), w);
      QL.ntx = (L.maxn[0] + 2 * w + TX - 1) / TX;
      const bool near = l == 0 || s == 2;
      QL.boxes = near ? L.runs2.p : L.runs.p;
      QL.chunks = near ? L.chunk_runs2.p : L.chunk_runs.p;
    }
    q.tasks = Q.d_tasks + 4 * Q.task_off[k];
    q.ntasks = Q.task_n[k];
    q.need = Q.d_need + (size_t)k * np;
    q.done = Q.d_ctr;
    q.head = Q.d_ctr + np;
    q.abort = (int*)(Q.d_ctr + np + 1);
    q.err = ctx->d_err;
    q.wait_ns = 500000000ull;  // 0.5 s
    cudaMemsetAsync(Q.d_ctr, 0, sizeof(unsigned int) * ((size_t)np + 2), ctx->stream);
    ctx->ops->advance_queue(q, Q.variant, ctx->stream, nl);
    // levels whose sub-step ends with this batch: registers, then the flip
    for (int l = F; l >= 0; --l) {
      if (!ends_at(l, k, F)) break;
      op_level_registers(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), substep_at(l, k, F), q.L[F - l].a.bnd, nl);
      ctx->cur[l] ^= 1;
    }
    // levels whose second sub-step ended, fine to coarse
    for (int l = F; l >= 1; --l) {
      const int per = 1 << (F - l);
      if ((k + 1) % per != 0 || (((k + 1) / per) & 1) != 0) break;
      op_reflux_restrict(ctx, l, nl);
    }
  }
}

void op_coarse_step(amrmhd_ctx* ctx, int* nl) {
  if (queue_active(ctx)) {
    op_coarse_step_queue(ctx, nl);
    return;
  }
  if (ctx->opt_concurrent && ctx->cfl_stream && !ctx->after_fill) {
    cudaStream_t main = ctx->stream;
    cudaEventRecord(ctx->ev_cfl_fork, main);
    cudaStreamWaitEvent(ctx->cfl_stream, ctx->ev_cfl_fork, 0);
    ctx->stream = ctx->cfl_stream;
    op_cfl(ctx, ctx->d_hist, nl);
    cudaEventRecord(ctx->ev_cfl_join, ctx->cfl_stream);
    ctx->stream = main;
    if (direct_halo(ctx, 0)) ctx->start[0] = ctx->cur[0];
    else op_fill(ctx, 0, 1, nl);
    ctx->dt_ready = ctx->ev_cfl_join;
    op_level_step(ctx, 0, 1, nl, true);
    return;
  }
  op_cfl(ctx, ctx->d_hist, nl);
  op_level_step(ctx, 0, 1, nl);
}

// the ghost fills as one row per position (the ghost maps' rows split by kind:
// same-level (dst, [d,] Ld, src, Ls), prolongation (dst, [d,] Ld, srcC, Lc),
// boundaries as the map rows), per level, for the adjoint's transposed fills
amrmhd_status upload_fill_rows(amrmhd_ctx* ctx) {
  amrmhd::Hierarchy& H = ctx->H;
  H.expand_ghost_rows();
  cudaError_t e = cudaSuccess;
  auto upload = [&](const std::vector<int32_t>& v, DevList& out, int width) -> bool {
    out.n = (int64_t)v.size() / width;
    if (v.empty()) { out.p = nullptr; return true; }
    out.p = dbuf<int>(ctx, v.size(), &e);
    if (e != cudaSuccess) return false;
    e = cudaMemcpy(out.p, v.data(), sizeof(int) * v.size(), cudaMemcpyHostToDevice);
    return e == cudaSuccess;
  };
  std::vector<std::vector<int32_t>> sc(H.nlev), pc(H.nlev), sf(H.nlev), pf(H.nlev), bcc(H.nlev), bcf(H.nlev);
  for (size_t r = 0; r < H.ghost_cells.size(); r += 5) {
    const int32_t* g = &H.ghost_cells[r];
    const int l = H.p[g[0]].level;
    if (g[2] >= 2) {
      bcc[l].insert(bcc[l].end(), g, g + 5);
      continue;
    }
    std::vector<int32_t>& v = g[2] == 0 ? sc[l] : pc[l];
    v.insert(v.end(), {g[0], g[1], g[3], g[4]});
  }
  for (size_t r = 0; r < H.ghost_faces.size(); r += 6) {
    const int32_t* g = &H.ghost_faces[r];
    const int l = H.p[g[0]].level;
    if (g[3] >= 2) {
      bcf[l].insert(bcf[l].end(), g, g + 6);
      continue;
    }
    std::vector<int32_t>& v = g[3] == 0 ? sf[l] : pf[l];
    v.insert(v.end(), {g[0], g[1], g[2], g[4], g[5]});
  }
  for (int l = 0; l < H.nlev; ++l) {
    LevelDev& L = ctx->lev[l];
    const bool ok = upload(sc[l], L.row_same_cells, 4) && upload(pc[l], L.row_prol_cells, 4) &&
                    upload(sf[l], L.row_same_faces, 5) && upload(pf[l], L.row_prol_faces, 5) &&
                    upload(bcc[l], L.row_bc_cells, 5) && upload(bcf[l], L.row_bc_faces, 6);
    if (!ok) return fail(ctx, AMRMHD_ECUDA, std::string("fill row upload: ") + cudaGetErrorString(e));
  }
  return AMRMHD_OK;
}

amrmhd_status check_bound(amrmhd_ctx* ctx) {
  if (!ctx) return AMRMHD_EINVAL;
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "no hierarchy set");
  if (!ctx->bound) return fail(ctx, AMRMHD_ESTATE, "no arena bound");
  return AMRMHD_OK;
}

const std::vector<int32_t>* map_vec(amrmhd_ctx* ctx, int which, int* width) {
  amrmhd::Hierarchy& H = ctx->H;
  if (which == AMRMHD_MAP_GHOST_CELLS || which == AMRMHD_MAP_GHOST_FACES) H.expand_ghost_rows();
  else if (download_register_maps(ctx) != AMRMHD_OK) return nullptr;
  switch (which) {
    case AMRMHD_MAP_GHOST_CELLS: *width = 5; return &H.ghost_cells;
    case AMRMHD_MAP_GHOST_FACES: *width = 6; return &H.ghost_faces;
    case AMRMHD_MAP_CF_FACES: *width = 7; return &H.cf_faces;
    case AMRMHD_MAP_CF_EDGES: *width = 6; return &H.cf_edges;
    case AMRMHD_MAP_EMF_FACES: *width = 8; return &H.emf_faces;
    case AMRMHD_MAP_RESTRICT_CELLS: *width = 5; return &H.restrict_cells;
    case AMRMHD_MAP_RESTRICT_FACES: *width = 6; return &H.restrict_faces;
    case AMRMHD_MAP_REFLUX_CELLS: *width = 9; return &H.reflux_cells;
    default: return nullptr;
  }
}

}  // namespace amrapi

extern "C" {

amrmhd_status amrmhd_create(const amrmhd_config* cfg, void* cuda_stream, amrmhd_ctx** out) {
  if (!cfg || !out) return AMRMHD_EINVAL;
  *out = nullptr;
  if (cfg->dim != 2 && cfg->dim != 3) return AMRMHD_EINVAL;
  if (cfg->nghost != 4 || cfg->ratio != 2) return AMRMHD_EINVAL;
  if (cfg->precision != AMRMHD_FP64 && cfg->precision != AMRMHD_MIXED) return AMRMHD_EINVAL;
  if (!(cfg->gamma > 1.0) || !(cfg->cfl > 0.0) || cfg->max_level < 0 || cfg->max_level > 20) return AMRMHD_EINVAL;
  for (int d = 0; d < 3; ++d) {
    if (d < cfg->dim && (cfg->base[d] < 8 || !(cfg->hi[d] > cfg->lo[d]))) return AMRMHD_EINVAL;
    if (d >= cfg->dim && cfg->base[d] != 1) return AMRMHD_EINVAL;
    if (d >= cfg->dim) continue;
    for (int s = 0; s < 2; ++s)
      if (cfg->bc[d][s] < AMRMHD_BC_PERIODIC || cfg->bc[d][s] > AMRMHD_BC_INFLOW) return AMRMHD_EINVAL;
    if ((cfg->bc[d][0] == AMRMHD_BC_PERIODIC) != (cfg->bc[d][1] == AMRMHD_BC_PERIODIC)) return AMRMHD_EINVAL;
  }
  amrmhd_ctx* ctx = new amrmhd_ctx();
  ctx->cfg = *cfg;
  ctx->stream = (cudaStream_t)cuda_stream;
  if (cfg->precision == AMRMHD_MIXED) ctx->variant = amrk::V_MIXED;
  else ctx->variant = cfg->strict_fp64 ? amrk::V_FP64_STRICT : amrk::V_FP64;
  ctx->ops = ctx->variant == amrk::V_FP64_STRICT ? amrk::ops_strict(cfg->dim) : amrk::ops_fast(ctx->variant, cfg->dim);
  *out = ctx;
  return AMRMHD_OK;
}

amrmhd_status amrmhd_destroy(amrmhd_ctx* ctx) {
  if (!ctx) return AMRMHD_EINVAL;
  free_device(ctx);
  if (ctx->d_maps) cudaFree(ctx->d_maps);
  if (ctx->d_cluster) cudaFree(ctx->d_cluster);
  if (ctx->own_stream) cudaStreamDestroy(ctx->own_stream);
  delete ctx;
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_floors(amrmhd_ctx* ctx, double rho_min, double p_min) {
  if (!ctx) return AMRMHD_EINVAL;
  if (!(rho_min >= 0.0) || !(p_min >= 0.0) || !std::isfinite(rho_min) || !std::isfinite(p_min))
    return fail(ctx, AMRMHD_EINVAL, "floors must be finite and non-negative");
  ctx->floor_rho = rho_min;
  ctx->floor_p = p_min;
  for (int i = 0; i < 2; ++i)
    if (ctx->gexec[i]) { cudaGraphExecDestroy(ctx->gexec[i]); ctx->gexec[i] = nullptr; }
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_option(amrmhd_ctx* ctx, int32_t option, int64_t value) {
  if (!ctx) return AMRMHD_EINVAL;
  if (option == AMRMHD_OPT_ADVANCE && value >= 0 && value <= 3) ctx->opt_advance = value;
  else if (option == AMRMHD_OPT_GRAPH && (value == 0 || value == 1)) ctx->opt_graph = value;
  else if (option == AMRMHD_OPT_TILE && value >= -1 && value <= 4) ctx->opt_tile = value;
  else if (option == AMRMHD_OPT_ZCHUNK && value >= -2 && value <= 4096) ctx->opt_zchunk = value;
  else if (option == AMRMHD_OPT_CONCURRENT && (value == 0 || value == 1)) ctx->opt_concurrent = value;
  else if (option == AMRMHD_OPT_HOST_IO && (value == 0 || value == 1)) ctx->opt_host_io = value;
  else if (option == AMRMHD_OPT_DIRECT_HALO && (value == 0 || value == 1)) ctx->opt_direct_halo = value;
  else if (option == AMRMHD_OPT_QUEUE && (value == 0 || value == 1)) ctx->opt_queue = value;
  else if (option == AMRMHD_OPT_QUEUE_TILE && (value == 2 || value == 3)) ctx->opt_queue_tile = value;
  else if (option == AMRMHD_OPT_QUEUE_WITHHOLD && (value == 0 || value == 1)) ctx->opt_queue_withhold = value;
  else if (option == AMRMHD_OPT_QUEUE_BALANCE && (value == 0 || value == 1)) ctx->opt_queue_balance = value;
  else if (option == AMRMHD_OPT_DEVICE_MAPS && value >= -1 && value <= 1) ctx->opt_device_maps = value;
  else if (option == AMRMHD_OPT_DEVICE_CLUSTER && (value == 0 || value == 1)) ctx->opt_device_cluster = value;
  else if (option == AMRMHD_OPT_ADJOINT_KEEP && value >= -1) {
    ctx->opt_adjoint_keep = value;
    adj_limit(ctx);
  }
  else return fail(ctx, AMRMHD_EINVAL, "unknown option or value");
  for (int i = 0; i < 2; ++i)
    if (ctx->gexec[i]) { cudaGraphExecDestroy(ctx->gexec[i]); ctx->gexec[i] = nullptr; }
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_hierarchy(amrmhd_ctx* ctx, const amrmhd_patch* patches, int32_t n, size_t* arena_bytes) {
  if (!ctx || !patches || n <= 0) return fail(ctx, AMRMHD_EINVAL, "bad arguments");
  free_device(ctx);
  ctx->have_h = false;
  amrmhd::Hierarchy& H = ctx->H;
  H.dim = ctx->cfg.dim;
  for (int d = 0; d < 3; ++d) {
    H.base[d] = ctx->cfg.base[d];
    H.bc[d][0] = d < H.dim ? ctx->cfg.bc[d][0] : 0;
    H.bc[d][1] = d < H.dim ? ctx->cfg.bc[d][1] : 0;
    H.per[d] = d >= H.dim || H.bc[d][0] == AMRMHD_BC_PERIODIC;
  }
  H.max_level = ctx->cfg.max_level;
  H.ghost_from = ctx->stage_light ? ctx->stage_ghost_from : 0;
  if (ctx->d_maps) { cudaFree(ctx->d_maps); ctx->d_maps = nullptr; }
  ctx->dmaps = ctx->dmaps_host = false;
  bool dev_maps = ctx->opt_device_maps == 1;
  if (ctx->opt_device_maps < 0) {
    int ndev = 0;
    dev_maps = cudaGetDeviceCount(&ndev) == cudaSuccess && ndev > 0;
    cudaGetLastError();  // a host without a device reports an error here: not sticky, cleared
  }
  H.ghost_elsewhere = dev_maps;
  const bool dev_regs = dev_maps && !ctx->stage_light;
  H.with_registers = !ctx->stage_light && !dev_maps;
  std::vector<int32_t> rows(7 * (size_t)n);
  for (int i = 0; i < n; ++i) {
    rows[7 * i] = patches[i].level;
    for (int d = 0; d < 3; ++d) { rows[7 * i + 1 + d] = patches[i].lo[d]; rows[7 * i + 4 + d] = patches[i].hi[d]; }
    // the fill records carry field strides (x 8 fields) in 32 bits: reject a
    // patch over 2^28 elements per field before any map is built
    long long e = 1;
    for (int d = 0; d < H.dim; ++d) e *= std::max(0, patches[i].hi[d] - patches[i].lo[d]) + 9LL;
    if (8 * ((e + 63) / 64 * 64) > INT32_MAX)
      return fail(ctx, AMRMHD_EINVAL, "patch too large (over 2^28 elements per field)");
  }
  auto now = [] {
    return std::chrono::duration_cast<std::chrono::microseconds>(std::chrono::steady_clock::now().time_since_epoch())
        .count();
  };
  long long t0 = now();
  int st = H.build(rows.data(), n);
  ctx->maps_us[0] = now() - t0;
  ctx->maps_us[1] = ctx->maps_us[2] = 0;
  if (st != AMRMHD_OK) return fail(ctx, (amrmhd_status)st, H.err);
  if (dev_maps) {
    t0 = now();
    amrmhd_status ds = device_ghost_boxes(ctx);
    ctx->maps_us[1] = now() - t0;
    t0 = now();
    if (ds == AMRMHD_OK && dev_regs) ds = device_register_maps(ctx);
    ctx->maps_us[2] = now() - t0;
    if (ds != AMRMHD_OK) return ds;
  }
  // arena layout: patches in (level, id) order
  const int np = (int)H.p.size();
  const size_t elem = ctx->ops->elem;
  ctx->off.assign(np, 0);
  ctx->fs.assign(np, 0);
  ctx->soff.assign(np, 0);
  long long acc = 0, sacc = 0;
  for (int l = 0; l < H.nlev; ++l)
    for (int q : H.level_patches[l]) {
      const long long e = (long long)H.p[q].ext[0] * H.p[q].ext[1] * H.p[q].ext[2];
      const long long f = (e + 63) / 64 * 64;
      // the fill records carry field strides (x 8 fields) in 32 bits
      if (8 * f > INT32_MAX) return fail(ctx, AMRMHD_EINVAL, "patch too large (over 2^28 elements per field)");
      ctx->fs[q] = f;
      ctx->off[q] = acc;
      acc += 8 * f;
      ctx->soff[q] = sacc;
      if (!ctx->fused() && !ctx->stage_light) sacc += amrk::SC_N * f;
    }
  ctx->state_elems = acc;
  ctx->scr_elems = sacc;
  // boundary capture blocks of the fused 3D path: fluxes and EMFs on the
  // boundary planes of every patch above level 0 (read by the fine registers)
  ctx->boff.assign(np, -1);
  long long bacc = 0;
  if (H.dim == 3 && ctx->fused() && !ctx->stage_light)
    for (int l = 1; l < H.nlev; ++l)
      for (int q : H.level_patches[l]) {
        ctx->boff[q] = bacc;
        bacc += 5 * amrk::bnd_faces_total(H.p[q].n) + amrk::bnd_edges_total(H.p[q].n);
      }
  ctx->bnd_elems = bacc;
  ctx->ncf = ctx->dmaps ? ctx->dmap_n[0] : (int64_t)H.cf_faces.size() / 7;
  ctx->nce = ctx->dmaps ? ctx->dmap_n[1] : (int64_t)H.cf_edges.size() / 6;
  for (int k = 0; k < 4; ++k) {
    ctx->poff[k].assign(np, 0);
    long long t = 0;
    for (int q = 0; q < np; ++q) {
      ctx->poff[k][q] = t;
      long long c = 1;
      for (int d = 0; d < H.dim; ++d) c *= H.p[q].n[d] + (k == d + 1 ? 1 : 0);
      if (k == 3 && H.dim == 2) c = 0;
      t += c;
    }
    ctx->ptotal[k] = t;
  }
  ctx->stage_elems = std::max(std::max(ctx->ptotal[0], ctx->ptotal[1]), std::max(ctx->ptotal[2], ctx->ptotal[3]));
  size_t o = 0;
  ctx->o_state[0] = o; o = align256(o + (size_t)acc * elem);
  ctx->o_state[1] = o; o = align256(o + (size_t)acc * elem);
  ctx->o_scr = o; o = align256(o + (size_t)sacc * elem);
  ctx->o_creg = o; o = align256(o + (size_t)ctx->ncf * 6 * sizeof(double));
  ctx->o_freg = o; o = align256(o + (size_t)ctx->ncf * 12 * sizeof(double));
  ctx->o_ecreg = o; o = align256(o + (size_t)ctx->nce * sizeof(double));
  ctx->o_efreg = o; o = align256(o + (size_t)ctx->nce * 2 * sizeof(double));
  ctx->o_stage = o; o = align256(o + (size_t)ctx->stage_elems * sizeof(double));
  ctx->o_bnd = o; o = align256(o + (size_t)ctx->bnd_elems * elem);
  ctx->arena_bytes = o;
  ctx->have_h = true;
  if (arena_bytes) *arena_bytes = o;
  return AMRMHD_OK;
}

amrmhd_status amrmhd_bind_arena(amrmhd_ctx* ctx, void* dev_ptr, size_t bytes) {
  if (!ctx) return AMRMHD_EINVAL;
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "bind_arena before set_hierarchy");
  if (!dev_ptr || ((uintptr_t)dev_ptr & 255)) return fail(ctx, AMRMHD_EINVAL, "arena must be a 256-byte aligned device pointer");
  if (bytes < ctx->arena_bytes) return fail(ctx, AMRMHD_ENOMEM, "arena smaller than required");
  free_device(ctx);
  if (!ctx->stream) {
    // the legacy default stream cannot be captured into a graph: use our own
    if (!ctx->own_stream) CU(cudaStreamCreateWithFlags(&ctx->own_stream, cudaStreamNonBlocking));
    ctx->stream = ctx->own_stream;
  }
  ctx->arena = (char*)dev_ptr;
  const amrmhd::Hierarchy& H = ctx->H;
  const int np = (int)H.p.size(), nlev = H.nlev;
  cudaError_t e = cudaSuccess;
  // patch table
  std::vector<DPatch> hp(np);
  for (int q = 0; q < np; ++q) {
    DPatch& P = hp[q];
    for (int d = 0; d < 3; ++d) { P.lo[d] = H.p[q].lo[d]; P.n[d] = H.p[q].n[d]; P.ext[d] = H.p[q].ext[d]; }
    P.level = H.p[q].level;
    P.off = ctx->off[q];
    P.fs = ctx->fs[q];
    P.soff = ctx->soff[q];
    P.boff = ctx->boff[q];
  }
  // the patch table, patch ids, packed-I/O offsets, scalars, CFL slots, error
  // word, floor count and dt history: one device block, one copy
  size_t o = 0;
  auto carve = [&](size_t bytes) { const size_t r = o; o = align256(o + bytes); return r; };
  const size_t oP = carve(sizeof(DPatch) * np), oI = carve(sizeof(int) * np);
  size_t oO[4];
  for (int k = 0; k < 4; ++k) oO[k] = carve(sizeof(long long) * np);
  const size_t oT = carve(sizeof(long long*) * 4), oS = carve(sizeof(double) * (2 + nlev)),
               oL = carve(sizeof(unsigned long long) * (nlev + 1)), oE = carve(sizeof(unsigned int)),
               oF = carve(sizeof(unsigned long long)), oH = carve(sizeof(double) * kHistCap);
  char* blk = dbuf<char>(ctx, o, &e);
  if (e != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  std::vector<char> img(oH, 0);  // everything before the history (zero scalars, slots, counters)
  std::memcpy(img.data() + oP, hp.data(), sizeof(DPatch) * np);
  for (int q = 0; q < np; ++q) ((int*)(img.data() + oI))[q] = q;
  for (int k = 0; k < 4; ++k) {
    std::memcpy(img.data() + oO[k], ctx->poff[k].data(), sizeof(long long) * np);
    ctx->d_poff[k] = (long long*)(blk + oO[k]);
    ((long long**)(img.data() + oT))[k] = ctx->d_poff[k];
  }
  CU(cudaMemcpy(blk, img.data(), img.size(), cudaMemcpyHostToDevice));
  ctx->dP = (DPatch*)(blk + oP);
  ctx->d_iota = (int*)(blk + oI);
  ctx->d_poff_tab = (const long long**)(blk + oT);
  ctx->d_scal = (double*)(blk + oS);
  ctx->d_slots = (unsigned long long*)(blk + oL);
  ctx->d_err = (unsigned int*)(blk + oE);
  ctx->d_floor_events = (unsigned long long*)(blk + oF);
  ctx->hist_cap = kHistCap;
  ctx->d_hist = (double*)(blk + oH);
  // per-level lists: gathered into one host image (each list 256-byte aligned),
  // then one device allocation and one copy
  const auto tb0 = std::chrono::steady_clock::now();
  ctx->lev.assign(nlev, LevelDev());
  std::vector<int32_t> pack;
  std::vector<std::pair<DevList*, size_t>> pend;  // list -> element offset in pack
  auto upload = [&](const std::vector<int32_t>& v, DevList& out, int width) -> bool {
    out.n = (int64_t)v.size() / width;
    out.p = nullptr;
    if (v.empty()) return true;
    const size_t o = (pack.size() + 63) / 64 * 64;
    pack.resize(o + v.size());
    std::copy(v.begin(), v.end(), pack.begin() + o);
    pend.push_back({&out, o});
    return true;
  };
  std::vector<DevList> id_lists(nlev);
  // the ghost boxes of each level in list order (cells, then faces)
  std::vector<std::vector<const int32_t*>> level_boxes(nlev);
  std::vector<int64_t> level_cell_boxes(nlev, 0);
  for (int faces = 0; faces < 2; ++faces) {
    const std::vector<int32_t>& gb = faces ? H.ghost_box_faces : H.ghost_box_cells;
    for (size_t r = 0; r < gb.size(); r += amrmhd::GHOST_BOX_W) level_boxes[H.p[gb[r]].level].push_back(&gb[r]);
    if (!faces)
      for (int l = 0; l < nlev; ++l) level_cell_boxes[l] = (int64_t)level_boxes[l].size();
  }
  for (int l = 0; l < nlev; ++l) {
    LevelDev& L = ctx->lev[l];
    const std::vector<int>& ids = H.level_patches[l];
    L.npatch = (int)ids.size();
    for (int d = 0; d < 3; ++d) {
      L.maxn[d] = 1;
      for (int q : ids) L.maxn[d] = std::max(L.maxn[d], H.p[q].n[d]);
      ctx->maxn_all[d] = std::max(ctx->maxn_all[d], L.maxn[d]);
    }
    upload(ids, id_lists[l], 1);
    // ghost fill lists of this level from the hierarchy's boxes (see LevelDev),
    // written straight into the upload image: a count pass over the level's
    // boxes (cells, then faces), prefix sums per list, then a write pass, both
    // over the boxes in parallel
    enum { RR, CR, PCB, PCC, PFB, PFC, BCB, BCC, BFB, BFC, RR2, CR2, BCB2, BCC2, BFB2, BFC2, NLIST };
    const int GW = amrmhd::GHOST_BOX_W, FW = amrk::FILL_BOX_W;
    static const int LW[NLIST] = {amrk::FILL_BOX_W, 4, amrmhd::GHOST_BOX_W, 2, amrmhd::GHOST_BOX_W, 2,
                                  amrmhd::GHOST_BOX_W, 2, amrmhd::GHOST_BOX_W, 2, amrk::FILL_BOX_W, 4,
                                  amrmhd::GHOST_BOX_W, 2, amrmhd::GHOST_BOX_W, 2};
    const std::vector<const int32_t*>& lb = level_boxes[l];
    const int64_t nb = (int64_t)lb.size(), nbc = level_cell_boxes[l];
    // a box clipped to the ghosts within 2 cells of the interior (faces: either
    // adjacent cell within 2); false if nothing is left
    auto clip_near = [&](const int32_t* b, int32_t* o) {
      const amrmhd::HPatch& P = H.p[b[0]];
      std::copy(b, b + GW, o);
      for (int e = 0; e < H.dim; ++e) {
        const int lo = std::max(b[4 + e], 2), hi = std::min(b[4 + e] + b[7 + e], P.n[e] + 6 + (e == b[1] ? 1 : 0));
        if (hi <= lo) return false;
        o[4 + e] = lo;
        o[7 + e] = hi - lo;
      }
      return true;
    };
    // the ints box b adds to each list (count), or writes them at cur[] (write)
    auto proc = [&](const int32_t* b, bool faces, bool write, int64_t* cur, int32_t* pk, const int64_t* base) {
      // a same-level box as a self-contained copy record (see k_fill_runs):
      // element offsets of the first destination and source positions (with
      // the face field for a face box), both patches' x/y extents and field
      // strides, the box's nx, ny, the number of fields, cx = min(nx, 64) and
      // the multipliers of the lane -> (x, row) and row -> (y, z) divisions;
      // chunks (box, x0, q0, nrows) of whole rows q = y + ny z of cx positions.
      // Every listed box has a chunk: a range of k chunks spans at most k boxes
      auto add_run = [&](const int32_t* r, int lr, int lc) {
        if (r[7] <= 0 || r[8] <= 0 || r[9] <= 0) return;
        const int nx = r[7], ny = r[8], nz = r[9];
        const int cx = std::min(nx, amrk::FILL_CHUNK);
        const int rows = ny * nz, per = amrk::FILL_CHUNK / cx;
        const int64_t nch = (int64_t)((rows + per - 1) / per) * ((nx + cx - 1) / cx);
        if (!write) {
          cur[lr] += FW;
          cur[lc] += 4 * nch;
          return;
        }
        const amrmhd::HPatch &D = H.p[r[0]], &S = H.p[r[3]];
        const long long Ld = r[4] + (long long)D.ext[0] * (r[5] + (long long)D.ext[1] * r[6]);
        const long long Ls = (r[4] + r[10]) + (long long)S.ext[0] * ((r[5] + r[11]) + (long long)S.ext[1] * (r[6] + r[12]));
        const long long fd = ctx->fs[r[0]], fsrc = ctx->fs[r[3]];
        const int fl = r[1] < 0 ? 0 : 5 + r[1];  // B_x, B_y, B_z are fields 5, 6, 7
        const long long db = ctx->off[r[0]] + fl * fd + Ld, sb = ctx->off[r[3]] + fl * fsrc + Ls;
        const int nv = r[1] >= 0 ? 1 : (H.dim == 3 ? 5 : 6);
        const uint64_t two31 = 1ull << 31;
        const uint32_t mcx = (uint32_t)((two31 + cx - 1) / cx), mny = (uint32_t)((two31 + ny - 1) / ny);
        const int bi = (int)((cur[lr] - base[lr]) / FW);
        const int32_t rec[amrk::FILL_BOX_W] = {(int32_t)(db & 0xffffffffLL), (int32_t)(db >> 32),
                                               (int32_t)(sb & 0xffffffffLL), (int32_t)(sb >> 32),
                                               D.ext[0], D.ext[1], S.ext[0], S.ext[1],
                                               (int32_t)fd, (int32_t)fsrc, nx, ny,
                                               nv, cx, (int32_t)mcx, (int32_t)mny};
        std::copy(rec, rec + FW, pk + cur[lr]);
        cur[lr] += FW;
        int32_t* c = pk + cur[lc];
        for (int q0 = 0; q0 < rows; q0 += per)
          for (int x0 = 0; x0 < nx; x0 += cx) {
            c[0] = bi;
            c[1] = x0;
            c[2] = q0;
            c[3] = std::min(per, rows - q0);
            c += 4;
          }
        cur[lc] += 4 * nch;
      };
      auto add_box = [&](const int32_t* r, int lr, int lc) {
        const int vol = r[7] * r[8] * r[9];
        const int64_t nch = (vol + amrk::FILL_CHUNK - 1) / amrk::FILL_CHUNK;
        if (!write) {
          cur[lr] += GW;
          cur[lc] += 2 * nch;
          return;
        }
        const int bi = (int)((cur[lr] - base[lr]) / GW);
        std::copy(r, r + GW, pk + cur[lr]);
        cur[lr] += GW;
        int32_t* c = pk + cur[lc];
        for (int k = 0; k < vol; k += amrk::FILL_CHUNK) {
          c[0] = bi;
          c[1] = k;
          c += 2;
        }
        cur[lc] += 2 * nch;
      };
      int32_t nbx[amrmhd::GHOST_BOX_W];
      const bool near = clip_near(b, nbx);
      if (b[2] == 0) {
        add_run(b, RR, CR);
        if (near) add_run(nbx, RR2, CR2);
      } else if (b[2] == 1) {
        add_box(b, faces ? PFB : PCB, faces ? PFC : PCC);
      } else {
        add_box(b, faces ? BFB : BCB, faces ? BFC : BCC);
        if (near) add_box(nbx, faces ? BFB2 : BCB2, faces ? BFC2 : BCC2);
      }
    };
    // count pass: offs[i] holds box i's ints per list, then the exclusive prefix
    std::vector<int64_t> offs((size_t)(nb + 1) * NLIST, 0);
#pragma omp parallel for schedule(static) if (nb > 4096)
    for (int64_t i = 0; i < nb; ++i) proc(lb[i], i >= nbc, false, &offs[(size_t)i * NLIST], nullptr, nullptr);
    int64_t tot[NLIST];
    for (int k = 0; k < NLIST; ++k) {
      int64_t acc = 0;
      for (int64_t i = 0; i <= nb; ++i) {
        const int64_t v = offs[(size_t)i * NLIST + k];
        offs[(size_t)i * NLIST + k] = acc;
        acc += v;
      }
      tot[k] = acc;
    }
    // the lists' places in the upload image (each 64-int aligned, in list order)
    int64_t base[NLIST];
    size_t psz = pack.size();
    for (int k = 0; k < NLIST; ++k) {
      psz = (psz + 63) / 64 * 64;
      base[k] = (int64_t)psz;
      psz += (size_t)tot[k];
    }
    pack.resize(psz);
    // the host copies the queue advance needs: per copy record its destination
    // patch and its first chunk
    L.h_dst.assign((size_t)(tot[RR] / FW), 0);
    L.h_dst2.assign((size_t)(tot[RR2] / FW), 0);
    L.h_chunk0.assign((size_t)(tot[RR] / FW) + 1, (int32_t)(tot[CR] / 4));
    L.h_chunk0_2.assign((size_t)(tot[RR2] / FW) + 1, (int32_t)(tot[CR2] / 4));
    int32_t* pk = pack.data();
#pragma omp parallel for schedule(static) if (nb > 4096)
    for (int64_t i = 0; i < nb; ++i) {
      int64_t cur[NLIST];
      const int64_t* o = &offs[(size_t)i * NLIST];
      for (int k = 0; k < NLIST; ++k) cur[k] = base[k] + o[k];
      const int32_t* b = lb[i];
      if (b[2] == 0) {
        if (o[(size_t)NLIST + RR] > o[RR]) {  // this box has a record (every box but empty ones)
          L.h_dst[o[RR] / FW] = b[0];
          L.h_chunk0[o[RR] / FW] = (int32_t)(o[CR] / 4);
        }
        if (o[(size_t)NLIST + RR2] > o[RR2]) {
          L.h_dst2[o[RR2] / FW] = b[0];
          L.h_chunk0_2[o[RR2] / FW] = (int32_t)(o[CR2] / 4);
        }
      }
      proc(b, i >= nbc, true, cur, pk, base);
    }
    L.runs_split = offs[(size_t)nbc * NLIST + CR] / 4;
    L.runs2_split = offs[(size_t)nbc * NLIST + CR2] / 4;
    L.has_bc = tot[BCB] + tot[BFB] > 0;
    DevList* outs[NLIST] = {&L.runs, &L.chunk_runs, &L.prol_cells, &L.chunk_pcells, &L.prol_faces, &L.chunk_pfaces,
                            &L.bc_cells, &L.chunk_bcells, &L.bc_faces, &L.chunk_bfaces, &L.runs2, &L.chunk_runs2,
                            &L.bc_cells2, &L.chunk_bcells2, &L.bc_faces2, &L.chunk_bfaces2};
    for (int k = 0; k < NLIST; ++k) {
      outs[k]->n = tot[k] / LW[k];
      outs[k]->p = nullptr;
      if (tot[k]) pend.push_back({outs[k], (size_t)base[k]});
    }
    bool ok = true;
    if (l > 0 && ok) {
      auto slice = [&](const std::vector<int32_t>& v, const std::array<int64_t, 2>& r, int w) {
        return std::vector<int32_t>(v.begin() + r[0] * w, v.begin() + r[1] * w);
      };
      if (ctx->dmaps) {
        // built on the device: the level's slices of the six lists
        auto dslice = [&](int list, const std::array<int64_t, 2>& r, int w, DevList& out) {
          out.n = r[1] - r[0];
          out.p = out.n ? ctx->d_maps + ctx->dmap_off[list] + w * r[0] : nullptr;
        };
        dslice(0, H.rng_cf_faces[l], 7, L.cf_faces);
        dslice(1, H.rng_cf_edges[l], 6, L.cf_edges);
        dslice(2, H.rng_emf_faces[l], 8, L.emf_faces);
        dslice(3, H.rng_restrict_cells[l], 5, L.restrict_cells);
        dslice(4, H.rng_restrict_faces[l], 6, L.restrict_faces);
        dslice(5, H.rng_reflux_cells[l], 9, L.reflux_cells);
      } else {
        ok = upload(slice(H.cf_faces, H.rng_cf_faces[l], 7), L.cf_faces, 7) &&
             upload(slice(H.cf_edges, H.rng_cf_edges[l], 6), L.cf_edges, 6) &&
             upload(slice(H.emf_faces, H.rng_emf_faces[l], 8), L.emf_faces, 8) &&
             upload(slice(H.restrict_cells, H.rng_restrict_cells[l], 5), L.restrict_cells, 5) &&
             upload(slice(H.restrict_faces, H.rng_restrict_faces[l], 6), L.restrict_faces, 6) &&
             upload(slice(H.reflux_cells, H.rng_reflux_cells[l], 9), L.reflux_cells, 9);
      }
      L.cf_face0 = H.rng_cf_faces[l][0];
      L.cf_edge0 = H.rng_cf_edges[l][0];
    }
    // direct halo reads: the 3D base level of a one-level hierarchy whose
    // equal patches tile the periodic domain (every halo position lies in the
    // interior of the neighbour patch in the patch grid, at a shift of one
    // patch; every advance of the level updates the interior only, w = 0)
    L.direct_halo = false;
    if (H.dim == 3 && l == 0 && nlev == 1 && !ctx->stage_light && !ids.empty()) {
      bool periodic = true;
      for (int d = 0; d < 3; ++d)
        for (int side = 0; side < 2; ++side) periodic = periodic && ctx->cfg.bc[d][side] == AMRMHD_BC_PERIODIC;
      const int* n0 = H.p[ids[0]].n;
      int N[3], G[3];
      bool uniform = periodic;
      for (int d = 0; d < 3 && uniform; ++d) {
        N[d] = ctx->cfg.base[d] << l;
        uniform = n0[d] >= 4 && N[d] % n0[d] == 0;
        G[d] = uniform ? N[d] / n0[d] : 0;
      }
      std::vector<int> grid;
      if (uniform && (long long)G[0] * G[1] * G[2] == (long long)ids.size()) {
        grid.assign(ids.size(), -1);
        for (int q : ids) {
          const amrmhd::HPatch& Q = H.p[q];
          int g[3];
          for (int d = 0; d < 3 && uniform; ++d) {
            uniform = Q.n[d] == n0[d] && Q.lo[d] % n0[d] == 0;
            g[d] = Q.lo[d] / n0[d];
          }
          if (!uniform) break;
          int& slot = grid[g[0] + G[0] * (g[1] + G[1] * g[2])];
          if (slot >= 0) { uniform = false; break; }
          slot = q;
        }
        if (uniform) {
          std::vector<int32_t> nb;
          nb.reserve(27 * ids.size());
          for (int q : ids) {
            const amrmhd::HPatch& Q = H.p[q];
            const int g[3] = {Q.lo[0] / n0[0], Q.lo[1] / n0[1], Q.lo[2] / n0[2]};
            for (int dz = -1; dz <= 1; ++dz)
              for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                  const int gx = (g[0] + dx + G[0]) % G[0], gy = (g[1] + dy + G[1]) % G[1],
                            gz = (g[2] + dz + G[2]) % G[2];
                  nb.push_back(grid[gx + G[0] * (gy + G[1] * gz)]);
                }
          }
          L.direct_halo = upload(nb, L.nbr, 27);
        }
      }
    }
    if (!ok) return fail(ctx, AMRMHD_ECUDA, std::string("map upload: ") + cudaGetErrorString(e));
  }
  const auto tb1 = std::chrono::steady_clock::now();
  if (!pack.empty()) {
    int* dlists = dbuf<int>(ctx, pack.size(), &e);
    if (e != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, "cudaMalloc");
    CU(cudaMemcpy(dlists, pack.data(), sizeof(int) * pack.size(), cudaMemcpyHostToDevice));
    for (auto& pr : pend) pr.first->p = dlists + pr.second;
  }
  if (std::getenv("AMRMHD_REGRID_TRACE"))
    std::fprintf(stderr, "amrmhd bind: lists %lld us, upload of %.1f MB %lld us\n",
                 (long long)std::chrono::duration_cast<std::chrono::microseconds>(tb1 - tb0).count(),
                 4e-6 * pack.size(),
                 (long long)std::chrono::duration_cast<std::chrono::microseconds>(std::chrono::steady_clock::now() - tb1)
                     .count());
  for (int l = 0; l < nlev; ++l) ctx->lev[l].ids = id_lists[l].p;
  ctx->cur.assign(nlev, 0);
  ctx->start.assign(nlev, 0);
  // side streams for concurrent levels (a regrid's light stages never step)
  for (int l = 0; l + 1 < nlev && !ctx->stage_light; ++l) {
    cudaStream_t st = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    CU(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    CU(cudaEventCreateWithFlags(&a, cudaEventDisableTiming));
    CU(cudaEventCreateWithFlags(&b, cudaEventDisableTiming));
    ctx->side.push_back(st);
    ctx->ev_fork.push_back(a);
    ctx->ev_join.push_back(b);
  }
  if (!ctx->stage_light) {
    CU(cudaStreamCreateWithFlags(&ctx->cfl_stream, cudaStreamNonBlocking));
    CU(cudaEventCreateWithFlags(&ctx->ev_cfl_fork, cudaEventDisableTiming));
    CU(cudaEventCreateWithFlags(&ctx->ev_cfl_join, cudaEventDisableTiming));
  }
  ctx->tile_level.assign(nlev, {-1, -1});
  ctx->zlen_level.assign(nlev, {0, 0});
  ctx->shape_rule = false;
  if (H.dim == 3 && ctx->cfg.precision == AMRMHD_MIXED && !ctx->stage_light) {
    int dev = 0, sms = 0;
    CU(cudaGetDevice(&dev));
    CU(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    ctx->shape_rule = true;
    for (int l = 0; l < nlev; ++l) {
      std::map<std::array<int, 3>, int> patches;
      for (int q : H.level_patches[l]) ++patches[{H.p[q].n[0], H.p[q].n[1], H.p[q].n[2]}];
      for (int wi = 0; wi < (l > 0 ? 2 : 1); ++wi)
        default_shape(patches, 4 * wi, std::max(sms, 1), &ctx->tile_level[l][wi], &ctx->zlen_level[l][wi]);
    }
  }
  ctx->ops->prepare();
  CU(cudaGetLastError());
  ctx->bound = true;
  return AMRMHD_OK;
}

static amrmhd_status io_one(amrmhd_ctx* ctx, int32_t patch, int32_t field, void* buf, int32_t on_device,
                            int to_state, bool packed) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  const amrmhd::Hierarchy& H = ctx->H;
  if (field < 0 || field > 7) return fail(ctx, AMRMHD_EINVAL, "bad field");
  if (!packed && (patch < 0 || patch >= (int)H.p.size())) return fail(ctx, AMRMHD_EINVAL, "bad patch");
  int kind = (field >= 5 && !(H.dim == 2 && field == 7)) ? field - 4 : 0;
  long long count;
  if (packed) count = ctx->ptotal[kind];
  else {
    count = 1;
    for (int d = 0; d < H.dim; ++d) count *= H.p[patch].n[d] + (kind == d + 1 ? 1 : 0);
  }
  double* stage = (double*)(ctx->arena + ctx->o_stage);
  double* dev = on_device ? (double*)buf : stage;
  // the I/O kernel addresses packed[poff[pid] + t]; for a single patch shift the base
  double* kbase = packed ? dev : dev - ctx->poff[kind][patch];
  const int* ids = packed ? ctx->d_iota : ctx->d_iota + patch;
  const int npatch = packed ? (int)H.p.size() : 1;
  const int* maxn = packed ? ctx->maxn_all : H.p[patch].n;
  void* state = state_buf(ctx, ctx->cur[H.p[packed ? 0 : patch].level]);
  if (packed) {
    // patches of different levels may sit in different buffers: one launch per level
    if (to_state && !on_device) CU(cudaMemcpyAsync(stage, buf, count * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    for (int l = 0; l < H.nlev; ++l) {
      const LevelDev& L = ctx->lev[l];
      int lm[3] = {L.maxn[0], L.maxn[1], L.maxn[2]};
      int nl = 0;
      ctx->ops->io(ctx->dP, L.ids, L.npatch, lm, state_buf(ctx, ctx->cur[l]), dev, ctx->d_poff[kind], field, to_state,
                   ctx->stream, &nl);
    }
    if (!to_state && !on_device) {
      CU(cudaMemcpyAsync(buf, stage, count * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
      CU(cudaStreamSynchronize(ctx->stream));
    }
    CU(cudaGetLastError());
    return AMRMHD_OK;
  }
  if (to_state && !on_device) CU(cudaMemcpyAsync(stage, buf, count * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
  int nl = 0;
  ctx->ops->io(ctx->dP, ids, npatch, maxn, state, kbase, ctx->d_poff[kind], field, to_state, ctx->stream, &nl);
  if (!to_state && !on_device) {
    CU(cudaMemcpyAsync(buf, stage, count * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CU(cudaStreamSynchronize(ctx->stream));
  }
  CU(cudaGetLastError());
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_state(amrmhd_ctx* ctx, int32_t patch, int32_t field, const void* src, int32_t on_device) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  if (!src) return fail(ctx, AMRMHD_EINVAL, "null source");
  return io_one(ctx, patch, field, (void*)src, on_device, 1, false);
}

amrmhd_status amrmhd_get_state(amrmhd_ctx* ctx, int32_t patch, int32_t field, void* dst, int32_t on_device) {
  if (!dst) return fail(ctx, AMRMHD_EINVAL, "null destination");
  return io_one(ctx, patch, field, dst, on_device, 0, false);
}

amrmhd_status amrmhd_packed_size(amrmhd_ctx* ctx, int32_t field, int64_t* count) {
  if (!ctx || !count) return AMRMHD_EINVAL;
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "no hierarchy set");
  if (field < 0 || field > 7) return fail(ctx, AMRMHD_EINVAL, "bad field");
  int kind = (field >= 5 && !(ctx->H.dim == 2 && field == 7)) ? field - 4 : 0;
  *count = ctx->ptotal[kind];
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_state_packed(amrmhd_ctx* ctx, int32_t field, const double* src, int32_t on_device) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  if (!src) return fail(ctx, AMRMHD_EINVAL, "null source");
  return io_one(ctx, 0, field, (void*)src, on_device, 1, true);
}

amrmhd_status amrmhd_get_state_packed(amrmhd_ctx* ctx, int32_t field, double* dst, int32_t on_device) {
  if (!dst) return fail(ctx, AMRMHD_EINVAL, "null destination");
  return io_one(ctx, 0, field, dst, on_device, 0, true);
}

// all 8 packed fields one after the other (the amrmhd_backward layout)
static amrmhd_status io_all(amrmhd_ctx* ctx, void* buf, int32_t on_device, int to_state, int f32) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  const amrmhd::Hierarchy& H = ctx->H;
  const size_t esz = f32 ? sizeof(float) : sizeof(double);
  long long total = 0, off[8];
  for (int f = 0; f < 8; ++f) {
    const int kind = (f >= 5 && !(H.dim == 2 && f == 7)) ? f - 4 : 0;
    off[f] = total;
    total += ctx->ptotal[kind];
  }
  void* dev = buf;
  bool mapped = false;
  if (!on_device) {
    // page-locked host memory mapped into the device address space: the packing
    // kernels read or write it directly over the host link (one pass, no
    // staging copy); other host memory goes through a device staging buffer
    cudaPointerAttributes pa;
    if (ctx->opt_host_io == 0 && cudaPointerGetAttributes(&pa, buf) == cudaSuccess && pa.type == cudaMemoryTypeHost &&
        pa.devicePointer) {
      dev = pa.devicePointer;
      mapped = true;
    } else {
      cudaGetLastError();  // an unregistered pointer is not an error here
      if (!ctx->d_stage_all) {
        cudaError_t e = cudaSuccess;
        ctx->d_stage_all = dbuf<double>(ctx, (size_t)total, &e);  // room for either element type
        if (e != cudaSuccess) return fail(ctx, AMRMHD_ENOMEM, "staging buffer");
      }
      dev = ctx->d_stage_all;
      if (to_state) CU(cudaMemcpyAsync(dev, buf, total * esz, cudaMemcpyHostToDevice, ctx->stream));
    }
  }
  // all 8 fields of a level per launch
  for (int l = 0; l < H.nlev; ++l) {
    const LevelDev& L = ctx->lev[l];
    int lm[3] = {L.maxn[0], L.maxn[1], L.maxn[2]};
    int nl = 0;
    ctx->ops->io_all(ctx->dP, L.ids, L.npatch, lm, state_buf(ctx, ctx->cur[l]), dev, f32, ctx->d_poff_tab, off,
                     to_state, ctx->stream, &nl);
  }
  if (!to_state && !on_device && !mapped)
    CU(cudaMemcpyAsync(buf, dev, total * esz, cudaMemcpyDeviceToHost, ctx->stream));
  if (!on_device) CU(cudaStreamSynchronize(ctx->stream));
  return AMRMHD_OK;
}

amrmhd_status amrmhd_set_state_all(amrmhd_ctx* ctx, const double* src, int32_t on_device) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  if (!src) return fail(ctx, AMRMHD_EINVAL, "null source");
  return io_all(ctx, (void*)src, on_device, 1, 0);
}

amrmhd_status amrmhd_get_state_all(amrmhd_ctx* ctx, double* dst, int32_t on_device) {
  if (!dst) return fail(ctx, AMRMHD_EINVAL, "null destination");
  return io_all(ctx, dst, on_device, 0, 0);
}

amrmhd_status amrmhd_set_state_all_f32(amrmhd_ctx* ctx, const float* src, int32_t on_device) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  if (!src) return fail(ctx, AMRMHD_EINVAL, "null source");
  return io_all(ctx, (void*)src, on_device, 1, 1);
}

amrmhd_status amrmhd_get_state_all_f32(amrmhd_ctx* ctx, float* dst, int32_t on_device) {
  if (!dst) return fail(ctx, AMRMHD_EINVAL, "null destination");
  return io_all(ctx, dst, on_device, 0, 1);
}

amrmhd_status amrmhd_export_map(amrmhd_ctx* ctx, int32_t which, int32_t* dst, int64_t cap, int64_t* len,
                                int32_t* width) {
  if (!ctx || !len) return AMRMHD_EINVAL;
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "no hierarchy set");
  std::vector<int32_t> tmp;
  const std::vector<int32_t>* v = nullptr;
  int w = 0;
  if (which == AMRMHD_MAP_NEIGHBORS) {
    w = 5;
    for (size_t q = 0; q < ctx->H.nbr.size(); ++q)
      for (const amrmhd::Nbr& x : ctx->H.nbr[q]) {
        tmp.push_back((int32_t)q); tmp.push_back(x.q); tmp.push_back(x.s[0]); tmp.push_back(x.s[1]); tmp.push_back(x.s[2]);
      }
    v = &tmp;
  } else {
    v = map_vec(ctx, which, &w);
    if (!v) return fail(ctx, AMRMHD_EINVAL, "unknown map");
  }
  *len = (int64_t)v->size();
  if (width) *width = w;
  if (dst && cap > 0) std::memcpy(dst, v->data(), sizeof(int32_t) * (size_t)std::min<int64_t>(cap, *len));
  return AMRMHD_OK;
}

amrmhd_status amrmhd_fill_ghosts(amrmhd_ctx* ctx, int32_t level, int32_t substep) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  if (level < 0 || level >= ctx->H.nlev || (substep != 1 && substep != 2)) return fail(ctx, AMRMHD_EINVAL, "bad level/substep");
  int nl = 0;
  op_fill(ctx, level, substep, &nl);
  ctx->launches += nl;
  CU(cudaGetLastError());
  return AMRMHD_OK;
}

amrmhd_status amrmhd_advance_level(amrmhd_ctx* ctx, int32_t level, double dt, int32_t substep) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  if (level < 0 || level >= ctx->H.nlev || (substep != 1 && substep != 2) || !(dt >= 0.0))
    return fail(ctx, AMRMHD_EINVAL, "bad level/substep/dt");
  int nl = 1;
  double* slot = ctx->d_scal + 1 + level;
  amrk::launch_set_scalar(slot, dt, ctx->stream);
  op_advance(ctx, level, slot, 1.0, substep, &nl);
  ctx->launches += nl;
  CU(cudaGetLastError());
  return AMRMHD_OK;
}

amrmhd_status amrmhd_reflux_restrict(amrmhd_ctx* ctx, int32_t fine_level) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  if (fine_level < 1 || fine_level >= ctx->H.nlev) return fail(ctx, AMRMHD_EINVAL, "bad fine level");
  int nl = 0;
  op_reflux_restrict(ctx, fine_level, &nl);
  ctx->launches += nl;
  CU(cudaGetLastError());
  return AMRMHD_OK;
}

amrmhd_status amrmhd_cfl_dt(amrmhd_ctx* ctx, double* dt0) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  int nl = 0;
  op_cfl(ctx, nullptr, &nl);
  ctx->launches += nl;
  double v = 0;
  unsigned int err = 0;
  CU(cudaMemcpyAsync(&v, ctx->d_scal, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaMemcpyAsync(&err, ctx->d_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  if (err) {
    CU(cudaMemset(ctx->d_err, 0, sizeof(unsigned int)));
    return fail(ctx, AMRMHD_ENONPHYS, "non-finite or non-positive density or pressure");
  }
  if (dt0) *dt0 = v;
  return AMRMHD_OK;
}

// waits for the context's stream, then reports and clears the error word
static amrmhd_status report_device_error(amrmhd_ctx* ctx) {
  unsigned int err = 0;
  CU(cudaMemcpyAsync(&err, ctx->d_err, sizeof(unsigned int), cudaMemcpyDeviceToHost, ctx->stream));
  CU(cudaStreamSynchronize(ctx->stream));
  if (err) {
    CU(cudaMemset(ctx->d_err, 0, sizeof(unsigned int)));
    if (err & amrk::ERR_QUEUE_TIMEOUT)
      return fail(ctx, AMRMHD_ETIMEOUT, "a wait of the queue advance ran out (a fill signal never came)");
    return fail(ctx, AMRMHD_ENONPHYS, "non-finite or non-positive density or pressure");
  }
  return AMRMHD_OK;
}

// n_coarse coarse steps; wait: synchronise and report device errors
static amrmhd_status step_impl(amrmhd_ctx* ctx, int32_t n_coarse, double* dt_used, bool wait) {
  if (ctx) ++ctx->state_version;  // a recorded forward (amrmhd_step_dt_ckpt) no longer matches
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  if (n_coarse < 0) return fail(ctx, AMRMHD_EINVAL, "negative step count");
  if (n_coarse == 0) return AMRMHD_OK;
  const int nlev = ctx->H.nlev;
  if (queue_active(ctx)) {
    st = build_queue_plan(ctx);
    if (st) return st;
  }
  for (int32_t done = 0; done < n_coarse;) {
    const int32_t chunk = (int32_t)std::min<int64_t>(kHistCap, n_coarse - done);
    CU(cudaMemsetAsync(ctx->d_slots + nlev, 0, sizeof(unsigned long long), ctx->stream));
    for (int it = 0; it < chunk; ++it) {
      if (ctx->opt_graph) {
        const int par = ctx->cur[0];
        // a graph bakes in every level's buffer choice: recapture when direct
        // level calls have changed the finer levels' buffers since the capture
        if (ctx->gexec[par] && ctx->g_cur_before[par] != ctx->cur) {
          cudaGraphExecDestroy(ctx->gexec[par]);
          ctx->gexec[par] = nullptr;
        }
        if (!ctx->gexec[par]) {
          std::vector<int> c0 = ctx->cur, s0 = ctx->start;
          cudaGraph_t g = nullptr;
          CU(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
          int nl = 0;
          op_coarse_step(ctx, &nl);
          cudaError_t ce = cudaStreamEndCapture(ctx->stream, &g);
          if (ce != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
          ce = cudaGraphInstantiate(&ctx->gexec[par], g, 0);
          cudaGraphDestroy(g);
          if (ce != cudaSuccess) return fail(ctx, AMRMHD_ECUDA, std::string("graph instantiate: ") + cudaGetErrorString(ce));
          ctx->g_cur_before[par] = c0;
          ctx->g_cur_after[par] = ctx->cur;
          ctx->g_start_after[par] = ctx->start;
          ctx->g_launches[par] = nl;
          ctx->cur = c0;
          ctx->start = s0;
        }
        CU(cudaGraphLaunch(ctx->gexec[par], ctx->stream));
        ctx->cur = ctx->g_cur_after[par];
        ctx->start = ctx->g_start_after[par];
        ctx->launches += ctx->g_launches[par];
      } else {
        int nl = 0;
        op_coarse_step(ctx, &nl);
        ctx->launches += nl;
        CU(cudaGetLastError());
      }
    }
    if (dt_used)
      CU(cudaMemcpyAsync(dt_used + done, ctx->d_hist, sizeof(double) * chunk, cudaMemcpyDeviceToHost, ctx->stream));
    done += chunk;
  }
  return wait ? report_device_error(ctx) : AMRMHD_OK;
}

amrmhd_status amrmhd_step(amrmhd_ctx* ctx, int32_t n_coarse, double* dt_used) {
  return step_impl(ctx, n_coarse, dt_used, true);
}

amrmhd_status amrmhd_step_async(amrmhd_ctx* ctx, int32_t n_coarse) { return step_impl(ctx, n_coarse, nullptr, false); }

amrmhd_status amrmhd_sync(amrmhd_ctx* ctx) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  return report_device_error(ctx);
}

amrmhd_status amrmhd_autotune(amrmhd_ctx* ctx, int32_t trials, int32_t* tiles) {
  amrmhd_status st = check_bound(ctx);
  if (st) return st;
  if (trials < 1) return fail(ctx, AMRMHD_EINVAL, "trials must be positive");
  const int nlev = ctx->H.nlev;
  if (!ctx->fused()) {
    if (tiles)
      for (int l = 0; l < nlev; ++l) tiles[l] = -1;
    return AMRMHD_OK;
  }
  // a CFL dt for the timed advances (the state is not changed: an advance
  // reads the current buffer and writes the other one)
  int nl = 0;
  op_cfl(ctx, nullptr, &nl);
  cudaEvent_t e0, e1;
  CU(cudaEventCreate(&e0));
  CU(cudaEventCreate(&e1));
  const int64_t keep = ctx->opt_tile, keepz = ctx->opt_zchunk;
  ctx->shape_rule = false;
  ctx->opt_tile = -1;
  ctx->opt_zchunk = -1;
  for (int l = 0; l < nlev; ++l) {
    // sub-step 1 of a level above 0 advances 2 extended ghost layers, sub-step 2
    // (and level 0) the interior only: each gets its own tile and z chunk (the
    // whole column, or 4, 8 or 16 planes per CTA: shorter marches in more
    // CTAs for levels of few or tall patches; or whole columns with those of
    // the launch's last partial wave halved, for a level of many columns)
    for (int s = 1; s <= (l > 0 ? 2 : 1); ++s) {
      const int wi = (l > 0 && s == 1) ? 1 : 0;
      float best = 0.0f;
      int bv = -1, bz = 0;
      const int ez = ctx->lev[l].maxn[2] + (wi ? 4 : 0);
      static const int zlens[5] = {0, -2, 4, 8, 16};
      for (int k = 0; k < 25; ++k) {
        const int v = k % 5, zl = zlens[k / 5];
        if (zl > 0 && zl >= ez) continue;  // one chunk: the whole column, timed already
        ctx->tile_level[l][wi] = v;
        ctx->zlen_level[l][wi] = zl;
        const int c0 = ctx->cur[l];
        op_advance(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), s, &nl);  // warm-up
        ctx->cur[l] = c0;
        if (cudaGetLastError() != cudaSuccess) continue;
        CU(cudaEventRecord(e0, ctx->stream));
        for (int t = 0; t < trials; ++t) {
          op_advance(ctx, l, ctx->d_scal, 1.0 / (double)(1 << l), s, &nl);
          ctx->cur[l] = c0;
        }
        CU(cudaEventRecord(e1, ctx->stream));
        CU(cudaEventSynchronize(e1));
        if (cudaGetLastError() != cudaSuccess) continue;
        float ms = 0.0f;
        CU(cudaEventElapsedTime(&ms, e0, e1));
        if (bv < 0 || ms < best) { best = ms; bv = v; bz = zl; }
      }
      ctx->tile_level[l][wi] = bv;
      ctx->zlen_level[l][wi] = bv < 0 ? 0 : bz;
      if (tiles && wi == 0) tiles[l] = bv;
    }
  }
  ctx->opt_tile = keep;
  ctx->opt_zchunk = keepz;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  for (int i = 0; i < 2; ++i)
    if (ctx->gexec[i]) { cudaGraphExecDestroy(ctx->gexec[i]); ctx->gexec[i] = nullptr; }
  CU(cudaStreamSynchronize(ctx->stream));
  return AMRMHD_OK;
}

amrmhd_status amrmhd_tile_choice(amrmhd_ctx* ctx, int32_t level, int32_t kind, int32_t* tile, int32_t* zlen) {
  if (!ctx || !tile || !zlen) return AMRMHD_EINVAL;
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "no hierarchy set");
  if (level < 0 || level >= ctx->H.nlev || (kind != 0 && kind != 1)) return fail(ctx, AMRMHD_EINVAL, "level or kind");
  if (!ctx->fused()) {
    *tile = -1;
    *zlen = 0;
  } else {
    *tile = ctx->tile_of(level, kind);
    *zlen = ctx->zlen_of(level, kind);
  }
  return AMRMHD_OK;
}

amrmhd_status amrmhd_query(amrmhd_ctx* ctx, int32_t what, int64_t* value) {
  if (!ctx || !value) return AMRMHD_EINVAL;
  if (what == AMRMHD_Q_KERNEL_LAUNCHES) { *value = ctx->launches; return AMRMHD_OK; }
  if (!ctx->have_h) return fail(ctx, AMRMHD_ESTATE, "no hierarchy set");
  const amrmhd::Hierarchy& H = ctx->H;
  switch (what) {
    case AMRMHD_Q_NPATCH: *value = (int64_t)H.p.size(); return AMRMHD_OK;
    case AMRMHD_Q_NLEVEL: *value = H.nlev; return AMRMHD_OK;
    case AMRMHD_Q_CELLS:
    case AMRMHD_Q_CELL_UPDATES_PER_STEP: {
      int64_t t = 0;
      for (const auto& P : H.p) {
        int64_t c = (int64_t)P.n[0] * P.n[1] * P.n[2];
        t += what == AMRMHD_Q_CELLS ? c : (c << P.level);
      }
      *value = t;
      return AMRMHD_OK;
    }
    case AMRMHD_Q_ARENA_BYTES: *value = (int64_t)ctx->arena_bytes; return AMRMHD_OK;
    case AMRMHD_Q_REGRID_FLAG_US:
    case AMRMHD_Q_REGRID_CLUSTER_US:
    case AMRMHD_Q_REGRID_BUILD_US:
    case AMRMHD_Q_REGRID_TRANSFER_US:
    case AMRMHD_Q_REGRID_MAPS_US: *value = ctx->regrid_us[what - AMRMHD_Q_REGRID_FLAG_US]; return AMRMHD_OK;
    case AMRMHD_Q_REGRID_TRANSFER_MAPS_US: *value = ctx->regrid_us[5]; return AMRMHD_OK;
    case AMRMHD_Q_MAPS_HOST_US:
    case AMRMHD_Q_MAPS_GHOST_US:
    case AMRMHD_Q_MAPS_REGISTERS_US: *value = ctx->maps_us[what - AMRMHD_Q_MAPS_HOST_US]; return AMRMHD_OK;
    case AMRMHD_Q_FLOOR_EVENTS: {
      unsigned long long v = 0;
      if (ctx->bound && ctx->d_floor_events) {
        CU(cudaMemcpyAsync(&v, ctx->d_floor_events, sizeof(v), cudaMemcpyDeviceToHost, ctx->stream));
        CU(cudaStreamSynchronize(ctx->stream));
      }
      *value = (int64_t)v;
      return AMRMHD_OK;
    }
    default: return fail(ctx, AMRMHD_EINVAL, "unknown query");
  }
}

const char* amrmhd_last_error(const amrmhd_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

amrmhd_status amrmhd_grad_velocity(int64_t ncells, const double* u0, const double* dL_dU0, double* dL_dv0,
                                   void* cuda_stream) {
  if (ncells < 0 || (ncells > 0 && (!u0 || !dL_dU0 || !dL_dv0))) return AMRMHD_EINVAL;
  if (ncells == 0) return AMRMHD_OK;
  amrk::launch_grad_velocity(ncells, u0, dL_dU0, dL_dv0, (cudaStream_t)cuda_stream);
  return cudaGetLastError() == cudaSuccess ? AMRMHD_OK : AMRMHD_ECUDA;
}

amrmhd_status amrmhd_alu_peak(int32_t fp64, double* flops_per_s, int32_t* sms) {
  if ((fp64 != 0 && fp64 != 1) || !flops_per_s) return AMRMHD_EINVAL;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
    return AMRMHD_ECUDA;
  if (sms) *sms = nsm;
  const int threads = 256, blocks = nsm * 8;  // 64 warps per SM
  void* out = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaMalloc(&out, sizeof(double) * blocks) != cudaSuccess) return AMRMHD_ECUDA;
  amrmhd_status st = AMRMHD_OK;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) st = AMRMHD_ECUDA;
  // iterations sized for about 50-100 ms at the expected rate; best of 5
  const int iters = fp64 ? 4096 : 1 << 17;
  float best = 0.0f;
  for (int rep = 0; rep < 6 && st == AMRMHD_OK; ++rep) {
    cudaEventRecord(e0, 0);
    amrk::launch_fma_peak(fp64, blocks, threads, iters, out, 0);
    cudaEventRecord(e1, 0);
    float ms = 0.0f;
    if (cudaGetLastError() != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
        cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
      st = AMRMHD_ECUDA;
      break;
    }
    if (rep > 0 && (best == 0.0f || ms < best)) best = ms;  // the first run warms up
  }
  if (st == AMRMHD_OK) *flops_per_s = 2.0 * 8.0 * (double)iters * threads * (double)blocks / (best * 1e-3);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(out);
  return st;
}

amrmhd_status amrmhd_recover_mixed(int64_t n, const float* u, const float* bl, const float* br, double gamma,
                                   float* w) {
  if (n < 0 || (n > 0 && (!u || !bl || !br || !w)) || !(gamma > 1.0)) return AMRMHD_EINVAL;
  if (n == 0) return AMRMHD_OK;
  const size_t nf = sizeof(float) * (size_t)n;
  char* buf = nullptr;
  if (cudaMalloc(&buf, 19 * nf) != cudaSuccess) return AMRMHD_ECUDA;
  float* du = (float*)buf;
  float* dl = du + 5 * n;
  float* dr = dl + 3 * n;
  float* dw = dr + 3 * n;
  amrmhd_status st = AMRMHD_OK;
  if (cudaMemcpy(du, u, 5 * nf, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(dl, bl, 3 * nf, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(dr, br, 3 * nf, cudaMemcpyHostToDevice) != cudaSuccess) {
    st = AMRMHD_ECUDA;
  } else {
    amrk::launch_recover_mixed(n, du, dl, dr, gamma - 1.0, dw, 0);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(w, dw, 8 * nf, cudaMemcpyDeviceToHost) != cudaSuccess)
      st = AMRMHD_ECUDA;
  }
  cudaFree(buf);
  return st;
}

amrmhd_status amrmhd_fp_convert(int32_t on_device, int64_t n, const double* x, const float* y, float* x_narrow,
                                double* y_widen, float* x_narrow_hw, double* y_widen_hw) {
  if ((on_device != 0 && on_device != 1) || n < 0 ||
      (n > 0 && (!x || !y || !x_narrow || !y_widen || !x_narrow_hw || !y_widen_hw)))
    return AMRMHD_EINVAL;
  if (n == 0) return AMRMHD_OK;
  if (!on_device) {
    for (int64_t i = 0; i < n; ++i) {
      x_narrow[i] = amrdev::narrow_bits(x[i]);
      y_widen[i] = amrdev::widen_bits(y[i]);
      x_narrow_hw[i] = (float)x[i];
      y_widen_hw[i] = (double)y[i];
    }
    return AMRMHD_OK;
  }
  // one allocation: x, y_widen, y_widen_hw (doubles), then y, x_narrow, x_narrow_hw
  char* buf = nullptr;
  const size_t nd = sizeof(double) * (size_t)n, nf = sizeof(float) * (size_t)n;
  if (cudaMalloc(&buf, 3 * nd + 3 * nf) != cudaSuccess) return AMRMHD_ECUDA;
  double* dx = (double*)buf;
  double* dyw = dx + n;
  double* dywh = dyw + n;
  float* dy = (float*)(buf + 3 * nd);
  float* dxn = dy + n;
  float* dxnh = dxn + n;
  amrmhd_status st = AMRMHD_OK;
  if (cudaMemcpy(dx, x, nd, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(dy, y, nf, cudaMemcpyHostToDevice) != cudaSuccess) {
    st = AMRMHD_ECUDA;
  } else {
    amrk::launch_fp_convert(n, dx, dy, dxn, dyw, dxnh, dywh, 0);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(x_narrow, dxn, nf, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(x_narrow_hw, dxnh, nf, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(y_widen, dyw, nd, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(y_widen_hw, dywh, nd, cudaMemcpyDeviceToHost) != cudaSuccess)
      st = AMRMHD_ECUDA;
  }
  cudaFree(buf);
  return st;
}

}  // extern "C"
