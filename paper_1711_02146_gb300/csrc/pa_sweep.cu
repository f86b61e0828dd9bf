// pa_sweep.cu — launches of the +-1 sweep kernels (pa_sweep_tile.cuh): the table of
// launch shapes and the split of a mostly empty last wave.
#include <algorithm>

#include "pa_sweep_tile.cuh"

namespace pa {

namespace {

// Candidate launch shapes of the +-1 sweep: words per site row W (32W replicas
// per tile), threads per CTA, CTAs per SM the kernel is compiled for (its
// register cap).  The first entry of each L is the default; the autotuner may
// pick another, and a run too small to give every SM a tile takes the shape
// with the most tiles (the W = 8 entries exist for those).  All give identical
// results.  At L = 14 the partitions of a
// warp may straddle the two parity classes (it then runs both colour offsets).
ShapeList shapes_of(int L) {
  switch (L) {
    case 2: return sweep_shapes_2();
    case 4: return sweep_shapes_4();
    case 6: return sweep_shapes_6();
    case 8: return sweep_shapes_8();
    case 10: return sweep_shapes_10();
    case 12: return sweep_shapes_12();
    case 14: return sweep_shapes_14();
    case 16: return sweep_shapes_16();
    default: return {nullptr, 0};
  }
}

const ShapeEntry* shape_of(int L, int i) {
  const ShapeList s = shapes_of(L);
  return i >= 0 && i < s.n ? &s.e[i] : nullptr;
}

}  // namespace

bool sweep_supported(int L) { return L >= 2 && L <= kMaxL && L % 2 == 0; }

int sweep_shape_count(int L) { return shapes_of(L).n; }

bool sweep_shape_info(int L, int i, SweepShapeInfo* out) {
  const ShapeEntry* e = shape_of(L, i);
  if (!e || !out) return false;
  out->L = e->L;
  out->W = e->W;
  out->NT = e->NT;
  out->MB = e->MB;
  out->smem = (int32_t)e->smem;
  return true;
}

static int sweep_launches(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, int t, int n_sweeps,
                          const uint32_t met_thr[3], bool fresh, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  const ShapeEntry* shape = shape_of(g.L, g.sweep_shape);
  if (!shape) return (int)cudaErrorInvalidValue;
  const ShapeEntry* tail = g.tail_shape >= 0 ? shape_of(g.L, g.tail_shape) : nullptr;
  for (int i = 0; i < g.n_pop; ++i) {
    SweepArgs args;
    fill_sweep_args(args, pops[i], jtab, g.n_levels, t, cur, n_sweeps, 32 * shape->W, met_thr);
    args.slot_base = g.slot_base;
    args.fam = g.shard ? 0 : 1;
    args.fresh = fresh ? 1 : 0;
    args.split = tail ? g.tail_from : 0x7fffffff;
    args.chained = i > 0 ? 1 : 0;
    args.tj_tail = tail ? 32 * tail->W : 32 * shape->W;
    int e = shape->launch(g, args, s);
    if (e == 0 && tail) {
      // not chained: the SMs that finish first would take two of its tiles each, where the
      // idle chip spreads them one to an SM (L = 10, R = 1e6: 213 against 207 ms a run)
      args.tile_base = g.tail_from;
      args.chained = 0;
      e = tail->launch(g, args, s);
    }
    if (e != 0) return e;
  }
  return 0;
}

int launch_sweep(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, int t, int n_sweeps,
                 const uint32_t met_thr[3], void* stream) {
  return sweep_launches(g, pops, cur, jtab, t, n_sweeps, met_thr, false, stream);
}

int launch_sweep_initial(const RunGeom& g, PopDev* pops, const uint32_t* jtab, void* stream) {
  const uint32_t none[3] = {0u, 0u, 0u};
  return sweep_launches(g, pops, 1, jtab, 0, 0, none, true, stream);
}

int sweep_tile_slots(int L, int shape) {
  const ShapeEntry* e = shape_of(L, shape);
  return e ? 32 * e->W : 0;
}

int launch_group_sweep(int L, int shape, const GroupUnit* units, const int32_t* list, const int32_t* off, int n,
                       int n_blocks, const int32_t* round, void* stream) {
  const ShapeEntry* e = shape_of(L, shape);
  if (!e || n <= 0) return (int)cudaErrorInvalidValue;
  return e->launch_group(units, list, off, n, n_blocks, round, (cudaStream_t)stream);
}

void sweep_tail_plan(int L, int shape, int64_t R, int n_sm, int32_t* tail_shape, int32_t* tail_from) {
  *tail_shape = -1;
  *tail_from = 0;
  const ShapeEntry* m = shape_of(L, shape);
  if (!m || n_sm <= 0) return;
  const int64_t tj = 32LL * m->W, slots = (int64_t)n_sm * m->MB, tiles = (R + tj - 1) / tj;
  const int64_t full = tiles / slots, rest = tiles - full * slots;
  if (full < 1 || rest == 0 || 10 * rest > 6 * slots) return;  // the last wave is more than 60 % full
  int best = -1;
  for (int i = 0; i < sweep_shape_count(L); ++i) {  // the largest smaller tile
    const ShapeEntry* e = shape_of(L, i);
    if (e->W < m->W && (best < 0 || e->W > shape_of(L, best)->W)) best = i;
  }
  if (best < 0) return;
  *tail_shape = best;
  *tail_from = (int32_t)(full * slots * tj);
}

}  // namespace pa
