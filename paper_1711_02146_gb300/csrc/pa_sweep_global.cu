// pa_sweep_global.cu — the sweep for lattices too large for a tile in shared
// memory (16 < L <= 64, +-1 couplings).  A step transposes the resampled population
// (the rows of the parents, §II) into site-major words in global memory, word w of a
// site holding slots 32 w .. 32 w + 31 as the tile kernel's words do, runs every
// half-sweep as one launch over all sites of one colour, in place, counts the energy
// levels of the words, and transposes them back into rows.  The half-sweep is the
// tile kernel's bit-sliced Metropolis test (pa_metropolis.cuh), with the words still
// undecided after eight bit planes queued per warp and finished by whole warps.
//
// One bit per spin keeps the words of moderate populations in the L2 cache (35 MB at
// L = 24 and 2e4 replicas) for all half-sweeps of a step, so a half-sweep is bound by
// integer issue, as the tile kernel is.  L = 24, R = 2e4, ten steps of ten sweeps: 14.4 ms
// for the whole run, from 328 ms with int8 spins (276 MB) and eight replicas per thread
// decided one bit at a time (233 ms of half-sweeps, 90 ms of level counts).
#include <cuda_runtime.h>

#include "pa_bits.cuh"
#include "pa_device.cuh"
#include "pa_internal.h"
#include "pa_metropolis.cuh"

namespace pa {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// The scratch of population P behind the rows of its buffer `buf`: site-major words
// [N][wp] and the step's site records [N].  The buffer's N pitch bytes hold the rows
// (about N pitch / 8), the words (N pitch / 8) and the records (32 N) for every L > 16.
struct Lattice {
  uint32_t* words;
  SiteRec* recs;
  int wp;  // words per site
};

__host__ __device__ inline Lattice lattice_of(const RunGeom& g, const PopDev& P, int buf) {
  Lattice lat;
  lat.wp = (int)(g.pitch / 32);
  lat.words = P.spins[buf] + (size_t)g.pitch * g.sw;
  lat.recs = reinterpret_cast<SiteRec*>(lat.words + (size_t)g.N * lat.wp);
  return lat;
}

struct LatticeArgs : MetropolisArgs {
  RunGeom g;
  PopDev P;
  const uint32_t* jtab;
  int cur, t, fresh;
};

__global__ void __launch_bounds__(kThreads) k_lattice_records(const __grid_constant__ LatticeArgs a) {
  const int n = blockIdx.x * kThreads + threadIdx.x;
  if (n < a.g.N) lattice_of(a.g, a.P, 1 - a.cur).recs[n] = site_record(a.g.L, n, a.jtab, (uint32_t)a.t, a);
}

// Rows <-> site-major words: a warp takes the 32 slots of one word and 32 words of
// their rows (1024 sites), lanes along the row, so that the row accesses are whole
// lines; each lane transposes its 32 x 32 bits, and the block's eight words of a site
// go through shared memory to be accessed together (one sector).  to_rows: words ->
// rows of the new buffer; else rows of the parents in the old buffer -> words.
template <bool TO_ROWS>
__global__ void __launch_bounds__(kThreads) k_lattice_transpose(const __grid_constant__ LatticeArgs a) {
  __shared__ uint32_t sh[32 * 32 * (kWarps + 1)];  // [site in block][lane][word], padded
  const RunGeom& g = a.g;
  const int R = a.P.rec[a.t].R_tilde;
  const Lattice lat = lattice_of(g, a.P, 1 - a.cur);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w0 = blockIdx.x * kWarps, w = w0 + warp, blk = blockIdx.y * 32 + lane;
  if (32 * w0 >= R) return;
  uint32_t m[32];
  auto words = [&](bool load) {  // the block's words of each of its 1024 sites, eight at a time
    for (int idx = threadIdx.x; idx < 1024 * kWarps; idx += kThreads) {
      const int k = idx % kWarps, s = idx / kWarps;  // s = 32 lane' + i: site 32 (32 blockIdx.y + lane') + i
      const int n = 1024 * blockIdx.y + s;
      if (n >= g.N) break;
      uint32_t* p = lat.words + (size_t)n * lat.wp + w0 + k;
      uint32_t& v = sh[((s & 31) * 32 + (s >> 5)) * (kWarps + 1) + k];
      if (load) v = *p; else *p = v;
    }
  };
  if (TO_ROWS) {
    words(true);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 32; ++i) m[i] = 32 * blk + i < g.N ? sh[(i * 32 + lane) * (kWarps + 1) + warp] : 0u;
    transpose32(m);
    if (blk < g.sw) {
#pragma unroll
      for (int i = 0; i < 32; ++i) a.P.spins[1 - a.cur][(size_t)(32 * w + i) * g.sw + blk] = m[i];
    }
  } else {
    const uint32_t* old = a.P.spins[a.cur];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int j = 32 * w + i;
      const int p = j < R ? (a.fresh ? j : a.P.parents[j]) : -1;
      m[i] = p >= 0 && blk < g.sw ? old[(size_t)p * g.sw + blk] : 0u;
    }
    transpose32(m);
#pragma unroll
    for (int i = 0; i < 32; ++i) sh[(i * 32 + lane) * (kWarps + 1) + warp] = m[i];
    __syncthreads();
    words(false);
  }
}

// One half-sweep (colour c, index q = 2 s + c): thread idx takes word idx mod n_words of
// the colour sites of row idx div n_words, so that a warp reads neighbouring words of a
// site together whatever the population.
struct __align__(16) LatticeDeferred {
  uint32_t loc, eq, u0, u1;  // loc: lane of the owner | colour site in its row << 5
};

template <int FORM>
__global__ void __launch_bounds__(kThreads) k_lattice_sweep(const __grid_constant__ LatticeArgs a, int q) {
  __shared__ LatticeDeferred queues[kWarps][64];
  const RunGeom& g = a.g;
  const int L = g.L, H = L / 2, c = q & 1;
  const int n_words = (a.P.rec[a.t].R_tilde + 31) / 32;
  const Lattice lat = lattice_of(g, a.P, 1 - a.cur);
  const int64_t idx = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  LatticeDeferred* dq = queues[threadIdx.x >> 5];
  const bool on = idx < (int64_t)L * L * n_words;  // lanes past the last row only help with the queue
  if (!__any_sync(0xffffffffu, on)) return;
  const int r = on ? (int)(idx / n_words) : 0, word = on ? (int)(idx % n_words) : 0;
  const int y = r % L, z = r / L, X0 = (c + y + z) & 1;
  const int64_t wp = lat.wp;
  uint32_t* p0 = lat.words + (int64_t)r * L * wp + word;
  const uint32_t* pyp = lat.words + ((int64_t)(y == L - 1 ? 0 : y + 1) + (int64_t)L * z) * L * wp + word;
  const uint32_t* pym = lat.words + ((int64_t)(y == 0 ? L - 1 : y - 1) + (int64_t)L * z) * L * wp + word;
  const uint32_t* pzp = lat.words + (y + (int64_t)L * (z == L - 1 ? 0 : z + 1)) * L * wp + word;
  const uint32_t* pzm = lat.words + (y + (int64_t)L * (z == 0 ? L - 1 : z - 1)) * L * wp + word;
  const uint32_t g8 = 8u * ((uint32_t)(g.slot_base >> 5) + (uint32_t)word);
  const ThreadPhilox tp[2] = {thread_philox(g8, (uint32_t)q, a.k0, a.k1),
                              thread_philox(g8 + 1u, (uint32_t)q, a.k0, a.k1)};
  int head = 0, cnt = 0;  // the same in every lane of the warp
  auto finish = [&](bool have) {  // every lane calls it; `have` lanes finish one queued word each
    const LatticeDeferred d = dq[(head + lane) & 63];
    const int owner = have ? (int)(d.loc & 31u) : 0, xh = (int)(d.loc >> 5);
    const int ro = __shfl_sync(0xffffffffu, r, owner), wo = __shfl_sync(0xffffffffu, word, owner);
    const int xo = __shfl_sync(0xffffffffu, X0, owner);
    const uint32_t go = __shfl_sync(0xffffffffu, g8, owner);
    if (have) {
      const int n = ro * L + 2 * xh + xo;
      lat.words[(int64_t)n * wp + wo] ^=
          compare_rest(d.eq, d.u0, d.u1, (uint32_t)n, lat.recs[n], go, (uint32_t)q, a);
    }
  };
#pragma unroll 1
  for (int xh = 0; xh < H; ++xh) {
    const int x = 2 * xh + X0;
    uint32_t eq = 0;
    BondCount b{};
    if (on) {
      const int xp = x == L - 1 ? 0 : x + 1, xm = x == 0 ? L - 1 : x - 1;
      const SiteRec sr = lat.recs[r * L + x];
      const int64_t at = x * wp;
      const uint32_t s0 = p0[at];
      b = bond_count(s0, sr, p0[xp * wp], p0[xm * wp], pyp[at], pym[at], pzp[at], pzm[at], a);
      uint32_t lt;
      compare_planes8<FORM>(kM0 * ((uint32_t)(r * L + x) >> 1), sr, tp, b, a, lt, eq);
      p0[at] = s0 ^ (lt | b.always);
    }
    const unsigned dm = __ballot_sync(0xffffffffu, eq != 0u);
    if (eq) dq[(head + cnt + __popc(dm & below)) & 63] = LatticeDeferred{(uint32_t)lane | (uint32_t)xh << 5, eq, b.u0, b.u1};
    cnt += __popc(dm);
    __syncwarp();
    if (cnt >= 32) {
      finish(true);
      __syncwarp();
      head = (head + 32) & 63;
      cnt -= 32;
    }
  }
  finish(lane < cnt);
}

// Unsatisfied forward bonds, added per replica into levels (zero before).  A block takes
// 32 words (a lane each, so that a site's words are one line) and kLevelRows rows for each
// of its warps, counts in bit planes, and adds its warps' counts in shared memory before
// one global addition per replica.  Bound by the latency of the words' loads from L2:
// with eight rows to a thread and a thread per word (216 blocks at L = 24, R = 2e4) it
// took 125 us per step; a run of ten steps 15.0 -> 14.4 ms.
constexpr int kLevelRows = 2;

__global__ void __launch_bounds__(kThreads) k_lattice_levels(const __grid_constant__ LatticeArgs a) {
  constexpr int CB = 9;  // 3 * 64 * kLevelRows = 384 bonds at most
  __shared__ int sums[32 * 32];  // [word][replica]
  const RunGeom& g = a.g;
  const int L = g.L, R = a.P.rec[a.t].R_tilde, n_words = (R + 31) / 32;
  const int w0 = 32 * blockIdx.x, lane = threadIdx.x & 31, word = w0 + lane;
  if (w0 >= n_words) return;
  const Lattice lat = lattice_of(g, a.P, 1 - a.cur);
  const int64_t wp = lat.wp;
  for (int i = threadIdx.x; i < 32 * 32; i += kThreads) sums[i] = 0;
  __syncthreads();
  uint32_t c[CB];
#pragma unroll
  for (int i = 0; i < CB; ++i) c[i] = 0;
  const int row0 = (blockIdx.y * kWarps + (threadIdx.x >> 5)) * kLevelRows;
  const int row1 = word < n_words ? min(row0 + kLevelRows, L * L) : row0;
  for (int r = row0; r < row1; ++r) {
    const int y = r % L, z = r / L;
    const uint32_t* p0 = lat.words + (int64_t)r * L * wp + word;
    const uint32_t* pyp = lat.words + ((int64_t)(y == L - 1 ? 0 : y + 1) + (int64_t)L * z) * L * wp + word;
    const uint32_t* pzp = lat.words + (y + (int64_t)L * (z == L - 1 ? 0 : z + 1)) * L * wp + word;
    const uint32_t first = p0[0];
    uint32_t s = first;
#pragma unroll 4
    for (int x = 0; x < L; ++x) {
      const SiteRec sr = lat.recs[r * L + x];
      const uint32_t nx = x == L - 1 ? first : p0[(x + 1) * wp];
      const uint32_t e0 = s ^ nx ^ sr.jxp, e1 = s ^ pyp[x * wp] ^ sr.jyp, e2 = s ^ pzp[x * wp] ^ sr.jzp;
      const uint32_t sum = e0 ^ e1 ^ e2, two = majority(e0, e1, e2);  // e0 + e1 + e2 = sum + 2 two
      uint32_t carry = c[0] & sum;
      c[0] ^= sum;
      const uint32_t c1 = c[1] ^ two ^ carry;
      carry = majority(c[1], two, carry);
      c[1] = c1;
#pragma unroll
      for (int i = 2; i < CB; ++i) {
        const uint32_t ci = c[i] ^ carry;
        carry &= c[i];
        c[i] = ci;
      }
      s = nx;
    }
  }
#pragma unroll 1
  for (int bb = 0; bb < 32; ++bb) {
    const int b = (bb + lane) & 31;  // the lanes of a warp hit different banks
    int k = 0;
#pragma unroll
    for (int i = 0; i < CB; ++i) k |= (int)((c[i] >> b) & 1u) << i;
    if (k) atomicAdd(&sums[32 * lane + b], k);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 32 * 32; i += kThreads)
    if (32 * w0 + i < R) atomicAdd(&a.P.levels[32 * w0 + i], sums[i]);
}

__global__ void __launch_bounds__(kThreads) k_lattice_hist(const __grid_constant__ LatticeArgs a) {
  const int j = blockIdx.x * kThreads + threadIdx.x;
  if (j < a.P.rec[a.t].R_tilde) atomicAdd(&a.P.hist[(size_t)a.t * a.g.n_levels + a.P.levels[j]], 1u);
}

int lattice_step(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, int t, int n_sweeps,
                 const uint32_t met_thr[3], bool fresh, cudaStream_t st) {
  const int n_words = (int)((g.R_cap + 31) / 32);
  for (int p = 0; p < g.n_pop; ++p) {
    LatticeArgs a;
    fill_metropolis(a, pops[p].key_met, met_thr);
    a.g = g;
    a.P = pops[p];
    a.jtab = jtab;
    a.cur = cur;
    a.t = t;
    a.fresh = fresh ? 1 : 0;
    const dim3 tiles((n_words + kWarps - 1) / kWarps, (g.sw + 31) / 32);
    k_lattice_records<<<(g.N + kThreads - 1) / kThreads, kThreads, 0, st>>>(a);
    k_lattice_transpose<false><<<tiles, kThreads, 0, st>>>(a);
    const int64_t threads = (int64_t)g.L * g.L * n_words;
    const unsigned blocks = (unsigned)((threads + kThreads - 1) / kThreads);
    auto* sweep = a.form == 3   ? k_lattice_sweep<3>
                  : a.form == 2 ? k_lattice_sweep<2>
                  : a.form == 1 ? k_lattice_sweep<1>
                                : k_lattice_sweep<0>;
    for (int q = 0; q < 2 * n_sweeps; ++q) sweep<<<blocks, kThreads, 0, st>>>(a, q);
    int e = (int)cudaMemsetAsync(pops[p].levels, 0, sizeof(int32_t) * (size_t)g.R_cap, st);
    if (e) return e;
    const int rows = kWarps * kLevelRows;  // of a block
    k_lattice_levels<<<dim3((n_words + 31) / 32, (g.L * g.L + rows - 1) / rows), kThreads, 0, st>>>(a);
    k_lattice_hist<<<(g.R_cap + kThreads - 1) / kThreads, kThreads, 0, st>>>(a);
    k_lattice_transpose<true><<<tiles, kThreads, 0, st>>>(a);
    e = (int)cudaGetLastError();
    if (e) return e;
  }
  return 0;
}

}  // namespace

bool lattice_supported(int L) { return L >= 2 && L <= kMaxLGlobal && L % 2 == 0; }

int launch_sweep_global(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, int t, int n_sweeps,
                        const uint32_t met_thr[3], void* stream) {
  return lattice_step(g, pops, cur, jtab, t, n_sweeps, met_thr, false, (cudaStream_t)stream);
}

int launch_sweep_global_initial(const RunGeom& g, PopDev* pops, const uint32_t* jtab, void* stream) {
  const uint32_t none[3] = {0u, 0u, 0u};
  return lattice_step(g, pops, 1, jtab, 0, 0, none, true, (cudaStream_t)stream);
}

}  // namespace pa
