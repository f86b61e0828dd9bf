// pa_sweep_tile.cuh — the +-1 Metropolis sweep kernels (the dominant cost of a PA step),
// compiled per lattice size by the pa_sweep_l*.cu files.
//
// One CTA owns a tile of consecutive slots of the NEW population and all N sites
// of those replicas in shared memory.  It
//   1. gathers each slot's spins from its parent in the old population (the
//      replica copy of the resampling, §II, fused into the load),
//   2. runs S checkerboard Metropolis sweeps at beta_t in shared memory (colour
//      c = (x + y + z) & 1, colour 0 then colour 1; the neighbours of a site all
//      have the other colour, so all sites of one colour update independently),
//   3. counts each replica's energy and adds the tile to the histogram of step t,
//   4. writes the tile to the new population buffer,
//   5. (+-1 couplings) adds the families of its slots to the step's family
//      statistics (§III.A), so the step needs no family launch of its own.
// HBM traffic is one read and one write of the tile per step, whatever S is, at one
// bit per spin (pa_bits.cuh): a replica is a row of spin_words(N) words, and the
// gather and the store each transpose 32 x 32 bits in registers between 32 rows and
// 32 site words.
//
// +-1 couplings (k_sweep): bit-sliced tiles.  Word w of a site row holds slots
// tile0 + 32w + b as bit b (set for spin -1), so one 32-bit logic instruction
// tests a bond, adds a bit or takes a comparison step for 32 replicas.  Flipping
// s_n costs dE = 12 - 4u, u = unsatisfied bonds at n; u comes from the six
// bond bits by a tree of full adders as three bit planes.  u >= 3 (dE <= 0)
// always flips; otherwise the flip is taken when the replica's 32-bit uniform r
// is below thr(u) = floor(2^32 exp(-beta dE)).  r is the replica's bit column:
// bit 31 - p of r is bit b of word p mod 4 of Philox4x32-10 at counter
// (n >> 1, 2s + c, 8 (slot >> 5) + p / 4, t) keyed by (run_seed, Metropolis,
// population), so one block gives four bit planes of 32 replicas' uniforms.
// A replica is decided at the first plane, from the top, where its bit differs
// from its threshold's (accepted if the threshold has the 1): two planes on
// average.  Blocks 0 and 1 (planes 0..7) are always drawn and compared as one
// 8-bit bit-sliced subtraction (its borrow is "below", plus an "equal so far"
// mask); the words with replicas still equal draw further blocks on demand.
//
// Philox hoisting (same function, fewer multiplies): with counter words
// (h, q, g, t) = (site, half-sweep, group, step), the round-1 and round-2
// products depend either on the site and step only (tabulated once per launch
// in shared memory) or on the thread and half-sweep only (registers), so each
// block costs the 16 wide multiplies of rounds 3..10.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "pa_bits.cuh"
#include "pa_device.cuh"
#include "pa_family.cuh"
#include "pa_internal.h"
#include "pa_metropolis.cuh"

namespace pa {

struct SweepArgs : MetropolisArgs {
  PopDev pop;
  const uint32_t* jtab;  // [N][4] forward-bond masks (non-zero for J = -1)
  int32_t n_levels;
  int32_t t;
  int32_t cur;
  int32_t n_sweeps;
  int32_t slot_base;  // global slot of local slot 0 (Philox groups are global); 0 for a whole population
  int32_t fam;        // 1: add the tile's families to the step record (not for one rank's share)
  int32_t fresh;      // 1: step 0, every slot is its own parent
  // this launch's first local slot (tile 0 of the grid), and the split of a two-launch
  // sweep: slots below `split` in tiles of tj_main, the rest in tiles of tj_tail
  int32_t tile_base, split, tj_main, tj_tail;
  int32_t chained;  // 1: may start while the launch before it, another population's sweep, still runs (launch_tiles)
};

// Row k of a partition: rows of one parity class (y + z) & 1 = p, interleaved
// across the partitions of that class.
template <int L, int NP>
__device__ __forceinline__ int row_index(int part, int k, int p) {
  constexpr int H = L / 2, PC = NP / 2;
  const int i = (part % PC) + k * PC;  // index within the class
  const int z = i / H;
  const int y = 2 * (i % H) + ((p + z) & 1);
  return y + L * z;
}

// Per partition and row (rows of the partition's parity class, row_index), the
// word offsets of the row and of its four neighbour rows in a tile of W words per
// site and the row's first site: {row, y+1, y-1, z+1, first site, z-1}.  A
// thread's rows never change, so each tile fills this once.
template <int L, int W, int NP>
__device__ __forceinline__ void fill_row_table(int* rowtab, int tid, int nthreads) {
  constexpr int RPP = L * L / NP;
  for (int e = tid; e < NP * RPP; e += nthreads) {
    const int pt = e / RPP, kr = e % RPP;
    const int r = row_index<L, NP>(pt, kr, pt / (NP / 2));
    const int y = r % L, z = r / L;
    const int yp = y == L - 1 ? 0 : y + 1, ym = y == 0 ? L - 1 : y - 1;
    const int zp = z == L - 1 ? 0 : z + 1, zm = z == 0 ? L - 1 : z - 1;
    int* o = rowtab + 8 * e;
    o[0] = r * L * W;
    o[1] = (yp + L * z) * L * W;
    o[2] = (ym + L * z) * L * W;
    o[3] = (y + L * zp) * L * W;
    o[4] = r * L;
    o[5] = (y + L * zm) * L * W;
  }
}

// ---- phases of a tile

// Site records (bond masks, site/step parts of Philox rounds 1-3); all
// `nthreads` threads of the CTA help.
template <int L>
__device__ __forceinline__ void init_tables(const SweepArgs& a, SiteRec* recs, int tid, int nthreads) {
  constexpr int N = L * L * L;
  for (int n = tid; n < N; n += nthreads) {
    recs[n] = site_record(L, n, a.jtab, (uint32_t)a.t, a);
  }
}

// The parent (old slot) of new slot j, -1 past R~.
__device__ __forceinline__ int parent_of(const SweepArgs& a, int j, int R_new) {
  return j < R_new ? (a.fresh ? j : a.pop.parents[j]) : -1;
}

// ---- +-1 couplings: the bit-sliced sweep

// Bits needed to hold 0..n.
constexpr int bits_for(int n) { return n < 2 ? 1 : 1 + bits_for(n / 2); }

// A word whose replicas the first two Philox blocks (bit planes 0..7) leave
// undecided: its site n and word (n | word << 16), the undecided replicas, and
// bits 0 and 1 of their unsatisfied-bond counts.
struct __align__(16) Deferred {
  uint32_t loc, eq, u0, u1;
};
constexpr int kQueueCap = 64;  // words a warp queues; it finishes 32 of them as soon as there are

template <int L, int W, int NT, int MB>
struct BitShape {
  static constexpr int LL = L, WW = W, THREADS = NT, CTAS = MB;
  static constexpr int N = L * L * L;
  static constexpr int ROWS = L * L;
  static constexpr int NP = NT / W;       // row partitions
  static constexpr int TJ = 32 * W;       // replicas per tile
  static constexpr int SLOTS = 33 * W;    // parents (padded by one per word), then level counts
  static constexpr int CB = bits_for(3 * L * (ROWS / NP));  // bit planes of a thread's level counter
  static constexpr size_t SMEM_TILE = (size_t)N * W * 4 + (size_t)N * sizeof(SiteRec) + (size_t)SLOTS * 4;
  static constexpr size_t SMEM_QUEUES = (size_t)(NT / 32) * kQueueCap * sizeof(Deferred);
  static constexpr int RPP = ROWS / NP;  // rows per partition
  static constexpr size_t SMEM_ROWS = (size_t)NP * RPP * 8 * sizeof(int);
  // Deferred comparisons need whole warps that each stay inside one parity class
  // (every lane of a warp then runs the same half-sweep code in step), and room
  // for the queues without fewer than MB CTAs per SM (228 KB per SM, 1 KB of it
  // reserved per CTA).
  static constexpr bool DEFER = NT % 32 == 0 && ((NP / 2) * W) % 32 == 0 &&
                                (size_t)MB * (SMEM_TILE + SMEM_QUEUES + SMEM_ROWS + 1024) <= 233472;
  static constexpr int NQ = DEFER ? NT / 32 : 0;  // one queue per warp
  static constexpr size_t SMEM = SMEM_TILE + (DEFER ? SMEM_QUEUES + SMEM_ROWS : 0);
  static constexpr size_t SLOT_TABLE = SMEM_TILE - (size_t)SLOTS * 4 + (DEFER ? SMEM_QUEUES : 0);  // its offset
  static_assert(NT % W == 0 && 32 % W == 0 && NT <= 1024, "threads must tile the words of a row");
  static_assert(L % 2 == 0 && L / 2 <= 8, "even L up to 16");
  static_assert(NP % 2 == 0 && (ROWS / 2) % (NP / 2) == 0, "row partitions must split each parity class");
  static_assert(1024 % TJ == 0, "a tile never crosses the 1024-slot pitch unit");
};

// One half-sweep of the rows of partition `part` (parity class p, colour sites at
// x = X0 mod 2).  spw points at this thread's word of site 0; tp[b] are the
// thread's hoisted Philox parts of block b for this half-sweep q; g8 = 8 x the
// thread's global word index (the group of block b is g8 + b).
template <int L, int W, int NP, int X0>
__device__ __forceinline__ void sweep_rows_bits(uint32_t* spw, const SiteRec* recs, int part, int p,
                                                const ThreadPhilox (&tp)[4], uint32_t q, uint32_t g8,
                                                const SweepArgs& a) {
  constexpr int H = L / 2, RPP = L * L / NP;
#pragma unroll 1
  for (int k = 0; k < RPP; ++k) {
    const int r = row_index<L, NP>(part, k, p);
    const int y = r % L, z = r / L;
    const int yp = y == L - 1 ? 0 : y + 1, ym = y == 0 ? L - 1 : y - 1;
    const int zp = z == L - 1 ? 0 : z + 1, zm = z == 0 ? L - 1 : z - 1;
    uint32_t* p0 = spw + (size_t)r * L * W;
    const uint32_t* pyp = spw + (size_t)(yp + L * z) * L * W;
    const uint32_t* pym = spw + (size_t)(ym + L * z) * L * W;
    const uint32_t* pzp = spw + (size_t)(y + L * zp) * L * W;
    const uint32_t* pzm = spw + (size_t)(y + L * zm) * L * W;
    const SiteRec* rr = recs + r * L;
    const uint32_t h0 = (uint32_t)(r * L) >> 1;
#pragma unroll 2  // two sites in flight: measured 3 % faster than one, as fast as all
    for (int xh = 0; xh < H; ++xh) {
      const int x = 2 * xh + X0;
      const int xp = x == L - 1 ? 0 : x + 1, xm = x == 0 ? L - 1 : x - 1;
      const SiteRec sr = rr[x];
      const uint32_t s0 = p0[x * W];
      // unsatisfied bonds (one bit per replica) and their count u in three planes
      const uint32_t b0 = s0 ^ p0[xp * W] ^ sr.jxp, b1 = s0 ^ p0[xm * W] ^ sr.jxm;
      const uint32_t b2 = s0 ^ pyp[x * W] ^ sr.jyp, b3 = s0 ^ pym[x * W] ^ sr.jym;
      const uint32_t b4 = s0 ^ pzp[x * W] ^ sr.jzp, b5 = s0 ^ pzm[x * W] ^ sr.jzm;
      const uint32_t sa = b0 ^ b1 ^ b2, ca = majority(b0, b1, b2);
      const uint32_t sb = b3 ^ b4 ^ b5, cb = majority(b3, b4, b5);
      const uint32_t u0 = sa ^ sb, k2 = sa & sb;
      const uint32_t u1 = ca ^ cb ^ k2, u2 = majority(ca, cb, k2);
      const uint32_t always = u2 | (u1 & u0);  // u >= 3: dE <= 0
      // replicas to compare: u = 0, 1, 2 (dE = 12, 8, 4) with thr(u) > 0
      uint32_t eq = ~always & threshold_bits(a.live, u0, u1);
      uint32_t acc = 0;
      const uint32_t uc = kM0 * (h0 + (uint32_t)xh);  // lo(M0 h), h = n >> 1
      {
        uint32_t w0[4], w1[4];
        philox_block(uc, sr, tp[0], a.k0, a.k1, w0);
        philox_block(uc, sr, tp[1], a.k0, a.k1, w1);
#pragma unroll
        for (int i = 0; i < 4; ++i) compare_plane(w0[i], u0, u1, a.tm[i], eq, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) compare_plane(w1[i], u0, u1, a.tm[4 + i], eq, acc);
      }
      if (eq) {
        uint32_t w[4];
        philox_block(uc, sr, tp[2], a.k0, a.k1, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) compare_plane(w[i], u0, u1, a.tm[8 + i], eq, acc);
      }
      if (eq) {
        uint32_t w[4];
        philox_block(uc, sr, tp[3], a.k0, a.k1, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) compare_plane(w[i], u0, u1, a.tm[12 + i], eq, acc);
      }
#pragma unroll 1
      for (int b = 4; b < 8 && eq; ++b) {  // rare: some replica matched its threshold for 16 bits
        const ThreadPhilox tb = thread_philox(g8 + (uint32_t)b, q, a.k0, a.k1);
        uint32_t w[4];
        philox_block(uc, sr, tb, a.k0, a.k1, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) compare_plane(w[i], u0, u1, a.tm[4 * b + i], eq, acc);
      }
      p0[x * W] = s0 ^ (acc | always);
    }
  }
}

// Finishes a deferred word: Philox blocks 2, 3, ... of its site and group until
// every queued replica is decided, then flips the accepted ones (the word's owner
// has already applied the flips decided in planes 0..7).  Any lane of the owner's
// warp may run it: the same-colour sites of a half-sweep are independent.
template <int W>
__device__ __forceinline__ void finish_deferred(uint32_t* sp, const SiteRec* recs, const Deferred d, uint32_t q,
                                                uint32_t gbase, const SweepArgs& a) {
  const int n = (int)(d.loc & 0xffffu), word = (int)(d.loc >> 16);
  sp[n * W + word] ^=
      compare_rest(d.eq, d.u0, d.u1, (uint32_t)n, recs[n], 8u * (gbase + (uint32_t)word), q, a);
}

// One half-sweep of the rows of partition `part`, as sweep_rows_bits, for shapes
// whose warps stay inside one parity class: a word still undecided after blocks
// 0 and 1 (about one in eight) goes to the warp's queue dq, and whenever 32 are
// queued the warp finishes them with all lanes (finish_deferred); the rest are
// finished at the end of the half-sweep.  The decisions are the same; only the
// lanes that take them change.  sp: the tile (word-major within a site row);
// gbase: the tile's first word index (Philox group 8 (gbase + word) + b); rowtab:
// per partition and row the word offsets of the row and its four neighbour rows
// and the row's first site (built once per tile: a thread's rows never change).
//
// The sites of a row are unrolled, so every column offset is a constant, and form one
// straight piece of code: the row's spins stay in registers, its new words are stored
// and its undecided words queued after the last site.  The multiplies of one site's
// Philox blocks (the FMA pipe, 32 wide products of 4 cycles each per warp) then run
// beside the logic of another's (the ALU pipe, 2 cycles per operation).
template <int L, int W, int NP, int X0, int FORM>
__device__ __forceinline__ void sweep_rows_bits_dq(uint32_t* sp, int word, const SiteRec* recs, int part, int p,
                                                   const ThreadPhilox (&tp)[2], uint32_t q, uint32_t gbase,
                                                   Deferred* dq, const int* rowtab, const SweepArgs& a) {
  constexpr int H = L / 2, RPP = L * L / NP;
  const int lane = (int)(threadIdx.x & 31u);
  const unsigned below = (1u << lane) - 1u;
  uint32_t* spw = sp + word;
  int head = 0, cnt = 0;  // the same in every lane of the warp
  auto push = [&](int n, uint32_t eq, const BondCount& c, unsigned dm) {
    if (eq) dq[(head + cnt + __popc(dm & below)) & (kQueueCap - 1)] =
        Deferred{(uint32_t)n | ((uint32_t)word << 16), eq, c.u0, c.u1};
    cnt += __popc(dm);
  };
  auto finish = [&]() {  // the 32 oldest, or all there are
    __syncwarp();
    if (lane < cnt) finish_deferred<W>(sp, recs, dq[(head + lane) & (kQueueCap - 1)], q, gbase, a);
    __syncwarp();
    const int done = min(cnt, 32);
    head = (head + done) & (kQueueCap - 1);
    cnt -= done;
  };
#pragma unroll 1
  for (int k = 0; k < RPP; ++k) {
    const int4 e0 = *reinterpret_cast<const int4*>(rowtab + 8 * (part * RPP + k));
    const int rL = rowtab[8 * (part * RPP + k) + 4];
    uint32_t* p0 = spw + e0.x;
    const uint32_t* pyp = spw + e0.y;
    const uint32_t* pym = spw + e0.z;
    const uint32_t* pzp = spw + e0.w;
    const uint32_t* pzm = spw + rowtab[8 * (part * RPP + k) + 5];
    const SiteRec* rr = recs + rL;
    const uint32_t h0 = (uint32_t)rL >> 1;
    uint32_t row[L];
#pragma unroll
    for (int x = 0; x < L; ++x) row[x] = p0[x * W];
    uint32_t eq[H];
    BondCount c[H];
#pragma unroll
    for (int xh = 0; xh < H; ++xh) {
      const int x = 2 * xh + X0;
      const int xp = x == L - 1 ? 0 : x + 1, xm = x == 0 ? L - 1 : x - 1;
      const SiteRec sr = rr[x];
      c[xh] = bond_count(row[x], sr, row[xp], row[xm], pyp[x * W], pym[x * W], pzp[x * W], pzm[x * W], a);
      uint32_t lt;
      compare_planes8<FORM>(kM0 * (h0 + (uint32_t)xh), sr, tp, c[xh], a, lt, eq[xh]);  // lo(M0 h), h = n >> 1
      row[x] ^= lt | c[xh].always;
    }
#pragma unroll
    for (int xh = 0; xh < H; ++xh) p0[(2 * xh + X0) * W] = row[2 * xh + X0];
    unsigned dm[H];
    int total = cnt;
#pragma unroll
    for (int xh = 0; xh < H; ++xh) {
      dm[xh] = __ballot_sync(0xffffffffu, eq[xh] != 0u);
      total += __popc(dm[xh]);
    }
    if (total <= kQueueCap) {
#pragma unroll
      for (int xh = 0; xh < H; ++xh) push(rL + 2 * xh + X0, eq[xh], c[xh], dm[xh]);
    } else {  // the row does not fit beside what is queued: room for each site's words first
#pragma unroll
      for (int xh = 0; xh < H; ++xh) {
        while (cnt > kQueueCap - 32) finish();
        push(rL + 2 * xh + X0, eq[xh], c[xh], dm[xh]);
      }
    }
    while (cnt >= 32) finish();
  }
  finish();
}

// How a shape moves its tile between the rows of its slots and its site-major words.
// A thread transposes the 32 x 32 BW bits of 32 slots (a word column of the tile) and
// BW words of their rows; BW = 2 where 64 words fit the registers.
//
// STAGED: the rows of the whole tile lie in shared memory in between, in place of the
// tile's words (every thread holds its bits in registers while the layout changes, so
// one pass must take the tile, and the rows must fit before the slot table).  The rows
// then come in by 16-byte asynchronous copies, all in flight at once, and go out as
// one bulk copy of contiguous memory.  Otherwise each thread reads and writes its
// pieces of 4 BW bytes in global memory.  At L = 10 (1024 slots, 128 KB) the pieces
// took 10.5 us to gather and 11 to 21 us to store.
// S: the tile's shape (lattice size LL, WW words per site, THREADS, CTAS per SM, and the
// bytes from the tile's words to its slot table).
template <typename S>
struct RowMove : Row<S::LL> {
  using Row<S::LL>::N;
  using Row<S::LL>::SW;
  using Row<S::LL>::NB;
  static constexpr int W = S::WW, NT = S::THREADS, MB = S::CTAS;
  static constexpr int BW = SW % 2 == 0 && NT * MB <= 640 ? 2 : 1;
  static constexpr int GATHER_UNITS = W * ((NB + BW - 1) / BW);
  static constexpr int STORE_UNITS = W * (SW / BW);  // the padding of a row too: its bits stay 0
  static constexpr int ROW_WORDS = 32 * W * SW;
  static constexpr bool STAGED = STORE_UNITS <= NT && (size_t)ROW_WORDS * 4 <= S::SLOT_TABLE;
  // Shared memory of the measurements after the store (level counts of the tile, then
  // the families): behind the rows while they are copied out, or in their place.
  static constexpr int LEVELS = 3 * N + 1;
  static constexpr int FAM_WORDS = ((32 * W + 1 + W + 2) & ~1) + 128;
  static constexpr int POST_WORDS = LEVELS > FAM_WORDS ? LEVELS : FAM_WORDS;
  static constexpr bool POST_BEHIND = STAGED && (size_t)(ROW_WORDS + POST_WORDS) * 4 <= S::SLOT_TABLE;
  static constexpr int POST = POST_BEHIND ? ROW_WORDS : 0;
};

// The unit's word column and first row word.  Neighbouring lanes take neighbouring
// word columns, and (STAGED) row words one step apart, which spreads both the rows and
// the words over the banks.
template <typename M, int UNITS>
__device__ __forceinline__ void move_unit(int u, int& word, int& blk) {
  constexpr int W = M::W, NBLK = UNITS / W;
  word = u % W;
  blk = (M::STAGED ? (u / W + word) % NBLK : u / W) * M::BW;
}

template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src, bool zero) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES),
               "r"(zero ? 0 : BYTES)
               : "memory");
}

// Gather the tile's spins from the parents of its slots into bit words; spar
// holds the tile's parents (-1 past R~), slot i at index 33 (i >> 5) + (i & 31).
// Ends with the words written but not yet synchronised; the site records may be
// written from then on, not before (STAGED).
template <typename S>
__device__ __forceinline__ void gather_bits(const SweepArgs& a, uint32_t* sp, const int* spar) {
  using M = RowMove<S>;
  constexpr int W = M::W, NT = M::NT;
  const uint32_t* src = a.pop.spins[a.cur];
  if constexpr (M::STAGED) {
    constexpr int CW = M::SW % 4 == 0 ? 4 : M::SW;  // words per copy
    constexpr int CPR = M::SW / CW;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sp);
    for (int e = threadIdx.x; e < 32 * W * CPR; e += NT) {
      const int r = e / CPR, o = e % CPR * CW;
      const int p = spar[33 * (r >> 5) + (r & 31)];
      copy_async<4 * CW>(base + 4u * (uint32_t)(r * M::SW + o), src + (size_t)(p >= 0 ? p : 0) * M::SW + o, p < 0);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }
  for (int u0 = 0; u0 < M::GATHER_UNITS; u0 += NT) {  // one pass when STAGED
    const int u = u0 + threadIdx.x;
    const bool on = u < M::GATHER_UNITS;
    uint32_t m[M::BW][32];
    int word = 0, blk = 0;
    if (on) {
      move_unit<M, M::GATHER_UNITS>(u, word, blk);
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const int p = M::STAGED ? 32 * word + i : spar[33 * word + i];
        const uint32_t* row = (M::STAGED ? sp : src) + (size_t)(p >= 0 ? p : 0) * M::SW + blk;
        if constexpr (M::BW == 2) {
          const uint2 v = p >= 0 ? *reinterpret_cast<const uint2*>(row) : make_uint2(0u, 0u);
          m[0][i] = v.x;
          m[1][i] = v.y;
        } else {
          m[0][i] = p >= 0 ? *row : 0u;
        }
      }
#pragma unroll
      for (int h = 0; h < M::BW; ++h) transpose32(m[h]);
    }
    if (M::STAGED) __syncthreads();
    if (on) {
#pragma unroll
      for (int h = 0; h < M::BW; ++h)
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int n = 32 * (blk + h) + i;
          if (M::N % (32 * M::BW) == 0 || n < M::N) sp[n * W + word] = m[h][i];
        }
    }
  }
}

// a + b + c = (the new a) + 2 (the result), bitwise.
__device__ __forceinline__ uint32_t add3(uint32_t& a, uint32_t b, uint32_t c) {
  const uint32_t carry = majority(a, b, c);
  a = a ^ b ^ c;
  return carry;
}

// Unsatisfied forward bonds of every replica of the tile, counted per thread in
// CB bit planes and then added per replica into ecnt (slot i at index i).  Two sites
// enter the planes together by full adders, so that the carries run through the upper
// planes once per pair: 14 operations per site and word where a carry chain per site
// takes 22.  The planes of four replicas are then read a byte each at a time (CB <= 8).
template <int L, int W, int NP, int CB>
__device__ __forceinline__ void count_levels_bits(const uint32_t* sp, const SiteRec* recs, int* ecnt, int word,
                                                  int part) {
  constexpr int ROWS = L * L;
  uint32_t c[CB > 3 ? CB : 4];
#pragma unroll
  for (int i = 0; i < (CB > 3 ? CB : 4); ++i) c[i] = 0;
  for (int r = part; r < ROWS; r += NP) {
    const int y = r % L, z = r / L;
    const int yp = y == L - 1 ? 0 : y + 1, zp = z == L - 1 ? 0 : z + 1;
    const uint32_t* p0 = sp + (size_t)r * L * W + word;
    const uint32_t* pyp = sp + (size_t)(yp + L * z) * L * W + word;
    const uint32_t* pzp = sp + (size_t)(y + L * zp) * L * W + word;
    const SiteRec* rr = recs + r * L;
#pragma unroll
    for (int x = 0; x < L; x += 2) {
      uint32_t one[2], two[2];  // the three bonds of a site: one + 2 two
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int xx = x + h, xp = xx == L - 1 ? 0 : xx + 1;
        const uint32_t s0 = p0[xx * W];
        one[h] = s0 ^ p0[xp * W] ^ rr[xx].jxp;
        two[h] = add3(one[h], s0 ^ pyp[xx * W] ^ rr[xx].jyp, s0 ^ pzp[xx * W] ^ rr[xx].jzp);
      }
      const uint32_t t0 = add3(c[0], one[0], one[1]);
      const uint32_t f0 = add3(c[1], two[0], two[1]);
      const uint32_t f1 = c[1] & t0;
      c[1] ^= t0;
      uint32_t carry = add3(c[2], f0, f1);
#pragma unroll
      for (int i = 3; i < CB; ++i) {
        const uint32_t ci = c[i] ^ carry;
        carry &= c[i];
        c[i] = ci;
      }
    }
  }
  if constexpr (CB <= 8) {
#pragma unroll 1
    for (int mm = 0; mm < 8; ++mm) {
      const int m = (mm + word) & 7;  // replicas m, m + 8, m + 16, m + 24
      uint32_t k4 = 0;
#pragma unroll
      for (int i = 0; i < CB; ++i) k4 |= ((c[i] >> m) & 0x01010101u) << i;
#pragma unroll
      for (int bb = 0; bb < 4; ++bb) {
        const int b = (bb + (word >> 3)) & 3;  // lanes of a warp hit different banks
        atomicAdd(&ecnt[32 * word + m + 8 * b], (int)((k4 >> (8 * b)) & 0xffu));
      }
    }
  } else {
#pragma unroll 1
    for (int bb = 0; bb < 32; ++bb) {
      const int b = (bb + word) & 31;
      int k = 0;
#pragma unroll
      for (int i = 0; i < CB; ++i) k |= (int)((c[i] >> b) & 1u) << i;
      if (k) atomicAdd(&ecnt[32 * word + b], k);
    }
  }
}

// Levels of the tile's slots (ecnt), and their histogram added to the step's: the tile
// is counted in shared memory first (hist, LEVELS words), lanes of a warp with the same
// level by one addition, so that the step's histogram gets one global addition per
// tile and occupied level.  With one per slot the tiles of a wave queued up at the few
// levels a population occupies: 2.5 to 23 us per tile at L = 10, and at L = 4, beta = 3
// (a handful of levels) 0.68 of a step's 0.73 ms at R = 1e6.
template <int TJ, int NT, int LEVELS>
__device__ __forceinline__ void publish_levels(const SweepArgs& a, const int* ecnt, int* hist, int tile0, int R_new) {
  const int tid = threadIdx.x;
  for (int k = tid; k < LEVELS; k += NT) hist[k] = 0;
  __syncthreads();
  const unsigned mask = warp_lanes(tid, NT);
  for (int base = 0; base < TJ; base += NT) {  // the same iterations in every lane of a warp
    const int i = base + tid, j = tile0 + i;
    const bool on = i < TJ && j < R_new;
    const int k = on ? ecnt[i] : -1;
    const unsigned peers = __match_any_sync(mask, k);
    if (on) {
      a.pop.levels[j] = k;
      if ((tid & 31) == __ffs(peers) - 1) atomicAdd(&hist[k], __popc(peers));
    }
  }
  __syncthreads();
  uint32_t* out = a.pop.hist + (size_t)a.t * a.n_levels;
  for (int k = tid; k < LEVELS; k += NT)
    if (hist[k]) atomicAdd(&out[k], (uint32_t)hist[k]);
}

// Write the tile back to the rows of its slots, the gather's split reversed.  STAGED:
// thread 0 has issued the bulk copy of the rows [0, ROW_WORDS) of shared memory when
// this returns (store_done waits for it); the caller synchronises either way.
template <typename S>
__device__ __forceinline__ void store_bits(const SweepArgs& a, uint32_t* sp, int tile0) {
  using M = RowMove<S>;
  constexpr int W = M::W, NT = M::NT;
  uint32_t* dst = a.pop.spins[1 - a.cur] + (size_t)tile0 * M::SW;
  for (int u0 = 0; u0 < M::STORE_UNITS; u0 += NT) {  // one pass when STAGED
    const int u = u0 + threadIdx.x;
    const bool on = u < M::STORE_UNITS;
    uint32_t m[M::BW][32];
    int word = 0, blk = 0;
    if (on) {
      move_unit<M, M::STORE_UNITS>(u, word, blk);
#pragma unroll
      for (int h = 0; h < M::BW; ++h) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const int n = 32 * (blk + h) + i;
          m[h][i] = n < M::N ? sp[n * W + word] : 0u;
        }
        transpose32(m[h]);
      }
    }
    if (M::STAGED) __syncthreads();
    if (on) {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        uint32_t* row = (M::STAGED ? sp : dst) + (size_t)(32 * word + i) * M::SW + blk;
        if constexpr (M::BW == 2)
          *reinterpret_cast<uint2*>(row) = make_uint2(m[0][i], m[1][i]);
        else
          *row = m[0][i];
      }
    }
  }
  if constexpr (M::STAGED) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the rows before the copy reads them
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                   "r"((uint32_t)__cvta_generic_to_shared(sp)), "r"(4 * M::ROW_WORDS)
                   : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      if (!M::POST_BEHIND) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
  }
}

// The bulk copy of store_bits is complete (the thread that issued it waits).
template <typename M>
__device__ __forceinline__ void store_done() {
  if (M::STAGED && threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Families (a7) of the tile's new slots, so that a step needs no family launch
// of its own: a family is a run of equal labels along the slots (labels ascend).
// sh (shared memory, free by now) holds labs[0..TJ] (the slot before the tile,
// then the tile's slots; -1 past R~), a bit mask per 32 slots of the slots that
// start a run, and 64 words for the final sum.  The thread at a run's first slot
// takes its end from the next start in the tile, or, for the tile's last run, by
// galloping through the labels after the tile (run_end), and records the family
// (pa_family.cuh); the last tile to finish adds the entropy.
template <int TJ, int NT>
__device__ __forceinline__ void tile_families(const SweepArgs& a, int* sh, int tile0, int R_new, int tid) {
  constexpr int NC = TJ / 32;  // chunks of 32 slots (TJ <= 1024)
  static_assert(NT % 32 == 0 || TJ <= NT, "the lanes of a warp take whole chunks");
  int* labs = sh;
  unsigned* bm = reinterpret_cast<unsigned*>(sh + TJ + 1);  // [NC + 1]: start bits per chunk, then chunks with starts
  long long* red = reinterpret_cast<long long*>(sh + ((TJ + 1 + NC + 2) & ~1));
  const int32_t* lab = a.pop.labels[1 - a.cur];
  const unsigned mask = warp_lanes(tid, NT);
  for (int i = tid; i <= TJ; i += NT) {
    const int j = tile0 - 1 + i;
    labs[i] = (j >= 0 && j < R_new) ? lab[j] : -1;
  }
  __syncthreads();
  // run starts, one ballot per chunk (lanes of a warp take consecutive slots)
  for (int base = 0; base < TJ; base += NT) {
    const int i = base + tid;
    const bool start = i < TJ && labs[i + 1] != labs[i];
    const unsigned b = __ballot_sync(mask, start);
    if ((i & 31) == 0 && i < TJ) bm[i >> 5] = b;
  }
  __syncthreads();
  if (tid < 32) {  // chunks that hold a run start
    const unsigned nzb = __ballot_sync(0xffffffffu, tid < NC && bm[tid] != 0u);
    if (tid == 0) bm[NC] = nzb;
  }
  __syncthreads();
  const unsigned nz = bm[NC];
  FamilyAcc f;
  for (int base = 0; base < TJ; base += NT) {  // the same iterations in every lane of a warp
    const int i = base + tid, j = tile0 + i, c = i >> 5, l = i & 31;
    int eta = 0;
    if (i < TJ && j < R_new && (bm[c] >> l & 1u)) {
      const unsigned above = l == 31 ? 0u : bm[c] & (~0u << (l + 1));
      const unsigned later = c == 31 ? 0u : nz & (~0u << (c + 1));
      int end;
      if (above) {
        end = tile0 + 32 * c + __ffs(above) - 1;
      } else if (later) {
        const int c2 = __ffs(later) - 1;
        end = tile0 + 32 * c2 + __ffs(bm[c2]) - 1;
      } else {
        end = run_end(lab, labs[i + 1], tile0 + TJ, R_new);
      }
      eta = end - j;
      f.add(eta);
    }
    family_size(a.pop, eta, mask);
  }
  family_flush(f, mask, &a.pop.rec[a.t]);
  // the tiles of both launches that hold slots take part
  const int in_main = min(R_new, a.split);
  const int participants = (in_main + a.tj_main - 1) / a.tj_main +
                           (R_new > a.split ? (R_new - a.split + a.tj_tail - 1) / a.tj_tail : 0);
  family_entropy_last(a.pop, &a.pop.rec[a.t], R_new, participants, tid, NT, red);
}

template <int F>
struct Form {
  static constexpr int value = F;
};

// One tile of the bit-sliced sweep (+-1 couplings): the slots tile0 .. tile0 + TJ - 1
// of the new population (R_new slots), in the dynamic shared memory sm.
template <int L, int W, int NT, int MB>
__device__ __forceinline__ void sweep_tile(const SweepArgs& a, uint32_t* sm, int tile0, int R_new) {
  using S = BitShape<L, W, NT, MB>;
  constexpr int N = S::N, NP = S::NP, TJ = S::TJ;
  uint32_t* sp = sm;                                               // spins [N][W]
  SiteRec* recs = reinterpret_cast<SiteRec*>(sm + (size_t)N * W);  // [N]
  Deferred* queues = reinterpret_cast<Deferred*>(recs + N);        // [NQ][kQueueCap]
  int* slots = reinterpret_cast<int*>(queues + S::NQ * kQueueCap);  // [33 W]: parents, then level counts
  int* rowtab = slots + S::SLOTS;  // [NP][RPP][8]: word offsets of a row and its four neighbour rows, its first site
  const int tid = threadIdx.x, word = tid % W, part = tid / W;
  Deferred* dq = queues + (S::DEFER ? (tid >> 5) * kQueueCap : 0);
  using M = RowMove<S>;
  if constexpr (S::DEFER) fill_row_table<L, W, NP>(rowtab, tid, NT);
  for (int i = tid; i < TJ; i += NT) slots[33 * (i >> 5) + (i & 31)] = parent_of(a, tile0 + i, R_new);
  __syncthreads();
  gather_bits<S>(a, sp, slots);
  init_tables<L>(a, recs, tid, NT);
  __syncthreads();
  for (int i = tid; i < S::SLOTS; i += NT) slots[i] = 0;
  __syncthreads();

  // sweeps: partition `part` owns rows of parity class p = (y + z) & 1; in
  // half-sweep c its colour sites sit at x = p ^ c mod 2 in every row.
  const uint32_t gbase = (uint32_t)((a.slot_base + tile0) >> 5);  // global index of the tile's first word
  const uint32_t g8 = 8u * (gbase + (uint32_t)word);             // Philox group of block 0 of this word
  const int pclass = part / (NP / 2);
  if constexpr (S::DEFER) {
    auto sweeps = [&](auto form) {
      constexpr int FORM = decltype(form)::value;
      for (uint32_t q = 0; q < 2u * (uint32_t)a.n_sweeps; ++q) {
        const ThreadPhilox tp[2] = {thread_philox(g8, q, a.k0, a.k1), thread_philox(g8 + 1u, q, a.k0, a.k1)};
        if ((pclass ^ (int)(q & 1u)) == 0)  // the same in every lane of the warp
          sweep_rows_bits_dq<L, W, NP, 0, FORM>(sp, word, recs, part, pclass, tp, q, gbase, dq, rowtab, a);
        else
          sweep_rows_bits_dq<L, W, NP, 1, FORM>(sp, word, recs, part, pclass, tp, q, gbase, dq, rowtab, a);
        __syncthreads();
      }
    };
    switch (a.form) {  // the same in every thread: the step's thresholds decide
      case 3: sweeps(Form<3>{}); break;
      case 2: sweeps(Form<2>{}); break;
      case 1: sweeps(Form<1>{}); break;
      default: sweeps(Form<0>{}); break;
    }
  } else {
    uint32_t* spw = sp + word;
#pragma unroll 1
    for (uint32_t q = 0; q < 2u * (uint32_t)a.n_sweeps; ++q) {
      const ThreadPhilox tp[4] = {thread_philox(g8, q, a.k0, a.k1), thread_philox(g8 + 1u, q, a.k0, a.k1),
                                  thread_philox(g8 + 2u, q, a.k0, a.k1), thread_philox(g8 + 3u, q, a.k0, a.k1)};
      if ((pclass ^ (int)(q & 1u)) == 0)
        sweep_rows_bits<L, W, NP, 0>(spw, recs, part, pclass, tp, q, g8, a);
      else
        sweep_rows_bits<L, W, NP, 1>(spw, recs, part, pclass, tp, q, g8, a);
      __syncthreads();
    }
  }
  count_levels_bits<L, W, NP, S::CB>(sp, recs, slots, word, part);
  __syncthreads();
  store_bits<S>(a, sp, tile0);
  if (!M::POST_BEHIND) __syncthreads();  // the words (or their rows) are dead
  int* post = reinterpret_cast<int*>(sm) + M::POST;
  publish_levels<TJ, NT, M::LEVELS>(a, slots, post, tile0, R_new);
  if (a.fam) {
    __syncthreads();  // the level counts are dead
    tile_families<TJ, NT>(a, post, tile0, R_new, tid);
  }
  store_done<M>();
}

// The sweeps of a step's two populations are independent of each other, so the second's is
// launched over the end of the first's: its tiles fill the SMs that the first's last wave
// leaves idle.  A launch lets the next one begin once all of its own tiles have
// (launch_dependents), which also means that the step's resampling is done; and so that
// the step's later kernels, which follow the last launch, find both done, the CTA of a
// launch's last tile waits for the launch before (griddepcontrol.wait; all of that
// launch's CTAs are running or done by then).  Two populations of 1e5, L = 8: +-1 run of
// 201 temperatures 76.8 -> 71.0 ms, Gaussian of 61 71.8 -> 67.2 ms (391 tiles each, 1.29
// and 0.64 waves).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// n_tiles: this launch's tiles that hold slots.
__device__ __forceinline__ void wait_launch_before(int n_tiles) {
  if ((int)blockIdx.x == min(max(n_tiles, 1), (int)gridDim.x) - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launches a sweep kernel of args (SweepArgs a among them) as above.
template <typename K, typename Args>
inline int launch_tiles(K* kernel, unsigned n_blocks, int threads, size_t smem, const SweepArgs& a, const Args& args,
                        cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute overlap{};
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &overlap;
  cfg.numAttrs = a.chained ? 1u : 0u;
  return (int)cudaLaunchKernelEx(&cfg, kernel, args);
}

// Bit-sliced sweep kernel (+-1 couplings): one tile per CTA.
template <int L, int W, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_sweep(const __grid_constant__ SweepArgs a) {
  extern __shared__ __align__(16) uint32_t sm[];
  constexpr int TJ = BitShape<L, W, NT, MB>::TJ;
  launch_dependents();
  const int R_new = a.pop.rec[a.t].R_tilde;
  const int tile0 = a.tile_base + blockIdx.x * TJ;
  if (tile0 < R_new) sweep_tile<L, W, NT, MB>(a, sm, tile0, R_new);
  wait_launch_before((R_new - a.tile_base + TJ - 1) / TJ);
}

// The sweep arguments of population P at step t from buffer cur with thresholds
// thr (dE = 4, 8, 12), as launch_sweep sets them for a run of one launch.
__host__ __device__ inline void fill_sweep_args(SweepArgs& a, const PopDev& P, const uint32_t* jtab,
                                                int n_levels, int t, int cur, int n_sweeps, int tj,
                                                const uint32_t thr[3]) {
  a.pop = P;
  fill_metropolis(a, P.key_met, thr);
  a.jtab = jtab;
  a.n_levels = n_levels;
  a.t = t;
  a.cur = cur;
  a.n_sweeps = n_sweeps;
  a.slot_base = 0;
  a.fam = 1;
  a.fresh = 0;
  a.tile_base = 0;
  a.split = 0x7fffffff;
  a.tj_main = tj;
  a.tj_tail = tj;
  a.chained = 0;
}

// The sweeps of a batch's units of one lattice size and launch shape: unit list[k]
// takes the CTAs off[k] .. off[k+1]-1, one tile each; each CTA builds its unit's
// arguments for the round's step in shared memory.
template <int L, int W, int NT, int MB>
__global__ void __launch_bounds__(NT, MB)
    k_sweep_group(const GroupUnit* __restrict__ units, const int32_t* __restrict__ list,
                  const int32_t* __restrict__ off, int n, const int32_t* __restrict__ round) {
  constexpr int TJ = BitShape<L, W, NT, MB>::TJ;
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ SweepArgs sa;
  __shared__ int hdr[3];  // unit, tile0, R_new (tile0 < 0: nothing to do)
  if (threadIdx.x == 0) {
    int lo = 0, hi = n - 1;
    const int b = (int)blockIdx.x;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (off[mid] <= b) lo = mid; else hi = mid - 1;
    }
    const GroupUnit& u = units[list[lo]];
    const int r = *round, t = u.t0 + 1 + r;
    const int tile0 = (b - off[lo]) * TJ;
    const int R_new = t <= u.last_t ? u.P.rec[t].R_tilde : 0;
    hdr[0] = list[lo];
    hdr[1] = tile0 < R_new ? tile0 : -1;
    hdr[2] = R_new;
    if (tile0 < R_new) {
      const GroupStep& st = u.steps[t];
      fill_sweep_args(sa, u.P, u.jtab, u.g.n_levels, t, u.cur0 ^ (r & 1), st.n_sweeps, TJ, st.thr);
    }
  }
  __syncthreads();
  if (hdr[1] < 0) return;
  sweep_tile<L, W, NT, MB>(sa, sm, hdr[1], hdr[2]);
}

template <int L, int W, int NT, int MB>
static int launch_group_t(const GroupUnit* units, const int32_t* list, const int32_t* off, int n, int n_blocks,
                          const int32_t* round, cudaStream_t s) {
  using S = BitShape<L, W, NT, MB>;
  static std::atomic<int> done[64];
  const cudaError_t e = smem_limit_once(k_sweep_group<L, W, NT, MB>, (int)S::SMEM, done);
  if (e != cudaSuccess) return (int)e;
  if (n_blocks <= 0) return 0;
  k_sweep_group<L, W, NT, MB><<<n_blocks, NT, S::SMEM, s>>>(units, list, off, n, round);
  return (int)cudaGetLastError();
}

template <int L, int W, int NT, int MB>
static int launch_t(const RunGeom& g, const SweepArgs& args, cudaStream_t s) {
  using S = BitShape<L, W, NT, MB>;
  static std::atomic<int> done[64];
  const cudaError_t e = smem_limit_once(k_sweep<L, W, NT, MB>, (int)S::SMEM, done);
  if (e != cudaSuccess) return (int)e;
  // tiles from tile_base up to the split (main launch) or to the capacity (tail launch)
  const int64_t end = args.tile_base < args.split ? std::min<int64_t>(args.split, g.R_cap) : g.R_cap;
  if (end <= args.tile_base) return 0;
  const unsigned grid = (unsigned)((end - args.tile_base + S::TJ - 1) / S::TJ);
  return launch_tiles(k_sweep<L, W, NT, MB>, grid, NT, S::SMEM, args, args, s);
}

// One launch shape of the +-1 sweep.
struct ShapeEntry {
  int L, W, NT, MB;
  size_t smem;
  int (*launch)(const RunGeom&, const SweepArgs&, cudaStream_t);
  int (*launch_group)(const GroupUnit*, const int32_t*, const int32_t*, int, int, const int32_t*, cudaStream_t);
};
#define PA_SHAPE(L, W, NT, MB) \
  {L, W, NT, MB, BitShape<L, W, NT, MB>::SMEM, &launch_t<L, W, NT, MB>, &launch_group_t<L, W, NT, MB>}

// The shapes of one lattice size, default first.
struct ShapeList {
  const ShapeEntry* e;
  int n;
};
ShapeList sweep_shapes_2();
ShapeList sweep_shapes_4();
ShapeList sweep_shapes_6();
ShapeList sweep_shapes_8();
ShapeList sweep_shapes_10();
ShapeList sweep_shapes_12();
ShapeList sweep_shapes_14();
ShapeList sweep_shapes_16();

}  // namespace pa
