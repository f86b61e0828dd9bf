// pa_sweep_gauss.cu — the Metropolis sweep kernel of the Gaussian-coupling model
// (§II.A), in the tiles of the +-1 kernel (pa_sweep_tile.cuh): one bit per replica, 32
// replicas per word, N sites, rows staged through shared memory.
//
// The acceptance comes from a per-site table (k_g_site_tables) for the step's beta: for
// each of the 64 patterns of antiparallel neighbours (bit k: bond k, in the order x+1,
// x-1, y+1, y-1, z+1, z-1) the threshold of the flip, 0xFFFFFFFF when it costs dE <= 0
// (always taken) and otherwise min(floor(2^32 exp(-beta dE)), 2^32 - 2); the flip is
// taken when the replica's 32-bit uniform U is below it.  The upper 16 bits of U are half
// (slot & 1) of word (slot >> 1) & 3 of the Philox block at counter (h, q, slot >> 3, t),
// h = site >> 1, its lower 16 bits the upper half of word slot & 3 at counter (h, q,
// (slot >> 2) | 2^31, t).  With T the threshold's upper half and u that of U, u < T
// flips for sure and u > T stays for sure; only u = T (probability 2^-16) needs the
// lower halves (g_ties).
//
// A thread updates the 32 replicas of a word at one site:
//  - six XORs give the bond planes, an 8 x 8 transpose of every byte lane turns them into
//    the patterns of the 32 replicas, a byte each, already scaled to a table offset;
//  - a replica then takes a byte permute (the shared-memory address of its threshold:
//    table base and pattern), the load, and one subtraction with its borrow: with T in
//    the upper half and zeros below, U - T 2^16 borrows exactly when u < T, whatever lies
//    below u, and the borrow is shifted into the word of flips; the difference is below
//    2^16 exactly when u = T, so the least of eight differences tells whether any replica
//    of the block needs the lower halves.
// The tables (256 bytes per site, from L2) are copied to shared memory a site ahead.
// Energies are recounted afterwards, E = -sum J + 2 sum over antiparallel bonds of J
// (exact integers), by the same means: the six forward bonds of two neighbouring sites
// index a table of 64 sums.
//
// Bound: issue (some 15 instructions per update, about half of them on the ALU pipe).
// L = 10, R = 1e6: 6.2 ms per step of ten sweeps, where nibble tiles (eight replicas per
// word, the table read through 64-bit addresses, two compares and two predicated ORs per
// replica: 19.8 integer instructions per update) took 9.7, 1.5 of them outside the sweeps.
// The comparison as a difference of FP32 numbers (2^23 + u, its sign shifted into the
// flips, a product of eight differences to find u = T) took 6.6, a compare and a
// predicated addition 6.5.
#include <cuda_runtime.h>

#include <algorithm>

#include "pa_sweep_tile.cuh"

namespace pa {

namespace {

struct GSweepArgs {
  SweepArgs base;
  const uint32_t* gtab;  // [N][64] acceptance thresholds of this step
  const uint32_t* utab;  // [N][64] their upper halves, in place
  const int32_t* etab;   // [N / 2][64] sums of the forward couplings of sites 2 i, 2 i + 1 over a pattern
  long long Jtot;        // sum of all couplings
};

__global__ void __launch_bounds__(256) k_g_sweep_tables(int L, const uint32_t* __restrict__ gtab,
                                                        const int32_t* __restrict__ Jq, uint32_t* utab, int32_t* etab) {
  const int i = blockIdx.x * 256 + threadIdx.x, N = L * L * L;
  if (i < N * kGPatterns && gtab) utab[i] = gtab[i] & 0xFFFF0000u;
  if (i < N / 2 * kGPatterns) {
    const int n = 2 * (i / kGPatterns), b = i % kGPatterns;
    int sum = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if ((b >> k) & 1) sum += Jq[3 * n + k];  // couplings 3 n .. 3 n + 5: both sites' forward bonds
    etab[i] = sum;
  }
}

template <int L, int W, int NT, int MB>
struct GShape {
  static constexpr int LL = L, WW = W, THREADS = NT, CTAS = MB;
  static constexpr int N = L * L * L;
  static constexpr int ROWS = L * L;
  static constexpr int NP = NT / W;      // partitions of the colour sites
  static constexpr int TJ = 32 * W;      // replicas per tile
  // shared memory: two tables of 256 bytes per partition, the tile's words, the sites'
  // Philox parts, energies (low and high sums), the slot table, the row table
  static constexpr size_t TABLES = (size_t)NP * 512;
  static constexpr size_t SLOT_TABLE = (size_t)N * W * 4 + (size_t)N * 8 + (size_t)TJ * 8;  // from the words on
  static constexpr size_t SMEM = TABLES + SLOT_TABLE + (size_t)33 * W * 4 + (size_t)ROWS * 8 * sizeof(int) + 16;
  static_assert(NT % W == 0 && 32 % W == 0 && NT <= 1024, "threads must tile the words of a row");
  static_assert(NT % 32 == 0 && NP <= ROWS * (L / 2), "whole warps, and a site for every partition");
  static_assert(1024 % TJ == 0, "a tile never crosses the 1024-slot pitch unit");
  static_assert((long long)((N / 2 + NP - 1) / NP) * 2 * 3 * 5 * (1 << 20) < (1ll << 31),
                "a thread's energy sum fits 32 bits");
};

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// The W lanes of a partition copy one 256-byte table into their buffer.
template <int W>
__device__ __forceinline__ void fetch_table(uint32_t dst, const void* src, int word) {
  if constexpr (W == 32) {
    copy_async<8>(dst + 8u * (uint32_t)word, static_cast<const char*>(src) + 8 * word, false);
  } else {
#pragma unroll
    for (int i = 0; i < 16 / W; ++i) {
      const int o = 16 * (word + W * i);
      copy_async<16>(dst + (uint32_t)o, static_cast<const char*>(src) + o, false);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// The tables of a partition's sites, one ahead of use, in two buffers of 256 bytes.
// Every lane of the partition (mask) calls next() together: it starts the copy of table
// `ahead` (null: none) and returns with the one started before ready at `cur`.
template <int W>
struct TableStream {
  uint32_t cur;  // shared-memory address of the current table (256-byte aligned)
  unsigned mask;
  int word;
  __device__ __forceinline__ TableStream(uint32_t buffers, unsigned lanes, int w, const void* first)
      : cur(buffers + 256u), mask(lanes), word(w) {
    fetch_table<W>(buffers, first, word);
  }
  __device__ __forceinline__ void next(const void* ahead) {
    __syncwarp(mask);  // every lane is done with the buffer that the copy overwrites
    if (ahead) {
      fetch_table<W>(cur, ahead, word);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    cur ^= 256u;
    __syncwarp(mask);
  }
};

// Six planes of 32 replicas -> their patterns: byte a of p[m] is, times four, the
// pattern of replica 8 a + m (plane k in bit k of the pattern).
__device__ __forceinline__ void patterns(const uint32_t (&d)[6], uint32_t (&p)[8]) {
  p[0] = p[1] = 0u;
#pragma unroll
  for (int k = 0; k < 6; ++k) p[k + 2] = d[k];
#pragma unroll
  for (int j = 4; j >= 1; j >>= 1) {
    const uint32_t lo = j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int g = 0; g < 8; g += 2 * j)
#pragma unroll
      for (int k = g; k < g + j; ++k) {
        const uint32_t x = p[k], y = p[k + j];
        p[k] = (x & lo) | ((y << j) & ~lo);
        p[k + j] = ((x >> j) & lo) | (y & ~lo);
      }
  }
}

// Table address of byte a of a pattern word (base: a multiple of 256).
__device__ __forceinline__ uint32_t entry(uint32_t p, uint32_t base, int a) {
  return __byte_perm(p, base, 0x7650u | (uint32_t)a);
}

// The flips of the replicas whose u equals T in the blocks `blocks` (bit a: replicas
// 8 a .. 8 a + 7) of the word of slot slot0: decided by the lower halves.
__device__ __noinline__ uint32_t g_ties(uint32_t blocks, uint32_t d0, uint32_t d1, uint32_t d2, uint32_t d3,
                                        uint32_t d4, uint32_t d5, const uint32_t* thr_site, uint32_t h, uint32_t q,
                                        uint32_t slot0, uint32_t t, uint32_t k0, uint32_t k1) {
  uint32_t flip = 0;
  for (int r = 0; r < 32; ++r) {
    if (!((blocks >> (r >> 3)) & 1u)) continue;
    const uint32_t slot = slot0 + (uint32_t)r;
    const uint32_t b = ((d0 >> r) & 1u) | ((d1 >> r) & 1u) << 1 | ((d2 >> r) & 1u) << 2 | ((d3 >> r) & 1u) << 3 |
                       ((d4 >> r) & 1u) << 4 | ((d5 >> r) & 1u) << 5;
    const uint32_t thr = thr_site[b];
    const uint32_t w = word_of(philox4x32_10(make_uint4(h, q, slot >> 3, t), k0, k1), (int)(slot >> 1) & 3);
    const uint32_t u = (slot & 1u) ? w >> 16 : w & 0xffffu;
    if (u != thr >> 16) continue;
    const uint32_t lo =
        word_of(philox4x32_10(make_uint4(h, q, (slot >> 2) | 0x80000000u, t), k0, k1), (int)(slot & 3u)) >> 16;
    if (thr == 0xFFFFFFFFu || (u << 16 | lo) < thr) flip |= 1u << r;
  }
  return flip;
}

// Word offsets of row r and its neighbour rows in the tile, and its first site.
struct RowAt {
  int p0, pyp, pym, pzp, site, pzm, parity;
};
__device__ __forceinline__ RowAt row_at(const int* rowtab, int r) {
  const int4 e0 = *reinterpret_cast<const int4*>(rowtab + 8 * r), e1 = *reinterpret_cast<const int4*>(rowtab + 8 * r + 4);
  return {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z};
}

// One half-sweep of the colour sites of a partition: the i-th colour site of the tile is
// number i mod H of row i div H, and partition `part` takes i = part, part + NP, ..., so
// that any number of warps shares the sites evenly.  A site is about 480 instructions, so
// it is not unrolled: ten copies (75 KB) overran the instruction cache, and the warps
// spent four fifths of their time waiting for instructions.
template <int L, int W, int NP>
__device__ __forceinline__ void sweep_sites_g(uint32_t* sp, const uint2* phil, const int* rowtab, uint32_t buffers,
                                              unsigned lanes, int part, int word, const ThreadPhilox (&tp)[4],
                                              uint32_t q, uint32_t slot0, const GSweepArgs& ga) {
  constexpr int H = L / 2, SITES = L * L * H;
  const SweepArgs& a = ga.base;
  const int c = (int)(q & 1u);
  auto column = [&](const RowAt& r, int i) { return 2 * (i % H) + (r.parity ^ c); };
  RowAt r = row_at(rowtab, part / H);
  int x = column(r, part);
  TableStream<W> tab(buffers, lanes, word, ga.utab + (size_t)(r.site + x) * kGPatterns);
#pragma unroll 1
  for (int i = part; i < SITES; i += NP) {
    const int ia = min(i + NP, SITES - 1);
    const RowAt ra = row_at(rowtab, ia / H);
    const int xa = column(ra, ia);
    tab.next(i + NP < SITES ? ga.utab + (size_t)(ra.site + xa) * kGPatterns : nullptr);
    const int xp = x == L - 1 ? 0 : x + 1, xm = x == 0 ? L - 1 : x - 1;
    const int n = r.site + x;
    uint32_t* p0 = sp + r.p0;
    const uint32_t s0 = p0[x * W];
    const uint32_t d[6] = {s0 ^ p0[xp * W], s0 ^ p0[xm * W], s0 ^ sp[r.pyp + x * W],
                           s0 ^ sp[r.pym + x * W], s0 ^ sp[r.pzp + x * W], s0 ^ sp[r.pzm + x * W]};
    uint32_t pat[8];
    patterns(d, pat);
    const uint2 ph = phil[n];
    const uint32_t uc = kM0 * ((uint32_t)n >> 1);
    uint32_t flip = 0, tied = 0;
#pragma unroll
    for (int b = 3; b >= 0; --b) {  // replicas 8 b + 7 .. 8 b, so that the signs shift in from the top one
      uint32_t w[4];
      philox_block(uc, ph.x, ph.y, tp[b], a.k0, a.k1, w);
      uint32_t least = ~0u;
#pragma unroll
      for (int m = 7; m >= 0; --m) {
        const uint32_t u = (m & 1) ? w[m >> 1] : w[m >> 1] << 16;  // the 16 random bits in the upper half
        uint32_t diff, below;  // u - T and, if that is negative, -1
        asm("sub.cc.u32 %0, %2, %3;\n\tsubc.u32 %1, 0, 0;"
            : "=&r"(diff), "=r"(below)
            : "r"(u), "r"(lds_u32(entry(pat[m], tab.cur, b))));
        flip = 2u * flip - below;
        least = min(least, diff);
      }
      if (least < 0x10000u) tied |= 1u << b;
    }
    if (tied)
      flip |= g_ties(tied, d[0], d[1], d[2], d[3], d[4], d[5], ga.gtab + (size_t)n * kGPatterns, (uint32_t)n >> 1, q,
                     slot0, (uint32_t)a.t, a.k0[0], a.k1[0]);
    p0[x * W] = s0 ^ flip;
    r = ra;
    x = xa;
  }
}

// Antiparallel forward bonds of every replica of the tile weighted by J, two sites at a
// time, added per replica to elo and ehi (the sums' low 16 bits and the rest).
template <int L, int W, int NP>
__device__ __forceinline__ void count_energies_g(const uint32_t* sp, const int* rowtab, uint32_t buffers,
                                                 unsigned lanes, int part, int word,
                                                 const int32_t* __restrict__ etab, int* elo, int* ehi) {
  constexpr int H = L / 2, PAIRS = L * L * H;
  int acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = 0;
  TableStream<W> tab(buffers, lanes, word, etab + (size_t)part * kGPatterns);
#pragma unroll 1
  for (int i = part; i < PAIRS; i += NP) {  // the pair of sites 2 i, 2 i + 1
    tab.next(i + NP < PAIRS ? etab + (size_t)(i + NP) * kGPatterns : nullptr);
    const RowAt r = row_at(rowtab, i / H);
    const int x = 2 * (i % H), x2 = x + 2 < L ? x + 2 : 0;
    const uint32_t* p0 = sp + r.p0;
    const uint32_t s0 = p0[x * W], s1 = p0[(x + 1) * W];
    const uint32_t d[6] = {s0 ^ s1, s0 ^ sp[r.pyp + x * W], s0 ^ sp[r.pzp + x * W],
                           s1 ^ p0[x2 * W], s1 ^ sp[r.pyp + (x + 1) * W], s1 ^ sp[r.pzp + (x + 1) * W]};
    uint32_t pat[8];
    patterns(d, pat);
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int m = 0; m < 8; ++m) acc[8 * b + m] += (int)lds_u32(entry(pat[m], tab.cur, b));
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    atomicAdd(&elo[32 * word + i], acc[i] & 0xffff);
    atomicAdd(&ehi[32 * word + i], acc[i] >> 16);
  }
}

template <int L, int W, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_sweep_g(const __grid_constant__ GSweepArgs ga) {
  using S = GShape<L, W, NT, MB>;
  constexpr int N = S::N, NP = S::NP, TJ = S::TJ;
  const SweepArgs& a = ga.base;
  extern __shared__ __align__(1024) uint32_t smg[];
  launch_dependents();
  const int R_new = a.pop.rec[a.t].R_tilde;
  const int tile0 = blockIdx.x * TJ;
  if (tile0 >= R_new) {
    wait_launch_before((R_new + TJ - 1) / TJ);
    return;
  }
  uint32_t* sp = smg + S::TABLES / 4;
  uint2* phil = reinterpret_cast<uint2*>(sp + (size_t)N * W);
  int* elo = reinterpret_cast<int*>(phil + N);
  int* ehi = elo + TJ;
  int* slots = ehi + TJ;
  int* rowtab = reinterpret_cast<int*>((reinterpret_cast<uintptr_t>(slots + 33 * W) + 15) & ~(uintptr_t)15);
  const int tid = threadIdx.x, word = tid % W, part = tid / W;
  const unsigned lanes = (W == 32 ? 0xffffffffu : (1u << (W & 31)) - 1u) << ((tid & 31) / W * W);
  const uint32_t buffers = (uint32_t)__cvta_generic_to_shared(smg) + 512u * (uint32_t)part;
  for (int r = tid; r < S::ROWS; r += NT) {  // rows in site order
    const int y = r % L, z = r / L;
    const int yp = y == L - 1 ? 0 : y + 1, ym = y == 0 ? L - 1 : y - 1;
    const int zp = z == L - 1 ? 0 : z + 1, zm = z == 0 ? L - 1 : z - 1;
    int* o = rowtab + 8 * r;
    o[0] = r * L * W;
    o[1] = (yp + L * z) * L * W;
    o[2] = (ym + L * z) * L * W;
    o[3] = (y + L * zp) * L * W;
    o[4] = r * L;
    o[5] = (y + L * zm) * L * W;
    o[6] = (y + z) & 1;
    o[7] = 0;
  }
  for (int i = tid; i < TJ; i += NT) slots[33 * (i >> 5) + (i & 31)] = parent_of(a, tile0 + i, R_new);
  __syncthreads();
  gather_bits<S>(a, sp, slots);
  for (int n = tid; n < N; n += NT) phil[n] = site_philox((uint32_t)n, (uint32_t)a.t, a);
  for (int i = tid; i < 2 * TJ; i += NT) elo[i] = 0;
  __syncthreads();
  const uint32_t slot0 = (uint32_t)tile0 + 32u * (uint32_t)word;  // the word's first replica
#pragma unroll 1
  for (uint32_t q = 0; q < 2u * (uint32_t)a.n_sweeps; ++q) {
    ThreadPhilox tp[4];  // Philox groups of eight replicas
#pragma unroll
    for (int b = 0; b < 4; ++b) tp[b] = thread_philox((slot0 >> 3) + (uint32_t)b, q, a.k0, a.k1);
    sweep_sites_g<L, W, NP>(sp + word, phil, rowtab, buffers, lanes, part, word, tp, q, slot0, ga);
    __syncthreads();
  }
  count_energies_g<L, W, NP>(sp + word, rowtab, buffers, lanes, part, word, ga.etab, elo, ehi);
  __syncthreads();
  for (int i = tid; i < TJ; i += NT) {
    const int j = tile0 + i;
    if (j < R_new) a.pop.E64[j] = -ga.Jtot + 2 * ((long long)ehi[i] * 65536 + elo[i]);
  }
  __syncthreads();  // the energies are read before the rows take their place
  store_bits<S>(a, sp, tile0);
  store_done<RowMove<S>>();
  wait_launch_before((R_new + TJ - 1) / TJ);
}

template <int L, int W, int NT, int MB>
int launch_g_t(const RunGeom& g, const GSweepArgs& args, cudaStream_t s) {
  using S = GShape<L, W, NT, MB>;
  static std::atomic<int> done[64];
  const cudaError_t e = smem_limit_once(k_sweep_g<L, W, NT, MB>, (int)S::SMEM, done);
  if (e != cudaSuccess) return (int)e;
  const unsigned grid = (unsigned)((g.R_cap + S::TJ - 1) / S::TJ);
  return launch_tiles(k_sweep_g<L, W, NT, MB>, grid, NT, S::SMEM, args.base, args, s);
}

int g_sweep_launches(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, const int32_t* Jq, long long Jtot,
                     const uint32_t* gtab, int t, int n_sweeps, bool fresh, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  // the kernel's tables, behind the rows that the sweep of population 0 writes
  uint32_t* utab = reinterpret_cast<uint32_t*>(pops[0].spins[1 - cur] + (size_t)g.pitch * g.sw);
  int32_t* etab = reinterpret_cast<int32_t*>(utab + (size_t)g.N * kGPatterns);
  k_g_sweep_tables<<<(g.N * kGPatterns + 255) / 256, 256, 0, s>>>(g.L, gtab, Jq, utab, etab);
  for (int i = 0; i < g.n_pop; ++i) {
    GSweepArgs ga;
    SweepArgs& args = ga.base;
    args.pop = pops[i];
    const uint32_t none[3] = {0u, 0u, 0u};  // its thresholds are in gtab
    fill_metropolis(args, pops[i].key_met, none);
    args.jtab = jtab;
    args.n_levels = g.n_levels;
    args.t = t;
    args.cur = cur;
    args.n_sweeps = n_sweeps;
    args.slot_base = 0;
    args.fam = 0;
    args.fresh = fresh ? 1 : 0;
    args.tile_base = 0;
    args.split = 0x7fffffff;
    args.tj_main = args.tj_tail = 1;
    args.chained = i > 0 ? 1 : 0;
    ga.gtab = gtab;
    ga.utab = utab;
    ga.etab = etab;
    ga.Jtot = Jtot;
    int e;
    // One launch shape per L.  Tiles of 256 slots, four to an SM, leave the last wave of
    // tiles short: at L = 10, R = 1e6 6.2 ms against 6.5 for two of 512 and 7.2 for one of
    // 1024; the larger lattices take what fits beside the site's words.
    switch (g.L) {
      case 2: e = launch_g_t<2, 32, 128, 2>(g, ga, s); break;
      case 4: e = launch_g_t<4, 32, 256, 2>(g, ga, s); break;
      case 6: e = launch_g_t<6, 16, 128, 4>(g, ga, s); break;
      case 8: e = launch_g_t<8, 8, 128, 4>(g, ga, s); break;
      case 10: e = launch_g_t<10, 8, 128, 4>(g, ga, s); break;
      case 12: e = launch_g_t<12, 8, 256, 2>(g, ga, s); break;
      case 14: e = launch_g_t<14, 8, 512, 1>(g, ga, s); break;
      case 16: e = launch_g_t<16, 4, 512, 1>(g, ga, s); break;
      default: e = (int)cudaErrorInvalidValue;
    }
    if (e != 0) return e;
  }
  return 0;
}

}  // namespace

int launch_g_sweep(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, const int32_t* Jq, long long Jtot,
                   const uint32_t* gtab, int t, int n_sweeps, void* stream) {
  return g_sweep_launches(g, pops, cur, jtab, Jq, Jtot, gtab, t, n_sweeps, false, stream);
}

int launch_g_sweep_initial(const RunGeom& g, PopDev* pops, const uint32_t* jtab, const int32_t* Jq, long long Jtot,
                           void* stream) {
  return g_sweep_launches(g, pops, 1, jtab, Jq, Jtot, nullptr, 0, 0, true, stream);
}

}  // namespace pa
