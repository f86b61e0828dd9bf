// pa_sweep_gauss.cu — the Metropolis sweep kernel of the Gaussian-coupling model.
#include <cuda_runtime.h>

#include <algorithm>

#include "pa_sweep_tile.cuh"

namespace pa {

// Nibble tiles of the Gaussian kernel: 8 replicas per word.
template <int L, int W, int NT>
struct SweepShape {
  static constexpr int N = L * L * L;
  static constexpr int ROWS = L * L;
  static constexpr int NP = NT / W;  // row partitions
  static constexpr int TJ = 8 * W;   // replicas per tile
  static constexpr int RPP = ROWS / NP;  // rows per partition
  static constexpr size_t SMEM = (size_t)N * W * 4 + (size_t)N * sizeof(SiteRec) + (size_t)TJ * 4;
  static constexpr size_t SMEM_ROWS = (size_t)NP * RPP * 8 * sizeof(int);  // the row table
  static_assert(NT % W == 0, "threads must tile the words of a row");
  static_assert(32 % W == 0, "a warp must cover whole rows");
  static_assert(L % 2 == 0 && L / 2 <= 8, "even L up to 16");
  static_assert(NP % 2 == 0 && (ROWS / 2) % (NP / 2) == 0, "row partitions must split each parity class");
};

// Bits 0..7 of x -> bit 0 of nibbles 0..7, and back.
__device__ __forceinline__ uint32_t bits_to_nibbles(uint32_t x) {
  x &= 0xffu;
  x = (x | (x << 12)) & 0x000F000Fu;
  x = (x | (x << 6)) & 0x03030303u;
  return (x | (x << 3)) & 0x11111111u;
}
__device__ __forceinline__ uint32_t nibbles_to_bits(uint32_t x) {
  x &= 0x11111111u;
  x = (x | (x >> 3)) & 0x03030303u;
  x = (x | (x >> 6)) & 0x000F000Fu;
  return (x | (x >> 12)) & 0xffu;
}

// Gather the tile's spins from the parents of its slots (nibble-packed): 32 slots
// and 32 sites per thread, as gather_bits.
template <int L, int W, int NT>
__device__ __forceinline__ void gather_tile(const SweepArgs& a, uint32_t* sp, int tile0, int R_new) {
  constexpr int N = Row<L>::N, SW = Row<L>::SW, NB = Row<L>::NB, GW = W / 4;  // groups of 32 slots
  const uint32_t* src = a.pop.spins[a.cur];
  for (int u = threadIdx.x; u < GW * NB; u += NT) {
    const int gw = u % GW, blk = u / GW;
    uint32_t m[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int p = parent_of(a, tile0 + 32 * gw + i, R_new);
      m[i] = p >= 0 ? src[(size_t)p * SW + blk] : 0u;
    }
    transpose32(m);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int n = 32 * blk + i;
      if (N % 32 == 0 || n < N)
        *reinterpret_cast<uint4*>(sp + n * W + 4 * gw) =
            make_uint4(bits_to_nibbles(m[i]), bits_to_nibbles(m[i] >> 8), bits_to_nibbles(m[i] >> 16),
                       bits_to_nibbles(m[i] >> 24));
    }
  }
}

// Write the tile back to the rows of its slots, their padding included.
template <int L, int W, int NT>
__device__ __forceinline__ void store_tile(const SweepArgs& a, const uint32_t* sp, int tile0) {
  constexpr int N = Row<L>::N, SW = Row<L>::SW, GW = W / 4;
  uint32_t* dst = a.pop.spins[1 - a.cur];
  for (int u = threadIdx.x; u < GW * SW; u += NT) {
    const int gw = u % GW, blk = u / GW;
    uint32_t m[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int n = 32 * blk + i;
      const uint4 v = n < N ? *reinterpret_cast<const uint4*>(sp + n * W + 4 * gw)
                                           : make_uint4(0u, 0u, 0u, 0u);
      m[i] = nibbles_to_bits(v.x) | nibbles_to_bits(v.y) << 8 | nibbles_to_bits(v.z) << 16 | nibbles_to_bits(v.w) << 24;
    }
    transpose32(m);
#pragma unroll
    for (int i = 0; i < 32; ++i) dst[(size_t)(tile0 + 32 * gw + i) * SW + blk] = m[i];
  }
}

// ---- Gaussian couplings (§II.A): nibble tiles (eight replicas per word, four
// bits each: gather_tile, store_tile) and one Philox block per site for the eight
// replicas of a word, whose 16-bit halves are the upper halves of their 32-bit
// uniforms (sweep_rows_g).  The acceptance comes from a per-site table built on the
// host for the step's beta: for each of the 64 patterns of antiparallel neighbours
// (bit k: bond k, in the order x+1, x-1, y+1, y-1, z+1, z-1) the threshold of the
// flip, 0xFFFFFFFF when it costs dE <= 0 (always taken) and otherwise
// min(floor(2^32 exp(-beta dE)), 2^32 - 2); the flip is taken when the uniform is
// below it.  Energies are recounted from scratch after the sweeps:
// E = -sum J + 2 sum over antiparallel bonds of J (exact integers).

struct GSweepArgs {
  SweepArgs base;
  const uint32_t* gtab;   // [N][64] acceptance thresholds of this step
  const int32_t* Jq;      // [3N] fixed-point couplings of the forward bonds
  long long Jtot;         // sum of all couplings
};

// The Metropolis uniform U of a replica (Gaussian couplings): its upper 16 bits are
// half (slot & 1) of word (slot >> 1) & 3 of the Philox block at counter
// (h, q, slot >> 3, t) (one block per site for the eight replicas of a nibble word),
// its lower 16 bits the upper half of word slot & 3 at counter (h, q, (slot >> 2) | 2^31,
// t).  With u = the upper half in place, U < thr holds for sure when (u | 0xffff) <
// thr and fails for sure when u >= thr; only in between (probability 2^-16 per
// update) is the second word drawn (g_tie_word).
__device__ __noinline__ uint32_t g_tie_word(uint32_t h, uint32_t q, uint32_t slot, uint32_t t, uint32_t k0,
                                            uint32_t k1) {
  return word_of(philox4x32_10(make_uint4(h, q, (slot >> 2) | 0x80000000u, t), k0, k1), (int)(slot & 3u)) >> 16;
}

template <int L, int W, int NP, int X0>
__device__ __forceinline__ void sweep_rows_g(uint32_t* sp, const SiteRec* recs, int part, const int* rowtab,
                                             const ThreadPhilox& tp, const uint32_t* k0, const uint32_t* k1,
                                             const uint32_t* __restrict__ gtab, uint32_t slot0, uint32_t q,
                                             uint32_t t) {
  constexpr int H = L / 2, RPP = L * L / NP;
#pragma unroll 1
  for (int k = 0; k < RPP; ++k) {
    const int4 e0 = *reinterpret_cast<const int4*>(rowtab + 8 * (part * RPP + k));
    const int rL = rowtab[8 * (part * RPP + k) + 4];  // the row's first site
    uint32_t* p0 = sp + e0.x;
    const uint32_t* pyp = sp + e0.y;
    const uint32_t* pym = sp + e0.z;
    const uint32_t* pzp = sp + e0.w;
    const uint32_t* pzm = sp + rowtab[8 * (part * RPP + k) + 5];
    uint32_t row[L];
#pragma unroll
    for (int x = 0; x < L; ++x) row[x] = p0[x * W];
#pragma unroll
    for (int xh = 0; xh < H; ++xh) {
      const int x = 2 * xh + X0;
      const int xp = x == L - 1 ? 0 : x + 1;
      const int xm = x == 0 ? L - 1 : x - 1;
      const uint32_t h = (uint32_t)rL / 2u + (uint32_t)xh;
      uint32_t w4[4];
      philox_block(kM0 * h, recs[rL + x], tp, k0, k1, w4);
      const uint32_t s0 = row[x];
      const uint32_t P1 = (s0 ^ row[xp]) | ((s0 ^ row[xm]) << 1) | ((s0 ^ pyp[x * W]) << 2);
      const uint32_t P2 = (s0 ^ pym[x * W]) | ((s0 ^ pzp[x * W]) << 1) | ((s0 ^ pzm[x * W]) << 2);
      const uint32_t* tb = gtab + (size_t)(rL + x) * kGPatterns;
      // byte k of Qe (Qo) is the pattern of replica 2k (2k + 1): its P1 bits, then its P2 bits
      const uint32_t Qe = (P1 & 0x0F0F0F0Fu) | ((P2 & 0x0F0F0F0Fu) << 3);
      const uint32_t Qo = ((P1 >> 4) & 0x0F0F0F0Fu) | (((P2 >> 4) & 0x0F0F0F0Fu) << 3);
      uint32_t flip = 0, tie = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t b = __byte_perm((i & 1) ? Qo : Qe, 0u, 0x4440u + (uint32_t)(i >> 1));  // the replica's pattern
        const uint32_t thr = __ldg(tb + b);
        const uint32_t u = (i & 1) ? (w4[i >> 1] & 0xffff0000u) : (w4[i >> 1] << 16);
        // a flip with dE <= 0 (thr = 0xFFFFFFFF) passes here unless u = 0xFFFF0000,
        // which the tie path takes
        if ((u | 0xffffu) < thr) flip |= 1u << (4 * i);
        else if (u < thr) tie |= 1u << i;
      }
      while (tie) {  // rare: the lower 16 bits decide
        const int i = __ffs(tie) - 1;
        tie &= tie - 1;
        const uint32_t b = ((P1 >> (4 * i)) & 7u) | (((P2 >> (4 * i)) & 7u) << 3);
        const uint32_t u = (i & 1) ? (w4[i >> 1] & 0xffff0000u) : (w4[i >> 1] << 16);
        const uint32_t thr = __ldg(tb + b);
        if (thr == 0xFFFFFFFFu || (u | g_tie_word(h, q, slot0 + (uint32_t)i, t, k0[0], k1[0])) < thr)
          flip |= 1u << (4 * i);
      }
      p0[x * W] = s0 ^ flip;
    }
  }
}

// Antiparallel forward bonds of every replica of the tile weighted by J, summed into ecnt.
template <int L, int W, int NP>
__device__ __forceinline__ void count_energies_g(const uint32_t* sp, const int32_t* __restrict__ Jq, long long* ecnt,
                                                 int word, int part) {
  constexpr int ROWS = L * L;
  int acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // |sum| < 2^31 for every launch shape in use
  for (int r = part; r < ROWS; r += NP) {
    const int y = r % L, z = r / L;
    const int yp = y == L - 1 ? 0 : y + 1, zp = z == L - 1 ? 0 : z + 1;
    const uint32_t* p0 = sp + (size_t)r * L * W + word;
    const uint32_t* pyp = sp + (size_t)(yp + L * z) * L * W + word;
    const uint32_t* pzp = sp + (size_t)(y + L * zp) * L * W + word;
#pragma unroll
    for (int x = 0; x < L; ++x) {
      const int xp = x == L - 1 ? 0 : x + 1;
      const int n = r * L + x;
      const uint32_t s0 = p0[x * W];
      const uint32_t ax = s0 ^ p0[xp * W], ay = s0 ^ pyp[x * W], az = s0 ^ pzp[x * W];
      const int jx = __ldg(Jq + 3 * n), jy = __ldg(Jq + 3 * n + 1), jz = __ldg(Jq + 3 * n + 2);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        acc[i] += (jx & -(int)((ax >> (4 * i)) & 1u)) + (jy & -(int)((ay >> (4 * i)) & 1u)) +
                  (jz & -(int)((az >> (4 * i)) & 1u));
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    atomicAdd(reinterpret_cast<unsigned long long*>(&ecnt[8 * word + i]), (unsigned long long)(long long)acc[i]);
}

template <int L, int W, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_sweep_g(const __grid_constant__ GSweepArgs ga) {
  using S = SweepShape<L, W, NT>;
  constexpr int N = S::N, NP = S::NP, TJ = S::TJ;
  const SweepArgs& a = ga.base;
  extern __shared__ __align__(16) uint32_t sm[];
  uint32_t* sp = sm;
  SiteRec* recs = reinterpret_cast<SiteRec*>(sm + (size_t)N * W);
  long long* ecnt = reinterpret_cast<long long*>(recs + N);
  int* rowtab = reinterpret_cast<int*>(ecnt + TJ);  // [NP][RPP][8], as the +-1 kernel's
  const int R_new = a.pop.rec[a.t].R_tilde;
  const int tile0 = blockIdx.x * TJ;
  if (tile0 >= R_new) return;
  const int tid = threadIdx.x, word = tid % W, part = tid / W;
  init_tables<L>(a, recs, tid, NT);
  fill_row_table<L, W, NP>(rowtab, tid, NT);
  for (int i = tid; i < TJ; i += NT) ecnt[i] = 0;
  gather_tile<L, W, NT>(a, sp, tile0, R_new);
  __syncthreads();
  const uint32_t slot0 = (uint32_t)tile0 + 8u * (uint32_t)word;  // the word's first replica
  const uint32_t g = slot0 >> 3;                                     // Philox group of its eight replicas
  const int pclass = part / (NP / 2);
  uint32_t* spw = sp + word;
  for (int s = 0; s < a.n_sweeps; ++s) {
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const uint32_t q = 2u * (uint32_t)s + (uint32_t)c;
      const ThreadPhilox tp = thread_philox(g, q, a.k0, a.k1);
      if ((pclass ^ c) == 0)
        sweep_rows_g<L, W, NP, 0>(spw, recs, part, rowtab, tp, a.k0, a.k1, ga.gtab, slot0, q, (uint32_t)a.t);
      else
        sweep_rows_g<L, W, NP, 1>(spw, recs, part, rowtab, tp, a.k0, a.k1, ga.gtab, slot0, q, (uint32_t)a.t);
      __syncthreads();
    }
  }
  count_energies_g<L, W, NP>(sp, ga.Jq, ecnt, word, part);
  __syncthreads();
  for (int i = tid; i < TJ; i += NT) {
    const int j = tile0 + i;
    if (j < R_new) a.pop.E64[j] = -ga.Jtot + 2 * ecnt[i];
  }
  store_tile<L, W, NT>(a, sp, tile0);
}

template <int L, int W, int NT, int MB>
static int launch_g_t(const RunGeom& g, const GSweepArgs& args, cudaStream_t s) {
  using S = SweepShape<L, W, NT>;
  const size_t smem = S::SMEM + (size_t)S::TJ * 4 + S::SMEM_ROWS;  // energy counters are 8 bytes, not 4
  static std::atomic<int> done[64];
  const cudaError_t e = smem_limit_once(k_sweep_g<L, W, NT, MB>, (int)smem, done);
  if (e != cudaSuccess) return (int)e;
  dim3 grid((unsigned)((g.R_cap + S::TJ - 1) / S::TJ));
  k_sweep_g<L, W, NT, MB><<<grid, NT, smem, s>>>(args);
  return (int)cudaGetLastError();
}

static int g_sweep_launches(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, const int32_t* Jq,
                            long long Jtot, const uint32_t* gtab, int t, int n_sweeps, bool fresh, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
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
    ga.gtab = gtab;
    ga.Jq = Jq;
    ga.Jtot = Jtot;
    int e;
    switch (g.L) {  // one launch shape per L, compiled for one CTA per SM (no register spills)
      case 2: e = launch_g_t<2, 32, 128, 1>(g, ga, s); break;
      case 4: e = launch_g_t<4, 32, 256, 1>(g, ga, s); break;
      case 6: e = launch_g_t<6, 32, 384, 1>(g, ga, s); break;
      case 8: e = launch_g_t<8, 32, 512, 1>(g, ga, s); break;
      case 10: e = launch_g_t<10, 32, 640, 1>(g, ga, s); break;
      case 12: e = launch_g_t<12, 16, 576, 1>(g, ga, s); break;
      case 14: e = launch_g_t<14, 8, 784, 1>(g, ga, s); break;
      case 16: e = launch_g_t<16, 4, 512, 1>(g, ga, s); break;
      default: e = (int)cudaErrorInvalidValue;
    }
    if (e != 0) return e;
  }
  return 0;
}

int launch_g_sweep(const RunGeom& g, PopDev* pops, int cur, const uint32_t* jtab, const int32_t* Jq, long long Jtot,
                   const uint32_t* gtab, int t, int n_sweeps, void* stream) {
  return g_sweep_launches(g, pops, cur, jtab, Jq, Jtot, gtab, t, n_sweeps, false, stream);
}

int launch_g_sweep_initial(const RunGeom& g, PopDev* pops, const uint32_t* jtab, const int32_t* Jq, long long Jtot,
                           void* stream) {
  return g_sweep_launches(g, pops, 1, jtab, Jq, Jtot, nullptr, 0, 0, true, stream);
}

}  // namespace pa
