// pa_metropolis.cuh — the bit-sliced Metropolis test of the +-1 sweeps (32 replicas
// per word) and the Philox blocks behind it, shared by the shared-memory sweep
// (pa_sweep_tile.cuh), its Gaussian counterpart (Philox only) and the sweep of large
// lattices in global memory (pa_sweep_global.cu).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace pa {

constexpr uint32_t kM0 = 0xD2511F53u;
constexpr uint32_t kM1 = 0xCD9E8D57u;

// Round keys of a population's Metropolis stream and the thresholds of a step.
struct MetropolisArgs {
  uint32_t k0[10];  // Metropolis round keys of this population
  uint32_t k1[10];
  // +-1: plane p's threshold bit as a function of the unsatisfied-bond count u
  // (bits u0, u1; u = 0, 1, 2): T(u) = bit 31 - p of thr(u) as an all-zero / all-one
  // word, stored as tm[p] = {T(0), T(0) ^ T(1), T(0) ^ T(2)}, so that the bit of a
  // replica is tm[p][0] ^ (u0 & tm[p][1]) ^ (u1 & tm[p][2]) (u >= 3 never compares)
  uint32_t tm[32][4];
  uint32_t live[4];    // +-1: the same form of "thr(u) > 0" (a replica with thr(u) = 0 never flips)
  // Leading zero bits of the thresholds, for the comparison's cheaper forms: `lead`
  // Philox blocks (four planes each) in which every threshold's bits are 0, and the
  // form of planes 0..7 (compare_planes8).
  int32_t lead, form;
};

// Sets them from the population's key and the thresholds of dE = 4, 8, 12.
__host__ __device__ inline void fill_metropolis(MetropolisArgs& a, const uint32_t key[2], const uint32_t thr[3]) {
  uint32_t k0 = key[0], k1 = key[1];
  for (int r = 0; r < 10; ++r) {
    a.k0[r] = k0;
    a.k1[r] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  const uint32_t thr_u[3] = {thr[2], thr[1], thr[0]};  // u = 0, 1, 2: dE = 12, 8, 4
  for (int p = 0; p < 32; ++p) {
    uint32_t T[3];
    for (int u = 0; u < 3; ++u) T[u] = ((thr_u[u] >> (31 - p)) & 1u) ? ~0u : 0u;
    a.tm[p][0] = T[0];
    a.tm[p][1] = T[0] ^ T[1];
    a.tm[p][2] = T[0] ^ T[2];
    a.tm[p][3] = 0u;
  }
  uint32_t live[3];
  for (int u = 0; u < 3; ++u) live[u] = thr_u[u] ? ~0u : 0u;
  a.live[0] = live[0];
  a.live[1] = live[0] ^ live[1];
  a.live[2] = live[0] ^ live[2];
  a.live[3] = 0u;
  int clz[2] = {0, 0};  // of thr(2) (dE = 4), the largest, and thr(1) (dE = 8)
  for (int i = 0; i < 2; ++i)
    while (clz[i] < 32 && !(thr[i] >> (31 - clz[i]) & 1u)) ++clz[i];
  a.lead = clz[0] / 4;
  a.form = clz[0] >= 8 ? 3 : clz[0] >= 4 && clz[1] >= 8 ? 2 : clz[0] >= 2 && clz[1] >= 4 ? 1 : 0;
}

// Per-site shared-memory record: the six bond masks of the site (all ones for
// J = -1), and the site/step-dependent parts of Philox rounds 2-3 for h = n >> 1
// (the third, lo(M0 h), is one multiply and is recomputed).
struct __align__(16) SiteRec {
  uint32_t jxp, jxm, jyp, jym;
  uint32_t jzp, jzm, ua, ub;
};

// 32 x 32 -> 64-bit product as one wide multiply (2.4 % faster sweep than the
// separate high and low products).
__device__ __forceinline__ void mulhilo(uint32_t m, uint32_t a, uint32_t& hi, uint32_t& lo) {
  uint64_t p;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(m));
  hi = (uint32_t)(p >> 32);
  lo = (uint32_t)p;
}

// The site/step part of Philox rounds 1-3: ua and ub of a SiteRec.
__device__ __forceinline__ uint2 site_philox(uint32_t n, uint32_t t, const MetropolisArgs& a) {
  uint32_t hi0, lo0, hi1, lo1;
  mulhilo(kM0, n >> 1, hi0, lo0);
  const uint32_t c1 = hi0 ^ t ^ a.k1[0];
  mulhilo(kM1, c1, hi1, lo1);
  return make_uint2(hi1 ^ a.k0[1], lo1 ^ a.k0[2]);
}

// The record of site n at step t; jtab: the forward-bond masks (non-zero for J = -1).
__device__ __forceinline__ SiteRec site_record(int L, int n, const uint32_t* __restrict__ jtab, uint32_t t,
                                               const MetropolisArgs& a) {
  const int x = n % L, y = (n / L) % L, z = n / (L * L);
  const int nxm = (x == 0 ? L - 1 : x - 1) + L * (y + L * z);
  const int nym = x + L * ((y == 0 ? L - 1 : y - 1) + L * z);
  const int nzm = x + L * (y + L * (z == 0 ? L - 1 : z - 1));
  SiteRec r;
  r.jxp = jtab[4 * n + 0] ? ~0u : 0u;
  r.jyp = jtab[4 * n + 1] ? ~0u : 0u;
  r.jzp = jtab[4 * n + 2] ? ~0u : 0u;
  r.jxm = jtab[4 * nxm + 0] ? ~0u : 0u;
  r.jym = jtab[4 * nym + 1] ? ~0u : 0u;
  r.jzm = jtab[4 * nzm + 2] ? ~0u : 0u;
  const uint2 u = site_philox((uint32_t)n, t, a);
  r.ua = u.x;
  r.ub = u.y;
  return r;
}

// Per-thread, per-half-sweep part of rounds 1-3 of one group g.
struct ThreadPhilox {
  uint32_t ta;   // lo(M1 g): XORed with the site's ua to give round-2 word 0
  uint32_t tb;   // hi(M0 A1) ^ k1_2: XORed with lo(M0 h) to give round-2 word 2
  uint32_t tdk;  // lo(M0 A1) ^ k1_3: round-3 word 2 is hi(M0 A2) ^ tdk
};

__device__ __forceinline__ ThreadPhilox thread_philox(uint32_t g, uint32_t q, const uint32_t* k0,
                                                      const uint32_t* k1) {
  uint32_t h1, l1;
  mulhilo(kM1, g, h1, l1);
  const uint32_t a1 = h1 ^ q ^ k0[0];
  uint32_t ha, la;
  mulhilo(kM0, a1, ha, la);
  ThreadPhilox tp;
  tp.ta = l1;
  tp.tb = ha ^ k1[1];
  tp.tdk = la ^ k1[2];
  return tp;
}

__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a ^ b)); }

// One Philox block (rounds 3..10 from the hoisted parts) of site h, uc = lo(M0 h),
// for the thread's group of block index b (its ThreadPhilox tp).
__device__ __forceinline__ void philox_block(uint32_t uc, uint32_t ua, uint32_t ub, const ThreadPhilox& tp,
                                             const uint32_t* k0, const uint32_t* k1, uint32_t (&w)[4]) {
  uint32_t hh, l, h2, l2;
  mulhilo(kM1, tp.tb ^ uc, hh, l);
  mulhilo(kM0, ua ^ tp.ta, h2, l2);
  w[0] = hh ^ ub;
  w[1] = l;
  w[2] = h2 ^ tp.tdk;
  w[3] = l2;
#pragma unroll
  for (int rr = 3; rr < 10; ++rr) {  // rounds 4..10 (key index rr)
    mulhilo(kM1, w[2], hh, l);
    mulhilo(kM0, w[0], h2, l2);
    const uint32_t n0 = hh ^ w[1] ^ k0[rr];
    const uint32_t n2 = h2 ^ w[3] ^ k1[rr];
    w[0] = n0;
    w[1] = l;
    w[2] = n2;
    w[3] = l2;
  }
}

__device__ __forceinline__ void philox_block(uint32_t uc, const SiteRec& sr, const ThreadPhilox& tp, const uint32_t* k0,
                                             const uint32_t* k1, uint32_t (&w)[4]) {
  philox_block(uc, sr.ua, sr.ub, tp, k0, k1, w);
}

// The plane's threshold bit of each replica of a word (MetropolisArgs::tm), from bits
// u0, u1 of its unsatisfied-bond count.
__device__ __forceinline__ uint32_t threshold_bits(const uint32_t* tm, uint32_t u0, uint32_t u1) {
  return tm[0] ^ (u0 & tm[1]) ^ (u1 & tm[2]);
}

// One plane of the comparison uniform < threshold for the 32 replicas of a word,
// most significant plane first: r holds the plane's bit of every replica's
// uniform.  eq: replicas whose uniform has matched its threshold so far; acc:
// replicas decided below it.
__device__ __forceinline__ void compare_plane(uint32_t r, uint32_t u0, uint32_t u1, const uint32_t* tm, uint32_t& eq,
                                              uint32_t& acc) {
  const uint32_t t = threshold_bits(tm, u0, u1);
  acc |= eq & t & ~r;
  eq &= ~(r ^ t);
}

// Unsatisfied bonds of a site of 32 replicas: u's bits 0 and 1, the replicas that
// always flip (u >= 3: dE <= 0), and those to compare (u = 0, 1, 2 with thr(u) > 0).
struct BondCount {
  uint32_t u0, u1, always, cmp;
};

__device__ __forceinline__ BondCount bond_count(uint32_t s0, const SiteRec& sr, uint32_t sxp, uint32_t sxm,
                                                uint32_t syp, uint32_t sym, uint32_t szp, uint32_t szm,
                                                const MetropolisArgs& a) {
  const uint32_t b0 = s0 ^ sxp ^ sr.jxp, b1 = s0 ^ sxm ^ sr.jxm;
  const uint32_t b2 = s0 ^ syp ^ sr.jyp, b3 = s0 ^ sym ^ sr.jym;
  const uint32_t b4 = s0 ^ szp ^ sr.jzp, b5 = s0 ^ szm ^ sr.jzm;
  const uint32_t sa = b0 ^ b1 ^ b2, ca = majority(b0, b1, b2);
  const uint32_t sb = b3 ^ b4 ^ b5, cb = majority(b3, b4, b5);
  BondCount c;
  c.u0 = sa ^ sb;
  const uint32_t k2 = sa & sb;
  c.u1 = ca ^ cb ^ k2;
  const uint32_t u2 = majority(ca, cb, k2);
  c.always = u2 | (c.u1 & c.u0);
  c.cmp = ~c.always & threshold_bits(a.live, c.u0, c.u1);
  return c;
}

// Bit planes 0..7 (Philox blocks 0 and 1) of the comparison for the replicas in
// c.cmp: lt = below the threshold in those planes, eq = equal so far.
//
// FORM says how many leading bits of the thresholds are 0 (thr(u) = 2^32 e^-beta(12-4u)
// loses 5.8 beta, 11.5 beta and 17.3 beta leading bits at u = 2, 1, 0):
//   3: all eight planes of every threshold are 0 (beta >= 1.39): a replica stays equal
//      while its bits are 0 and is never below: one operation per two planes;
//   2: planes 0..3 are 0, planes 4..7 only where u = 2 may not be (beta >= 0.69);
//   1: planes 0, 1 are 0, 2, 3 only where u = 2 may not be (beta >= 0.35);
//   0: any thresholds.
// A plane costs four operations in general (threshold bit 2, borrow, equality), three
// where only u = 2 has a threshold bit, half to one where none has: 34, 24, 15 and 4
// per word for the forms 0 to 3, of some 150 per word and site in all.  With form 0 for
// every step: L = 8, 201 temperatures to beta = 5, two populations of 1e5 97.9 ms, with
// the forms 89.2; 64 runs of L = 4 to 10 on 101 temperatures 382 and 344 ms; L = 10,
// R = 1e6 adaptive (most of its steps below beta = 0.7) 224.7 and 221.8 ms.
template <int FORM>
__device__ __forceinline__ void compare_planes8(uint32_t uc, const SiteRec& sr, const ThreadPhilox (&tp)[2],
                                                const BondCount& c, const MetropolisArgs& a, uint32_t& lt,
                                                uint32_t& eq) {
  constexpr int ZERO = FORM == 3 ? 8 : FORM == 2 ? 4 : FORM == 1 ? 2 : 0;  // planes without any threshold bit
  constexpr int TWO = FORM == 2 ? 8 : FORM == 1 ? 4 : ZERO;                // planes before this: only u = 2 has one
  uint32_t w[2][4];
  philox_block(uc, sr, tp[0], a.k0, a.k1, w[0]);
  philox_block(uc, sr, tp[1], a.k0, a.k1, w[1]);
  uint32_t same = c.cmp;
#pragma unroll
  for (int p = 0; p < ZERO; ++p) same &= ~w[p / 4][p & 3];
  lt = 0;
  eq = same;
#pragma unroll
  for (int p = 7; p >= ZERO; --p) {
    const uint32_t r = w[p / 4][p & 3];
    const uint32_t t = p < TWO ? c.u1 & a.tm[p][2] : threshold_bits(a.tm[p], c.u0, c.u1);
    lt = (~r & t) | (~(r ^ t) & lt);
    eq &= ~(r ^ t);
  }
  lt &= same;
}

// Bit planes 8.. (Philox blocks 2..7) of site n, record sr, for the replicas in eq of
// the word whose block 0 is Philox group g8: those accepted.
__device__ __forceinline__ uint32_t compare_rest(uint32_t eq, uint32_t u0, uint32_t u1, uint32_t n, const SiteRec& sr,
                                                 uint32_t g8, uint32_t q, const MetropolisArgs& a) {
  uint32_t acc = 0;
  const uint32_t uc = kM0 * (n >> 1);
#pragma unroll 1
  for (int b = 2; b < 8 && eq; ++b) {
    const ThreadPhilox tb = thread_philox(g8 + (uint32_t)b, q, a.k0, a.k1);
    uint32_t w[4];
    philox_block(uc, sr, tb, a.k0, a.k1, w);
    if (b < a.lead) {  // no threshold bits in these planes
      eq &= ~(w[0] | w[1] | w[2] | w[3]);
      continue;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) compare_plane(w[i], u0, u1, a.tm[4 * b + i], eq, acc);
  }
  return acc;
}

}  // namespace pa
