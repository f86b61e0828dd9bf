// pa_noalloc.cu — pa_resample_counts_noalloc: the copy numbers, scan and parent
// map of one resampling, for callers that cannot allocate device memory.
//
// The block totals of the scan live in a file-scope __device__ array of fixed
// size instead of memory allocated per call.  Every GPU that loads libpa.so
// holds this array (32 KiB) until the process exits; all calls on a device share
// it, so calls whose work overlaps on the GPU (different streams, or different
// host threads) race on it and must be serialised by the caller.  Each call
// writes every entry it later reads (the block totals), so nothing has to start at
// zero.
//
// Host code must not pass the array's name to a kernel: in host code it is a
// host-side stand-in, not a device address.  The device address is looked up
// with cudaGetSymbolAddress once per device, with that device current, on the
// first call made on it.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "../../include/pa.h"
#include "pa_device.cuh"
#include "pa_internal.h"

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaSlotsPerBlock = 1024;  // four old slots per thread
constexpr int kNaMaxDevices = 64;

// [0, n_blocks): block totals (64-bit: a block of 1024 slots may hold up to 2^41
// copies); a block whose inputs are invalid writes -1 as its total.
__device__ __align__(256) long long g_na_scratch[PA_NOALLOC_MAX_BLOCKS];

__device__ __forceinline__ long long warp_inclusive_scan_ll(long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Exclusive block scan of one 64-bit value per thread; sh holds 33 entries.
__device__ long long block_exclusive_scan_ll(long long v, long long* sh, long long* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long long inc = warp_inclusive_scan_ll(v);
  if (lane == 31) sh[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const long long x = lane < nw ? sh[lane] : 0;
    const long long xi = warp_inclusive_scan_ll(x);
    if (lane < nw) sh[lane] = xi - x;
    if (lane == nw - 1) sh[32] = xi;
  }
  __syncthreads();
  const long long out = sh[warp] + inc - v;
  if (total) *total = sh[32];
  __syncthreads();
  return out;
}

// Copy numbers n_i = fl(k_i) + [r_i < thr(k_i)] of 1024 old slots per block; the
// block total goes to the static scratch.  A level outside [0, n_levels) or a
// floor entry outside [0, 2^31 - 2] is invalid: that slot's count is written as 0
// and the block's total as -1.
__global__ void __launch_bounds__(kNaThreads) k_na_counts(const int32_t* __restrict__ levels, int n_old,
                                                          const int32_t* __restrict__ fl,
                                                          const uint32_t* __restrict__ thr, int n_levels,
                                                          uint32_t k0, uint32_t k1, int t, int32_t* counts,
                                                          long long* scratch) {
  __shared__ long long red[kNaThreads / 32];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int i0 = blockIdx.x * kNaSlotsPerBlock + 4 * threadIdx.x;
  long long sum = 0;
  int bad = 0;
  if (i0 < n_old) {
    const uint4 r = pa::philox4x32_10(make_uint4((uint32_t)(i0 >> 2), 0u, 0u, (uint32_t)t), k0, k1);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = i0 + b;
      if (i < n_old) {
        const int k = levels[i];
        int n = 0;
        if (k < 0 || k >= n_levels) {
          bad = 1;
        } else {
          const int f = fl[k];
          if (f < 0 || f == INT_MAX)
            bad = 1;
          else
            n = f + (pa::word_of(r, b) < thr[k] ? 1 : 0);
        }
        counts[i] = n;
        sum += n;
      }
    }
  }
  bad = __syncthreads_or(bad);
  sum = pa::warp_sum(sum);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long s = 0;
    for (int w = 0; w < kNaThreads / 32; ++w) s += red[w];
    scratch[blockIdx.x] = bad ? -1 : s;
  }
}

// Parents of the new slots j < cap: slot offset_i + q (q < n_i) descends from old
// slot i.  A block takes the slots of PER counting blocks.  It reads all block totals: those
// before its own give its offset, and a negative one anywhere means invalid input, for which
// nothing is written but *n_new = -1; the last block writes the grand total, the new
// population size.  (A scan kernel of one block in between cost 1.9 us and a launch: 18.5 us
// per call at 1e6 slots against 14.6.)  The totals are read blocks x totals times: with
// PER = 1 the 4096 blocks of the largest population read 134 MB of them, 39.0 us per call at
// 4 194 304 slots where the scan kernel's form took 37.3; PER = 2 takes 36.8, and 24.7 at
// 2.5e6 (26.0).  PER = 2 from 1 048 577 slots on is slower there (16.5 us against 14.5: half
// the chip's places stay empty), and eight slots in a row per thread (up to 38.9 at
// 4 194 304) and the counts of both blocks loaded ahead (39.0 at 4e6) are no faster than PER = 1.
// With PER = 1 a thread loads its counts before the scan of the totals, and the total is
// written before the parents (15.0 us at 1e6 slots otherwise, 14.5 so).
// The launch overlaps the counting kernel's end; griddepcontrol.wait orders the reads.
constexpr int kNaScatterBlocks = 2048;  // PER = 1 up to these many, 2 beyond

template <int PER>
__global__ void __launch_bounds__(kNaThreads) k_na_scatter(const int32_t* __restrict__ counts, int n_old, int n_blocks,
                                                           const long long* __restrict__ scratch, int32_t* parents,
                                                           long long cap, int64_t* n_new) {
  __shared__ long long sh[33];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  long long before = 0;
  int bad = 0;
  for (int b = threadIdx.x; b < n_blocks; b += kNaThreads) {
    const long long v = __ldcg(scratch + b);
    bad |= v < 0;
    if (b < PER * (int)blockIdx.x) before += v;
  }
  bad = __syncthreads_or(bad);
  long long n[4], base, mine;
  auto load = [&](int i0) {
#pragma unroll
    for (int b = 0; b < 4; ++b) n[b] = !bad && i0 + b < n_old ? __ldcg(counts + i0 + b) : 0;
  };
  if (PER == 1) load(blockIdx.x * kNaSlotsPerBlock + 4 * threadIdx.x);
  block_exclusive_scan_ll(before, sh, &base);
  const int first = PER * blockIdx.x, last = min(first + PER, n_blocks);
  for (int blk = first; blk == first || blk < last; ++blk) {  // the slots of one counting block after the other
    const int i0 = blk * kNaSlotsPerBlock + 4 * threadIdx.x;
    if (PER > 1) load(i0);
    long long off = base + block_exclusive_scan_ll(n[0] + n[1] + n[2] + n[3], sh, &mine);
    base += mine;
    if (PER == 1 && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_new = bad ? -1 : base;
    if (PER == 1 && bad) return;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      for (long long j = off; j < off + n[b] && j < cap; ++j)
        if (j >= 0) parents[j] = i0 + b;
      off += n[b];
    }
    if (PER == 1) return;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *n_new = bad ? -1 : base;
}

std::mutex g_na_mutex;
long long* g_na_scratch_dev[kNaMaxDevices] = {};

// Device address of the scratch on the current device (looked up on first use).
int na_scratch(long long** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNaMaxDevices) return PA_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_scratch_dev[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || !p) return PA_ERR_CUDA;
    g_na_scratch_dev[dev] = static_cast<long long*>(p);
  }
  *out = g_na_scratch_dev[dev];
  return PA_OK;
}

}  // namespace

extern "C" int pa_resample_counts_noalloc(const int32_t* levels, int64_t n_old, const int32_t* fl,
                                          const uint32_t* thr, int32_t n_levels, uint64_t run_seed, int32_t pop,
                                          int32_t t, int32_t* counts, int32_t* parents, int64_t parents_cap,
                                          int64_t* n_new, void* cuda_stream) {
  if (n_old < 0 || n_old > (int64_t)PA_NOALLOC_MAX_BLOCKS * kNaSlotsPerBlock) return PA_ERR_INVALID;
  if (!n_new || n_levels < 1 || parents_cap < 0 || pop < 0 || pop > 15 || t < 0 ||
      run_seed >= ((uint64_t)1 << 56))
    return PA_ERR_INVALID;
  if (n_old > 0 && (!levels || !fl || !thr || !counts)) return PA_ERR_INVALID;
  if (parents_cap > 0 && !parents) return PA_ERR_INVALID;
  long long* scratch = nullptr;
  int rc = na_scratch(&scratch);
  if (rc != PA_OK) return rc;
  const uint32_t k0 = (uint32_t)(run_seed & 0xffffffffu);
  const uint32_t k1 = (uint32_t)(run_seed >> 32) | ((uint32_t)pa::kResample << 28) | ((uint32_t)pop << 24);
  const int n_blocks = (int)((n_old + kNaSlotsPerBlock - 1) / kNaSlotsPerBlock);
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (n_blocks > 0)
    k_na_counts<<<n_blocks, kNaThreads, 0, s>>>(levels, (int)n_old, fl, thr, n_levels, k0, k1, t, counts, scratch);
  cudaLaunchConfig_t cfg{};
  const int per = n_blocks > kNaScatterBlocks ? 2 : 1;
  cfg.gridDim = dim3((unsigned)std::max((n_blocks + per - 1) / per, 1));  // an empty population: one block writes the total
  cfg.blockDim = dim3(kNaThreads);
  cfg.stream = s;
  cudaLaunchAttribute overlap{};
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &overlap;
  cfg.numAttrs = n_blocks > 0 ? 1u : 0u;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, per == 2 ? k_na_scatter<2> : k_na_scatter<1>, (const int32_t*)counts,
                                           (int)n_old, n_blocks, (const long long*)scratch, parents,
                                           (long long)parents_cap, n_new);
  if (e != cudaSuccess) return PA_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}
