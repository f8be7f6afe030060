// noalloc.cu -- per-receiver reduction of caller-provided path records that
// allocates no device memory.
//
// Some callers cannot allocate device memory at the time they need the
// received power: a host framework that owns the whole device memory pool
// and forbids allocations outside it, or a real-time loop that must not call
// cudaMalloc after start-up (cudaMalloc can synchronise the device and stall
// the loop). dcem_reduce_paths_noalloc serves them: the caller passes device
// buffers for the inputs and outputs, and the only scratch the kernels need
// lives in one file-scope device array of fixed size. The CUDA runtime may
// load this file's kernels and reserve that array lazily, at the first use
// on a device; a set-up call (n_paths = 0, nrx = 0) made once per device at
// start-up does that work, so that later calls allocate nothing.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "dcem_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kNaMaxRx = 4096;          // receivers per call
constexpr int kNaMaxPaths = 1 << 16;    // path records per call
constexpr int kNaMaxPerRx = 4096;       // paths of one receiver (sorted in shared memory)
constexpr int kNaThreads = 256;
constexpr int kNaMaxDevices = 64;

enum : unsigned { NA_ERR_RX_RANGE = 1u, NA_ERR_PER_RX = 2u };

struct NaScratch {
  unsigned count[kNaMaxRx];    // paths per receiver
  unsigned offset[kNaMaxRx];   // exclusive prefix sum of count
  int order[kNaMaxPaths];      // path indices grouped by receiver
};

// The scratch of every call on a device (about 295 KB per device, held from
// the first use on that device until the process exits). Host code reaches it
// only through the address returned by cudaGetSymbolAddress.
static __device__ __align__(256) NaScratch g_na_scratch;

// The records grouped by receiver, by one cluster of eight CTAs: each counts
// the receivers of its eighth of the records in shared memory (a record's
// rank among them stays in a register), each then scans its eighth of the
// receivers over the eight counts, and places its records: 9 us for 16,384
// records and 1024 receivers. As four kernels with counters in device memory
// (clear, count, scan, place) it was 13 us and three launches more; one CTA
// alone (25 us) reads the records' receiver numbers, 224 bytes apart, at one
// SM's rate.
constexpr int kNaCluster = 8, kNaGroupThreads = 1024;
constexpr int kNaPerThread = kNaMaxPaths / (kNaCluster * kNaGroupThreads);
constexpr int kNaSlice = kNaMaxRx / kNaCluster;
static_assert(kNaSlice <= kNaGroupThreads, "one receiver of the slice per thread");

__global__ void __cluster_dims__(kNaCluster, 1, 1) __launch_bounds__(kNaGroupThreads)
    k_na_group(NaScratch* s, unsigned* err, const dcem_path* __restrict__ p, int n, int nrx) {
  __shared__ unsigned cnt[kNaMaxRx];          // paths per receiver, then their first places
  __shared__ unsigned total[kNaCluster], errs[kNaCluster], part[32];
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, me = (int)cl.block_rank();
  for (int r = tid; r < nrx; r += kNaGroupThreads) cnt[r] = 0u;
  __syncthreads();
  const int per_cta = (n + kNaCluster - 1) / kNaCluster, i0 = me * per_cta, i1 = min(n, i0 + per_cta);
  int rx[kNaPerThread];
  unsigned rank[kNaPerThread];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < kNaPerThread; ++k) {
    const int i = i0 + k * kNaGroupThreads + tid;
    rx[k] = i < i1 ? p[i].rx : -1;
    if (i < i1 && (rx[k] < 0 || rx[k] >= nrx)) {
      bad = true;
      rx[k] = -1;
    }
  }
#pragma unroll
  for (int k = 0; k < kNaPerThread; ++k) rank[k] = rx[k] >= 0 ? atomicAdd(&cnt[rx[k]], 1u) : 0u;
  const int any_bad = __syncthreads_or(bad);
  cl.sync();
  // this CTA's slice of the receivers, one per thread
  const int slice = (nrx + kNaCluster - 1) / kNaCluster, r = me * slice + tid;
  const bool own = tid < slice && r < nrx;
  unsigned h[kNaCluster], sum = 0;
#pragma unroll
  for (int c = 0; c < kNaCluster; ++c) {
    h[c] = own ? cl.map_shared_rank(cnt, c)[r] : 0u;
    sum += h[c];
  }
  unsigned x = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) part[tid >> 5] = x;
  const int any_long = __syncthreads_or(sum > (unsigned)kNaMaxPerRx);
  for (int w = 0; w < (tid >> 5); ++w) x += part[w];
  const unsigned first = x - sum;   // within the slice
  if (own) {
    unsigned at = first;
#pragma unroll
    for (int c = 0; c < kNaCluster; ++c) {
      cl.map_shared_rank(cnt, c)[r] = at;
      at += h[c];
    }
    s->count[r] = sum;
  }
  if (tid == kNaGroupThreads - 1)
    for (int c = 0; c < kNaCluster; ++c) cl.map_shared_rank(total, c)[me] = x;
  if (tid == 0) cl.map_shared_rank(errs, 0)[me] = (any_bad ? NA_ERR_RX_RANGE : 0u) | (any_long ? NA_ERR_PER_RX : 0u);
  cl.sync();   // no CTA reaches into another's shared memory from here on
  if (tid < kNaCluster) {
    unsigned before = 0;
    for (int c = 0; c < tid; ++c) before += total[c];
    part[tid] = before;
  }
  __syncthreads();
  if (own) s->offset[r] = part[me] + first;
#pragma unroll
  for (int k = 0; k < kNaPerThread; ++k)
    if (rx[k] >= 0)
      s->order[part[rx[k] / slice] + cnt[rx[k]] + rank[k]] = i0 + k * kNaGroupThreads + tid;
  if (me == 0 && tid == 0) {
    unsigned e = 0;
    for (int c = 0; c < kNaCluster; ++c) e |= errs[c];
    *err = e;
  }
}

// Each receiver's paths sorted by key, records with equal keys (the same
// sequence from two transmitters) by record index, then the same fixed-order
// sums as the frame reduction (sorted position i goes to partial sum i mod
// 256, in order, then a fixed binary tree). The order, and so every bit of
// the sums, depends only on the records, not on the order in which the
// grouping's atomics placed them; for one transmitter's records (distinct
// keys) it is the frame's order, so the results match dcem_trace_frame's.
// One warp per receiver with up to 32 paths, its keys and sums in registers
// (the tree's upper levels would add zeros), then the CTA together for each
// with more, in shared memory. One CTA per receiver took 21 us for 1024
// receivers with 16 paths each, this 10 us.
constexpr int kNaWarps = kNaThreads / 32;

__device__ __forceinline__ bool na_after(unsigned long long x, int xi, unsigned long long y, int yi) {
  return x != y ? x > y : (unsigned)xi > (unsigned)yi;   // padding (~0, -1) sorts last
}

__global__ void __launch_bounds__(kNaThreads) k_na_reduce(const NaScratch* s, const dcem_path* __restrict__ p,
                                                          int nrx, int per, double tx_power, double* field,
                                                          double* pc, double* pi) {
  extern __shared__ unsigned long long skey[];  // kNaMaxPerRx keys, then as many ints
  int* sidx = reinterpret_cast<int*>(skey + kNaMaxPerRx);
  __shared__ double red[3][kNaThreads], sums[kNaWarps][3];
  __shared__ int scnt[kNaWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int r0 = blockIdx.x * per, rw = wid < per ? r0 + wid : nrx;
  const int cnt = rw < nrx ? (int)min(s->count[rw], (unsigned)kNaMaxPerRx) : 0;
  if (lane == 0) scnt[wid] = cnt;
  if (cnt <= 32) {
    unsigned long long key = ~0ull;
    int idx = -1;
    if (lane < cnt) {
      idx = s->order[s->offset[rw] + lane];
      key = p[idx].key;
    }
    for (int k = 2; k < 2 * cnt; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, j);
        const int oi = __shfl_xor_sync(0xffffffffu, idx, j);
        const bool low = (lane & j) == 0, up = (lane & k) == 0;
        if (low == up ? na_after(key, idx, ok, oi) : na_after(ok, oi, key, idx)) {
          key = ok;
          idx = oi;
        }
      }
    double sre = 0.0, sim = 0.0, sinc = 0.0;
    if (lane < cnt) {
      const dcem_path& q = p[idx];
      sre += q.amp_re;
      sim += q.amp_im;
      sinc += q.amp_re * q.amp_re + q.amp_im * q.amp_im;
    }
    for (int o = 16; o > 0; o >>= 1) {
      sre += __shfl_down_sync(0xffffffffu, sre, o);
      sim += __shfl_down_sync(0xffffffffu, sim, o);
      sinc += __shfl_down_sync(0xffffffffu, sinc, o);
    }
    if (lane == 0) {
      sums[wid][0] = sre;
      sums[wid][1] = sim;
      sums[wid][2] = sinc;
    }
  }
  __syncthreads();
  for (int w = 0; w < per; ++w) {  // receivers with more paths, the CTA together
    const int n = scnt[w];
    if (n <= 32) continue;
    const unsigned off = s->offset[r0 + w];
    int np2 = 64;
    while (np2 < n) np2 <<= 1;
    for (int i = tid; i < np2; i += kNaThreads) {
      const int u = i < n ? s->order[off + i] : -1;
      skey[i] = u >= 0 ? p[u].key : ~0ull;
      sidx[i] = u;
    }
    __syncthreads();
    for (int k = 2; k <= np2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = tid; i < np2; i += kNaThreads) {
          const int o = i ^ j;
          if (o > i) {
            const unsigned long long x = skey[i], y = skey[o];
            const int xi = sidx[i], yi = sidx[o];
            if (na_after(x, xi, y, yi) == ((i & k) == 0)) {
              skey[i] = y;
              skey[o] = x;
              sidx[i] = yi;
              sidx[o] = xi;
            }
          }
        }
        __syncthreads();
      }
    double sre = 0.0, sim = 0.0, sinc = 0.0;
    for (int i = tid; i < n; i += kNaThreads) {
      const dcem_path& q = p[sidx[i]];
      sre += q.amp_re;
      sim += q.amp_im;
      sinc += q.amp_re * q.amp_re + q.amp_im * q.amp_im;
    }
    red[0][tid] = sre;
    red[1][tid] = sim;
    red[2][tid] = sinc;
    __syncthreads();
    for (int h = kNaThreads / 2; h > 0; h >>= 1) {
      if (tid < h)
        for (int k = 0; k < 3; ++k) red[k][tid] += red[k][tid + h];
      __syncthreads();
    }
    if (tid < 3) sums[w][tid] = red[tid][0];
    __syncthreads();
  }
  // a logarithm is some 60 dependent FP64 operations: the coherent power by
  // one thread, the incoherent by another, the CTA's receivers side by side
  const int n = min(per, nrx - r0);
  if (tid < 2 * n) {
    const int k = tid < n ? tid : tid - n;
    const size_t r = (size_t)r0 + k;
    const double fr = sums[k][0], fi = sums[k][1], w = tid < n ? fr * fr + fi * fi : sums[k][2];
    if (tid < n && field) {
      field[2 * r] = fr;
      field[2 * r + 1] = fi;
    }
    double* out = tid < n ? pc : pi;
    if (out) out[r] = 10.0 * log10(tx_power * w) + 30.0;
  }
}

// Per-device address of g_na_scratch, looked up once per device.
std::mutex g_na_mutex;
NaScratch* g_na_addr[kNaMaxDevices] = {};
unsigned* g_na_err[kNaMaxDevices] = {};   // error bits of the current call, in mapped host memory
bool g_na_attr[kNaMaxDevices] = {};

int na_status(cudaError_t e) {
  if (e == cudaSuccess) return DCEM_OK;
  cudaGetLastError();
  return DCEM_ERR_CUDA;
}

}  // namespace

extern "C" int dcem_reduce_paths_noalloc(const dcem_path* paths, int32_t n_paths, int32_t nrx,
                                         double tx_power_w, double* field, double* p_coh_dbm,
                                         double* p_inc_dbm, void* stream) {
  if (n_paths < 0 || nrx < 0 || (n_paths > 0 && !paths)) return DCEM_ERR_ARG;
  if (!(tx_power_w > 0.0)) return DCEM_ERR_ARG;
  if (n_paths > kNaMaxPaths || nrx > kNaMaxRx) return DCEM_ERR_CAPACITY;
  if (nrx == 0 && n_paths > 0) return DCEM_ERR_ARG;  // no receiver can hold them
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return na_status(e);
  if (dev < 0 || dev >= kNaMaxDevices) return DCEM_ERR_CUDA;
  NaScratch* s = nullptr;
  unsigned *err = nullptr, *err_d = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
      // set-up on the first call on this device, with the device current
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_na_scratch);
      if (e != cudaSuccess) return na_status(e);
      g_na_addr[dev] = static_cast<NaScratch*>(ptr);
    }
    if (!g_na_err[dev]) {
      void* ptr = nullptr;
      e = cudaHostAlloc(&ptr, 64, cudaHostAllocMapped);
      if (e != cudaSuccess) return na_status(e);
      g_na_err[dev] = static_cast<unsigned*>(ptr);
    }
    if (!g_na_attr[dev]) {
      size_t smem = (size_t)kNaMaxPerRx * (sizeof(unsigned long long) + sizeof(int));
      e = cudaFuncSetAttribute(k_na_reduce, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return na_status(e);
      // the other kernel too, so that a lazily loading runtime loads it now
      // rather than at a later call
      cudaFuncAttributes fa;
      e = cudaFuncGetAttributes(&fa, k_na_group);
      if (e != cudaSuccess) return na_status(e);
      g_na_attr[dev] = true;
    }
    s = g_na_addr[dev];
    err = g_na_err[dev];
    void* ptr = nullptr;
    e = cudaHostGetDevicePointer(&ptr, err, 0);
    if (e != cudaSuccess) return na_status(e);
    err_d = static_cast<unsigned*>(ptr);
  }
  if (nrx == 0) return DCEM_OK;  // the set-up call
  cudaStream_t st = (cudaStream_t)stream;
  k_na_group<<<kNaCluster, kNaGroupThreads, 0, st>>>(s, err_d, paths, n_paths, nrx);
  // receivers per CTA: enough CTAs for every SM (four fit by shared memory),
  // no more than a warp each
  const int per = std::min(kNaWarps, (nrx + 511) / 512);
  size_t smem = (size_t)kNaMaxPerRx * (sizeof(unsigned long long) + sizeof(int));
  k_na_reduce<<<(nrx + per - 1) / per, kNaThreads, smem, st>>>(s, paths, nrx, per, tx_power_w, field, p_coh_dbm,
                                                              p_inc_dbm);
  e = cudaGetLastError();
  if (e != cudaSuccess) return na_status(e);
  // the error bits come with the end of the kernels, without a copy of their own
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return na_status(e);
  const unsigned bits = *static_cast<volatile unsigned*>(err);
  if (bits & NA_ERR_RX_RANGE) return DCEM_ERR_ARG;
  if (bits & NA_ERR_PER_RX) return DCEM_ERR_CAPACITY;
  return DCEM_OK;
}
