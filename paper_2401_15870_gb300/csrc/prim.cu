// prim.cu -- scan, radix sort, compaction and fills (see prim.cuh).
#include <atomic>
#include "kernel_limits.cuh"
#include "prim.cuh"

namespace dfpr {

static std::atomic<unsigned long long> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void note_launches(unsigned long long k) { g_launches.fetch_add(k, std::memory_order_relaxed); }
unsigned long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

// allocations until the injected failure (0: none armed)
static std::atomic<long long> g_fail_in{0};

void arm_alloc_failure(long long k) { g_fail_in.store(k > 0 ? k : 0); }

cudaError_t dev_malloc_raw(void** p, size_t bytes) {
  if (g_fail_in.load(std::memory_order_relaxed) > 0 && g_fail_in.fetch_sub(1) == 1) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMalloc(p, bytes);
}

static int g_sms = 0;

int num_sms() {
  if (g_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_sms <= 0) g_sms = 152;
  }
  return g_sms;
}

int grid_for(int64_t n, int block) {
  int64_t want = cdiv(n > 0 ? n : 1, block);
  int64_t cap = (int64_t)num_sms() * 16;
  return (int)(want < cap ? want : cap);
}

namespace {
struct CudaLimits {
  using Error = cudaError_t;
  static constexpr Error ok = cudaSuccess, does_not_fit = cudaErrorInvalidConfiguration;
  static Error device(int* d) { return cudaGetDevice(d); }
  static Error raise(const void* fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  }
  static Error blocks(int* b, const void* fn, int threads, size_t smem) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(b, fn, threads, smem);
  }
};
}  // namespace

cudaError_t kernel_occupancy(const void* fn, int threads, size_t smem, int* bps) {
  static KernelLimits<CudaLimits> limits;
  return limits.get(fn, threads, smem, bps);
}

// ================================================================== scan

constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 8;
constexpr int SC_CHUNK = SC_THREADS * SC_ITEMS;  // 2048

int64_t scan_tmp_elems(int64_t n) { return cdiv(n > 0 ? n : 1, SC_CHUNK) + 1; }

// inclusive block scan of one value per thread; returns the inclusive prefix,
// *total receives the block total
template <typename T>
__device__ __forceinline__ T block_incl_scan(T x, T* total) {
  __shared__ T wsum[SC_THREADS / WARP];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    T s = lane < SC_THREADS / WARP ? wsum[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < SC_THREADS / WARP) wsum[lane] = s;
  }
  __syncthreads();
  T add = w > 0 ? wsum[w - 1] : T(0);
  *total = wsum[SC_THREADS / WARP - 1];
  __syncthreads();
  return x + add;
}

template <typename T>
__global__ void k_scan_reduce(const T* __restrict__ in, int64_t n, T* __restrict__ sums) {
  int64_t base = (int64_t)blockIdx.x * SC_CHUNK + (int64_t)threadIdx.x * SC_ITEMS;
  T s = 0;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; i++) {
    int64_t j = base + i;
    if (j < n) s += in[j];
  }
  T tot;
  block_incl_scan<T>(s, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// one block: exclusive scan of sums[0..nb) in place, sums[nb] = total
template <typename T>
__global__ void k_scan_top(T* sums, int64_t nb) {
  T carry = 0;
  for (int64_t base = 0; base < nb; base += SC_THREADS) {
    int64_t j = base + threadIdx.x;
    T x = j < nb ? sums[j] : T(0);
    T tot;
    T inc = block_incl_scan<T>(x, &tot);
    if (j < nb) sums[j] = carry + inc - x;
    carry += tot;
  }
  if (threadIdx.x == 0) sums[nb] = carry;
}

template <typename T>
__global__ void k_scan_down(const T* in, int64_t n, const T* __restrict__ sums, T* out, int64_t nb) {
  int64_t base = (int64_t)blockIdx.x * SC_CHUNK + (int64_t)threadIdx.x * SC_ITEMS;
  T v[SC_ITEMS];
  T s = 0;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; i++) {
    int64_t j = base + i;
    v[i] = j < n ? in[j] : T(0);
    s += v[i];
  }
  T tot;
  T inc = block_incl_scan<T>(s, &tot);
  T run = sums[blockIdx.x] + inc - s;
#pragma unroll
  for (int i = 0; i < SC_ITEMS; i++) {
    int64_t j = base + i;
    if (j < n) out[j] = run;
    run += v[i];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = sums[nb];
}

template <typename T>
cudaError_t scan_excl(const T* in, T* out, int64_t n, T* tmp, cudaStream_t s) {
  int64_t nb = cdiv(n > 0 ? n : 1, SC_CHUNK);
  if (n == 0) return cudaMemsetAsync(out, 0, sizeof(T), s);
  note_launch(); k_scan_reduce<T><<<(unsigned)nb, SC_THREADS, 0, s>>>(in, n, tmp);
  note_launch(); k_scan_top<T><<<1, SC_THREADS, 0, s>>>(tmp, nb);
  note_launch(); k_scan_down<T><<<(unsigned)nb, SC_THREADS, 0, s>>>(in, n, tmp, out, nb);
  return cudaGetLastError();
}

template cudaError_t scan_excl<int32_t>(const int32_t*, int32_t*, int64_t, int32_t*, cudaStream_t);
template cudaError_t scan_excl<int64_t>(const int64_t*, int64_t*, int64_t, int64_t*, cudaStream_t);

// ================================================================== radix sort

constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / WARP;
constexpr int RS_ITEMS = 16;
constexpr int RS_KPW = WARP * RS_ITEMS;       // keys per warp
constexpr int RS_TILE = RS_WARPS * RS_KPW;    // 8192 keys per tile
// digits of at most RS_BITS bits: the 2 x 25-bit edge keys of a 2^25-vertex
// graph take 5 passes instead of the 7 of 8-bit digits.  A sort takes the
// narrowest digits that need no more passes: the fewer digits, the longer the
// runs of a tile's keys that go to one place (8 keys on average with 10 bits)
constexpr int RS_BITS = 10;
constexpr int RS_BINS = 1 << RS_BITS;

static int64_t rs_tiles(int64_t n) { return cdiv(n > 0 ? n : 1, RS_TILE); }

size_t radix_tmp_bytes(int64_t n) {
  int64_t cnt = (int64_t)RS_BINS * rs_tiles(n);
  return sizeof(int32_t) * (size_t)(cnt + 1 + scan_tmp_elems(cnt));
}

// (both kernels load a thread's RS_ITEMS keys before they use the first: one
// memory latency per tile, not RS_ITEMS)
__global__ void __launch_bounds__(RS_THREADS, 2) k_rs_hist(const uint64_t* __restrict__ keys, int64_t n, int shift, int bits,
                                                           int32_t* __restrict__ counts, int64_t ntiles) {
  __shared__ int hist[RS_BINS];
  const int bins = 1 << bits;
  const int64_t base = (int64_t)blockIdx.x * RS_TILE + threadIdx.x;
  uint64_t k[RS_ITEMS];
#pragma unroll
  for (int i = 0; i < RS_ITEMS; i++) {
    const int64_t j = base + (int64_t)i * RS_THREADS;
    k[i] = j < n ? keys[j] : 0;
  }
  for (int i = threadIdx.x; i < bins; i += RS_THREADS) hist[i] = 0;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RS_ITEMS; i++)
    if (base + (int64_t)i * RS_THREADS < n) atomicAdd(&hist[(int)((k[i] >> shift) & (bins - 1))], 1);
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += RS_THREADS) counts[(int64_t)d * ntiles + blockIdx.x] = hist[d];
}

// stable scatter: a warp owns a contiguous run of RS_KPW keys of the tile and
// ranks its keys item by item, so (warp, item, lane) order is input order.
// The tile's keys are first placed in shared memory in digit order (each at
// its position among the tile's keys of its digit), then written out by
// consecutive threads, so the keys of one digit leave as one coalesced run
// instead of each warp's 32 keys going to up to 32 places.
// Dynamic shared memory: the staged tile, the per-warp digit counts (16 bits: a
// tile holds 8192 keys) and two words per digit, 104 KB, so two blocks share an SM
// (32-bit counts: 132 KB and one block).  A pass over 35.6M keys of 42 bits took
// 336 us for the scatter and 91 for the counts with 10-bit digits, one block and
// the loads one by one; 259 and 52 now (0.57 and 0.28 GB moved).  What is left is
// instructions (60% of the issue slots: the ballots) and shared memory.
constexpr size_t RS_STAGE_BYTES =
    sizeof(uint64_t) * RS_TILE + sizeof(uint16_t) * (size_t)RS_WARPS * RS_BINS + 2 * sizeof(int) * (size_t)RS_BINS;

__global__ void __launch_bounds__(RS_THREADS, 2) k_rs_scatter(const uint64_t* __restrict__ keys, uint64_t* __restrict__ out,
                                                              int64_t n, int shift, int bits,
                                                              const int32_t* __restrict__ offs,
                                                              int64_t ntiles) {
  extern __shared__ uint64_t stage[];   // RS_TILE keys, then dstart, gofs and wcnt
  int* dstart = reinterpret_cast<int*>(stage + RS_TILE);   // first position of each digit
  int* gofs = dstart + RS_BINS;                            // its place in the output, less that position
  uint16_t (*wcnt)[RS_BINS] = reinterpret_cast<uint16_t (*)[RS_BINS]>(gofs + RS_BINS);
  __shared__ int wtot[RS_WARPS];
  const int bins = 1 << bits;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t tile0 = (int64_t)blockIdx.x * RS_TILE;
  const int64_t base = tile0 + (int64_t)w * RS_KPW;
  uint64_t k[RS_ITEMS];
#pragma unroll
  for (int i = 0; i < RS_ITEMS; i++) {
    const int64_t j = base + i * WARP + lane;
    k[i] = j < n ? keys[j] : 0;
  }
  int32_t goff[2] = {0, 0};
  if (2 * threadIdx.x < bins) {   // (bins: at least two)
    goff[0] = offs[(int64_t)(2 * threadIdx.x) * ntiles + blockIdx.x];
    goff[1] = offs[(int64_t)(2 * threadIdx.x + 1) * ntiles + blockIdx.x];
  }
  for (int i = threadIdx.x; i < RS_WARPS * RS_BINS / 2; i += RS_THREADS) reinterpret_cast<uint32_t*>(wcnt)[i] = 0u;
  __syncthreads();
  uint32_t rank[RS_ITEMS / 2] = {};   // two ranks of 16 bits each
  const unsigned lt = lanemask_lt();
#pragma unroll
  for (int i = 0; i < RS_ITEMS; i++) {
    const bool valid = base + i * WARP + lane < n;
    const int d = (int)((k[i] >> shift) & (bins - 1));
    // lanes of the same digit, from a ballot per bit (__match_any_sync takes
    // longer than the ten of them)
    unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < RS_BITS; b++) {   // (bits past the digit's are zero in every lane)
      const bool bit = (d >> b) & 1;
      const unsigned m = __ballot_sync(0xffffffffu, bit);
      peers &= bit ? m : ~m;
    }
    const int before = valid ? wcnt[w][d] : 0;
    rank[i / 2] |= (uint32_t)(before + __popc(peers & lt)) << (16 * (i & 1));
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) wcnt[w][d] = (uint16_t)(before + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  // per digit (thread t: digits 2 t and 2 t + 1): the warps' counts turned into
  // offsets within the digit, the totals into the digits' first positions, and
  // the place of the tile's run of the digit in the output less that position
  static_assert(RS_BINS == 2 * RS_THREADS, "two digits per thread");
  int run[2] = {0, 0};
  uint32_t* const col = reinterpret_cast<uint32_t*>(&wcnt[0][2 * threadIdx.x]);
#pragma unroll
  for (int ww = 0; ww < RS_WARPS; ww++) {
    const uint32_t t = col[ww * (RS_BINS / 2)];
    col[ww * (RS_BINS / 2)] = (uint32_t)run[0] | (uint32_t)run[1] << 16;
    run[0] += (int)(t & 0xffffu);
    run[1] += (int)(t >> 16);
  }
  int incl = run[0] + run[1];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) wtot[w] = incl;
  __syncthreads();
  int first = incl - run[0] - run[1];
  for (int ww = 0; ww < w; ww++) first += wtot[ww];
  dstart[2 * threadIdx.x] = first;
  dstart[2 * threadIdx.x + 1] = first + run[0];
  gofs[2 * threadIdx.x] = goff[0] - first;
  gofs[2 * threadIdx.x + 1] = goff[1] - first - run[0];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < RS_ITEMS; i++) {
    if (base + i * WARP + lane < n) {
      const int d = (int)((k[i] >> shift) & (bins - 1));
      stage[dstart[d] + wcnt[w][d] + (rank[i / 2] >> (16 * (i & 1)) & 0xffffu)] = k[i];
    }
  }
  __syncthreads();
  const int valid_keys = (int)(n - tile0 < RS_TILE ? n - tile0 : RS_TILE);
#pragma unroll 4
  for (int t = threadIdx.x; t < valid_keys; t += RS_THREADS) {
    const uint64_t key = stage[t];
    const int d = (int)((key >> shift) & (bins - 1));
    out[(int64_t)gofs[d] + t] = key;
  }
}

// packed pairs (a, b) as (b, a)
__global__ void k_swap_keys(const uint64_t* __restrict__ in, int64_t n, int bits, uint64_t* __restrict__ out) {
  const uint64_t mask = (1ull << bits) - 1;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = ((in[i] & mask) << bits) | (in[i] >> bits);
}

cudaError_t swap_keys_u64(const uint64_t* in, int64_t n, int bits, uint64_t* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  note_launch(); k_swap_keys<<<grid_for(n, 256), 256, 0, s>>>(in, n, bits, out);
  return cudaGetLastError();
}

cudaError_t radix_sort_u64(uint64_t* keys, uint64_t* alt, int64_t n, int lo_bit, int hi_bit, void* tmp,
                           cudaStream_t s) {
  if (n <= 1 || hi_bit <= lo_bit) return cudaSuccess;
  if (n >= (int64_t(1) << 31)) return cudaErrorInvalidValue;
  int bps;   // (raises the kernel's shared memory limit)
  const cudaError_t limit = kernel_occupancy((const void*)k_rs_scatter, RS_THREADS, RS_STAGE_BYTES, &bps);
  if (limit != cudaSuccess) return limit;
  int64_t ntiles = rs_tiles(n);
  const int passes = (hi_bit - lo_bit + RS_BITS - 1) / RS_BITS;
  const int bits = (hi_bit - lo_bit + passes - 1) / passes;
  const int64_t cnt = ((int64_t)1 << bits) * ntiles;
  int32_t* counts = (int32_t*)tmp;
  int32_t* scratch = counts + (int64_t)RS_BINS * ntiles + 1;
  uint64_t* src = keys;
  uint64_t* dst = alt;
  for (int p = 0; p < passes; p++) {
    const int shift = lo_bit + p * bits;
    note_launch(); k_rs_hist<<<(unsigned)ntiles, RS_THREADS, 0, s>>>(src, n, shift, bits, counts, ntiles);
    cudaError_t e = scan_excl<int32_t>(counts, counts, cnt, scratch, s);
    if (e != cudaSuccess) return e;
    note_launch(); k_rs_scatter<<<(unsigned)ntiles, RS_THREADS, RS_STAGE_BYTES, s>>>(src, dst, n, shift, bits, counts, ntiles);
    uint64_t* t = src;
    src = dst;
    dst = t;
  }
  if (src != keys) return cudaMemcpyAsync(keys, src, sizeof(uint64_t) * (size_t)n, cudaMemcpyDeviceToDevice, s);
  return cudaGetLastError();
}

// ================================================================== compaction

size_t compact_tmp_bytes(int64_t n) { return sizeof(int64_t) * (size_t)(n + 1 + scan_tmp_elems(n)); }

__global__ void k_flag_to_i64(const uint8_t* __restrict__ f, int64_t n, int64_t* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = f[i] ? 1 : 0;
}

__global__ void k_compact_scatter(const uint64_t* __restrict__ in, const uint8_t* __restrict__ f,
                                  const int64_t* __restrict__ pos, int64_t n, uint64_t* __restrict__ out,
                                  int64_t* count_dev) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (f[i]) out[pos[i]] = in[i];
  if (blockIdx.x == 0 && threadIdx.x == 0) *count_dev = pos[n];
}

cudaError_t compact_u64(const uint64_t* in, const uint8_t* flag, int64_t n, uint64_t* out, int64_t* count_dev,
                        void* tmp, cudaStream_t s) {
  if (n == 0) return cudaMemsetAsync(count_dev, 0, sizeof(int64_t), s);
  int64_t* pos = (int64_t*)tmp;
  int64_t* scr = pos + n + 1;
  note_launch(); k_flag_to_i64<<<grid_for(n, 256), 256, 0, s>>>(flag, n, pos);
  cudaError_t e = scan_excl<int64_t>(pos, pos, n, scr, s);
  if (e != cudaSuccess) return e;
  note_launch(); k_compact_scatter<<<grid_for(n, 256), 256, 0, s>>>(in, flag, pos, n, out, count_dev);
  return cudaGetLastError();
}

__global__ void k_flag_unique(const uint64_t* __restrict__ k, int64_t n, uint8_t* __restrict__ f) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    f[i] = (i == 0 || k[i] != k[i - 1]) ? 1 : 0;
}

cudaError_t flag_unique_sorted(const uint64_t* k, int64_t n, uint8_t* flag, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  note_launch(); k_flag_unique<<<grid_for(n, 256), 256, 0, s>>>(k, n, flag);
  return cudaGetLastError();
}

// ================================================================== fills

template <typename T>
__global__ void k_fill(T* p, T v, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}
__global__ void k_iota(int32_t* p, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = (int32_t)i;
}

cudaError_t fill_i32(int32_t* p, int32_t v, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  note_launch(); k_fill<int32_t><<<grid_for(n, 256), 256, 0, s>>>(p, v, n);
  return cudaGetLastError();
}
cudaError_t fill_i64(int64_t* p, int64_t v, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  note_launch(); k_fill<int64_t><<<grid_for(n, 256), 256, 0, s>>>(p, v, n);
  return cudaGetLastError();
}
cudaError_t iota_i32(int32_t* p, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  note_launch(); k_iota<<<grid_for(n, 256), 256, 0, s>>>(p, n);
  return cudaGetLastError();
}

}  // namespace dfpr
