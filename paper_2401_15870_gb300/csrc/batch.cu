// batch.cu -- a batch of edge deletions and insertions applied to the device
// CSR and transpose-CSR in place (Sec. 3.2).
//
//   E_t = (E_{t-1} \ D) u I      (deletions first; self-loop deletions are
//                                 ignored because self-loops are re-added with
//                                 every batch, Sec. 5.1.4 / 4.2.2)
//   Delta- = E_{t-1} \ E_t,  Delta+ = E_t \ E_{t-1}   (the effective change)
//
// Steps: packed keys -> radix sort -> first occurrences -> effective flags by
// binary search in the sorted rows -> compaction (Delta-, Delta+ sorted by
// (src, dst)) -> the same sorted by (dst, src) -> touched rows with their edit
// plans -> the rows rewritten in place, padding slots set to the sentinel.  A
// batch of at most SMALL_MAX edges does the steps up to the plans in two
// kernels.  A row whose new degree exceeds its capacity triggers a repack of
// that direction (a full rebuild with fresh slack).
#include <algorithm>
#include <climits>
#include <cstring>
#include <new>
#include "batch.cuh"
#include "edit_marks.cuh"
#include "frontier.cuh"
#include "prim.cuh"
#include "sweep.cuh"

namespace dfpr {

constexpr uint64_t DROP = ~0ull;

struct Carve {
  char* p;
  size_t used = 0;
  explicit Carve(void* base) : p((char*)base) {}
  template <typename T>
  T* take(int64_t n) {
    size_t off = (used + 255) & ~(size_t)255;
    used = off + sizeof(T) * (size_t)(n > 0 ? n : 1);
    return (T*)(p + off);
  }
};

#define GRID_STRIDE(i, n) \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

#define TRY(x)                                          \
  do {                                                  \
    cudaError_t _e = (x);                               \
    if (_e != cudaSuccess) return cuda_fail(g, _e, #x); \
  } while (0)

// ------------------------------------------------------------------ kernels

__global__ void k_validate(const int32_t* __restrict__ s, const int32_t* __restrict__ d, int64_t k, int32_t n,
                           unsigned long long* bad) {
  unsigned long long c = 0;
  GRID_STRIDE(i, k) c += (s[i] < 0 || s[i] >= n || d[i] < 0 || d[i] >= n) ? 1 : 0;
  if (c) atomicAdd(bad, c);
}

// user ids -> packed internal keys; self-loops become DROP
__global__ void k_make_keys(const int32_t* __restrict__ s, const int32_t* __restrict__ d, int64_t k,
                            const int32_t* __restrict__ perm, int bits, uint64_t* __restrict__ out) {
  GRID_STRIDE(i, k) {
    int32_t u = s[i], v = d[i];
    out[i] = (u == v) ? DROP : (((uint64_t)perm[u] << bits) | (uint64_t)perm[v]);
  }
}

__device__ __forceinline__ bool in_row(const int32_t* col, int64_t base, int32_t deg, int32_t x) {
  int32_t lo = 0, hi = deg;
  while (lo < hi) {
    int32_t mid = (lo + hi) >> 1;
    if (col[base + mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo < deg && col[base + lo] == x;
}

__device__ __forceinline__ bool key_in(const uint64_t* k, int64_t len, uint64_t x) {
  int64_t lo = 0, hi = len;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (k[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo < len && k[lo] == x;
}

__device__ __forceinline__ int64_t lower_key(const uint64_t* k, int64_t lo, int64_t hi, uint64_t x) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (k[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// effective deletion: first occurrence, present in E_{t-1}, not re-inserted
__global__ void k_flag_del(const uint64_t* __restrict__ dk, int64_t nd, const uint64_t* __restrict__ ik, int64_t ni,
                           const int64_t* __restrict__ oo, const int32_t* __restrict__ od,
                           const int32_t* __restrict__ oc, int bits, uint8_t* __restrict__ f) {
  uint64_t mask = (1ull << bits) - 1;
  GRID_STRIDE(i, nd) {
    uint64_t k = dk[i];
    bool e = k != DROP && (i == 0 || dk[i - 1] != k);
    if (e) {
      int32_t u = (int32_t)(k >> bits), v = (int32_t)(k & mask);
      e = in_row(oc, oo[u], od[u], v) && !key_in(ik, ni, k);
    }
    f[i] = e;
  }
}

// effective insertion: first occurrence, absent from E_{t-1}
__global__ void k_flag_ins(const uint64_t* __restrict__ ik, int64_t ni, const int64_t* __restrict__ oo,
                           const int32_t* __restrict__ od, const int32_t* __restrict__ oc, int bits,
                           uint8_t* __restrict__ f) {
  uint64_t mask = (1ull << bits) - 1;
  GRID_STRIDE(i, ni) {
    uint64_t k = ik[i];
    bool e = k != DROP && (i == 0 || ik[i - 1] != k);
    if (e) {
      int32_t u = (int32_t)(k >> bits), v = (int32_t)(k & mask);
      e = !in_row(oc, oo[u], od[u], v);
    }
    f[i] = e;
  }
}

constexpr int32_t REPACK_SHORT = 64;     // rows of at most this degree are rewritten by one thread
constexpr int32_t REPACK_HUB = 16384;    // rows above this degree are spread over many blocks
constexpr int64_t REPACK_CHUNK = 8192;   // elements of a hub row per block

// repack of a direction, pass 1: per row the new degree and the new capacity:
// round4(degree) + 8 slots of slack, a quarter of the degree more for a row
// that received insertions (rows that grew tend to grow again -- a hub of a
// temporal stream -- and geometric slack makes their repacks rare), an eighth
// more for every row of degree >= 64 once the direction has been repacked
// before (the graph keeps growing), and never less than the row had
// (also each row's first deletion and insertion, dstart / istart[0..n], and
// the list of rows above REPACK_HUB with their count and largest degree in
// hinfo[0..1], for pass 2)
__global__ void k_repack_plan(const int64_t* __restrict__ off, const int32_t* __restrict__ deg, int32_t n,
                              const uint64_t* __restrict__ dl, int64_t nd, const uint64_t* __restrict__ il, int64_t ni,
                              int bits, bool growing, int32_t* __restrict__ newdeg, int64_t* __restrict__ cap,
                              int64_t* __restrict__ dstart, int64_t* __restrict__ istart, int32_t* __restrict__ hubs,
                              int32_t* __restrict__ hinfo) {
  GRID_STRIDE(r, n) {
    const int32_t od = deg[r];
    const int slot = warp_append(hinfo, od > REPACK_HUB);
    if (od > REPACK_HUB) {
      hubs[slot] = (int32_t)r;
      atomicMax(hinfo + 1, od);
    }
    const uint64_t rk = (uint64_t)r << bits, rk1 = (uint64_t)(r + 1) << bits;
    const int64_t d0 = lower_key(dl, 0, nd, rk), d1 = lower_key(dl, d0, nd, rk1);
    const int64_t i0 = lower_key(il, 0, ni, rk), i1 = lower_key(il, i0, ni, rk1);
    dstart[r] = d0;
    istart[r] = i0;
    if (r == n - 1) {
      dstart[n] = nd;
      istart[n] = ni;
    }
    const int64_t d = deg[r] - (d1 - d0) + (i1 - i0);
    newdeg[r] = (int32_t)d;
    const int64_t extra = i1 > i0 ? round4(d >> 2) : (growing && d >= 64 ? round4(d >> 3) : 0);
    const int64_t want = round4(d) + 8 + extra, had = off[r + 1] - off[r];
    cap[r] = want > had ? want : had;
  }
}

// pass 2 for the rows longer than REPACK_SHORT: the surviving old elements
// and the insertions merged into the new column array (both are sorted, so
// each element's output position is its rank: survivors x -> i - #deletions
// below x + #insertions below x, insertion y -> k + #old below y - #deletions
// below y), then the padding slots get the sentinel.  part / nparts: this
// call's share of the row -- elements [part * chunk, (part + 1) * chunk) and
// the same share of its insertions and of its padding -- worked by `step`
// threads from t0.
__device__ __forceinline__ void repack_row_part(int64_t r, int64_t part, int64_t nparts, int64_t chunk, int64_t t0,
                                                int64_t step, const int64_t* __restrict__ off,
                                                const int32_t* __restrict__ deg, const int32_t* __restrict__ col,
                                                int32_t n, const uint64_t* __restrict__ dl,
                                                const uint64_t* __restrict__ il, const int64_t* __restrict__ dstart,
                                                const int64_t* __restrict__ istart, int bits,
                                                const int64_t* __restrict__ noff, const int32_t* __restrict__ ndeg,
                                                int32_t* __restrict__ ncol) {
  const uint64_t mask = (1ull << bits) - 1;
  const int64_t dg = deg[r];
  const uint64_t rk = (uint64_t)r << bits;
  const int64_t d0 = dstart[r], d1 = dstart[r + 1];
  const int64_t i0 = istart[r], i1 = istart[r + 1];
  const int64_t base = off[r], nbase = noff[r];
  const int32_t* row = col + base;
  const int64_t x1 = min(dg, (part + 1) * chunk);
  for (int64_t x = part * chunk + t0; x < x1; x += step) {
    const int32_t v = row[x];
    const uint64_t key = rk | (uint64_t)v;
    const int64_t dlt = lower_key(dl, d0, d1, key);
    if (dlt < d1 && dl[dlt] == key) continue;   // deleted
    ncol[nbase + x - (dlt - d0) + (lower_key(il, i0, i1, key) - i0)] = v;
  }
  const int64_t ish = cdiv(i1 - i0, nparts);
  const int64_t k1 = min(i1, i0 + (part + 1) * ish);
  for (int64_t k = i0 + part * ish + t0; k < k1; k += step) {
    const int32_t y = (int32_t)(il[k] & mask);
    int64_t a = 0, b = dg;   // old elements below y
    while (a < b) {
      const int64_t mid = (a + b) >> 1;
      if (row[mid] < y) a = mid + 1;
      else b = mid;
    }
    ncol[nbase + (k - i0) + a - (lower_key(dl, d0, d1, rk | (uint64_t)y) - d0)] = y;
  }
  const int64_t f0 = ndeg[r], f1 = noff[r + 1] - nbase;
  const int64_t fsh = cdiv(f1 - f0, nparts);
  const int64_t e1 = min(f1, f0 + (part + 1) * fsh);
  for (int64_t x = f0 + part * fsh + t0; x < e1; x += step) ncol[nbase + x] = n;
}

// rows of degree in (REPACK_SHORT, REPACK_HUB], one warp per row
__global__ void k_repack_rows(const int64_t* __restrict__ off, const int32_t* __restrict__ deg,
                              const int32_t* __restrict__ col, int32_t n, const uint64_t* __restrict__ dl,
                              const uint64_t* __restrict__ il, const int64_t* __restrict__ dstart,
                              const int64_t* __restrict__ istart, int bits, const int64_t* __restrict__ noff,
                              const int32_t* __restrict__ ndeg, int32_t* __restrict__ ncol) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; r < n; r += nw) {
    const int64_t dg = deg[r];
    if (dg <= REPACK_SHORT || dg > REPACK_HUB) continue;   // k_repack_short / k_repack_hub
    repack_row_part(r, 0, 1, dg, lane, 32, off, deg, col, n, dl, il, dstart, istart, bits, noff, ndeg, ncol);
  }
}

// rows of degree above REPACK_HUB (listed by k_repack_plan): block (x, y)
// works share x of hub row hubs[y], REPACK_CHUNK elements each, so a row of
// a million edges is spread over the grid instead of one warp
__global__ void k_repack_hub(const int32_t* __restrict__ hubs, const int64_t* __restrict__ off,
                             const int32_t* __restrict__ deg, const int32_t* __restrict__ col, int32_t n,
                             const uint64_t* __restrict__ dl, const uint64_t* __restrict__ il,
                             const int64_t* __restrict__ dstart, const int64_t* __restrict__ istart, int bits,
                             const int64_t* __restrict__ noff, const int32_t* __restrict__ ndeg,
                             int32_t* __restrict__ ncol) {
  const int64_t r = hubs[blockIdx.y];
  const int64_t nparts = cdiv((int64_t)deg[r], REPACK_CHUNK);
  if ((int64_t)blockIdx.x >= nparts) return;
  repack_row_part(r, blockIdx.x, nparts, REPACK_CHUNK, threadIdx.x, blockDim.x, off, deg, col, n, dl, il, dstart,
                  istart, bits, noff, ndeg, ncol);
}

// pass 2 for the short rows (degree <= REPACK_SHORT), one thread per row: an
// untouched row is copied as whole quads (both offsets are multiples of four
// slots, so the copies are aligned 16-byte moves), a touched one is merged
// element by element (old elements ascending, deletions skipped, insertions
// placed in order: the effective deletions are present and the effective
// insertions absent, so the merge never meets an equal pair).  The rest of the
// new capacity gets the sentinel.  Longer rows are left to k_repack_rows.
__global__ void k_repack_short(const int64_t* __restrict__ off, const int32_t* __restrict__ deg,
                               const int32_t* __restrict__ col, int32_t n, const uint64_t* __restrict__ dl,
                               const uint64_t* __restrict__ il, const int64_t* __restrict__ dstart,
                               const int64_t* __restrict__ istart, int bits, const int64_t* __restrict__ noff,
                               int32_t* __restrict__ ncol) {
  const uint64_t mask = (1ull << bits) - 1;
  GRID_STRIDE(r, n) {
    const int32_t dg = deg[r];
    if (dg > REPACK_SHORT) continue;
    const int64_t d0 = dstart[r], d1 = dstart[r + 1], i0 = istart[r], i1 = istart[r + 1];
    const int32_t* row = col + off[r];
    int32_t* out = ncol + noff[r];
    const int64_t ncap = noff[r + 1] - noff[r];
    int64_t o = 0;
    if (d0 == d1 && i0 == i1) {
      const int64_t q = round4(dg);   // the last quad's slack slots already hold the sentinel
      for (int64_t k = 0; k < q; k += 4)
        *reinterpret_cast<int4*>(out + k) = *reinterpret_cast<const int4*>(row + k);
      o = q;
    } else {
      int64_t di = d0, ii = i0;
      for (int32_t x = 0; x < dg; x++) {
        const int32_t v = row[x];
        while (ii < i1 && (int32_t)(il[ii] & mask) < v) out[o++] = (int32_t)(il[ii++] & mask);
        while (di < d1 && (int32_t)(dl[di] & mask) < v) di++;
        if (di < d1 && (int32_t)(dl[di] & mask) == v) {
          di++;
          continue;
        }
        out[o++] = v;
      }
      while (ii < i1) out[o++] = (int32_t)(il[ii++] & mask);
    }
    for (; o < ncap; o++) out[o] = n;
  }
}

// ------------------------------------------------------------------ host

// a direction whose new rows do not fit their capacity is rebuilt with fresh
// slack: new degrees and capacities, their prefix as the new offsets, and the
// rows merged straight into a new column array (no sort: the old rows and the
// insertions are both sorted)
static int repack_direction(Graph* g, Csr* c, const uint64_t* dl, int64_t nd, const uint64_t* il, int64_t ni) {
  cudaStream_t s = g->stream;
  const int bits = g->id_bits;
  const int32_t n = g->n;
  int32_t* ndeg = nullptr;
  int64_t *cap = nullptr, *noff = nullptr, *scr = nullptr, *dstart = nullptr, *istart = nullptr;
  int32_t *ncol = nullptr, *hubs = nullptr, *hinfo = nullptr;
  auto release = [&] {
    cudaFree(ndeg);
    cudaFree(cap);
    cudaFree(noff);
    cudaFree(scr);
    cudaFree(dstart);
    cudaFree(istart);
    cudaFree(hubs);
    cudaFree(hinfo);
  };
  // rows above REPACK_HUB, each holding more than REPACK_HUB of the old edges
  const int64_t hub_cap = std::min<int64_t>(n, c->cap / REPACK_HUB + 1);
  cudaError_t e;
  if ((e = dev_malloc(&ndeg, sizeof(int32_t) * n)) != cudaSuccess ||
      (e = dev_malloc(&cap, sizeof(int64_t) * (n + 1))) != cudaSuccess ||
      (e = dev_malloc(&noff, sizeof(int64_t) * (n + 1))) != cudaSuccess ||
      (e = dev_malloc(&scr, sizeof(int64_t) * scan_tmp_elems(n))) != cudaSuccess ||
      (e = dev_malloc(&dstart, sizeof(int64_t) * (n + 1))) != cudaSuccess ||
      (e = dev_malloc(&istart, sizeof(int64_t) * (n + 1))) != cudaSuccess ||
      (e = dev_malloc(&hubs, sizeof(int32_t) * hub_cap)) != cudaSuccess ||
      (e = dev_malloc(&hinfo, sizeof(int32_t) * 2)) != cudaSuccess ||
      (e = cudaMemsetAsync(hinfo, 0, sizeof(int32_t) * 2, s)) != cudaSuccess) {
    release();
    return cuda_fail(g, e, "cudaMalloc(repack)");
  }
  note_launch(); k_repack_plan<<<grid_for(n, 256), 256, 0, s>>>(c->off, c->deg, n, dl, nd, il, ni, bits, c->repacks > 0,
                                                                 ndeg, cap, dstart, istart, hubs, hinfo);
  e = scan_excl<int64_t>(cap, noff, n, scr, s);
  int64_t total = 0;
  int32_t hinfo_h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&total, noff + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hinfo_h, hinfo, sizeof(hinfo_h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && (hinfo_h[0] < 0 || hinfo_h[0] > hub_cap || hinfo_h[0] > 65535)) e = cudaErrorUnknown;
  if (e == cudaSuccess) e = dev_malloc(&ncol, sizeof(int32_t) * (size_t)total);
  if (e != cudaSuccess) {
    release();
    return cuda_fail(g, e, "repack");
  }
  note_launch(); k_repack_short<<<grid_for(n, 256), 256, 0, s>>>(c->off, c->deg, c->col, n, dl, il, dstart, istart,
                                                                  bits, noff, ncol);
  note_launch(); k_repack_rows<<<num_sms() * 16, 256, 0, s>>>(c->off, c->deg, c->col, n, dl, il, dstart, istart, bits,
                                                              noff, ndeg, ncol);
  if (hinfo_h[0] > 0) {
    const dim3 hgrid((unsigned)cdiv(hinfo_h[1], REPACK_CHUNK), (unsigned)hinfo_h[0]);
    note_launch(); k_repack_hub<<<hgrid, 256, 0, s>>>(hubs, c->off, c->deg, c->col, n, dl, il, dstart, istart, bits, noff,
                                                       ndeg, ncol);
  }
  e = cudaMemcpyAsync(c->off, noff, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(c->deg, ndeg, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  release();
  if (e != cudaSuccess) {
    cudaFree(ncol);
    return cuda_fail(g, e, "repack");
  }
  // the new column array replaces the old one in the graph's allocations
  bool owned = false;
  for (auto& p : g->allocs)
    if (p == c->col) {
      cudaFree(p);
      p = ncol;
      owned = true;
    }
  if (!owned) g->allocs.push_back(ncol);
  c->col = ncol;
  c->cap = total;
  c->repacks++;
  return OK;
}

// ------------------------------------------------------------------ editing rows in place
//
// Touched rows of both directions with their plans, rewritten by these kernels:
//   k_edit_short  rows of at most EDIT_SHORT slots, eight lanes per row, the
//                 row in registers;
//   k_edit_long   the others in chunks of RW_CH slots, one warp per chunk
//                 staged in shared memory; a row of several chunks is copied to
//                 scratch first (k_edit_copy), because its chunks move into one
//                 another's places; chunks that take more insertions than they
//                 have slots go to its first blocks (edit_crowd).
// A survivor x goes to x - (deletions below it) + (insertions below it), an
// insertion to its rank among the insertions + old elements below it -
// deletions below it.  A chunk looks only at the changes that fall into it:
// held one per lane when they are few, else counted into the places where they
// take effect and summed over the chunk (a prefix sum per 32 elements), so an
// element costs no search.  Bound by reading and writing the rows: 2.7M
// changes of a graph of 271M edges touch rows that hold most of them, about
// 2 GB per direction.  Before, a warp searched both lists of the row in global
// memory for every element: 5.7 ms per direction there, with a scratch copy of
// every touched row.
constexpr int RW_CH = 1024;         // slots of a chunk
constexpr int EDIT_SHORT = 64;      // rows of at most this many slots: eight lanes
constexpr int EDIT_FEW = 8;         // changes of a chunk compared one by one

}  // namespace dfpr

struct dfpr::EditStatus {
  int32_t n_del, n_ins;   // effective deletions / insertions
  int32_t bad;            // an id out of range (nothing was changed)
  // per direction (out 0, in 1): touched rows, those of more than EDIT_SHORT
  // slots, their chunks, and the scratch chunks of rows of several; the device
  // leaves the direction unchanged (skip), because rows overflow (ovf) or the
  // scratch is too small (need)
  int32_t nr[2], nlong[2], chunks[2], scratch[2], skip[2], ovf[2], need[2];
};

// device arrays of one batch's edit, in one scratch buffer
struct dfpr::EditBufs {
  uint64_t *dl[2], *il[2];   // Delta-, Delta+ sorted by (src, dst) and by (dst, src)
  int32_t* rows[2];
  int4* plan[2];             // per touched row: its deletions [x, y) and insertions [z, w)
  int32_t* od[2];            // its degree before the batch
  // rows of more than EDIT_SHORT slots: index into rows, chunks and scratch
  // chunks before
  int32_t *lrow[2], *lpre[2], *lsc[2];
  EditStatus* st;
  EditStatus* st_h;          // small batches: the pinned host copy the ingest writes
  uint64_t* key;             // small batches: packed (src, dst, insertion, present)
};

namespace dfpr {

struct EditArgs {
  const int64_t* off[2];
  int32_t* deg[2];
  int32_t* col[2];
  int32_t* S[2];          // scratch: chunk c at c x RW_CH
  int32_t sent;
  const double* R;        // ranks, or null: no contributions to refresh
  long long* C;
  const double* tab_sc;
  int dirs;               // bit d: work on direction d
};

// the long row that chunk c belongs to
__device__ __forceinline__ int long_row(const int32_t* pre, int nlong, int c) {
  int lo = 0, hi = nlong - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// one warp: the first `len` (at most RW_CH) elements of src, a row position
// that is a multiple of four, to dst, in whole quads (a row's slots are a
// multiple of four), every load of a lane before its stores
__device__ __forceinline__ void copy_chunk(const int32_t* src, int32_t len, int32_t* dst) {
  const int lane = threadIdx.x & 31;
  int4 v[RW_CH / 128];
#pragma unroll
  for (int k = 0; k < RW_CH / 128; k++) {
    const int q = k * 32 + lane;
    if (4 * q < len) v[k] = reinterpret_cast<const int4*>(src)[q];
  }
#pragma unroll
  for (int k = 0; k < RW_CH / 128; k++) {
    const int q = k * 32 + lane;
    if (4 * q < len) reinterpret_cast<int4*>(dst)[q] = v[k];
  }
}

__global__ void __launch_bounds__(256) k_edit_copy(const __grid_constant__ EditBufs B, const __grid_constant__ EditArgs p) {
  const EditStatus& st = *B.st;
  const int nw = (gridDim.x * blockDim.x) >> 5, w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int d = 0; d < 2; d++) {
    if (!((p.dirs >> d) & 1) || st.skip[d] || st.scratch[d] == 0) continue;
    const int nc = st.chunks[d];
    for (int c = w0; c < nc; c += nw) {
      const int l = long_row(B.lpre[d], st.nlong[d], c);
      if (B.lpre[d][l + 1] - B.lpre[d][l] == 1) continue;   // edited straight from shared memory
      const int part = c - B.lpre[d][l], j = B.lrow[d][l];
      const int32_t x0 = part * RW_CH;
      copy_chunk(p.col[d] + p.off[d][B.rows[d][j]] + x0, min(B.od[d][j] - x0, RW_CH),
                 p.S[d] + (int64_t)(B.lsc[d][l] + part) * RW_CH);
    }
  }
}

__device__ __forceinline__ int32_t lower_i32(const int32_t* a, int32_t lo, int32_t hi, int32_t x) {
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// the row's new degree, and (out-rows) its source's contribution with it
__device__ __forceinline__ void finish_row(const EditArgs& p, int d, int32_t r, int32_t d_new) {
  p.deg[d][r] = d_new;
  if (d == 0 && p.R) {
    const double sc = d_new < TAB ? p.tab_sc[d_new] : FIX_ONE / (double)d_new;
    p.C[r] = __double2ll_rn(p.R[r] * sc);
  }
}

__global__ void __launch_bounds__(256) k_edit_short(const __grid_constant__ EditBufs B, const __grid_constant__ EditArgs p,
                                                    int bits) {
  const EditStatus& st = *B.st;
  const int lane = threadIdx.x & 31, l = lane & 7;
  const unsigned grp = 0xffu << (lane & 24);   // the eight lanes of this row
  const uint64_t mask = (1ull << bits) - 1;
  const int e0 = (p.dirs & 1) && !st.skip[0] ? st.nr[0] : 0, e1 = e0 + ((p.dirs & 2) && !st.skip[1] ? st.nr[1] : 0);
  const int stride = (gridDim.x * blockDim.x) >> 3;
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 3; w < e1; w += stride) {
    const int d = w >= e0 ? 1 : 0, j = w - (d ? e0 : 0);
    const int32_t r = B.rows[d][j], d_old = B.od[d][j];
    const int4 pl = B.plan[d][j];
    const int32_t d_new = d_old - (pl.y - pl.x) + (pl.w - pl.z);
    const int32_t len = (int32_t)round4(d_old > d_new ? d_old : d_new);
    if (len > EDIT_SHORT) continue;
    const int64_t base = p.off[d][r];
    const int32_t cap = (int32_t)min(p.off[d][r + 1] - base, (int64_t)INT32_MAX);
    int32_t* const row = p.col[d] + base;
    int32_t v[8];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      int4 q = make_int4(0, 0, 0, 0);
      if (8 * l + 4 * h < d_old) q = reinterpret_cast<const int4*>(row)[2 * l + h];
      v[4 * h] = q.x;
      v[4 * h + 1] = q.y;
      v[4 * h + 2] = q.z;
      v[4 * h + 3] = q.w;
    }
    int pos[8];
    unsigned keep = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) {
      pos[e] = 8 * l + e;
      if (pos[e] < d_old) keep |= 1u << e;
    }
    const unsigned old = keep;
    for (int k = pl.x; k < pl.y; k++) {
      const int32_t y = (int32_t)(B.dl[d][k] & mask);
#pragma unroll
      for (int e = 0; e < 8; e++) {
        pos[e] -= y < v[e];
        if (y == v[e]) keep &= ~(1u << e);
      }
    }
    __syncwarp(grp);   // every lane holds its elements before any is overwritten
    for (int k = pl.z; k < pl.w; k++) {
      const int32_t y = (int32_t)(B.il[d][k] & mask);
      int below = 0;
#pragma unroll
      for (int e = 0; e < 8; e++) {
        pos[e] += y < v[e];
        below += ((old >> e) & 1u) && v[e] < y ? 1 : 0;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) below += __shfl_xor_sync(grp, below, o);
      if (((k - pl.z) & 7) == l) {
        for (int i = pl.x; i < pl.y; i++) below -= (int32_t)(B.dl[d][i] & mask) < y;
        const int at = k - pl.z + below;
        if (at >= 0 && at < cap) row[at] = y;
      }
    }
#pragma unroll
    for (int e = 0; e < 8; e++) {
      const int x = 8 * l + e;
      if (((keep >> e) & 1u) && pos[e] != x && pos[e] >= 0 && pos[e] < cap) row[pos[e]] = v[e];
      if (x >= d_new && x < len && x < cap) row[x] = p.sent;
    }
    if (l == 0) finish_row(p, d, r, d_new);
  }
}

constexpr int EDIT_WARPS = 4;   // warps of a k_edit_long block

// Crowded chunks: those with more insertions than slots, because the batch
// refills a row that was emptied, or puts new ids behind a row's last one.  Work
// is shared out by insertions, 1024 of the whole sorted list to a warp, not by
// chunks of the old rows: with one warp per gap 10^6 insertions behind a hub's
// last element took 17.7 ms per batch (now 1.42), 10^5 1.53 (0.61).  A crowded chunk holds
// more insertions than a share, so the ones in a share are those of the chunk of
// its first and of the chunk of its last insertion.  The warp
//   - places them, each by searches between the places of the share's ends;
//   - moves the survivors of the chunk whose insertions begin in its share: an
//     element finds the changes below it by searches, the first of each 32 among
//     all of the chunk's, the others between two of those.
// The first blocks of k_edit_long, only for batches of more than 1024 insertions:
// nothing here reads what the others write, and a launch of its own cost a batch
// without crowded chunks 5 to 9 us.  Bound by the latency of the searches.

// the insertions [ia, ib) that fall into one chunk of a row, and what the row is
struct CrowdChunk {
  int32_t ch = 0, ia = 0, ib = 0;   // ia == ib: not crowded
  int32_t r = 0, d_old = 0, cap = 0;
  int4 pl = make_int4(0, 0, 0, 0);
  const int32_t* old = nullptr;
  int32_t* row = nullptr;
};

// the crowded chunk that insertion k of direction d belongs to, if it does
__device__ __forceinline__ CrowdChunk crowd_chunk(const EditBufs& B, const EditArgs& p, const EditStatus& st, int d,
                                                  int bits, int64_t k) {
  const uint64_t* il = B.il[d];
  const uint64_t key = il[k];
  CrowdChunk q;
  q.r = (int32_t)(key >> bits);
  const int j = lower_i32(B.rows[d], 0, st.nr[d], q.r);
  q.pl = B.plan[d][j];
  if (q.pl.w - q.pl.z <= RW_CH) return q;   // (more: a row of several chunks, so in the scratch)
  q.d_old = B.od[d][j];
  q.old = p.S[d] + (int64_t)B.lsc[d][lower_i32(B.lrow[d], 0, st.nlong[d], j)] * RW_CH;
  const int64_t base = p.off[d][q.r];
  q.cap = (int32_t)min(p.off[d][q.r + 1] - base, (int64_t)INT32_MAX);
  q.row = p.col[d] + base;
  // a chunk's insertions: those above the element before it and below its last
  // one (the last chunk: all that are left)
  const uint64_t rk = (uint64_t)q.r << bits, mask = (1ull << bits) - 1;
  q.ch = min(lower_i32(q.old, 0, q.d_old, (int32_t)(key & mask)), q.d_old - 1) / RW_CH;
  const int32_t x0 = q.ch * RW_CH;
  const int ia = x0 > 0 ? (int)lower_key(il, q.pl.z, q.pl.w, rk | (uint64_t)q.old[x0 - 1]) : q.pl.z;
  const int ib = x0 + (int64_t)RW_CH < q.d_old ? (int)lower_key(il, ia, q.pl.w, rk | (uint64_t)q.old[x0 + RW_CH - 1])
                                               : q.pl.w;
  if (ib - ia > RW_CH) {
    q.ia = ia;
    q.ib = ib;
  }
  return q;
}

// warps w0, w0 + nw, ... of the shares of both directions
__device__ __forceinline__ void edit_crowd(const EditBufs& B, const EditArgs& p, int bits, int w0, int nw) {
  const EditStatus& st = *B.st;
  const int lane = threadIdx.x & 31;
  const uint64_t mask = (1ull << bits) - 1;
  const int shares = (int)cdiv(st.n_ins, RW_CH);
  const int e0 = (p.dirs & 1) && !st.skip[0] ? shares : 0, e1 = e0 + ((p.dirs & 2) && !st.skip[1] ? shares : 0);
  for (int w = w0; w < e1; w += nw) {
    const int d = w >= e0 ? 1 : 0;
    const int64_t ka = (int64_t)(w - (d ? e0 : 0)) * RW_CH, kb = min((int64_t)st.n_ins, ka + RW_CH);
    const uint64_t *dl = B.dl[d], *il = B.il[d];
    for (int end = 0; end < 2; end++) {
      const CrowdChunk q = crowd_chunk(B, p, st, d, bits, end ? kb - 1 : ka);
      if (q.ia == q.ib || (end && q.ia <= ka)) continue;   // (the second time: the chunk seen first)
      const uint64_t rk = (uint64_t)q.r << bits;
      const int64_t k0 = max(ka, (int64_t)q.ia), k1 = min(kb, (int64_t)q.ib);
      {
        const uint64_t at_end = il[(lane & 1) ? k1 - 1 : k0];
        const int32_t pa = lower_i32(q.old, 0, q.d_old, (int32_t)(at_end & mask));
        const int32_t pd = (int32_t)lower_key(dl, q.pl.x, q.pl.y, at_end);
        const int32_t a0 = __shfl_sync(0xffffffffu, pa, 0), a1 = __shfl_sync(0xffffffffu, pa, 1);
        const int32_t b0 = __shfl_sync(0xffffffffu, pd, 0), b1 = __shfl_sync(0xffffffffu, pd, 1);
        for (int64_t k = k0 + lane; k < k1; k += 32) {
          const uint64_t key = il[k];
          const int32_t at = (int32_t)(k - q.pl.z) + lower_i32(q.old, a0, a1, (int32_t)(key & mask)) -
                             ((int32_t)lower_key(dl, b0, b1, key) - q.pl.x);
          if (at >= 0 && at < q.cap) q.row[at] = (int32_t)(key & mask);
        }
      }
      __syncwarp();
      if (q.ia < ka) continue;   // its survivors: the warp of the share before
      const int32_t x0 = q.ch * RW_CH, no = min(q.d_old - x0, RW_CH);
      const int da = (int)lower_key(dl, q.pl.x, q.pl.y, rk | (uint64_t)q.old[x0]);
      const int db = (int)lower_key(dl, da, q.pl.y, (rk | (uint64_t)q.old[x0 + no - 1]) + 1);
      const bool any = lane * 32 < no;
      const uint64_t head = any ? rk | (uint64_t)q.old[x0 + lane * 32] : 0;
      const int fi = any ? (int)lower_key(il, q.ia, q.ib, head) : q.ib, fd = any ? (int)lower_key(dl, da, db, head) : db;
      for (int32_t b = 0; b < no; b += 32) {
        const int g = b >> 5, h = g < 31 ? g + 1 : 31;
        const int i0 = __shfl_sync(0xffffffffu, fi, g), d0 = __shfl_sync(0xffffffffu, fd, g);
        const int ni = __shfl_sync(0xffffffffu, fi, h), nd = __shfl_sync(0xffffffffu, fd, h);
        const int i1 = g < 31 ? ni : q.ib, d1 = g < 31 ? nd : db;
        if (b + lane < no) {
          const int32_t x = x0 + b + lane, v = q.old[x];
          const uint64_t key = rk | (uint64_t)v;
          const int ki = (int)lower_key(il, i0, i1, key), kd = (int)lower_key(dl, d0, d1, key);
          const int32_t at = x - (kd - q.pl.x) + (ki - q.pl.z);
          if (!(kd < d1 && dl[kd] == key) && at != x && at >= 0 && at < q.cap) q.row[at] = v;
        }
      }
    }
  }
}

__global__ void __launch_bounds__(EDIT_WARPS * 32) k_edit_long(const __grid_constant__ EditBufs B,
                                                               const __grid_constant__ EditArgs p, int bits,
                                                               int crowd_blocks) {
  if ((int)blockIdx.x < crowd_blocks) {
    edit_crowd(B, p, bits, blockIdx.x * EDIT_WARPS + (threadIdx.x >> 5), crowd_blocks * EDIT_WARPS);
    return;
  }
  __shared__ __align__(16) int32_t stage[EDIT_WARPS][RW_CH];
  __shared__ int32_t delta[EDIT_WARPS][RW_CH + 1];     // edit_marks.cuh: change of the shift at an element
  __shared__ uint32_t gone[EDIT_WARPS][RW_CH / 32];    // and whether it is deleted
  const EditStatus& st = *B.st;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x - crowd_blocks) * EDIT_WARPS;
  const uint64_t mask = (1ull << bits) - 1;
  int32_t* const T = stage[threadIdx.x >> 5];
  int32_t* const D = delta[threadIdx.x >> 5];
  uint32_t* const dead = gone[threadIdx.x >> 5];
  const int e0 = (p.dirs & 1) && !st.skip[0] ? st.chunks[0] : 0;
  const int e1 = e0 + ((p.dirs & 2) && !st.skip[1] ? st.chunks[1] : 0);
  for (int w = (blockIdx.x - crowd_blocks) * EDIT_WARPS + (threadIdx.x >> 5); w < e1; w += nw) {
    const int d = w >= e0 ? 1 : 0, c = w - (d ? e0 : 0);
    const int li = long_row(B.lpre[d], st.nlong[d], c);
    const int j = B.lrow[d][li], part = c - B.lpre[d][li];
    const bool one = B.lpre[d][li + 1] - B.lpre[d][li] == 1;
    const int32_t r = B.rows[d][j], d_old = B.od[d][j];
    const int4 pl = B.plan[d][j];
    const int nd = pl.y - pl.x, ni = pl.w - pl.z;
    const int32_t d_new = d_old - nd + ni;
    const int32_t len = (int32_t)round4(d_old > d_new ? d_old : d_new);
    const int64_t base = p.off[d][r];
    const int32_t cap = (int32_t)min(p.off[d][r + 1] - base, (int64_t)INT32_MAX);
    int32_t* const row = p.col[d] + base;
    const int32_t x0 = part * RW_CH, no = max(0, min(d_old - x0, RW_CH));   // old elements of the chunk
    const uint64_t *dl = B.dl[d], *il = B.il[d];
    __syncwarp();
    copy_chunk(one ? row : p.S[d] + (int64_t)(B.lsc[d][li] + part) * RW_CH, no, T);
    int32_t before = 0;   // the element before the chunk
    if (part > 0 && no > 0) before = p.S[d][(int64_t)(B.lsc[d][li] + part) * RW_CH - 1];
    __syncwarp();
    // the chunk's changes: deletions [da, db) are those of its elements;
    // insertions [ia, ib) those above the element before it and below its last
    // one (the last chunk with elements: all that are left)
    int da = pl.x, db = pl.y, ia = pl.z, ib = pl.w;
    int32_t mine = 0;
    const bool few = nd + ni <= 32;
    if (few && lane < nd + ni) mine = (int32_t)((lane < nd ? dl[pl.x + lane] : il[pl.z + lane - nd]) & mask);
    if (no == 0) {
      da = db;
      ia = ib;
    } else if (!one) {
      const bool last = x0 + RW_CH >= d_old;
      const int32_t lo = T[0], hi = T[no - 1];
      if (few) {
        const bool del = lane < nd, ins = lane >= nd && lane < nd + ni;
        da = pl.x + __popc(__ballot_sync(0xffffffffu, del && mine < lo));
        db = pl.x + __popc(__ballot_sync(0xffffffffu, del && mine <= hi));
        const int bi = __popc(__ballot_sync(0xffffffffu, ins && part > 0 && mine < before));
        const int ei = __popc(__ballot_sync(0xffffffffu, ins && (last || mine < hi)));
        ia = pl.z + bi;
        ib = pl.z + ei;
      } else {
        const uint64_t rk = (uint64_t)r << bits;
        int at = 0;   // lanes 0 to 3 search one bound each
        if (lane == 0) at = (int)lower_key(dl, pl.x, pl.y, rk | (uint64_t)lo);
        if (lane == 1) at = (int)lower_key(dl, pl.x, pl.y, (rk | (uint64_t)hi) + 1);
        if (lane == 2) at = part > 0 ? (int)lower_key(il, pl.z, pl.w, rk | (uint64_t)before) : pl.z;
        if (lane == 3) at = last ? pl.w : (int)lower_key(il, pl.z, pl.w, rk | (uint64_t)hi);
        da = __shfl_sync(0xffffffffu, at, 0);
        db = __shfl_sync(0xffffffffu, at, 1);
        ia = __shfl_sync(0xffffffffu, at, 2);
        ib = __shfl_sync(0xffffffffu, at, 3);
      }
    }
    const int shift = (ia - pl.z) - (da - pl.x);   // of the chunk's first element
    const int cd = db - da, ci = ib - ia;
    if (ci > RW_CH) {
      // edit_crowd
    } else if (cd + ci <= EDIT_FEW) {
      // one change per lane, compared with every element
      int32_t y = 0;
      if (lane < cd + ci) y = (int32_t)((lane < cd ? dl[da + lane] : il[ia + lane - cd]) & mask);
      for (int32_t b = 0; b < no; b += 32) {
        const int32_t i = b + lane, v = i < no ? T[i] : 0;
        int sh = shift;
        bool dead = false;
        for (int k = 0; k < cd; k++) {
          const int32_t z = __shfl_sync(0xffffffffu, y, k);
          sh -= z < v;
          dead |= z == v;
        }
        for (int k = cd; k < cd + ci; k++) sh += __shfl_sync(0xffffffffu, y, k) < v;
        const int32_t at = x0 + i + sh;
        if (i < no && !dead && sh != 0 && at >= 0 && at < cap) row[at] = v;
      }
      if (lane >= cd && lane < cd + ci) {
        int below = da - pl.x;
        for (int k = 0; k < cd; k++) below += (int32_t)(dl[da + k] & mask) < y;
        const int32_t at = (ia + lane - cd - pl.z) + x0 + lower_i32(T, 0, no, y) - below;
        if (at >= 0 && at < cap) row[at] = y;
      }
    } else {
      for (int32_t i = lane; i <= no; i += 32) D[i] = 0;
      if (lane < RW_CH / 32) dead[lane] = 0u;
      __syncwarp();
      for (int k = da + lane; k < db; k += 32) {
        const int32_t i = lower_i32(T, 0, no, (int32_t)(dl[k] & mask));   // its element (present)
        editmarks::mark_deleted(D, dead, i);
      }
      for (int k = ia + lane; k < ib; k += 32) {
        const int32_t y = (int32_t)(il[k] & mask);
        const int32_t i = lower_i32(T, 0, no, y);
        editmarks::mark_inserted(D, i, 1);
        const int below = (int)(lower_key(dl, da, db, ((uint64_t)r << bits) | (uint64_t)y) - pl.x);
        const int32_t at = (k - pl.z) + x0 + i - below;
        if (at >= 0 && at < cap) row[at] = y;
      }
      __syncwarp();
      int run = shift;
      for (int32_t b = 0; b < no; b += 32) {
        const int32_t i = b + lane;
        int sh = i < no ? D[i] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, sh, o);
          if (lane >= o) sh += y;
        }
        const int all = __shfl_sync(0xffffffffu, sh, 31);
        sh += run;
        run += all;
        const int32_t at = x0 + i + sh;
        if (i < no && !editmarks::is_deleted(dead, i) && sh != 0 && at >= 0 && at < cap) row[at] = T[i];
      }
    }
    for (int32_t x = x0 + lane; x < min(x0 + RW_CH, len); x += 32)
      if (x >= d_new && x < cap) row[x] = p.sent;
    if (part == 0 && lane == 0) finish_row(p, d, r, d_new);
  }
}

// queue the edit of the directions in `dirs`; rows: touched rows of both, at
// most; ins: insertions, at most
static void launch_edit(Graph* g, const EditBufs& B, int32_t* const* S, int dirs, int64_t rows, int64_t ins) {
  cudaStream_t s = g->stream;
  EditArgs p;
  const Csr* c[2] = {&g->out, &g->in};
  for (int d = 0; d < 2; d++) {
    p.off[d] = c[d]->off;
    p.deg[d] = c[d]->deg;
    p.col[d] = c[d]->col;
    p.S[d] = S[d];
  }
  p.sent = g->n;
  p.R = g->has_ranks ? g->R : nullptr;
  p.C = g->C[g->ccur];
  p.tab_sc = g->tab_sc;
  p.dirs = dirs;
  note_launch(); k_edit_copy<<<num_sms() * 4, 256, 0, s>>>(B, p);
  note_launch(); k_edit_short<<<grid_for(8 * rows, 256), 256, 0, s>>>(B, p, g->id_bits);
  const int crowd = ins > RW_CH ? grid_for(2 * cdiv(ins, RW_CH), EDIT_WARPS) : 0;
  note_launch(); k_edit_long<<<crowd + num_sms() * 6, EDIT_WARPS * 32, 0, s>>>(B, p, g->id_bits, crowd);
}

// what a row of `len` slots adds to the lists of long rows: one entry, its
// chunks, and its scratch chunks (20 + 22 + 22 bits: at most SMALL_MAX entries
// here, and a direction holds fewer than 2^31 slots)
__device__ __forceinline__ uint64_t long_counts(int64_t len) {
  if (len <= EDIT_SHORT) return 0;
  const uint64_t c = (uint64_t)cdiv(len, RW_CH);
  return 1ull << 44 | c << 22 | (c > 1 ? c : 0);
}

// ------------------------------------------------------------------ small batches
//
// A batch of at most SMALL_MAX edges costs four launches and one host
// synchronisation (the status read at the end).  It is bound by latency, not
// by bytes: a chain of launches, of dependent loads and of block barriers.
//   k_small_keys    one thread per edge over the whole chip: ids checked,
//                   packed key, and whether the edge is in E_{t-1} (a search of
//                   its out-row, eight ways per step);
//   k_small_ingest  one block per direction, side by side: the keys sorted as
//                   (src, dst) and as (dst, src) in registers (bitonic: strides
//                   within a thread and a warp need no barrier), effective
//                   flags, compaction, touched rows with their edit plans;
// and then the row edit above, both directions at once, with the new degrees
// and the contributions of the sources.
// Device time of a batch: 50 us for 168 edges on a graph of 2^20 vertices, 115
// for 4000 and 145 for 6300 on one of 2.6M (k_small_keys 4 to 8, k_small_ingest
// 9 / 37 / 63).  Before, one block ran both directions in turn with the sort in
// shared memory (53 us at 168 edges, 143 at 1300, 312 at 4000) and five kernels
// per direction followed: 166 us in all for 168 edges, 450 for 4000; above 4096
// edges the path below, 930 us for 6300.
// A direction whose rows overflow their capacity, or whose scratch is too
// small, is left alone by the device and finished by the host.
constexpr int SMALL_MAX = 16384;                // edges of a batch (deletions + insertions)
constexpr int SMALL_THREADS = 1024;
constexpr uint64_t BAD = ~1ull;                  // key of an edge with an id out of range (no packed key: ids are below 2^31)

static size_t small_carve(void* base, int64_t cap, EditBufs* B) {
  Carve c(base);
  B->key = c.take<uint64_t>(cap);
  B->dl[0] = B->il[0] = nullptr;   // the graph's own buffers
  B->dl[1] = c.take<uint64_t>(cap);
  B->il[1] = c.take<uint64_t>(cap);
  for (int d = 0; d < 2; d++) {
    B->rows[d] = c.take<int32_t>(cap);
    B->plan[d] = c.take<int4>(cap);
    B->od[d] = c.take<int32_t>(cap);
    B->lrow[d] = c.take<int32_t>(cap);
    B->lpre[d] = c.take<int32_t>(cap + 1);
    B->lsc[d] = c.take<int32_t>(cap);
  }
  B->st = c.take<EditStatus>(1);
  return c.used;
}

__host__ __device__ __forceinline__ int pow2_at_least(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// whether x is in the sorted row[0..deg): seven pivots per step, their loads
// together, then the last few elements together
__device__ __forceinline__ bool in_sorted_row(const int32_t* __restrict__ row, int32_t deg, int32_t x) {
  int32_t lo = 0, hi = deg;   // the first element >= x is at [lo, hi]
  while (hi - lo > 8) {
    const int32_t s = (hi - lo) >> 3;
    int c = 0;
#pragma unroll
    for (int k = 1; k < 8; k++) c += row[lo + k * s] < x ? 1 : 0;
    const int32_t l2 = c > 0 ? lo + c * s + 1 : lo;
    hi = c < 7 ? lo + (c + 1) * s : hi;
    lo = l2;
  }
  bool found = false;
#pragma unroll
  for (int k = 0; k <= 8; k++) found |= lo + k <= hi && lo + k < deg && row[lo + k] == x;
  return found;
}

__global__ void __launch_bounds__(256) k_small_keys(const int32_t* __restrict__ ds, const int32_t* __restrict__ dd, int nd,
                                                    const int32_t* __restrict__ is, const int32_t* __restrict__ id,
                                                    int ni, int32_t n, int bits, const int32_t* __restrict__ perm,
                                                    const int64_t* __restrict__ oo, const int32_t* __restrict__ od,
                                                    const int32_t* __restrict__ oc, uint64_t* __restrict__ key) {
  GRID_STRIDE(i, nd + ni) {
    const bool del = i < nd;
    const int32_t u = del ? ds[i] : is[i - nd], v = del ? dd[i] : id[i - nd];
    uint64_t k = DROP;   // self-loops are re-added with every batch
    if (u < 0 || u >= n || v < 0 || v >= n) {
      k = BAD;
    } else if (u != v) {
      const int32_t a = perm[u], b = perm[v];
      const bool present = in_sorted_row(oc + oo[a], od[a], b);
      k = (((((uint64_t)a << bits) | (uint64_t)b) << 1 | (del ? 0u : 1u)) << 1) | (present ? 1u : 0u);
    }
    key[i] = k;
  }
}

// ascending bitonic sort of the block's P keys (a power of two, at most
// SMALL_THREADS x E), thread t holding keys [t E, t E + E); x: P keys of shared
// memory
template <int E>
__device__ __forceinline__ void block_sort(uint64_t (&k)[E], int P, uint64_t* x) {
  const int t = threadIdx.x;
  for (int size = 2; size <= P; size <<= 1)
    for (int j = size >> 1; j > 0; j >>= 1) {
      if (j < E) {
#pragma unroll
        for (int jj = E / 2; jj > 0; jj >>= 1)
          if (j == jj) {
#pragma unroll
            for (int e = 0; e < E; e++)
              if ((e & jj) == 0) {
                const bool up = ((t * E + e) & size) == 0;
                const uint64_t a = k[e], b = k[e | jj];
                const bool sw = (a > b) == up;
                k[e] = sw ? b : a;
                k[e | jj] = sw ? a : b;
              }
          }
      } else if (j < 32 * E) {
#pragma unroll
        for (int e = 0; e < E; e++) {
          const int i = t * E + e;
          const uint64_t o = __shfl_xor_sync(0xffffffffu, k[e], j / E);
          const bool low = ((i & j) == 0) == ((i & size) == 0);   // keeps the smaller
          k[e] = (o < k[e]) == low ? o : k[e];
        }
      } else {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; e++) x[e * SMALL_THREADS + t] = k[e];
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; e++) {
          const int i = t * E + e;
          const uint64_t o = x[e * SMALL_THREADS + (t ^ (j / E))];
          const bool low = ((i & j) == 0) == ((i & size) == 0);
          k[e] = (o < k[e]) == low ? o : k[e];
        }
      }
    }
}

// exclusive prefix of one value per thread over the block; *total the sum
__device__ __forceinline__ uint64_t block_excl(uint64_t v, uint64_t* wsum /* 33 */, uint64_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();   // wsum may still be read from the call before
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    uint64_t z = wsum[lane];
    const uint64_t own = z;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, z, o);
      if (lane >= o) z += y;
    }
    wsum[lane] = z - own;
    if (lane == 31) wsum[32] = z;
  }
  __syncthreads();
  *total = wsum[32];
  return wsum[w] + x - v;
}

struct SmallCsr {
  const int64_t* off;
  const int32_t* deg;
  int64_t scap;   // scratch elements for rows longer than a chunk
};

// shared memory: the keys, and per key the deletions before it and the first
// key of each row
template <int E>
constexpr size_t small_smem() {
  return (sizeof(uint64_t) + 2 * sizeof(uint16_t)) * (size_t)(SMALL_THREADS * E + 8);
}

template <int E>
__global__ void __launch_bounds__(SMALL_THREADS, 1)
    k_small_ingest(int N, int bits, const __grid_constant__ SmallCsr out, const __grid_constant__ SmallCsr in,
                   const __grid_constant__ EditBufs B) {
  extern __shared__ uint64_t K[];   // the sorted keys, then the effective changes (row, col, insertion)
  uint16_t* const DP = reinterpret_cast<uint16_t*>(K + SMALL_THREADS * E + 8);
  uint16_t* const RS = DP + SMALL_THREADS * E + 8;
  __shared__ uint64_t wsum[33];
  const int dir = blockIdx.x, t = threadIdx.x;
  const SmallCsr& c = dir == 0 ? out : in;
  const uint64_t mask = (1ull << bits) - 1;
  EditStatus& st = *B.st;
  uint64_t k[E];
  bool bad = false;
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int i = t * E + e;
    k[e] = i < N ? B.key[i] : DROP;
    bad |= k[e] == BAD;
    if (dir == 1 && k[e] != DROP) {
      const uint64_t edge = k[e] >> 2;
      k[e] = (((edge & mask) << bits | edge >> bits) << 2) | (k[e] & 3);
    }
  }
  if (__syncthreads_or(bad)) {
    if (t == 0) {
      st.bad = 1;
      st.nr[dir] = st.nlong[dir] = st.chunks[dir] = st.scratch[dir] = 0;
      st.skip[dir] = 1;
      *(volatile int32_t*)&B.st_h->bad = 1;
    }
    return;
  }
  const int P = pow2_at_least(N);
  block_sort<E>(k, P, K);
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; e++)
    if (t * E + e < P) K[t * E + e] = k[e];
  __syncthreads();
  // effective flags (Sec. 3.2): a deletion is a first occurrence, present in
  // E_{t-1} and not re-inserted; an insertion is a first occurrence absent from
  // E_{t-1}.  Equal edges lie together, deletions first.
  unsigned fd = 0, fi = 0;
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int i = t * E + e;
    const uint64_t x = k[e];
    if (i >= P || x == DROP || (i > 0 && K[i - 1] == x)) continue;
    if (x & 2) {
      if (!(x & 1)) fi |= 1u << e;
    } else if (x & 1) {
      int j = i + 1;
      while (j < P && K[j] == x) j++;
      if (!(j < P && (K[j] >> 1) == ((x >> 1) | 1))) fd |= 1u << e;
    }
  }
  uint64_t tot;
  uint64_t pre = block_excl((uint64_t)__popc(fd) | (uint64_t)__popc(fi) << 32, wsum, &tot);   // (its barriers end the reads of K)
  const int nde = (int)(uint32_t)tot, nie = (int)(tot >> 32), ne = nde + nie;
  {
    int pd = (int)(uint32_t)pre, pi = (int)(pre >> 32);
#pragma unroll
    for (int e = 0; e < E; e++) {
      const bool d = (fd >> e) & 1u, a = (fi >> e) & 1u;
      if (!d && !a) continue;
      K[pd + pi] = k[e] >> 1;
      DP[pd + pi] = (uint16_t)pd;
      if (d) B.dl[dir][pd++] = k[e] >> 2;
      else B.il[dir][pi++] = k[e] >> 2;
    }
  }
  if (t == 0) DP[ne] = (uint16_t)nde;
  __syncthreads();
  // touched rows
  unsigned heads = 0;
#pragma unroll
  for (int e = 0; e < E; e++) {
    const int i = t * E + e;
    if (i < ne && (i == 0 || K[i] >> (bits + 1) != K[i - 1] >> (bits + 1))) heads |= 1u << e;
  }
  pre = block_excl((uint64_t)__popc(heads), wsum, &tot);
  const int nr = (int)tot;
  {
    int j = (int)pre;
#pragma unroll
    for (int e = 0; e < E; e++)
      if ((heads >> e) & 1u) RS[j++] = (uint16_t)(t * E + e);
  }
  if (t == 0) RS[nr] = (uint16_t)ne;
  __syncthreads();
  // their edit plans; rows longer than a chunk are listed with their chunks
  bool ovf = false;
  uint64_t carry = 0;
  for (int j0 = 0; j0 < nr; j0 += SMALL_THREADS) {
    const int j = j0 + t;
    uint64_t longs = 0;
    if (j < nr) {
      const int a = RS[j], b = RS[j + 1];
      const int d0 = DP[a], d1 = DP[b], i0 = a - d0, i1 = b - d1;
      const int32_t r = (int32_t)(K[a] >> (bits + 1));
      const int32_t dg = c.deg[r];
      const int32_t dn = dg - (d1 - d0) + (i1 - i0);
      B.rows[dir][j] = r;
      B.plan[dir][j] = make_int4(d0, d1, i0, i1);
      B.od[dir][j] = dg;
      ovf |= round4(dn) > c.off[r + 1] - c.off[r];
      longs = long_counts(round4(dg > dn ? dg : dn));
    }
    if (__syncthreads_or(longs != 0)) {
      const uint64_t before = carry + block_excl(longs, wsum, &tot);
      if (longs) {
        const int at = (int)(before >> 44);
        B.lrow[dir][at] = j;
        B.lpre[dir][at] = (int32_t)(before >> 22 & 0x3fffff);
        B.lsc[dir][at] = (int32_t)(before & 0x3fffff);
      }
      carry += tot;
    }
  }
  const int any_ovf = __syncthreads_or(ovf);
  if (t == 0) {
    const int nlong = (int)(carry >> 44), chunks = (int)(carry >> 22 & 0x3fffff), scratch = (int)(carry & 0x3fffff);
    st.bad = 0;
    st.n_del = nde;
    st.n_ins = nie;
    st.nr[dir] = nr;
    st.nlong[dir] = nlong;
    st.chunks[dir] = chunks;
    st.scratch[dir] = scratch;
    B.lpre[dir][nlong] = chunks;
    st.ovf[dir] = any_ovf ? 1 : 0;
    st.need[dir] = (int64_t)scratch * RW_CH > c.scap ? 1 : 0;
    st.skip[dir] = st.ovf[dir] | st.need[dir];
    // the same to the host, which a copy engine after the edit would reach
    // about 10 us later
    volatile EditStatus& h = *B.st_h;
    h.n_del = nde;
    h.n_ins = nie;
    h.skip[dir] = st.skip[dir];
    h.ovf[dir] = st.ovf[dir];
    h.scratch[dir] = scratch;
  }
}

// grow-only scratch of one direction's long rows (scratch slot 5: out, 7: in)
static cudaError_t small_staging(Graph* g, int dir, int64_t elems, int32_t** out, int64_t* cap) {
  const int slot = dir == 0 ? 5 : 7;
  void* p;
  cudaError_t e = scratch_get(g, slot, sizeof(int32_t) * (size_t)(elems + 1), &p);
  if (e != cudaSuccess) return e;
  *out = (int32_t*)p;
  *cap = (int64_t)(g->scr[slot].bytes / sizeof(int32_t)) - 1;
  return cudaSuccess;
}

// the list of one side of the effective change with room for `need` keys,
// keeping the keys it holds (a batch that is refused leaves the last one's
// change in place)
static cudaError_t grow_delta(Graph* g, uint64_t** list, int64_t* cap, int64_t used, int64_t need) {
  if (*cap >= need) return cudaSuccess;
  uint64_t* p = nullptr;
  cudaError_t e = dev_malloc(&p, sizeof(uint64_t) * (size_t)(need + 1));
  if (e != cudaSuccess) return e;
  if (used > 0)
    e = cudaMemcpyAsync(p, *list, sizeof(uint64_t) * (size_t)used, cudaMemcpyDeviceToDevice, g->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
  if (e != cudaSuccess) {
    cudaFree(p);
    return e;
  }
  if (*list) cudaFree(*list);
  *list = p;
  *cap = need;
  return cudaSuccess;
}

template <int E>
static cudaError_t launch_ingest(Graph* g, int N, const SmallCsr& out, const SmallCsr& in, const EditBufs& B) {
  int bps;   // (raises the kernel's shared memory limit once)
  cudaError_t e = kernel_occupancy((const void*)k_small_ingest<E>, SMALL_THREADS, small_smem<E>(), &bps);
  if (e != cudaSuccess) return e;
  note_launch();
  k_small_ingest<E><<<2, SMALL_THREADS, small_smem<E>(), g->stream>>>(N, g->id_bits, out, in, B);
  return cudaGetLastError();
}

// phase 1 of a small batch: keys, ingest (which writes the status to the host's
// pinned copy) and row edit, queued on the graph's stream without waiting
static int small_launch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                        const int32_t* id, int64_t ni, SmallApply* A) {
  cudaStream_t s = g->stream;
  const int N = (int)(nd + ni);
  const int64_t cap = std::max(1024, pow2_at_least(N));
  EditBufs B;
  void* bp;
  TRY(scratch_get(g, 6, small_carve(nullptr, cap, &B) + 256, &bp));
  small_carve(bp, cap, &B);
  if (!g->small_h) TRY(cudaMallocHost(&g->small_h, sizeof(EditStatus)));
  B.st_h = (EditStatus*)g->small_h;
  B.st_h->bad = 0;
  TRY(grow_delta(g, &g->dmin, &g->cap_dmin, g->n_dmin, nd));
  TRY(grow_delta(g, &g->dplus, &g->cap_dplus, g->n_dplus, ni));
  B.dl[0] = g->dmin;
  B.il[0] = g->dplus;
  // scratch for at least 64 chunks of long rows per direction; more is handled by growing it
  SmallCsr csr[2];
  for (int d = 0; d < 2; d++) {
    const Csr& c = d == 0 ? g->out : g->in;
    TRY(small_staging(g, d, 65536, &A->S[d], &csr[d].scap));
    csr[d].off = c.off;
    csr[d].deg = c.deg;
  }
  A->B = new (std::nothrow) EditBufs(B);
  if (!A->B) return set_error(g, ENOMEM_, "pr_apply_batch: host memory");
  note_launch();
  k_small_keys<<<grid_for(N, 256), 256, 0, s>>>(ds, dd, (int)nd, is, id, (int)ni, g->n, g->id_bits, g->perm, g->out.off,
                                                g->out.deg, g->out.col, B.key);
  cudaError_t e = N <= SMALL_THREADS       ? launch_ingest<1>(g, N, csr[0], csr[1], B)
                  : N <= 2 * SMALL_THREADS ? launch_ingest<2>(g, N, csr[0], csr[1], B)
                  : N <= 4 * SMALL_THREADS ? launch_ingest<4>(g, N, csr[0], csr[1], B)
                  : N <= 8 * SMALL_THREADS ? launch_ingest<8>(g, N, csr[0], csr[1], B)
                                           : launch_ingest<16>(g, N, csr[0], csr[1], B);
  if (e == cudaSuccess) {
    launch_edit(g, B, A->S, 3, 2 * (int64_t)N, ni);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    delete A->B;
    A->B = nullptr;
    return cuda_fail(g, e, "pr_apply_batch");
  }
  return OK;
}

// phase 2: wait for the status, keep the effective change, and finish on the
// host what the device left (a larger scratch, or a repack)
static int small_complete(Graph* g, SmallApply* A) {
  cudaStream_t s = g->stream;
  const int32_t n = g->n;
  const EditBufs B = *A->B;
  struct Release {
    SmallApply* a;
    ~Release() {
      delete a->B;
      a->B = nullptr;
    }
  } release{A};
  TRY(cudaStreamSynchronize(s));
  g->stage_busy = false;
  const EditStatus h = *(EditStatus*)g->small_h;
  if (h.bad) return set_error(g, ERANGE_, "pr_apply_batch: vertex id out of range");
  const int64_t a = h.n_del, b = h.n_ins;
  g->n_dmin = a;
  g->n_dplus = b;
  if (a + b == 0) return OK;
  bool rep[2] = {false, false};
  for (int dir = 0; dir < 2; dir++) {
    if (!h.skip[dir]) continue;
    Csr* c = dir == 0 ? &g->out : &g->in;
    if (h.ovf[dir]) {
      int rc = repack_direction(g, c, B.dl[dir], a, B.il[dir], b);
      if (rc) return rc;
      rep[dir] = true;
    } else {
      int64_t cap;
      TRY(small_staging(g, dir, (int64_t)h.scratch[dir] * RW_CH, &A->S[dir], &cap));
      TRY(cudaMemsetAsync(&B.st->skip[dir], 0, sizeof(int32_t), s));
      launch_edit(g, B, A->S, 1 << dir, a + b, b);
    }
  }
  if (rep[1]) {
    int rc = refresh_full_tiles(g);
    if (rc) return rc;
  }
  if (rep[0] && g->has_ranks) {
    TRY(cudaMemsetAsync(g->aux, 0, sizeof(uint32_t) * (size_t)(cdiv(n, 32) + 1), s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
    TRY(launch_mark_sources(g->dmin, a, g->dplus, b, g->id_bits, g->aux, g->wl[0], &g->ctl->count[0], s));
    TRY(launch_contrib_list(g->wl[0], &g->ctl->count[0], g->R, g->C[g->ccur], g->out.deg, g->tab_sc, n, s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
  }
  TRY(cudaGetLastError());
  return OK;
}

// the endpoint arrays of a host batch where the device can read them: deletion
// sources and targets, insertion sources and targets, one after another.  A
// small batch's are read once, by k_small_keys, straight from the graph's
// pinned buffer; a larger one's are copied (scratch slot 0).
int stage_host_batch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is, const int32_t* id,
                     int64_t ni, int32_t** out) {
  cudaStream_t s = g->stream;
  const int32_t* src[4] = {ds, dd, is, id};
  const int64_t len[4] = {nd, nd, ni, ni};
  if (nd + ni <= SMALL_MAX) {
    if (!g->stage_h) TRY(cudaMallocHost(&g->stage_h, sizeof(int32_t) * 2 * SMALL_MAX));
    if (g->stage_busy) TRY(cudaDeviceSynchronize());   // the read of a call that failed after it
    int32_t* h = (int32_t*)g->stage_h;
    *out = h;
    g->stage_busy = nd + ni > 0;
    for (int k = 0; k < 4; k++)
      if (len[k]) {
        memcpy(h, src[k], sizeof(int32_t) * (size_t)len[k]);
        h += len[k];
      }
    return OK;
  }
  void* stage;
  TRY(scratch_get(g, 0, sizeof(int32_t) * (size_t)(2 * (nd + ni) + 4) + 1024, &stage));
  int32_t* b = (int32_t*)stage;
  *out = b;
  for (int k = 0; k < 4; k++)
    if (len[k]) {
      TRY(cudaMemcpyAsync(b, src[k], sizeof(int32_t) * (size_t)len[k], cudaMemcpyHostToDevice, s));
      b += len[k];
    }
  return OK;
}

int apply_batch_launch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                       const int32_t* id, int64_t ni, bool validated, SmallApply* pending) {
  const int64_t nk = nd + ni;
  pending->B = nullptr;
  if (nk > 0 && nk <= SMALL_MAX) return small_launch(g, ds, dd, nd, is, id, ni, pending);
  return apply_batch_device(g, ds, dd, nd, is, id, ni, validated);
}

int apply_batch_complete(Graph* g, SmallApply* pending) {
  if (!pending->B) return OK;
  return small_complete(g, pending);
}

// the touched rows' plans (row j of *nrp, zero counts for the rest up to mr):
// changes, old degree, whether the row overflows, and what it adds to the lists
// of long rows: ca entries << 32 | chunks, cb scratch chunks
__global__ void k_edit_plan(const __grid_constant__ EditBufs B, int d, const int32_t* nrp, int64_t mr, int64_t nd,
                            int64_t ni, int bits, const int64_t* __restrict__ off, const int32_t* __restrict__ deg,
                            int64_t* __restrict__ ca, int64_t* __restrict__ cb) {
  const int nr = *nrp;
  const uint64_t *dl = B.dl[d], *il = B.il[d];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    B.st->nr[d] = nr;
    B.st->n_ins = (int32_t)ni;
  }
  GRID_STRIDE(j, mr) {
    int64_t long_chunks = 0, scratch = 0;
    if (j < nr) {
      const int32_t r = B.rows[d][j];
      const uint64_t lo = (uint64_t)r << bits, hi = (uint64_t)(r + 1) << bits;
      const int64_t d0 = lower_key(dl, 0, nd, lo), d1 = lower_key(dl, d0, nd, hi);
      const int64_t i0 = lower_key(il, 0, ni, lo), i1 = lower_key(il, i0, ni, hi);
      const int32_t dg = deg[r];
      const int32_t dn = dg - (int32_t)(d1 - d0) + (int32_t)(i1 - i0);
      B.plan[d][j] = make_int4((int)d0, (int)d1, (int)i0, (int)i1);
      B.od[d][j] = dg;
      if (round4(dn) > off[r + 1] - off[r]) B.st->ovf[d] = 1;
      const int64_t len = round4(dg > dn ? dg : dn);
      if (len > EDIT_SHORT) {
        const int64_t c = cdiv(len, RW_CH);
        long_chunks = (1ll << 32) | c;
        scratch = c > 1 ? c : 0;
      }
    }
    ca[j] = long_chunks;
    cb[j] = scratch;
  }
}

// ca, cb: exclusive prefixes of what k_edit_plan wrote, totals at [mr]
__global__ void k_edit_lists(const __grid_constant__ EditBufs B, int d, int64_t mr, const int64_t* __restrict__ ca,
                             const int64_t* __restrict__ cb) {
  GRID_STRIDE(j, mr) {
    if (ca[j + 1] == ca[j]) continue;
    const int64_t at = ca[j] >> 32;
    B.lrow[d][at] = (int32_t)j;
    B.lpre[d][at] = (int32_t)(uint32_t)ca[j];
    B.lsc[d][at] = (int32_t)cb[j];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    EditStatus& st = *B.st;
    st.nlong[d] = (int32_t)(ca[mr] >> 32);
    st.chunks[d] = (int32_t)(uint32_t)ca[mr];
    st.scratch[d] = (int32_t)cb[mr];
    B.lpre[d][ca[mr] >> 32] = (int32_t)(uint32_t)ca[mr];
    st.skip[d] = st.ovf[d];
  }
}

int apply_batch_device(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                       const int32_t* id, int64_t ni, bool validated) {
  cudaStream_t s = g->stream;
  int bits = g->id_bits;
  int32_t n = g->n;
  int64_t nk = nd + ni;
  if (nk > 0 && nk <= SMALL_MAX) {
    SmallApply A;
    const int rc = small_launch(g, ds, dd, nd, is, id, ni, &A);
    return rc != OK ? rc : small_complete(g, &A);
  }
  size_t need;
  {
    Carve probe(nullptr);
    probe.take<uint64_t>(nd);
    probe.take<uint64_t>(ni);
    probe.take<uint64_t>(nk);
    probe.take<uint8_t>(nk);
    probe.take<char>((int64_t)std::max(radix_tmp_bytes(nk), compact_tmp_bytes(nk)));
    probe.take<unsigned long long>(4);
    need = probe.used + 4096;
  }
  void* base;
  TRY(scratch_get(g, 2, need, &base));
  Carve cv(base);
  uint64_t* dk = cv.take<uint64_t>(nd);
  uint64_t* ik = cv.take<uint64_t>(ni);
  uint64_t* alt = cv.take<uint64_t>(nk);
  uint8_t* flag = cv.take<uint8_t>(nk);
  void* tmp = cv.take<char>((int64_t)std::max(radix_tmp_bytes(nk), compact_tmp_bytes(nk)));
  unsigned long long* small = cv.take<unsigned long long>(4);
  if (!validated && nk) {
    TRY(cudaMemsetAsync(small, 0, sizeof(unsigned long long), s));
    if (nd) { note_launch(); k_validate<<<grid_for(nd, 256), 256, 0, s>>>(ds, dd, nd, n, small); }
    if (ni) { note_launch(); k_validate<<<grid_for(ni, 256), 256, 0, s>>>(is, id, ni, n, small); }
    unsigned long long bad = 0;
    TRY(cudaMemcpyAsync(&bad, small, sizeof(bad), cudaMemcpyDeviceToHost, s));
    TRY(cudaStreamSynchronize(s));
    if (bad) return set_error(g, ERANGE_, "pr_apply_batch: vertex id out of range");
  }
  // effective change lists (grow-only buffers owned by the graph)
  if (g->cap_dmin < nd) {
    if (g->dmin) cudaFree(g->dmin);
    g->dmin = nullptr;
    g->cap_dmin = 0;
    TRY(dev_malloc(&g->dmin, sizeof(uint64_t) * (nd + 1)));
    g->cap_dmin = nd;
  }
  if (g->cap_dplus < ni) {
    if (g->dplus) cudaFree(g->dplus);
    g->dplus = nullptr;
    g->cap_dplus = 0;
    TRY(dev_malloc(&g->dplus, sizeof(uint64_t) * (ni + 1)));
    g->cap_dplus = ni;
  }
  if (nd) {
    note_launch(); k_make_keys<<<grid_for(nd, 256), 256, 0, s>>>(ds, dd, nd, g->perm, bits, dk);
    TRY(radix_sort_u64(dk, alt, nd, 0, 2 * bits, tmp, s));
  }
  if (ni) {
    note_launch(); k_make_keys<<<grid_for(ni, 256), 256, 0, s>>>(is, id, ni, g->perm, bits, ik);
    TRY(radix_sort_u64(ik, alt, ni, 0, 2 * bits, tmp, s));
  }
  int64_t* cnts = (int64_t*)(small + 1);
  TRY(cudaMemsetAsync(cnts, 0, 2 * sizeof(int64_t), s));
  if (nd) {
    note_launch(); k_flag_del<<<grid_for(nd, 256), 256, 0, s>>>(dk, nd, ik, ni, g->out.off, g->out.deg, g->out.col, bits, flag);
    TRY(compact_u64(dk, flag, nd, g->dmin, cnts, tmp, s));
  }
  if (ni) {
    note_launch(); k_flag_ins<<<grid_for(ni, 256), 256, 0, s>>>(ik, ni, g->out.off, g->out.deg, g->out.col, bits, flag + nd);
    TRY(compact_u64(ik, flag + nd, ni, g->dplus, cnts + 1, tmp, s));
  }
  int64_t hc[2] = {0, 0};
  TRY(cudaMemcpyAsync(hc, cnts, sizeof(hc), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  g->n_dmin = hc[0];
  g->n_dplus = hc[1];
  if (hc[0] + hc[1] == 0) return OK;

  // both directions: the lists (in-CSR: the same keyed (dst, src); the lists are
  // sorted by (src, dst), so a stable sort by dst alone orders them), touched
  // rows from a bitmap, plans, long rows
  const int64_t a = hc[0], b = hc[1];
  const int64_t mr = std::min<int64_t>(a + b, n);   // touched rows, at most
  const int64_t tmp_bytes = (int64_t)std::max(radix_tmp_bytes(a + b), sizeof(int64_t) * (size_t)scan_tmp_elems(mr));
  auto carve = [&](void* at, EditBufs* B, uint64_t** alt2, void** tmp2, uint32_t** rbits, int32_t** btmp, int64_t** ca,
                   int64_t** cb, int32_t** cnt) {
    Carve c(at);
    B->key = nullptr;
    B->dl[0] = g->dmin;
    B->il[0] = g->dplus;
    B->dl[1] = c.take<uint64_t>(a);
    B->il[1] = c.take<uint64_t>(b);
    *alt2 = c.take<uint64_t>(std::max(a, b));
    *tmp2 = c.take<char>(tmp_bytes);
    *rbits = c.take<uint32_t>(cdiv(n, 32) + 1);
    *btmp = c.take<int32_t>(bits_to_list_tmp(n));
    *ca = c.take<int64_t>(mr + 1);
    *cb = c.take<int64_t>(mr + 1);
    *cnt = c.take<int32_t>(2);
    for (int d = 0; d < 2; d++) {
      B->rows[d] = c.take<int32_t>(mr);
      B->plan[d] = c.take<int4>(mr);
      B->od[d] = c.take<int32_t>(mr);
      B->lrow[d] = c.take<int32_t>(mr);
      B->lpre[d] = c.take<int32_t>(mr + 1);
      B->lsc[d] = c.take<int32_t>(mr);
    }
    B->st = c.take<EditStatus>(1);
    return c.used;
  };
  EditBufs B;
  uint64_t* alt2;
  void *tmp2, *ebase;
  uint32_t* rbits;
  int32_t *btmp, *rcnt;
  int64_t *ca, *cb;
  TRY(scratch_get(g, 1, carve(nullptr, &B, &alt2, &tmp2, &rbits, &btmp, &ca, &cb, &rcnt) + 256, &ebase));
  carve(ebase, &B, &alt2, &tmp2, &rbits, &btmp, &ca, &cb, &rcnt);
  if (a) {
    TRY(swap_keys_u64(g->dmin, a, bits, B.dl[1], s));
    TRY(radix_sort_u64(B.dl[1], alt2, a, bits, 2 * bits, tmp2, s));
  }
  if (b) {
    TRY(swap_keys_u64(g->dplus, b, bits, B.il[1], s));
    TRY(radix_sort_u64(B.il[1], alt2, b, bits, 2 * bits, tmp2, s));
  }
  TRY(cudaMemsetAsync(B.st, 0, sizeof(EditStatus), s));
  Csr* dirs[2] = {&g->out, &g->in};
  for (int d = 0; d < 2; d++) {
    const Csr* c = dirs[d];
    TRY(cudaMemsetAsync(rbits, 0, sizeof(uint32_t) * (size_t)(cdiv(n, 32) + 1), s));
    TRY(launch_source_bits(B.dl[d], a, bits, rbits, s));
    TRY(launch_source_bits(B.il[d], b, bits, rbits, s));
    TRY(launch_bits_to_list(rbits, nullptr, n, B.rows[d], rcnt, btmp, s));
    note_launch();
    k_edit_plan<<<grid_for(mr, 256), 256, 0, s>>>(B, d, rcnt, mr, a, b, bits, c->off, c->deg, ca, cb);
    TRY(scan_excl<int64_t>(ca, ca, mr, (int64_t*)tmp2, s));
    TRY(scan_excl<int64_t>(cb, cb, mr, (int64_t*)tmp2, s));
    note_launch(); k_edit_lists<<<grid_for(mr, 256), 256, 0, s>>>(B, d, mr, ca, cb);
  }
  if (!g->small_h) TRY(cudaMallocHost(&g->small_h, sizeof(EditStatus)));
  TRY(cudaMemcpyAsync(g->small_h, B.st, sizeof(EditStatus), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));
  const EditStatus h = *(EditStatus*)g->small_h;
  int32_t* S[2] = {nullptr, nullptr};
  int todo = 0;
  for (int d = 0; d < 2; d++) {
    if (h.ovf[d]) continue;
    int64_t cap;
    TRY(small_staging(g, d, (int64_t)h.scratch[d] * RW_CH, &S[d], &cap));
    todo |= 1 << d;
  }
  if (todo) launch_edit(g, B, S, todo, 2 * mr, b);
  TRY(cudaGetLastError());
  for (int d = 0; d < 2; d++)
    if (h.ovf[d]) {
      int rc = repack_direction(g, dirs[d], B.dl[d], a, B.il[d], b);
      if (rc) return rc;
      if (d == 1) {
        rc = refresh_full_tiles(g);
        if (rc) return rc;
      }
    }
  // contributions of sources whose out-degree changed (a3); the edit in place
  // has refreshed them
  if (h.ovf[0] && g->has_ranks) {
    TRY(cudaMemsetAsync(g->aux, 0, sizeof(uint32_t) * (size_t)(cdiv(n, 32) + 1), s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
    TRY(launch_mark_sources(g->dmin, a, g->dplus, b, bits, g->aux, g->wl[0], &g->ctl->count[0], s));
    TRY(launch_contrib_list(g->wl[0], &g->ctl->count[0], g->R, g->C[g->ccur], g->out.deg, g->tab_sc, n, s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
  }
  TRY(cudaGetLastError());
  return OK;
}

}  // namespace dfpr
