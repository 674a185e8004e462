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
// (src, dst)).  Each touched row is rewritten by one warp: the old row is
// copied to scratch, every surviving element and every insertion computes its
// output position by counting smaller deletions / insertions / old elements,
// and is written back in place; padding slots get the sentinel.  A row whose
// new degree exceeds its capacity triggers a repack of that direction (a full
// rebuild with fresh slack).
#include <algorithm>
#include <climits>
#include <cstring>
#include <new>
#include "batch.cuh"
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

__global__ void k_swap_keys(const uint64_t* __restrict__ in, int64_t k, int bits, uint64_t* __restrict__ out) {
  uint64_t mask = (1ull << bits) - 1;
  GRID_STRIDE(i, k) out[i] = ((in[i] & mask) << bits) | (in[i] >> bits);
}

__global__ void k_row_keys(const uint64_t* __restrict__ a, int64_t na, const uint64_t* __restrict__ b, int64_t nb,
                           int bits, uint64_t* __restrict__ out) {
  GRID_STRIDE(i, na + nb) out[i] = (i < na ? a[i] : b[i - na]) >> bits;
}

// per touched row: ranges in the deletion / insertion lists, old degree,
// chunk counts of the copy and write passes, overflow
constexpr int RW_CH = 1024;   // row elements per chunk (one warp works on a chunk)

__global__ void k_row_plan(const uint64_t* __restrict__ rows, int64_t nr, const uint64_t* __restrict__ dl, int64_t nd,
                           const uint64_t* __restrict__ il, int64_t ni, int bits, const int64_t* __restrict__ off,
                           const int32_t* __restrict__ deg, int64_t* __restrict__ plan, int64_t* __restrict__ olddeg,
                           int64_t* __restrict__ cchunks, int64_t* __restrict__ wchunks, unsigned long long* overflow) {
  GRID_STRIDE(j, nr) {
    uint64_t r = rows[j];
    int64_t d0 = lower_key(dl, 0, nd, r << bits), d1 = lower_key(dl, d0, nd, (r + 1) << bits);
    int64_t i0 = lower_key(il, 0, ni, r << bits), i1 = lower_key(il, i0, ni, (r + 1) << bits);
    int64_t dg = deg[r];
    int64_t nd2 = dg - (d1 - d0) + (i1 - i0);
    plan[4 * j + 0] = d0;
    plan[4 * j + 1] = d1;
    plan[4 * j + 2] = i0;
    plan[4 * j + 3] = i1;
    olddeg[j] = dg;
    cchunks[j] = cdiv(dg, RW_CH);
    wchunks[j] = cdiv(round4(dg > nd2 ? dg : nd2), RW_CH);
    if (round4(nd2) > off[r + 1] - off[r]) atomicAdd(overflow, 1ull);
  }
}

// row j of chunk c: largest j with pre[j] <= c
__device__ __forceinline__ int64_t chunk_row(const int64_t* pre, int64_t nr, int64_t c) {
  int64_t lo = 0, hi = nr - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// copy pass: the old elements of every touched row into scratch, one warp per chunk
__global__ void k_row_copy(const uint64_t* __restrict__ rows, const int64_t* __restrict__ nrp,
                           const int64_t* __restrict__ sofs, const int64_t* __restrict__ cpre,
                           const int64_t* __restrict__ off, const int32_t* __restrict__ deg,
                           const int32_t* __restrict__ col, int32_t* __restrict__ scratch) {
  const int64_t nr = *nrp;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = cpre[nr];
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < total; c += nw) {
    const int64_t j = chunk_row(cpre, nr, c);
    const int64_t r = (int64_t)rows[j];
    const int64_t x0 = (c - cpre[j]) * RW_CH;
    const int64_t x1 = min(x0 + (int64_t)RW_CH, (int64_t)deg[r]);
    const int64_t base = off[r];
    int32_t* S = scratch + sofs[j];
    for (int64_t x = x0 + lane; x < x1; x += 32) S[x] = col[base + x];
  }
}

// write pass over old positions: every surviving element moves to
// x - (#deletions below it) + (#insertions below it); slots from the new degree
// up to the old end get the sentinel
__global__ void k_row_survivors(const uint64_t* __restrict__ rows, const int64_t* __restrict__ nrp,
                                const int64_t* __restrict__ plan, const int64_t* __restrict__ sofs,
                                const int64_t* __restrict__ wpre, const uint64_t* __restrict__ dl,
                                const uint64_t* __restrict__ il, int bits, const int64_t* __restrict__ off,
                                const int32_t* __restrict__ deg, int32_t* __restrict__ col,
                                const int32_t* __restrict__ scratch, int32_t sent) {
  const int64_t nr = *nrp;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = wpre[nr];
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < total; c += nw) {
    const int64_t j = chunk_row(wpre, nr, c);
    const int64_t r = (int64_t)rows[j];
    const int64_t d0 = plan[4 * j], d1 = plan[4 * j + 1], i0 = plan[4 * j + 2], i1 = plan[4 * j + 3];
    const int64_t d_old = deg[r];
    const int64_t d_new = d_old - (d1 - d0) + (i1 - i0);
    const int64_t pad_end = round4(d_old > d_new ? d_old : d_new);
    const int64_t base = off[r], cap = off[r + 1] - base;
    const int32_t* S = scratch + sofs[j];
    const int64_t x0 = (c - wpre[j]) * RW_CH;
    const int64_t x1 = min(x0 + (int64_t)RW_CH, pad_end);
    for (int64_t x = x0 + lane; x < x1; x += 32) {
      if (x < d_old) {
        const int32_t v = S[x];
        const uint64_t key = ((uint64_t)r << bits) | (uint64_t)v;
        const int64_t dl_lt = lower_key(dl, d0, d1, key);
        if (!(dl_lt < d1 && dl[dl_lt] == key)) {
          const int64_t pos = x - (dl_lt - d0) + (lower_key(il, i0, i1, key) - i0);
          if (pos >= 0 && pos < cap) col[base + pos] = v;
        }
      }
      if (x >= d_new && x < cap) col[base + x] = sent;
    }
  }
}

// write pass over insertions: insertion k of row r goes to
// (#insertions below it) + (#old elements below it) - (#deletions below it)
__global__ void k_row_insertions(const uint64_t* __restrict__ rows, const int64_t* __restrict__ nrp,
                                 const int64_t* __restrict__ plan, const int64_t* __restrict__ sofs,
                                 const uint64_t* __restrict__ dl, const uint64_t* __restrict__ il,
                                 const int64_t* __restrict__ nip, int bits, const int64_t* __restrict__ off,
                                 const int32_t* __restrict__ deg, int32_t* __restrict__ col,
                                 const int32_t* __restrict__ scratch) {
  const int64_t nr = *nrp, ni = *nip;
  const uint64_t mask = (1ull << bits) - 1;
  GRID_STRIDE(k, ni) {
    const uint64_t r = il[k] >> bits;
    int64_t lo = 0, hi = nr - 1;   // touched-row index of r
    while (lo < hi) {
      int64_t mid = (lo + hi) >> 1;
      if (rows[mid] < r) lo = mid + 1;
      else hi = mid;
    }
    const int64_t j = lo;
    const int64_t d0 = plan[4 * j], d1 = plan[4 * j + 1], i0 = plan[4 * j + 2];
    const int32_t y = (int32_t)(il[k] & mask);
    const int32_t* S = scratch + sofs[j];
    int32_t a = 0, b = deg[r];
    while (a < b) {
      int32_t mid = (a + b) >> 1;
      if (S[mid] < y) a = mid + 1;
      else b = mid;
    }
    const int64_t dl_lt = lower_key(dl, d0, d1, (r << bits) | (uint64_t)y);
    const int64_t pos = (k - i0) + a - (dl_lt - d0);
    const int64_t base = off[r], cap = off[r + 1] - base;
    if (pos >= 0 && pos < cap) col[base + pos] = y;
  }
}

__global__ void k_row_degrees(const uint64_t* __restrict__ rows, const int64_t* __restrict__ nrp,
                              const int64_t* __restrict__ plan, int32_t* __restrict__ deg) {
  const int64_t nr = *nrp;
  GRID_STRIDE(j, nr) {
    const uint64_t r = rows[j];
    deg[r] = deg[r] - (int32_t)(plan[4 * j + 1] - plan[4 * j]) + (int32_t)(plan[4 * j + 3] - plan[4 * j + 2]);
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

__global__ void k_u64_to_i32_low(const uint64_t* __restrict__ in, int64_t k, int32_t* __restrict__ out) {
  GRID_STRIDE(i, k) out[i] = (int32_t)in[i];
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

static int edit_direction(Graph* g, Csr* c, const uint64_t* dl, int64_t nd, const uint64_t* il, int64_t ni,
                          const int64_t* ni_dev, bool* repacked) {
  cudaStream_t s = g->stream;
  int bits = g->id_bits;
  *repacked = false;
  int64_t nrk = nd + ni;
  if (nrk == 0) return OK;
  // touched rows: sorted distinct row ids
  size_t need = 0;
  {
    Carve probe(nullptr);
    probe.take<uint64_t>(nrk);
    probe.take<uint64_t>(nrk);
    probe.take<uint64_t>(nrk);
    probe.take<uint8_t>(nrk);
    probe.take<char>((int64_t)std::max(radix_tmp_bytes(nrk), compact_tmp_bytes(nrk)));
    probe.take<int64_t>(1);
    need = probe.used + 4096;
  }
  void* base;
  TRY(scratch_get(g, 3, need, &base));
  Carve cv(base);
  uint64_t* rk = cv.take<uint64_t>(nrk);
  uint64_t* alt = cv.take<uint64_t>(nrk);
  uint64_t* rows = cv.take<uint64_t>(nrk);
  uint8_t* flag = cv.take<uint8_t>(nrk);
  void* tmp = cv.take<char>((int64_t)std::max(radix_tmp_bytes(nrk), compact_tmp_bytes(nrk)));
  int64_t* cnt = cv.take<int64_t>(1);
  note_launch(); k_row_keys<<<grid_for(nrk, 256), 256, 0, s>>>(dl, nd, il, ni, bits, rk);
  TRY(radix_sort_u64(rk, alt, nrk, bits, tmp, s));
  TRY(flag_unique_sorted(rk, nrk, flag, s));
  TRY(compact_u64(rk, flag, nrk, rows, cnt, tmp, s));
  int64_t nr = 0;
  TRY(cudaMemcpyAsync(&nr, cnt, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));

  void* base2;
  size_t need2 = 0;
  {
    Carve probe(nullptr);
    probe.take<int64_t>(4 * nr);
    for (int i = 0; i < 3; i++) probe.take<int64_t>(nr + 1);
    probe.take<int64_t>(scan_tmp_elems(nr));
    probe.take<unsigned long long>(1);
    need2 = probe.used + 4096;
  }
  TRY(scratch_get(g, 4, need2, &base2));
  Carve c2(base2);
  int64_t* plan = c2.take<int64_t>(4 * nr);
  int64_t* sofs = c2.take<int64_t>(nr + 1);
  int64_t* cpre = c2.take<int64_t>(nr + 1);
  int64_t* wpre = c2.take<int64_t>(nr + 1);
  int64_t* sscr = c2.take<int64_t>(scan_tmp_elems(nr));
  unsigned long long* ovf = c2.take<unsigned long long>(1);
  TRY(cudaMemsetAsync(ovf, 0, sizeof(unsigned long long), s));
  note_launch(); k_row_plan<<<grid_for(nr, 256), 256, 0, s>>>(rows, nr, dl, nd, il, ni, bits, c->off, c->deg, plan, sofs,
                                                              cpre, wpre, ovf);
  TRY(scan_excl<int64_t>(sofs, sofs, nr, sscr, s));
  TRY(scan_excl<int64_t>(cpre, cpre, nr, sscr, s));
  TRY(scan_excl<int64_t>(wpre, wpre, nr, sscr, s));
  unsigned long long ovf_h = 0;
  int64_t stot = 0;
  TRY(cudaMemcpyAsync(&ovf_h, ovf, sizeof(ovf_h), cudaMemcpyDeviceToHost, s));
  TRY(cudaMemcpyAsync(&stot, sofs + nr, sizeof(stot), cudaMemcpyDeviceToHost, s));
  TRY(cudaStreamSynchronize(s));

  if (ovf_h == 0) {
    void* sp;
    TRY(scratch_get(g, 5, sizeof(int32_t) * (size_t)(stot + 1), &sp));
    int32_t* S = (int32_t*)sp;
    const int wgrid = num_sms() * 16;
    note_launch(); k_row_copy<<<wgrid, 256, 0, s>>>(rows, cnt, sofs, cpre, c->off, c->deg, c->col, S);
    note_launch(); k_row_survivors<<<wgrid, 256, 0, s>>>(rows, cnt, plan, sofs, wpre, dl, il, bits, c->off, c->deg, c->col,
                                                         S, g->n);
    if (ni) {
      note_launch(); k_row_insertions<<<grid_for(ni, 256), 256, 0, s>>>(rows, cnt, plan, sofs, dl, il, ni_dev, bits,
                                                                        c->off, c->deg, c->col, S);
    }
    note_launch(); k_row_degrees<<<grid_for(nr, 256), 256, 0, s>>>(rows, cnt, plan, c->deg);
    TRY(cudaGetLastError());
    return OK;
  }

  // repack this direction: survivors + insertions, sorted, rebuilt with more slack
  *repacked = true;
  return repack_direction(g, c, dl, nd, il, ni);
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
//   k_small_copy    the old elements of touched rows longer than a chunk into
//                   scratch (a row is edited in place, by many warps);
//   k_small_edit    one warp per touched row, staged in shared memory, or per
//                   chunk of a longer row; both directions at once, with the
//                   new degrees and the contributions of the sources.
// Device time of a batch: 50 us for 168 edges on a graph of 2^20 vertices, 115
// for 4000 and 145 for 6300 on one of 2.6M (k_small_keys 4 to 8, k_small_ingest
// 9 / 37 / 63, k_small_copy 6 to 8, k_small_edit 12 to 37).  Before, one block
// ran both directions in turn with the sort in shared memory (53 us at 168
// edges, 143 at 1300, 312 at 4000) and five kernels per direction followed: 166
// us in all for 168 edges, 450 for 4000; above 4096 edges the path below, 930
// us for 6300.
// A direction whose rows overflow their capacity, or whose scratch is too
// small, is left alone by the device and finished by the host.
constexpr int SMALL_MAX = 16384;                // edges of a batch (deletions + insertions)
constexpr int SMALL_THREADS = 1024;
constexpr uint64_t BAD = ~1ull;                  // key of an edge with an id out of range (no packed key: ids are below 2^31)

}  // namespace dfpr

struct dfpr::SmallStatus {
  int32_t n_del, n_ins;   // effective deletions / insertions
  int32_t bad;
  // per direction (out 0, in 1): touched rows, those longer than a chunk and
  // their chunks; the device left the direction unchanged (skip), because rows
  // overflow (ovf) or the scratch is too small (need)
  int32_t nr[2], nlong[2], chunks[2], skip[2], ovf[2], need[2];
};

// device arrays of one small batch, all in one scratch buffer
struct dfpr::SmallBufs {
  uint64_t* key;           // packed (src, dst, insertion, present)
  uint64_t *dl[2], *il[2];   // Delta-, Delta+ sorted by (src, dst) and by (dst, src)
  int32_t* rows[2];
  int4* plan[2];           // per touched row: its deletions [x, y) and insertions [z, w)
  int32_t* od[2];          // its degree before the batch
  int32_t *lrow[2], *lpre[2];   // rows longer than a chunk: index into rows, chunks before
  SmallStatus* st;
};

namespace dfpr {

static size_t small_carve(void* base, int64_t cap, SmallBufs* B) {
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
  }
  B->st = c.take<SmallStatus>(1);
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
                   const __grid_constant__ SmallBufs B) {
  extern __shared__ uint64_t K[];   // the sorted keys, then the effective changes (row, col, insertion)
  uint16_t* const DP = reinterpret_cast<uint16_t*>(K + SMALL_THREADS * E + 8);
  uint16_t* const RS = DP + SMALL_THREADS * E + 8;
  __shared__ uint64_t wsum[33];
  const int dir = blockIdx.x, t = threadIdx.x;
  const SmallCsr& c = dir == 0 ? out : in;
  const uint64_t mask = (1ull << bits) - 1;
  SmallStatus& st = *B.st;
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
      st.nr[dir] = st.nlong[dir] = st.chunks[dir] = 0;
      st.skip[dir] = 1;
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
      const int32_t len = dg > dn ? dg : dn;
      if (len > RW_CH) longs = 1ull << 32 | (uint64_t)cdiv(round4(len), RW_CH);
    }
    if (__syncthreads_or(longs != 0)) {
      const uint64_t before = carry + block_excl(longs, wsum, &tot);
      if (longs) {
        B.lrow[dir][before >> 32] = j;
        B.lpre[dir][before >> 32] = (int32_t)(uint32_t)before;
      }
      carry += tot;
    }
  }
  const int any_ovf = __syncthreads_or(ovf);
  if (t == 0) {
    const int64_t chunks = (int64_t)(uint32_t)carry;
    st.bad = 0;
    st.n_del = nde;
    st.n_ins = nie;
    st.nr[dir] = nr;
    st.nlong[dir] = (int32_t)(carry >> 32);
    st.chunks[dir] = (int32_t)chunks;
    B.lpre[dir][carry >> 32] = (int32_t)chunks;
    st.ovf[dir] = any_ovf ? 1 : 0;
    st.need[dir] = chunks * RW_CH > c.scap ? 1 : 0;
    st.skip[dir] = st.ovf[dir] | st.need[dir];
  }
}

struct SmallEdit {
  const int64_t* off[2];
  int32_t* deg[2];
  int32_t* col[2];
  int32_t* S[2];          // scratch of rows longer than a chunk: chunk c of the direction at c x RW_CH
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

__global__ void __launch_bounds__(256) k_small_copy(const __grid_constant__ SmallBufs B,
                                                    const __grid_constant__ SmallEdit p) {
  const SmallStatus& st = *B.st;
  const int nw = (gridDim.x * blockDim.x) >> 5, w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (int d = 0; d < 2; d++) {
    if (!((p.dirs >> d) & 1) || st.skip[d]) continue;
    const int nc = st.chunks[d];
    for (int c = w0; c < nc; c += nw) {
      const int l = long_row(B.lpre[d], st.nlong[d], c), j = B.lrow[d][l];
      const int32_t x0 = (c - B.lpre[d][l]) * RW_CH;
      const int32_t* row = p.col[d] + p.off[d][B.rows[d][j]];
      copy_chunk(row + x0, min(B.od[d][j] - x0, RW_CH), p.S[d] + (int64_t)c * RW_CH);
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

// one warp: positions [x0, x1) of a touched row (its old elements from x0 on in
// shared memory at T, all of them at S; the padding after them included) and its
// insertions [k0, k1) written to their new places: a survivor x goes to x - (deletions below it) + (insertions below
// it), an insertion to its rank among the insertions + old elements below it -
// deletions below it
__device__ __forceinline__ void edit_row_part(const int32_t* T, const int32_t* S, int32_t x0, int32_t x1, int k0, int k1, int32_t r, int4 pl,
                                              int32_t d_old, int32_t cap, const uint64_t* __restrict__ dl,
                                              const uint64_t* __restrict__ il, uint64_t mask, int bits,
                                              int32_t* __restrict__ row, int32_t sent) {
  const int lane = threadIdx.x & 31;
  const int nd = pl.y - pl.x, ni = pl.w - pl.z;
  const int32_t d_new = d_old - nd + ni;
  const bool few = nd + ni <= 32;   // the row's changes in registers, one per lane
  const int32_t mine = few && lane < nd + ni ? (int32_t)((lane < nd ? dl[pl.x + lane] : il[pl.z + lane - nd]) & mask) : 0;
  const uint64_t rk = (uint64_t)r << bits;
  for (int32_t xb = x0; xb < x1; xb += 32) {
    const int32_t x = xb + lane;
    const bool old = x < x1 && x < d_old;
    const int32_t v = old ? T[x - x0] : 0;
    int dlt = 0, ilt = 0;
    bool dead = false;
    if (few) {
      for (int k = 0; k < nd; k++) {
        const int32_t y = __shfl_sync(0xffffffffu, mine, k);
        dlt += y < v;
        dead |= y == v;
      }
      for (int k = nd; k < nd + ni; k++) ilt += __shfl_sync(0xffffffffu, mine, k) < v;
    } else if (old) {
      const int64_t a = lower_key(dl, pl.x, pl.y, rk | (uint64_t)v);
      dead = a < pl.y && dl[a] == (rk | (uint64_t)v);
      dlt = (int)(a - pl.x);
      ilt = (int)(lower_key(il, pl.z, pl.w, rk | (uint64_t)v) - pl.z);
    }
    if (old && !dead) {
      const int32_t pos = x - dlt + ilt;
      if (pos >= 0 && pos < cap) row[pos] = v;
    }
    if (x < x1 && x >= d_new && x < cap) row[x] = sent;
  }
  for (int k = k0 + lane; k < k1; k += 32) {
    const int32_t y = (int32_t)(il[k] & mask);
    const int32_t pos = (k - pl.z) + lower_i32(S, 0, d_old, y) - (int32_t)(lower_key(dl, pl.x, pl.y, rk | (uint64_t)y) - pl.x);
    if (pos >= 0 && pos < cap) row[pos] = y;
  }
}

__global__ void __launch_bounds__(256) k_small_edit(const __grid_constant__ SmallBufs B,
                                                    const __grid_constant__ SmallEdit p, int bits) {
  __shared__ __align__(16) int32_t stage[8][RW_CH];
  const SmallStatus& st = *B.st;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const uint64_t mask = (1ull << bits) - 1;
  // the work: touched rows of both directions, then chunks of both
  const bool on0 = (p.dirs & 1) && !st.skip[0], on1 = (p.dirs & 2) && !st.skip[1];
  const int e0 = on0 ? st.nr[0] : 0, e1 = e0 + (on1 ? st.nr[1] : 0);
  const int e2 = e1 + (on0 ? st.chunks[0] : 0), e3 = e2 + (on1 ? st.chunks[1] : 0);
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < e3; w += nw) {
    const bool chunk = w >= e1;
    const int d = chunk ? (w >= e2 ? 1 : 0) : (w >= e0 ? 1 : 0);
    const int item = chunk ? w - (d ? e2 : e1) : w - (d ? e0 : 0);
    const int l = chunk ? long_row(B.lpre[d], st.nlong[d], item) : 0;
    const int j = chunk ? B.lrow[d][l] : item;
    const int32_t r = B.rows[d][j], d_old = B.od[d][j];
    const int4 pl = B.plan[d][j];
    const int32_t d_new = d_old - (pl.y - pl.x) + (pl.w - pl.z);
    const int32_t len = d_old > d_new ? d_old : d_new;
    const int64_t base = p.off[d][r];
    const int64_t cap64 = p.off[d][r + 1] - base;
    const int32_t cap = (int32_t)(cap64 < INT32_MAX ? cap64 : INT32_MAX), end = (int32_t)round4(len);
    int32_t* const row = p.col[d] + base;
    if (!chunk && len > RW_CH) continue;   // a long row: its chunks are items of their own
    int32_t* const T = stage[threadIdx.x >> 5];
    const int part = chunk ? item - B.lpre[d][l] : 0, parts = chunk ? B.lpre[d][l + 1] - B.lpre[d][l] : 1;
    const int32_t x0 = part * RW_CH;
    const int32_t* const S = chunk ? p.S[d] + (int64_t)B.lpre[d][l] * RW_CH : T;
    __syncwarp();
    copy_chunk(chunk ? S + x0 : row, min(d_old - x0, RW_CH), T);
    __syncwarp();
    const int per = (pl.w - pl.z + parts - 1) / parts;
    const int k0 = min(pl.z + part * per, pl.w), k1 = min(k0 + per, pl.w);
    edit_row_part(T, S, x0, min(x0 + RW_CH, end), k0, k1, r, pl, d_old, cap, B.dl[d], B.il[d], mask, bits, row, p.sent);
    if (part > 0) continue;
    if (lane == 0) {
      p.deg[d][r] = d_new;
      if (d == 0 && p.R) {   // the source's contribution with its new out-degree
        const double sc = d_new < TAB ? p.tab_sc[d_new] : FIX_ONE / (double)d_new;
        p.C[r] = __double2ll_rn(p.R[r] * sc);
      }
    }
  }
}

static void launch_small_edit(Graph* g, const SmallApply* A, int dirs) {
  cudaStream_t s = g->stream;
  SmallEdit p;
  const Csr* c[2] = {&g->out, &g->in};
  for (int d = 0; d < 2; d++) {
    p.off[d] = c[d]->off;
    p.deg[d] = c[d]->deg;
    p.col[d] = c[d]->col;
    p.S[d] = A->S[d];
  }
  p.sent = g->n;
  p.R = g->has_ranks ? g->R : nullptr;
  p.C = g->C[g->ccur];
  p.tab_sc = g->tab_sc;
  p.dirs = dirs;
  note_launch(); k_small_copy<<<num_sms() * 2, 256, 0, s>>>(*A->B, p);
  note_launch(); k_small_edit<<<num_sms() * 4, 256, 0, s>>>(*A->B, p, g->id_bits);
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
static cudaError_t launch_ingest(Graph* g, int N, const SmallCsr& out, const SmallCsr& in, const SmallBufs& B) {
  int bps;   // (raises the kernel's shared memory limit once)
  cudaError_t e = gather_occupancy((const void*)k_small_ingest<E>, SMALL_THREADS, small_smem<E>(), &bps);
  if (e != cudaSuccess) return e;
  note_launch();
  k_small_ingest<E><<<2, SMALL_THREADS, small_smem<E>(), g->stream>>>(N, g->id_bits, out, in, B);
  return cudaGetLastError();
}

// phase 1 of a small batch: everything up to the status copy to the host,
// queued on the graph's stream without waiting
static int small_launch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is,
                        const int32_t* id, int64_t ni, SmallApply* A) {
  cudaStream_t s = g->stream;
  const int N = (int)(nd + ni);
  const int64_t cap = std::max(1024, pow2_at_least(N));
  SmallBufs B;
  void* bp;
  TRY(scratch_get(g, 6, small_carve(nullptr, cap, &B) + 256, &bp));
  small_carve(bp, cap, &B);
  if (!g->small_h) TRY(cudaMallocHost(&g->small_h, sizeof(SmallStatus)));
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
  A->B = new (std::nothrow) SmallBufs(B);
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
    launch_small_edit(g, A, 3);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(g->small_h, B.st, sizeof(SmallStatus), cudaMemcpyDeviceToHost, s);
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
  const SmallBufs B = *A->B;
  struct Release {
    SmallApply* a;
    ~Release() {
      delete a->B;
      a->B = nullptr;
    }
  } release{A};
  TRY(cudaStreamSynchronize(s));
  g->stage_busy = false;
  const SmallStatus h = *(SmallStatus*)g->small_h;
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
      TRY(small_staging(g, dir, (int64_t)h.chunks[dir] * RW_CH, &A->S[dir], &cap));
      TRY(cudaMemsetAsync(&B.st->skip[dir], 0, sizeof(int32_t), s));
      launch_small_edit(g, A, 1 << dir);
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

// the endpoint arrays of a host batch on the device (scratch slot 0): deletion
// sources and targets, insertion sources and targets, one after another.  A
// small batch goes through the graph's pinned buffer in one copy: four copies
// from pageable memory take about 8 us of host time each.
int stage_host_batch(Graph* g, const int32_t* ds, const int32_t* dd, int64_t nd, const int32_t* is, const int32_t* id,
                     int64_t ni, int32_t** out) {
  cudaStream_t s = g->stream;
  void* stage;
  TRY(scratch_get(g, 0, sizeof(int32_t) * (size_t)(2 * (nd + ni) + 4) + 1024, &stage));
  int32_t* b = (int32_t*)stage;
  *out = b;
  const int32_t* src[4] = {ds, dd, is, id};
  const int64_t len[4] = {nd, nd, ni, ni};
  if (nd + ni <= SMALL_MAX) {
    if (!g->stage_h) TRY(cudaMallocHost(&g->stage_h, sizeof(int32_t) * 2 * SMALL_MAX));
    if (g->stage_busy) TRY(cudaDeviceSynchronize());   // the copy of a call that failed after it
    int32_t* h = (int32_t*)g->stage_h;
    for (int k = 0; k < 4; k++)
      if (len[k]) {
        memcpy(h, src[k], sizeof(int32_t) * (size_t)len[k]);
        h += len[k];
      }
    if (nd + ni > 0) {
      g->stage_busy = true;
      TRY(cudaMemcpyAsync(b, g->stage_h, sizeof(int32_t) * 2 * (size_t)(nd + ni), cudaMemcpyHostToDevice, s));
    }
    return OK;
  }
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
    TRY(radix_sort_u64(dk, alt, nd, 2 * bits, tmp, s));
  }
  if (ni) {
    note_launch(); k_make_keys<<<grid_for(ni, 256), 256, 0, s>>>(is, id, ni, g->perm, bits, ik);
    TRY(radix_sort_u64(ik, alt, ni, 2 * bits, tmp, s));
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

  // out-CSR: lists are sorted by (src, dst)
  bool rep_out = false, rep_in = false;
  int rc = edit_direction(g, &g->out, g->dmin, hc[0], g->dplus, hc[1], cnts + 1, &rep_out);
  if (rc) return rc;
  // in-CSR: the same lists keyed (dst, src)
  {
    int64_t a = hc[0], b = hc[1];
    void* base2;
    size_t need2;
    {
      Carve probe(nullptr);
      probe.take<uint64_t>(a);
      probe.take<uint64_t>(b);
      probe.take<uint64_t>(a + b);
      probe.take<char>((int64_t)radix_tmp_bytes(a + b));
      need2 = probe.used + 4096;
    }
    TRY(scratch_get(g, 1, need2, &base2));
    Carve c2(base2);
    uint64_t* sd = c2.take<uint64_t>(a);
    uint64_t* si = c2.take<uint64_t>(b);
    uint64_t* alt2 = c2.take<uint64_t>(a + b);
    void* tmp2 = c2.take<char>((int64_t)radix_tmp_bytes(a + b));
    if (a) {
      note_launch(); k_swap_keys<<<grid_for(a, 256), 256, 0, s>>>(g->dmin, a, bits, sd);
      TRY(radix_sort_u64(sd, alt2, a, 2 * bits, tmp2, s));
    }
    if (b) {
      note_launch(); k_swap_keys<<<grid_for(b, 256), 256, 0, s>>>(g->dplus, b, bits, si);
      TRY(radix_sort_u64(si, alt2, b, 2 * bits, tmp2, s));
    }
    rc = edit_direction(g, &g->in, sd, a, si, b, cnts + 1, &rep_in);
    if (rc) return rc;
  }
  if (rep_in) {
    rc = refresh_full_tiles(g);
    if (rc) return rc;
  }
  // contributions of sources whose out-degree changed (a3)
  if (g->has_ranks) {
    // the sources: reuse worklist 0 and the aux bitset
    TRY(cudaMemsetAsync(g->aux, 0, sizeof(uint32_t) * (size_t)(cdiv(n, 32) + 1), s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
    TRY(launch_mark_sources(g->dmin, hc[0], g->dplus, hc[1], bits, g->aux, g->wl[0], &g->ctl->count[0], s));
    TRY(launch_contrib_list(g->wl[0], &g->ctl->count[0], g->R, g->C[g->ccur], g->out.deg, g->tab_sc, n, s));
    TRY(cudaMemsetAsync(&g->ctl->count[0], 0, sizeof(int32_t), s));
  }
  TRY(cudaGetLastError());
  return OK;
}

}  // namespace dfpr
