// loop.cu -- one graph's whole update (Static, ND, DF or DF-P) in one
// cooperative kernel, one grid barrier per iteration.
//
// What bounds it.  On graphs of up to about a million vertices a sweep takes
// microseconds, and the time of an update is the number of iterations times
// the latency of one: launches (three kernels per iteration in the CUDA graph,
// 18-21 us) or, in the group loop of group.cu, two grid barriers plus two
// phases of dependent loads (12-13 us at 2^14 vertices; here 4.5, and 4.0 at
// 2^10).  Of the 4 us the barrier is 1.6, the gather 0.6 and the epilogue 0.3
// when measured alone; the rest is the flush of a block's writes and the first
// misses after the L1 is invalidated.  Here every block owns a run of whole in-CSR rows, cut at equal
// shares of the quads, for the whole update: it gathers its rows' sums into
// shared memory, runs the epilogue of its own vertices from there, and only
// the new contributions and expanded flags leave the SM.  So there is one
// barrier per iteration, and the L-inf change of the iteration is read while
// the next gather is under way.  The columns and
// the row-start index stay in shared memory when they fit, and the degree
// tables, ranks and own contributions stay in registers when a block has at
// most one row per thread.
//
// Sums of row pieces need no atomics: a warp reduces 32 consecutive quads; the
// piece that holds a row's start is stored at the row, the piece that
// continues a row from the quads before (at most one per 32) at the word, and
// the epilogue adds a row's start and its words.  Integer sums, so the order
// does not change a bit: the ranks and statistics are those of the other loops.
#include <algorithm>
#include <atomic>
#include "loop.cuh"
#include "prim.cuh"
#include "pull_step.cuh"

namespace dfpr {

namespace {

constexpr int LT = 1024;                        // threads per block
constexpr int LW = LT / 32;
// polls of a barrier wait before it gives up, after the first 4096 with a short
// sleep each: about a second (2^20 polls took 0.33 s), against microseconds when
// every block runs
constexpr long long LOOP_SPINS = 3ll << 20;
constexpr long long LOOP_SPINS_STUCK = 1ll << 13;   // where a wait is made to run out (LOOP_STUCK)
// shared memory of a block: above STAGE_MAX the columns stay in L2.  The rest
// of the 256 KB is the L1 that the gathers land in: random 8-byte gathers of a
// 64 MB table ran at 236 G/s with 64 KB in shared memory, 217 with 128 KB and
// 127 with 192 KB
constexpr size_t STAGE_MAX = 64 << 10;
constexpr size_t LOOP_SMEM_MAX = 112 << 10;

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ uint32_t ld_byte(const uint8_t* p) {
  uint32_t v;
  asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
    x = y > x ? y : x;
  }
  return x;
}

// The grid barrier, called by thread 0 of every block after a block barrier:
// one counter that only grows, polled by one thread per block until it holds
// `target` arrivals.  False when a wait ran out, here or elsewhere (err set).
// Measured with 152 blocks of 1024 threads, nothing else in the loop: 1.6 us;
// an arrival counter plus a release word 2.1; a slot per block polled by 152
// threads of every block (no atomics) 3.9 to 5.2, the polls contending for a
// few L2 lines.
__device__ __forceinline__ bool grid_wait(LoopState* st, LoopOut* out, unsigned long long target, long long polls) {
  fence_acq_rel();   // this block's writes before its arrival
  atomicAdd(&st->count, 1ull);
  long long spins = 0;
  bool good = true;
  while (ld_relaxed_u64(&st->count) < target) {
    spins++;
    if ((spins & 255) == 0 && *(volatile int32_t*)&st->err) {
      good = false;
      break;
    }
    if (spins > polls) {
      atomicExch(&st->err, 1);
      *(volatile int32_t*)&out->err = 1;
      good = false;
      break;
    }
    if (spins > 4096) __nanosleep(64);
  }
  fence_acq_rel();   // the other blocks' writes before their arrivals
  return good;
}

// rows of the in-CSR that start below quad q
__device__ __forceinline__ int32_t rows_before(const uint32_t* rowbits, const int32_t* rowbase, int64_t q,
                                               int64_t nquads, int32_t n) {
  if (q >= nquads) return n;
  const int64_t w = q >> 5;
  return rowbase[w] + __popc(rowbits[w] & ((1u << (q & 31)) - 1u));
}
__host__ __device__ __forceinline__ int64_t share_start(int64_t nquads, int b, int NB) { return nquads * b / NB; }

// Eq. 1 / Eq. 2 and the frontier tests of Alg. 1 for one processed vertex, the
// operations of finish_pull_step (pull_step.cuh)
template <bool CLOSED, bool REL>
__device__ __forceinline__ void row_update(const LoopParams& p, double alpha_fix, bool same_tau, long long sum,
                                           long long cself, double Rv, int32_t d, double sc, double2 ab, double& r,
                                           long long& c, unsigned long long& drb, bool& stay, bool& expand) {
  if (CLOSED) r = fma(ab.x, fixconv::i64_to_f64_rn(sum - cself), ab.y);
  else r = fma(alpha_fix, fixconv::i64_to_f64_rn(sum), p.C0);
  drb = dbits(fabs(r - Rv));
  c = fixconv::f64_to_i64_rn(r * sc);
  const double mx = dbits(r) > dbits(Rv) ? r : Rv;
  const double mr = REL ? mx : measure_base(p.metric, mx, d);
  const unsigned long long tf = dbits(p.tau_f * mr);
  const unsigned long long tp = same_tau ? tf : dbits(p.tau_p * mr);
  stay = !CLOSED || drb > tp;
  expand = drb > tf;
}

// FRONTIER: DF / DF-P (else every vertex is processed: Static, ND).  REGS: at
// most one row per thread, its constants, rank and contribution in registers.
template <bool CLOSED, bool FRONTIER, bool REL, bool REGS>
__global__ void __launch_bounds__(LT, 1) k_loop(const __grid_constant__ LoopParams p) {
  constexpr int U = REGS ? 2 : 4;   // 32-quad words a warp has in flight
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long red[2 * LW];
  __shared__ long long tot[3][LW];
  int4* const scol = reinterpret_cast<int4*>(smem);                                  // staged: 32 per word
  long long* const acc = reinterpret_cast<long long*>(scol + (p.staged ? 32 * p.words_cap : 0));
  long long* const cont = acc + p.rows_cap;
  uint32_t* const sbits = reinterpret_cast<uint32_t*>(cont + p.words_cap);
  int32_t* const sbase = reinterpret_cast<int32_t*>(sbits + p.words_cap);
  uint8_t* const flag = reinterpret_cast<uint8_t*>(sbase + p.words_cap);             // 1: in S, 2: ever processed
  uint8_t* const accx = flag + p.rows_cap;                                           // an in-neighbour expanded
  uint8_t* const contx = accx + p.rows_cap;

  LoopState* const st = p.st;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int NB = gridDim.x;
  const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
  // barriers of the launches before (block 0 wrote it at the end of the last one)
  unsigned long long k = ld_relaxed_u64(&st->barriers);
  auto barrier = [&]() -> bool {
    __syncthreads();
    bool good = true;
    if (tid == 0) good = grid_wait(st, p.out, (k + 1) * NB, p.polls);
    k++;
    return __syncthreads_and(good) != 0;
  };

  // this block's rows, quads and 32-quad words
  const int32_t r0 = rows_before(p.rowbits, p.rowbase, share_start(p.nquads, blockIdx.x, NB), p.nquads, p.n);
  const int32_t r1 = rows_before(p.rowbits, p.rowbase, share_start(p.nquads, blockIdx.x + 1, NB), p.nquads, p.n);
  const int rows = r1 - r0;
  const int64_t qa = rows ? p.ioff[r0] >> 2 : 0, qe = rows ? p.ioff[r1] >> 2 : 0;
  const int64_t w0 = qa >> 5;
  const int nw = rows ? (int)(((qe + 31) >> 5) - w0) : 0;
  for (int i = tid; i < nw; i += LT) {
    sbits[i] = p.rowbits[w0 + i];
    sbase[i] = p.rowbase[w0 + i] - r0;
  }
  if (p.staged)
    for (int i = tid; i < nw * 32; i += LT) {
      const int64_t q = w0 * 32 + i;
      scol[i] = q < p.nquads ? ld_stream4(p.icol + 4 * q, pol_stream) : make_int4(p.n, p.n, p.n, p.n);
    }

  // the row of this thread (REGS)
  double rR = 0.0, rsc = 0.0;
  double2 rab = make_double2(0.0, 0.0);
  long long rc = 0;
  int32_t rd = 1, rdin = 0;
  int rw = 0, rwn = 0;   // words that continue the row: cont[rw .. rw + rwn)
  const bool have = REGS && tid < rows;
  const double r_init = 1.0 / (double)p.n;
  if (REGS) {
    if (have) {
      const int32_t v = r0 + tid;
      rd = p.odeg[v];
      rdin = p.ideg[v];
      const int64_t a = p.ioff[v] >> 2, b = p.ioff[v + 1] >> 2;
      rw = (int)((a >> 5) - w0) + 1;
      rwn = (int)(((b - 1) >> 5) - (a >> 5));
      rsc = rd < TAB ? p.tab_sc[rd] : FIX_ONE / (double)rd;
      if (CLOSED) rab = rd < TAB ? p.tab_ab[rd] : closed_coeffs(p.alpha, p.n, rd);
      if (p.method == 0 /* Static */) {
        rR = r_init;
        rc = __double2ll_rn(rR * rsc);
        p.R[v] = rR;
        p.C[0][v] = rc;
      } else {
        rR = p.R[v];
        rc = p.C[0][v];
      }
      if (FRONTIER) p.X[0][v] = 0;
      flag[tid] = FRONTIER ? 0 : 1;
    }
  } else {
    for (int i = tid; i < rows; i += LT) {
      const int32_t v = r0 + i;
      if (p.method == 0) {
        const int32_t d = p.odeg[v];
        p.R[v] = r_init;
        p.C[0][v] = __double2ll_rn(r_init * (d < TAB ? p.tab_sc[d] : FIX_ONE / (double)d));
      }
      if (FRONTIER) p.X[0][v] = 0;
      flag[i] = FRONTIER ? 0 : 1;
    }
  }
  if (FRONTIER) {
    const int64_t words = cdiv((int64_t)p.n, 32);
    for (int64_t i = blockIdx.x * (int64_t)LT + tid; i < words; i += (int64_t)NB * LT) p.S[i] = 0u;
  }
  if (blockIdx.x == 0 && tid < 3) st_relaxed_u64(&st->dR[tid], 0ull);
  if (!barrier()) return;
  if (FRONTIER) {
    // initial frontier F = S u out(X) (Alg. 1): X the sources of the effective
    // change, S the targets of its deletions
    const uint64_t mask = (1ull << p.id_bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)LT + tid; i < p.n_dmin + p.n_dplus; i += (int64_t)NB * LT) {
      const bool del = i < p.n_dmin;
      const uint64_t key = del ? p.dmin[i] : p.dplus[i - p.n_dmin];
      p.X[0][key >> p.id_bits] = 1;
      if (del) {
        const int32_t t = (int32_t)(key & mask);
        atomicOr(p.S + (t >> 5), 1u << (t & 31));
      }
    }
    if (!barrier()) return;
    for (int i = tid; i < rows; i += LT) flag[i] = (__ldcg(p.S + ((r0 + i) >> 5)) >> ((r0 + i) & 31)) & 1u;
    __syncthreads();
  }

  const double alpha_fix = p.alpha * FIX_INV;
  const bool same_tau = p.tau_f == p.tau_p;
  const unsigned upto = lane == 31 ? 0xffffffffu : ((2u << lane) - 1u);
  long long edges = 0, verts = 0, ever = 0;
  int cur = 0, it = 0, conv = 0;
  unsigned long long dR = 0ull, next_dR = 0ull;
  for (;;) {
    const long long* const C = p.C[cur];
    const uint8_t* const X = p.X[cur];
    const long long* const hub_end = C + p.l1_hub;
    // gather: the sums of the row pieces of every 32-quad word
    for (int wi = it < p.max_iter ? warp : nw; wi < nw; wi += U * LW) {
      int4 c[U];
      int own[U];
      long long s[U];
      unsigned wb[U], x[U];
      unsigned xv[REGS ? U : 1][4] = {};
#pragma unroll
      for (int j = 0; j < U; j++) {
        const int w = wi + j * LW;
        const int64_t q = (w0 + w) * 32 + lane;
        const bool valid = w < nw && q >= qa && q < qe;
        wb[j] = w < nw ? sbits[w] : 0u;
        own[j] = valid ? sbase[w] + __popc(wb[j] & upto) - 1 : -1;
        c[j] = valid ? (p.staged ? scol[w * 32 + lane] : ld_stream4(p.icol + 4 * q, pol_stream))
                     : make_int4(p.n, p.n, p.n, p.n);
      }
#pragma unroll
      for (int j = 0; j < U; j++) {
        const int32_t a[4] = {c[j].x, c[j].y, c[j].z, c[j].w};
        s[j] = 0;
#pragma unroll
        for (int e = 0; e < 4; e++) s[j] += a[e] == p.n ? 0ll : ld_weak_contrib(C + a[e], hub_end, pol_keep);
        x[j] = 0u;
        // (REGS: the bytes are kept apart until every load of the step is under
        // way; combined inside the branch they would be waited for there)
        if (FRONTIER && own[j] >= 0 && !(flag[own[j]] & 1)) {
          if (REGS) {
#pragma unroll
            for (int e = 0; e < 4; e++) xv[j][e] = a[e] == p.n ? 0u : ld_byte(X + a[e]);
          } else {
#pragma unroll
            for (int e = 0; e < 4; e++) x[j] |= a[e] == p.n ? 0u : ld_byte(X + a[e]);
          }
        }
      }
      if (REGS && FRONTIER)
#pragma unroll
        for (int j = 0; j < U; j++) x[j] = xv[j][0] | xv[j][1] | xv[j][2] | xv[j][3];
#pragma unroll
      for (int j = 0; j < U; j++) {
        const int w = wi + j * LW;
        if (w >= nw) break;   // the same in every lane
        long long sum = s[j];
        const unsigned vm = __ballot_sync(0xffffffffu, own[j] >= 0);
        const unsigned starts = wb[j] | 1u | (vm ^ (vm << 1));   // segment starts
        const unsigned later = starts & ~upto;
        const int end = later ? __ffs(later) - 1 : 32;       // this lane's row piece ends before it
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long os = __shfl_down_sync(0xffffffffu, sum, o);
          if (lane + o < end) sum += os;
        }
        unsigned any = 0u;
        if (FRONTIER) {
          const unsigned xm = __ballot_sync(0xffffffffu, x[j] != 0u);
          any = (xm & (unsigned)((1ull << end) - (1ull << lane))) != 0u;
        }
        if (own[j] >= 0 && ((starts >> lane) & 1u)) {
          if ((wb[j] >> lane) & 1u) {
            acc[own[j]] = sum;
            if (FRONTIER) accx[own[j]] = (uint8_t)any;
          } else {
            cont[w] = sum;
            if (FRONTIER) contx[w] = (uint8_t)any;
          }
        }
      }
    }
    if (tid == 0) red[LW] = next_dR;
    __syncthreads();
    // close the iteration before.  Its L-inf change is looked at only here, so
    // that its load overlaps the gather (which writes nothing but shared
    // memory); a block of more rows than threads has seen it after the barrier
    if (it > 0) {
      dR = red[LW];
      if (__longlong_as_double((long long)dR) <= p.tau) {
        conv = 1;
        break;
      }
    }
    if (it >= p.max_iter) break;
    // epilogue of the block's own vertices
    unsigned long long dmax = 0ull;
    if (REGS) {
      if (have) {
        const int32_t v = r0 + tid;
        long long sum = acc[tid];
        unsigned f = flag[tid];
        bool member = !FRONTIER || (f & 1) || accx[tid];
        for (int i = 0; i < rwn; i++) sum += cont[rw + i];
        if (FRONTIER && !member)
          for (int i = 0; i < rwn; i++) member = member || contx[rw + i];
        bool stay = false, expand = false;
        if (member) {
          double r;
          long long c;
          unsigned long long drb;
          row_update<CLOSED, REL>(p, alpha_fix, same_tau, sum, rc, rR, rd, rsc, rab, r, c, drb, stay, expand);
          dmax = drb;
          edges += rdin;
          verts += 1;
          rR = r;
          rc = c;
          p.R[v] = r;
          if (FRONTIER && !(f & 2)) ever++;
          f |= 2;
        }
        p.C[cur ^ 1][v] = rc;
        if (FRONTIER) {
          p.X[cur ^ 1][v] = expand;
          flag[tid] = (uint8_t)((f & 2) | (stay ? 1 : 0));
        }
      }
    } else {
      for (int i0 = tid; i0 < rows; i0 += 2 * LT) {
        double Rv[2];
        long long cs[2];
        int32_t d[2], din[2];
        int64_t a[2], b[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int i = i0 + u * LT;
          const bool in = i < rows;
          const int32_t v = r0 + (in ? i : 0);
          Rv[u] = in ? ld_weak(p.R + v) : 0.0;
          cs[u] = in ? ld_weak(C + v) : 0;
          d[u] = in ? __ldg(p.odeg + v) : 1;
          din[u] = in ? __ldg(p.ideg + v) : 0;
          a[u] = in ? __ldg(p.ioff + v) >> 2 : 0;
          b[u] = in ? __ldg(p.ioff + v + 1) >> 2 : 1;
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int i = i0 + u * LT;
          if (i >= rows) break;
          const int32_t v = r0 + i;
          long long sum = acc[i];
          unsigned f = flag[i];
          bool member = !FRONTIER || (f & 1) || accx[i];
          const int wa = (int)((a[u] >> 5) - w0) + 1, wn = (int)(((b[u] - 1) >> 5) - (a[u] >> 5));
          for (int e = 0; e < wn; e++) sum += cont[wa + e];
          if (FRONTIER && !member)
            for (int e = 0; e < wn; e++) member = member || contx[wa + e];
          bool stay = false, expand = false;
          if (member) {
            const double sc = d[u] < TAB ? __ldg(p.tab_sc + d[u]) : FIX_ONE / (double)d[u];
            double2 ab = make_double2(0.0, 0.0);
            if (CLOSED) ab = d[u] < TAB ? __ldg(p.tab_ab + d[u]) : closed_coeffs(p.alpha, p.n, d[u]);
            double r;
            unsigned long long drb;
            row_update<CLOSED, REL>(p, alpha_fix, same_tau, sum, cs[u], Rv[u], d[u], sc, ab, r, cs[u], drb, stay,
                                    expand);
            dmax = drb > dmax ? drb : dmax;
            edges += din[u];
            verts += 1;
            p.R[v] = r;
            if (FRONTIER && !(f & 2)) ever++;
            f |= 2;
          }
          p.C[cur ^ 1][v] = cs[u];
          if (FRONTIER) {
            p.X[cur ^ 1][v] = expand;
            flag[i] = (uint8_t)((f & 2) | (stay ? 1 : 0));
          }
        }
      }
    }
    // the block's change into the iteration's word, then the barrier.  Block 0
    // clears the next iteration's word: it was last read before the barrier
    // of the iteration before this one
    dmax = warp_max_u64(dmax);
    if (lane == 0) red[warp] = dmax;
    __syncthreads();
    bool good = true;
    if (warp == 0) {
      const unsigned long long m = warp_max_u64(red[lane]);
      if (lane == 0) {
        if (blockIdx.x == 0) st_relaxed_u64(&st->dR[(it + 1) % 3], 0ull);
        if (m) atomicMax(&st->dR[it % 3], m);
        good = grid_wait(st, p.out, (k + 1) * NB, p.polls);
        next_dR = ld_relaxed_u64(&st->dR[it % 3]);
        if (!REGS) red[LW] = next_dR;
      }
    }
    k++;
    if (!__syncthreads_and(good)) return;
    it++;
    cur ^= 1;
    if (!REGS && __longlong_as_double((long long)red[LW]) <= p.tau) {
      // no wasted gather where a gather takes tens of microseconds
      dR = red[LW];
      conv = 1;
      break;
    }
  }
  // outcome: the block's totals, and block 0's view of the loop (every block's
  // is the same)
  edges = warp_sum_ll(edges);
  verts = warp_sum_ll(verts);
  ever = warp_sum_ll(ever);
  if (lane == 0) {
    tot[0][warp] = edges;
    tot[1][warp] = verts;
    tot[2][warp] = ever;
  }
  __syncthreads();
  if (tid < 3) {
    long long s = 0;
    for (int i = 0; i < LW; i++) s += tot[tid][i];
    p.out->part[blockIdx.x][tid] = s;
  }
  if (blockIdx.x == 0 && tid == 0) {
    st->barriers = k;
    p.out->iter = it;
    p.out->converged = conv;
    p.out->cur = cur;
    p.out->dR_last = dR;
  }
}

__global__ void k_loop_shares(const int64_t* __restrict__ off, int32_t n, int64_t nquads,
                              const uint32_t* __restrict__ rowbits, const int32_t* __restrict__ rowbase, int NB,
                              int32_t* __restrict__ out) {
  for (int b = threadIdx.x; b < NB; b += blockDim.x) {
    const int32_t r0 = rows_before(rowbits, rowbase, share_start(nquads, b, NB), nquads, n);
    const int32_t r1 = rows_before(rowbits, rowbase, share_start(nquads, b + 1, NB), nquads, n);
    if (r1 <= r0) continue;
    atomicMax(out, r1 - r0);
    const int64_t q = (off[r1] - off[r0]) >> 2;
    atomicMax(out + 1, (int32_t)(q < INT32_MAX ? q : INT32_MAX));
  }
}

// default for a graph of fewer in-CSR slots, about 2.2M edges (larger ones run
// the CUDA graph, one launch pair and a control kernel per iteration).  Time per
// iteration here and there (us), ND, DF and DF-P from the previous ranks:
//   245K edges  4.5 / 16.6 (ND)
//   1.0M        7.5 / 18.7    9.9 / 19.1   13.9 / 23.5
//   2.1M       11.6 / 24.0   15.5 / 24.6   19.6 / 29.8
//   4.2M       19.5 / 32.5   26.4 / 33.1   31.2 / 37.2
//   6.6M       31.8 / 42.3   39.8 / 44.1   47.6 / 50.6
//   8.5M       41.8 / 46.8   47.6 / 48.0   55.8 / 54.0
// (above 10M a block's rows do not fit, loop_fits).  So the two cross near 8M
// edges for a graph that has the chip to itself.  The line is below that, at three
// times PR_ONE_KERNEL_SLOTS as dfpr.h says, because the loop holds every SM for
// the whole update and waits for every other such launch of the process, while
// the CUDA graph shares the chip with other streams' work: between 2.2M and 8M
// edges PR_OPT_ONE_KERNEL asks for it.
constexpr int64_t LOOP_SLOTS = 3ll << 20;

struct Layout {
  int32_t rows_cap, words_cap;
  bool staged;
  size_t bytes;
};
Layout layout(const Graph* g) {
  Layout l;
  l.rows_cap = (g->loop_rows + 15) / 16 * 16;
  l.words_cap = (g->loop_quads / 32 + 2 + 15) / 16 * 16;
  const size_t base = (8 + 2) * (size_t)l.rows_cap + (8 + 8 + 1) * (size_t)l.words_cap;
  const size_t cols = 512 * (size_t)l.words_cap;
  l.staged = base + cols <= STAGE_MAX;
  l.bytes = base + (l.staged ? cols : 0);
  return l;
}

}  // namespace

int loop_blocks() { return std::min(num_sms(), LOOP_MAX_BLOCKS); }
size_t loop_state_bytes() { return sizeof(LoopState); }

static std::atomic<int> g_loop_failure{0};   // of the next launch
void arm_loop_failure(int how) { g_loop_failure.store(how == LOOP_REFUSED || how == LOOP_STUCK ? how : 0); }

cudaError_t loop_reset(LoopState* st, cudaStream_t s) {
  return cudaMemsetAsync(st, 0, sizeof(*st), s);
}

bool loop_fits(const Graph* g) {
  if (g->loop_rows <= 0 || layout(g).bytes > LOOP_SMEM_MAX) return false;
  // one block works a whole row: a row much longer than a block's share would
  // leave the others waiting (4096 quads are four per thread, about 2 us)
  const int64_t share = cdiv(g->in.cap >> 2, loop_blocks());
  return g->loop_quads <= std::max<int64_t>(4096 + share, share + share / 2);
}

bool loop_default(const Graph* g) { return g->in.cap < LOOP_SLOTS && loop_fits(g); }

cudaError_t launch_loop_shares(const int64_t* off, int32_t n, int64_t nquads, const uint32_t* rowbits,
                               const int32_t* rowbase, int32_t* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, 2 * sizeof(int32_t), s);
  if (e != cudaSuccess) return e;
  note_launch();
  k_loop_shares<<<1, 256, 0, s>>>(off, n, nquads, rowbits, rowbase, loop_blocks(), out);
  return cudaGetLastError();
}

template <bool CLOSED, bool FRONTIER, bool REL>
static const void* loop_kernel(bool regs) {
  return regs ? (const void*)k_loop<CLOSED, FRONTIER, REL, true> : (const void*)k_loop<CLOSED, FRONTIER, REL, false>;
}

cudaError_t launch_loop(const Graph* g, LoopParams p, cudaStream_t s) {
  const int fail = g_loop_failure.exchange(0);
  if (fail == LOOP_REFUSED) return cudaErrorCooperativeLaunchTooLarge;
  p.polls = LOOP_SPINS;
  if (fail == LOOP_STUCK) {
    // barriers counted whose arrivals never come: every block's first wait runs out
    p.polls = LOOP_SPINS_STUCK;
    const unsigned long long far = 1ull << 40;
    const cudaError_t e = cudaMemcpyAsync(&p.st->barriers, &far, sizeof(far), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
  }
  const Layout l = layout(g);
  p.rows_cap = l.rows_cap;
  p.words_cap = l.words_cap;
  p.staged = l.staged ? 1 : 0;
  p.l1_hub = L1_HUB;
  const bool regs = g->loop_rows <= LT;
  const bool rel = p.metric == METRIC_RELATIVE;
  const void* fn;
  switch (p.method) {
    case 3: fn = rel ? loop_kernel<false, true, true>(regs) : loop_kernel<false, true, false>(regs); break;   // DF
    case 4: fn = rel ? loop_kernel<true, true, true>(regs) : loop_kernel<true, true, false>(regs); break;     // DF-P
    default: fn = loop_kernel<false, false, true>(regs); break;                                               // Static, ND
  }
  int bps = 0;
  cudaError_t e = kernel_occupancy(fn, LT, l.bytes, &bps);   // also raises the kernel's shared memory limit
  if (e != cudaSuccess) return e;
  void* args[] = {&p};
  note_launch();
  return cudaLaunchCooperativeKernel(fn, dim3(loop_blocks()), dim3(LT), args, l.bytes, s);
}

}  // namespace dfpr
