// loop.cuh -- the whole update of one graph in one cooperative kernel with one
// grid barrier per iteration (loop.cu).
#pragma once
#include "graph.cuh"
#include "sweep.cuh"

namespace dfpr {

constexpr int LOOP_MAX_BLOCKS = 256;
// the outcome of an update, written by the kernel to pinned host memory (a
// copy engine after the kernel adds about 10 us)
struct LoopOut {
  int32_t iter, converged, err, cur;
  unsigned long long dR_last;
  long long part[LOOP_MAX_BLOCKS][3];         // per block: in-edges, vertices, vertices ever affected
};
// what a launch leaves on the device for the next one
struct LoopState {
  unsigned long long count;      // arrivals at the grid barrier, over all launches
  unsigned long long pad0[15];
  unsigned long long dR[3];      // L-inf change of an iteration (mod 3), the bits of a non-negative double
  unsigned long long barriers;   // grid barriers completed, over all launches
  int32_t err;                   // 1: a wait ran out
  int32_t pad1;
};

struct LoopParams {
  int32_t n, method, max_iter, metric, id_bits;
  const int32_t* icol;
  const int64_t* ioff;
  const uint32_t* rowbits;
  const int32_t* rowbase;
  int64_t nquads;
  const int32_t* odeg;
  const int32_t* ideg;
  double* R;
  long long* C[2];          // C[0] holds the contributions of the ranks on entry
  uint8_t* X[2];            // n bytes each: the vertex expanded in the iteration before
  uint32_t* S;              // n bits: targets of deleted edges
  const uint64_t* dmin;
  const uint64_t* dplus;
  int64_t n_dmin, n_dplus;
  double alpha, C0, tau, tau_f, tau_p;
  const double* tab_sc;
  const double2* tab_ab;
  LoopState* st;
  LoopOut* out;             // pinned host memory; err must be 0 on entry
  int32_t rows_cap, words_cap, staged;
  int32_t l1_hub;           // contributions of internal ids below it are kept in L1
  long long polls;          // of a barrier wait before it gives up
};

// Whether a graph's rows can be shared out to the blocks as the loop wants it.
bool loop_fits(const Graph* g);
// Whether that loop is the default for it (when no flag names a loop).
bool loop_default(const Graph* g);
size_t loop_state_bytes();
// first use of a state, or after a launch that gave up
cudaError_t loop_reset(LoopState* st, cudaStream_t s);
// queue the update; p.rows_cap, words_cap, staged, l1_hub and polls are filled in here
cudaError_t launch_loop(const Graph* g, LoopParams p, cudaStream_t s);
int loop_blocks();
// the next launch fails (pr_debug_fail_loop): LOOP_REFUSED, the launch returns
// cudaErrorCooperativeLaunchTooLarge and nothing is launched; LOOP_STUCK, its
// first barrier waits for arrivals that never come and gives up after a short
// wait; 0 disarms
enum LoopFailure : int { LOOP_REFUSED = 1, LOOP_STUCK = 2 };
void arm_loop_failure(int how);

// the shares of the in-CSR's rows that loop_blocks() blocks get: writes
// {largest rows, largest quads} of a block to out[0..1]
cudaError_t launch_loop_shares(const int64_t* off, int32_t n, int64_t nquads, const uint32_t* rowbits,
                               const int32_t* rowbase, int32_t* out, cudaStream_t s);

}  // namespace dfpr
