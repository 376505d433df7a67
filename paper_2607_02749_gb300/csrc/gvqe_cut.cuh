// gvqe_cut.cuh -- evaluation of a circuit from its two halves (shared declarations).
//
// Cut the register between qubits h - 1 and h.  Every CNOT of an entangler layer
// (Section IV-B) that crosses the cut is sum_b |b><b| (x) X^b: for a fixed bit b the
// control's half is projected and the target's half is flipped, and nothing couples
// the halves any more.  With K crossing CNOTs in the whole circuit the final state is
//   psi(x_hi, x_lo) = sum_{a < 2^K} L_a(x_lo) R_a(x_hi),
// where a collects the bits and L_a, R_a are circuits on h and n - h qubits.  The
// energy of a diagonal H and the gradient's two contractions need psi only tile by
// tile (lambda = E(x) psi(x)):
//   E = sum lambda psi,  G_L(x_lo, a) = sum_{x_hi} lambda R_a,  G_R(x_hi, a) = sum_{x_lo} lambda L_a,
// and dE/dtheta of an RY in one half is the sum over a of <G_a| J |phi_a>, the adjoint
// sweep of that half's own circuit started from G_a.  No 2^n state is stored, read or
// written: one pass over E(x) per contraction replaces the tile passes of every layer.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace gvqe {

constexpr int CUT_MAX_LAYERS = 6;  // entangler layers, each with at least one crossing CNOT
constexpr int CUT_MAX_PATH = 6;    // crossing CNOTs in all: at most 64 terms
constexpr int CUT_MAX_M = 15;      // qubits of a half

// One entangler layer as seen by one half: the GF(2)-affine map of its basis indices
// for each value b of the layer's path bits, and its projections.
struct CutLayer {
  uint16_t fc[CUT_MAX_M];  // y = XOR of fc[q] over the set bits q of x, ^ fo[b]
  uint16_t ic[CUT_MAX_M];  // x = XOR of ic[q] over the set bits q of y, ^ io[b]
  uint16_t fo[4], io[4];
  uint16_t pm[2];          // projection k keeps x with parity(x & pm[k]) == bit b of pt[k]
  uint8_t pt[2];
  uint8_t np;              // projections of this layer in this half
  uint8_t shift, nb;       // the layer's path bits: (a >> shift) & (2^nb - 1)
};

struct CutHalf {
  int m, q0;  // qubits, and the first one's index
  CutLayer L[CUT_MAX_LAYERS];
};

struct CutDesc {
  int n, reps, kappa, D;  // D = 2^kappa terms
  CutHalf half[2];        // 0: qubits [0, h), 1: qubits [h, n)
};

// Workspace of one evaluation (byte offsets) and how its contractions are split.
struct CutLayout {
  long long tab[2];   // L and R: [a][x], amplitude type
  long long pack[2];  // FP32: their tensor-core operand images
  long long phi[2];   // the half states after layers 0 .. reps - 1, one per value of the path bits so far
  long long g[2];     // partial contractions: [split][a][x]
  long long gp;       // gradient partials (doubles): [half][a][(reps + 1) * 16]
  long long ep;       // per item of contraction 0: energy and norm (doubles)
  long long total;
  int rb[2], ns[2];   // row blocks and column splits of each contraction
};

// The caller's buffers of one batch instance (read when the kernels run).
struct BatchIO {
  const double *params;  // P doubles
  const uint8_t *mask;   // P bytes or NULL (all active)
  double *grad;          // P doubles or NULL
  double *energy;        // one double
};

// One evaluation: a launch over several vectors of one (ansatz, Hamiltonian) pair
// steps the pointers of job 0; a launch over different problems reads an array.
struct CutJob {
  const CutDesc *desc;
  const void *cs;       // (cos, sin) of theta/2 per parameter
  const void *table;    // E(x), amplitude type
  const void *table_t;  // FP32: E with the halves of its index exchanged
  char *ws;
  const uint8_t *mask;  // or NULL
  double *E, *grad;
  const BatchIO *io;    // or NULL: mask, E and grad come from here
  CutLayout lay;
};

struct CutArgs {
  CutJob job0;
  const CutJob *jobs;   // NULL: job k is job0 stepped k times
  const int4 *items;    // with jobs: (job, half, index, 0) of each block of this launch
  long long ws_stride, cs_stride;  // bytes
  int P;                // parameters per job (with jobs == NULL)
  int njobs, nblk;
  int blk0;             // blocks of half 0 per job (without items)
};

// The cut plan of a circuit; false when it has none (no layer, too many layers or
// crossing CNOTs, halves out of range).
bool cut_build(int n, int reps, int ent, int prec, CutDesc *d);
CutLayout cut_layout(const CutDesc &d, int prec, bool grad);

// What the launches of one evaluation cover: the largest low half and number of terms,
// and, for different problems in one launch, the blocks of the half circuits and of the
// contraction.  The threads of a half circuit's CTA fix the order of its sums, so only
// problems with equal cut_threads share a launch.
struct CutGrid {
  int m0, D;
  int half_blocks, con_blocks;
  const int4 *half_items, *con_items;
};
int cut_threads(int m0);
int cut_k(int D);  // terms of the tensor-core operands
// The kernels of one evaluation, in order.  `grad`: also the gradients.
cudaError_t launch_cut(int prec, const CutArgs &A, const CutGrid &g, bool grad, cudaStream_t s, int *launches);
// dst[x_lo][x_hi] = src[x_hi][x_lo], x_lo of m0 and x_hi of m1 bits (both at least 5):
// one table, or several at once (nmax: the largest m0 + m1).
struct TransposeJob {
  const float *src;
  float *dst;
  int m0, m1;
};
cudaError_t launch_transpose_table(const TransposeJob &t, cudaStream_t s);
cudaError_t launch_transpose_tables(const TransposeJob *jobs, int njobs, int nmax, cudaStream_t s);
// FP32 contraction on the tensor cores (gvqe_cut_tc.cu).
cudaError_t launch_cut_tc(const CutArgs &A, int K, bool grad, cudaStream_t s);

__device__ __forceinline__ CutJob cut_job(const CutArgs &A, int k) {
  if (A.jobs) {
    CutJob j = A.jobs[k];
    if (j.io) {
      j.mask = j.io->mask;
      j.E = j.io->energy;
      j.grad = j.io->grad;
    }
    return j;
  }
  CutJob j = A.job0;
  j.ws += (long long)k * A.ws_stride;
  j.cs = (const char *)j.cs + (long long)k * A.cs_stride;
  if (j.mask) j.mask += (long long)k * A.P;
  j.E += k;
  if (j.grad) j.grad += (long long)k * A.P;
  return j;
}

}  // namespace gvqe
