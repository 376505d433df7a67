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
#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

namespace gvqe {

constexpr int CUT_MAX_LAYERS = 6;  // entangler layers, each with at least one crossing CNOT
constexpr int CUT_MAX_PATH = 6;    // crossing CNOTs in all, at most 64 terms
constexpr int CUT_MAX_PATH64 = 8;  // FP64 to 16 qubits: at most 256
constexpr int CUT_MAX_M = 15;      // qubits of a half

// One entangler layer as seen by one half: the GF(2)-affine map of its basis indices
// for each value b of the layer's path bits.  Bits 16 and 17 carry the layer's projections
// through the map: an amplitude is kept where both come out 0.
struct CutLayer {
  uint32_t fc[CUT_MAX_M];  // y = XOR of fc[q] over the set bits q of x, ^ fo[b]
  uint32_t ic[CUT_MAX_M];  // x = XOR of ic[q] over the set bits q of y, ^ io[b]
  uint32_t fo[4], io[4];
  int shift, nb;           // the layer's path bits: (a >> shift) & (2^nb - 1)
};

struct CutHalf {
  int m, q0;  // qubits, and the first one's index
  CutLayer L[CUT_MAX_LAYERS];
};

struct CutDesc {
  int n, reps, kappa, D;  // D = 2^kappa terms
  int cx;                 // 1: RY then RZ (complex amplitudes), FP32
  CutHalf half[2];        // 0: qubits [0, h), 1: qubits [h, n)
};

// Workspace of one evaluation (byte offsets) and how its contractions are split.
struct CutLayout {
  // A state is kept as its amplitudes [x], the same in runs of 16 bytes, and (FP32, RY) its low
  // parts [x]: SR = 2 or 3 times 2^m numbers.
  long long tab[2];   // L and R: [a][SR][x]
  long long pack[2];  // FP32: their tensor-core operand images (as rows and as columns)
  long long packr[2]; // complex: as rows, (x, channel) by two real terms per term; pack as columns
  long long phi[2];   // the half states after layers 0 .. reps - 1 (complex: reps), one per value of
                      // the path bits so far
  long long g[2];     // partial contractions: [split][a][x]
  long long gp;       // gradient partials (doubles): [half][a][(reps + 1) * 16]
  long long ep;       // per item of contraction 0: energy and norm (doubles)
  long long total;
  int rb[2], ns[2];   // row blocks and column splits of each contraction
  int gs[2];          // slices of g the backward adds up: ns, and one more with X/Y strings
  // X/Y strings (gvqe_cut_xy.cu)
  long long rows[2];   // the tables as [x][a]
  long long mpart[2];  // M of every part: [run][part][a][b]
  long long mm[2];     // ... summed, FP64
  long long nn[2];     // N: [part][b][a] (-1 without gradients)
  long long exy;       // energies per part of half 0 (doubles)
  int xrun[2];         // rows in one run of M's sum
  int nexy;            // parts of half 0 (0: no X/Y strings)
};

// The X/Y strings of a Hamiltonian as parts on the two halves (device arrays): part u of half
// h flips xm and signs with zm; its strings t in [start[u], start[u + 1]) pair it with part
// other[t] of the other half and carry coef[t].  Parts in order of xm; gstart: where xm changes.
struct CutXyDims {
  int U[2], ng[2];
};
struct CutXy : CutXyDims {
  const uint32_t *xm[2], *zm[2];
  const int *start[2], *other[2], *gstart[2];
  const double *coef[2];
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
  const void *cs;       // (cos, sin) of theta/2 per parameter, double2
  const void *table;    // E(x): FP64 in index order, FP32 in contraction 0's tile order
  const void *table_t;  // FP32: in contraction 1's tile order
  char *ws;
  const uint8_t *mask;  // or NULL
  double *E, *grad;
  const BatchIO *io;    // or NULL: mask, E and grad come from here
  CutLayout lay;
};

struct CutArgs {
  CutJob job0;
  const CutXy *xy;      // or NULL (diagonal H)
  const CutJob *jobs;   // NULL: job k is job0 stepped k times
  const int4 *items;    // with jobs: (job, half, index, 0) of each block of this launch
  long long ws_stride, cs_stride;  // bytes
  int P;                // parameters per job (with jobs == NULL)
  int njobs, nblk;
  int blk0;             // blocks of half 0 per job (without items)
  float *state;         // launch_cut_state: the states, state_stride floats apart
  long long state_stride;
};

// The cut plan of a circuit; false when it has none (no layer, too many layers or
// crossing CNOTs, halves out of range).
bool cut_build(int n, int reps, int ent, int prec, int gates, CutDesc *d);
CutLayout cut_layout(const CutDesc &d, int prec, bool grad, const CutXyDims *xy = nullptr);

// What the launches of one evaluation cover: the largest half and number of terms, and,
// for different problems in one launch, the blocks of the half circuits, of the operand
// images and of the contraction.  Problems share launches when their larger halves have
// the same cut_class.
struct CutGrid {
  int cx;        // complex amplitudes
  int m0, m1, D;  // m1: the smallest half
  int reps, bits[CUT_MAX_LAYERS + 1];  // one problem: path bits up to each layer; several: the most layers
  int half_blocks, con_blocks, pack_blocks;
  const int4 *half_items, *con_items, *pack_items;  // (job, half, path value | index | 64-row tile, 0)
};
int cut_class(int prec, int m);
int cut_k(int D);  // terms of the tensor-core operands
// The kernels of one evaluation, in order.  `grad`: also the gradients.
struct CutMark {  // told before and after the contraction (for the event profiler)
  virtual void mark(bool begin) = 0;
};
cudaError_t launch_cut(int prec, const CutArgs &A, const CutGrid &g, bool grad, cudaStream_t s, int *launches,
                       const CutXyDims *xy = nullptr, CutMark *mark = nullptr);
int cut_xy_dp(int D);  // row length of its matrices
// The state itself, S of every tile, for circuits that go on after these layers (FP32, RY): the
// half tables of all jobs, then the states of some.
cudaError_t launch_cut_halves(const CutArgs &A, const CutGrid &g, cudaStream_t s, int *launches);
cudaError_t launch_cut_state(const CutArgs &A, const CutGrid &g, cudaStream_t s, int *launches);
cudaError_t launch_cut_xy(const CutArgs &A, const CutGrid &g, const CutXyDims &x, bool grad, cudaStream_t s, int *launches);
// The diagonal table in the order the FP32 contractions read it, rounded from FP64:
// d0 for contraction 0 (rows x_lo), d1 for contraction 1 (rows x_hi; may be NULL).  Tiles
// of 128 rows x 64 columns, a row block's tiles after one another, each [j / 4][row][j % 4]
// (cx: the rows are (x, channel), and a tile holds one value for both channels, 64 rows).
struct TableJob {
  const double *src;
  float *d0, *d1;
  int m0, m1, cx;
};
// one table, or several at once (nmax: the largest m0 + m1)
cudaError_t launch_tile_table(const TableJob &t, cudaStream_t s);
cudaError_t launch_tile_tables(const TableJob *jobs, int njobs, int nmax, cudaStream_t s);
// The half circuits: FP32 forward (gvqe_cut_fwd.cu); the rest (gvqe_cut_half.cu) by mode, 0
// forward, 1 forward keeping the states the backward reads, 2 backward; m: the class of the
// larger half.
constexpr int HALF_SMALL_M(int prec) { return prec ? 7 : 10; }  // halves up to here share one kernel
cudaError_t launch_cut_fwd32(const CutArgs &A, const CutGrid &g, bool grad, cudaStream_t s, int *launches);  // FP32 forward
template <typename T>
cudaError_t launch_half(const CutArgs &A, int m, int mode, int blocks, cudaStream_t s);
cudaError_t launch_halfc(const CutArgs &A, int m, int mode, int blocks, cudaStream_t s);  // complex (gvqe_cut_halfc.cu)
// A kernel's dynamic shared-memory limit, raised once per device.
struct SmemLimit {
  std::atomic<uint64_t> done{0};
  template <typename K>
  cudaError_t set(K k, size_t bytes) {
    int dev = 0;
    if (const cudaError_t e = cudaGetDevice(&dev)) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
  }
};
// FP32 contraction on the tensor cores (gvqe_cut_tc.cu).
enum CutUse { CUT_ENERGY = 0, CUT_GRAD = 1, CUT_STATE = 2 };
cudaError_t launch_cut_tc(const CutArgs &A, int K, CutUse use, cudaStream_t s);

// What a kernel uses of job k (the layout is indexed in place, not copied).
struct CutView {
  const CutDesc *desc;
  const CutLayout *lay;
  const void *cs, *table, *table_t;
  char *ws;
};
__device__ __forceinline__ CutView cut_view(const CutArgs &A, int k) {
  const CutJob &j = A.jobs ? A.jobs[k] : A.job0;
  CutView v{j.desc, &j.lay, j.cs, j.table, j.table_t, j.ws};
  if (!A.jobs) {
    v.ws += (long long)k * A.ws_stride;
    v.cs = (const char *)v.cs + (long long)k * A.cs_stride;
  }
  return v;
}
struct CutOut {
  const uint8_t *mask;
  double *E, *grad;
};
__device__ __forceinline__ CutOut cut_out(const CutArgs &A, int k) {
  const CutJob &j = A.jobs ? A.jobs[k] : A.job0;
  if (j.io) return {j.io->mask, j.io->energy, j.io->grad};
  const long long o = A.jobs ? 0 : k;
  return {j.mask ? j.mask + o * A.P : nullptr, j.E + o, j.grad ? j.grad + o * A.P : nullptr};
}

}  // namespace gvqe
