// gvqe_cut.cu -- evaluation of a circuit from its two halves: plan, half circuits,
// the FP64 contraction and the final sums (the FP32 contraction is gvqe_cut_tc.cu).
#include <cstring>
#include <utility>
#include <vector>

#include "gvqe_cut.cuh"
#include "gvqe_engine.cuh"

namespace gvqe {

// ------------------------------------------------------------------ plan --
// The CNOT list of entangler layer r.  FULL is taken as the reverse-linear list, the
// same unitary with one CNOT per bond instead of n (n - 1) / 2.
static std::vector<std::pair<int, int>> cnot_list(int ent, int n, int r) {
  std::vector<std::pair<int, int>> v;
  if (n < 2) return v;
  auto ring = [&]() {
    v.push_back({n - 1, 0});
    for (int i = 0; i + 1 < n; ++i) v.push_back({i, i + 1});
  };
  switch (ent) {
    case ENT_CIRCULAR:
      ring();
      break;
    case ENT_FULL:
    case ENT_REVERSE_LINEAR:
      for (int i = n - 2; i >= 0; --i) v.push_back({i, i + 1});
      break;
    case ENT_PAIRWISE:
      for (int i = 0; i + 1 < n; i += 2) v.push_back({i, i + 1});
      for (int i = 1; i + 1 < n; i += 2) v.push_back({i, i + 1});
      break;
    case ENT_SCA: {
      ring();
      const int s = (r - 1) % n;
      std::vector<std::pair<int, int>> w(v.end() - s, v.end());
      w.insert(w.end(), v.begin(), v.end() - s);
      v = w;
      if ((r - 1) & 1)
        for (auto &g : v) std::swap(g.first, g.second);
      break;
    }
    default:
      for (int i = 0; i + 1 < n; ++i) v.push_back({i, i + 1});
  }
  return v;
}

static int parity32(uint32_t x) { return __builtin_parity(x); }

bool cut_build(int n, int reps, int ent, int prec, CutDesc *d) {
  memset(d, 0, sizeof(*d));
  const int h = (n + 1) / 2;
  // FP32: 128-row and 64-column tiles in the contraction; FP64: 32 x 32 tiles, and a half's
  // state (with its padding) in one CTA's shared memory
  if (reps < 1 || reps > CUT_MAX_LAYERS || n - h < (prec ? 5 : 7) || h > (prec ? CUT_MAX_M - 1 : CUT_MAX_M)) return false;
  d->n = n;
  d->reps = reps;
  const int lo[3] = {0, h, n};
  for (int s = 0; s < 2; ++s) {
    d->half[s].m = lo[s + 1] - lo[s];
    d->half[s].q0 = lo[s];
  }
  int kappa = 0;
  for (int r = 1; r <= reps; ++r) {
    CutLayer *L[2] = {&d->half[0].L[r - 1], &d->half[1].L[r - 1]};
    // every bit of a half as an affine function of its input bits and the path bits
    uint32_t xm[2][CUT_MAX_M], bm[2][CUT_MAX_M];
    for (int s = 0; s < 2; ++s)
      for (int q = 0; q < d->half[s].m; ++q) {
        xm[s][q] = 1u << q;
        bm[s][q] = 0;
      }
    int nb = 0;
    for (const auto &g : cnot_list(ent, n, r)) {
      const int sc = g.first >= h, st = g.second >= h;
      const int c = g.first - lo[sc], t = g.second - lo[st];
      if (sc == st) {
        xm[st][t] ^= xm[sc][c];
        bm[st][t] ^= bm[sc][c];
        continue;
      }
      if (nb == 2 || L[sc]->np == 2) return false;
      const int k = L[sc]->np++;
      L[sc]->pm[k] = (uint16_t)xm[sc][c];
      uint8_t pt = 0;
      for (uint32_t b = 0; b < 4; ++b) pt |= (uint8_t)(parity32((bm[sc][c] ^ (1u << nb)) & b) << b);
      L[sc]->pt[k] = pt;
      bm[st][t] ^= 1u << nb;
      ++nb;
    }
    for (int s = 0; s < 2; ++s) {
      const int m = d->half[s].m;
      CutLayer &l = *L[s];
      l.shift = (uint8_t)kappa;
      l.nb = (uint8_t)nb;
      uint32_t rows[CUT_MAX_M], inv[CUT_MAX_M];
      for (int q = 0; q < m; ++q) {
        rows[q] = xm[s][q];
        inv[q] = 1u << q;
        for (int i = 0; i < m; ++i)
          if ((xm[s][q] >> i) & 1u) l.fc[i] |= (uint16_t)(1u << q);
        for (uint32_t b = 0; b < 4; ++b) l.fo[b] |= (uint16_t)(parity32(bm[s][q] & b) << q);
      }
      for (int col = 0; col < m; ++col) {
        int piv = col;
        while (piv < m && !((rows[piv] >> col) & 1u)) ++piv;
        if (piv == m) return false;  // a CNOT product is invertible
        std::swap(rows[col], rows[piv]);
        std::swap(inv[col], inv[piv]);
        for (int q = 0; q < m; ++q)
          if (q != col && ((rows[q] >> col) & 1u)) {
            rows[q] ^= rows[col];
            inv[q] ^= inv[col];
          }
      }
      for (int q = 0; q < m; ++q)  // bit q of x is parity(inv[q] & y)
        for (int i = 0; i < m; ++i)
          if ((inv[q] >> i) & 1u) l.ic[i] |= (uint16_t)(1u << q);
      for (uint32_t b = 0; b < 4; ++b) {
        uint32_t x = 0;
        for (int i = 0; i < m; ++i)
          if ((l.fo[b] >> i) & 1u) x ^= l.ic[i];
        l.io[b] = (uint16_t)x;
      }
    }
    kappa += nb;
    if (kappa > CUT_MAX_PATH) return false;
  }
  d->kappa = kappa;
  d->D = 1 << kappa;
  return true;
}

// Terms of the tensor-core operands: at least 16 (the smallest N of its MMAs).
int cut_k(int D) { return D < 16 ? 16 : D; }

constexpr int CUT_ROWS32 = 128, CUT_COLS32 = 64;  // FP32 contraction tile
constexpr int CUT_TILE64 = 32;                    // FP64 contraction tile (square)

CutLayout cut_layout(const CutDesc &d, int prec, bool grad) {
  CutLayout l;
  memset(&l, 0, sizeof(l));
  const long long es = prec ? 8 : 4;
  long long off = 0;
  auto take = [&](long long bytes) {
    const long long o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  };
  for (int s = 0; s < 2; ++s) {
    const long long S = 1LL << d.half[s].m;
    const int mo = d.half[1 - s].m;
    l.rb[s] = (int)(S / (prec ? CUT_TILE64 : CUT_ROWS32));
    const long long tiles = (1LL << mo) / (prec ? CUT_TILE64 : CUT_COLS32);
    // enough items for 152 SMs on a single vector, but runs long enough that an item's
    // set-up (its rows into tensor memory, the first tiles) stays small
    const long long per = prec ? 8 : 32;
    l.ns[s] = (int)(tiles / per < 1 ? 1 : tiles / per > 4 ? 4 : tiles / per);
    l.tab[s] = take(d.D * S * es);
    if (!prec) l.pack[s] = take(S * cut_k(d.D) * 16);
    if (grad) {
      long long states = 0;
      for (int r = 0; r < d.reps; ++r) states += 1LL << d.half[s].L[r].shift;
      l.phi[s] = take(states * S * es);
      l.g[s] = take((long long)l.ns[s] * d.D * S * es);
    }
  }
  if (grad) l.gp = take(2LL * d.D * (d.reps + 1) * 16 * 8);
  l.ep = take((long long)l.rb[0] * l.ns[0] * 16);
  l.total = off;
  return l;
}

// ---------------------------------------------------------- half circuits --
// One CTA runs one half's circuit for one value a of the path bits, its 2^m
// amplitudes in shared memory (padded by one element per 32 FP32 / 16 FP64 so that
// neither runs nor powers of two of stride share a bank).  A layer is a gather through
// the layer's affine map (amplitudes that fail a projection are zero) and RY on every
// qubit in register rounds of up to 5 (FP64: 4) qubits.  At m = 15 that is 132 KB and
// 1024 threads, 64 registers each: one CTA per SM, bound by its shared-memory rounds.
template <typename T>
struct CutT;
template <>
struct CutT<float> {
  using T2 = float2;
  static constexpr int PAD = 5, GMAX = 5;
};
template <>
struct CutT<double> {
  using T2 = double2;
  static constexpr int PAD = 4, GMAX = 4;
};
constexpr int CUT_NT = 1024;
template <typename T>
constexpr int CUT_EPT = sizeof(T) == 8 ? 16 : 32;  // elements a thread holds in a gather: 2^14 (FP64), 2^15 over 1024

template <typename T>
__device__ __forceinline__ int cpad(int i) {
  return i + (i >> CutT<T>::PAD);
}

__device__ __forceinline__ uint32_t cut_map(const uint16_t *col, uint32_t v) {
  uint32_t r = 0;
  while (v) {
    const int q = __ffs(v) - 1;
    v &= v - 1;
    r ^= col[q];
  }
  return r;
}

// st[y] = keep(y) ? st[src(y)] : 0 for the whole half.  fwd: src is A^-1 and the
// projections test the source; else src is A and they test the place itself.
template <typename T>
__device__ void cut_gather(T *st, const CutLayer &l, int m, int b, bool fwd) {
  const int NT = blockDim.x, tid = threadIdx.x, S = 1 << m;
  const uint16_t *col = fwd ? l.ic : l.fc;
  const uint32_t off = fwd ? l.io[b] : l.fo[b];
  const int np = l.np;
  const uint32_t p0 = l.pm[0], p1 = l.pm[1];
  const int t0 = (l.pt[0] >> b) & 1, t1 = (l.pt[1] >> b) & 1;
  T v[CUT_EPT<T>];
  uint32_t src = cut_map(col, tid) ^ off;
  const int lnt = 31 - __clz(NT);
#pragma unroll
  for (int e = 0; e < CUT_EPT<T>; ++e) {  // places in Gray order: one column per step
    const int gray = e ^ (e >> 1);
    if (e > 0) {
      const int bit = lnt + __ffs(e) - 1;
      if (bit < m) src ^= col[bit];
    }
    const int y = tid | (gray << lnt);
    T x = (T)0;
    if (y < S) {
      const uint32_t chk = fwd ? src : (uint32_t)y;
      bool ok = true;
      if (np > 0) ok = (__popc(chk & p0) & 1) == t0;
      if (np > 1) ok = ok && (__popc(chk & p1) & 1) == t1;
      if (ok) x = st[cpad<T>((int)src)];
    }
    v[e] = x;
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < CUT_EPT<T>; ++e) {
    const int y = tid | ((e ^ (e >> 1)) << lnt);
    if (y < S) st[cpad<T>(y)] = v[e];
  }
  __syncthreads();
}

// RY (sign = 1) or its inverse (sign = -1) on qubits [lo, lo + G)
template <typename T, int G>
__device__ __forceinline__ void cut_rotate(T *st, int m, int lo, const typename CutT<T>::T2 *cs, T sign) {
  const int items = 1 << (m - G), low = (1 << lo) - 1;
  typename CutT<T>::T2 w[G];
#pragma unroll
  for (int k = 0; k < G; ++k) {
    w[k] = cs[lo + k];
    w[k].y *= sign;
  }
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int base = (it & low) | ((it >> lo) << (lo + G));
    T v[1 << G];
#pragma unroll
    for (int s = 0; s < (1 << G); ++s) v[s] = st[cpad<T>(base + (s << lo))];
#pragma unroll
    for (int k = 0; k < G; ++k)
#pragma unroll
      for (int s = 0; s < (1 << G); ++s)
        if (!((s >> k) & 1)) {
          const T a = v[s], b = v[s | (1 << k)];
          v[s] = w[k].x * a - w[k].y * b;
          v[s | (1 << k)] = w[k].y * a + w[k].x * b;
        }
#pragma unroll
    for (int s = 0; s < (1 << G); ++s) st[cpad<T>(base + (s << lo))] = v[s];
  }
  __syncthreads();
}

// sums of G1 phi0 - G0 phi1 for qubits [lo, lo + G), one per warp into red[warp][qubit]
template <typename T, int G>
__device__ __forceinline__ void cut_grads(const T *st, const T *phi, int m, int lo, T *red) {
  const int items = 1 << (m - G), low = (1 << lo) - 1;
  T acc[G];
#pragma unroll
  for (int k = 0; k < G; ++k) acc[k] = (T)0;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int base = (it & low) | ((it >> lo) << (lo + G));
    T v[1 << G];
#pragma unroll
    for (int s = 0; s < (1 << G); ++s) v[s] = st[cpad<T>(base + (s << lo))];
#pragma unroll
    for (int s = 0; s < (1 << G); ++s) {
      const T p = phi[base + (s << lo)];
#pragma unroll
      for (int k = 0; k < G; ++k) {
        if ((s >> k) & 1)
          acc[k] -= v[s ^ (1 << k)] * p;
        else
          acc[k] += v[s ^ (1 << k)] * p;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < G; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if ((threadIdx.x & 31) == 0) red[(threadIdx.x >> 5) * 16 + lo + k] = acc[k];
  }
}

// the register rounds of one layer: about equal groups of at most GMAX qubits
template <typename T, typename F>
__device__ __forceinline__ void cut_rounds(int m, F f) {
  const int nr = (m + CutT<T>::GMAX - 1) / CutT<T>::GMAX;
  int lo = 0;
  for (int r = 0; r < nr; ++r) {
    const int g = (m - lo + nr - r - 1) / (nr - r);
    f(lo, g);
    lo += g;
  }
}
template <typename T>
__device__ __forceinline__ void cut_rotate_all(T *st, int m, const typename CutT<T>::T2 *cs, T sign) {
  cut_rounds<T>(m, [&](int lo, int g) {
    if (g == 5) {
      if constexpr (CutT<T>::GMAX >= 5) cut_rotate<T, 5>(st, m, lo, cs, sign);
    } else if (g == 4) {
      cut_rotate<T, 4>(st, m, lo, cs, sign);
    } else if (g == 3) {
      cut_rotate<T, 3>(st, m, lo, cs, sign);
    } else {
      cut_rotate<T, 2>(st, m, lo, cs, sign);
    }
  });
}
template <typename T>
__device__ __forceinline__ void cut_grads_all(const T *st, const T *phi, int m, T *red) {
  cut_rounds<T>(m, [&](int lo, int g) {
    if (g == 5) {
      if constexpr (CutT<T>::GMAX >= 5) cut_grads<T, 5>(st, phi, m, lo, red);
    } else if (g == 4) {
      cut_grads<T, 4>(st, phi, m, lo, red);
    } else if (g == 3) {
      cut_grads<T, 3>(st, phi, m, lo, red);
    } else {
      cut_grads<T, 2>(st, phi, m, lo, red);
    }
  });
}

// block -> (job, half, path value)
__device__ __forceinline__ int3 cut_half_item(const CutArgs &A) {
  if (A.items) {
    const int4 it = A.items[blockIdx.x];
    return make_int3(it.x, it.y, it.z);
  }
  const int per = 2 * A.blk0;  // blk0: the D of every job
  const int job = blockIdx.x / per, r = blockIdx.x % per;
  return make_int3(job, r / A.blk0, r % A.blk0);
}

// element (x, a) of the tensor-core images of a half's table: per 64 rows x the blocks
// [hi | lo] of the row form (K-major over a) and [hi | lo] of the column form (rows a,
// K-major over x); core matrices of 8 rows x 16 bytes
__device__ __forceinline__ void cut_pack(float *pack, int K, int x, int a, float v) {
  float hi;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=f"(hi) : "f"(v));
  const float lo = v - hi;
  float *t = pack + (size_t)(x >> 6) * (256 * K);
  const int r = x & 63;
  const int o1 = (r >> 3) * (K * 8) + (a >> 2) * 32 + (r & 7) * 4 + (a & 3);
  const int o2 = (a >> 3) * 512 + (r >> 2) * 32 + (a & 7) * 4 + (r & 3);
  t[o1] = hi;
  t[64 * K + o1] = lo;
  t[128 * K + o2] = hi;
  t[192 * K + o2] = lo;
}

template <typename T, bool GRAD>
__global__ void __launch_bounds__(CUT_NT) k_cut_fwd(const CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  T *st = reinterpret_cast<T *>(cut_smem);
  using T2 = typename CutT<T>::T2;
  __shared__ T2 cs[(CUT_MAX_LAYERS + 1) * CUT_MAX_M];
  __shared__ CutHalf H;
  const int3 it = cut_half_item(A);
  const CutJob J = cut_job(A, it.x);
  const int h = it.y, a = it.z, tid = threadIdx.x, NT = blockDim.x;
  const int n = J.desc->n, reps = J.desc->reps, D = J.desc->D;
  for (int i = tid; i < (int)(sizeof(CutHalf) / 4); i += NT)
    reinterpret_cast<int *>(&H)[i] = reinterpret_cast<const int *>(&J.desc->half[h])[i];
  __syncthreads();
  const int m = H.m, S = 1 << m;
  for (int i = tid; i < (reps + 1) * m; i += NT)
    cs[i] = reinterpret_cast<const T2 *>(J.cs)[(i / m) * n + H.q0 + i % m];
  __syncthreads();
  // layer 0: the product state
  for (int i = tid; i < S; i += NT) {
    T v = (T)1;
    for (int q = 0; q < m; ++q) v *= ((i >> q) & 1) ? cs[q].y : cs[q].x;
    st[cpad<T>(i)] = v;
  }
  __syncthreads();
  T *phi = reinterpret_cast<T *>(J.ws + J.lay.phi[h]);
  for (int r = 1; r <= reps; ++r) {
    const CutLayer &l = H.L[r - 1];
    if (GRAD) {
      // the state after layer r - 1 depends on the path bits below l.shift only: kept once
      if ((a >> l.shift) == 0)
        for (int i = tid; i < S; i += NT) phi[(size_t)a * S + i] = st[cpad<T>(i)];
      phi += (size_t)S << l.shift;
    }
    cut_gather<T>(st, l, m, (a >> l.shift) & ((1 << l.nb) - 1), true);
    cut_rotate_all<T>(st, m, cs + r * m, (T)1);
  }
  T *tab = reinterpret_cast<T *>(J.ws + J.lay.tab[h]) + (size_t)a * S;
  if constexpr (sizeof(T) == 4) {
    float *pack = reinterpret_cast<float *>(J.ws + J.lay.pack[h]);
    const int K = D < 16 ? 16 : D;
    for (int i = tid; i < S; i += NT) {
      const float v = st[cpad<T>(i)];
      if (GRAD) tab[i] = v;
      cut_pack(pack, K, i, a, v);
      for (int z = a + D; z < K; z += D) cut_pack(pack, K, i, z, 0.f);
    }
  } else {
    for (int i = tid; i < S; i += NT) tab[i] = st[cpad<T>(i)];
  }
}

// The adjoint sweep of one half's circuit for one path value, from G_a (the sum of
// its column splits): per layer the RY gradients of all its qubits against the stored
// state, RY(-theta), and the transposed map.
template <typename T>
__global__ void __launch_bounds__(CUT_NT) k_cut_bwd(const CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  T *st = reinterpret_cast<T *>(cut_smem);
  using T2 = typename CutT<T>::T2;
  __shared__ T2 cs[(CUT_MAX_LAYERS + 1) * CUT_MAX_M];
  __shared__ CutHalf H;
  __shared__ T red[32 * 16];
  const int3 it = cut_half_item(A);
  const CutJob J = cut_job(A, it.x);
  const int h = it.y, a = it.z, tid = threadIdx.x, NT = blockDim.x;
  const int n = J.desc->n, reps = J.desc->reps, D = J.desc->D;
  for (int i = tid; i < (int)(sizeof(CutHalf) / 4); i += NT)
    reinterpret_cast<int *>(&H)[i] = reinterpret_cast<const int *>(&J.desc->half[h])[i];
  __syncthreads();
  const int m = H.m, S = 1 << m;
  for (int i = tid; i < (reps + 1) * m; i += NT)
    cs[i] = reinterpret_cast<const T2 *>(J.cs)[(i / m) * n + H.q0 + i % m];
  const T *g = reinterpret_cast<const T *>(J.ws + J.lay.g[h]) + (size_t)a * S;
  const int ns = J.lay.ns[h];
  for (int i = tid; i < S; i += NT) {
    T v = g[i];
    for (int k = 1; k < ns; ++k) v += g[(size_t)k * D * S + i];
    st[cpad<T>(i)] = v;
  }
  __syncthreads();
  double *gp = reinterpret_cast<double *>(J.ws + J.lay.gp) + ((size_t)h * D + a) * (reps + 1) * 16;
  const T *phi = reinterpret_cast<const T *>(J.ws + J.lay.tab[h]) + (size_t)a * S;
  const T *base = reinterpret_cast<const T *>(J.ws + J.lay.phi[h]);
  for (int r = 0; r < reps; ++r) base += (size_t)S << H.L[r].shift;
  for (int r = reps;; --r) {
    cut_grads_all<T>(st, phi, m, red);
    __syncthreads();
    if (tid < m) {
      double s = 0.0;
      for (int w = 0; w < NT / 32; ++w) s += (double)red[w * 16 + tid];
      gp[r * 16 + tid] = s;
    }
    if (r == 0) break;
    cut_rotate_all<T>(st, m, cs + r * m, (T)-1);
    const CutLayer &l = H.L[r - 1];
    cut_gather<T>(st, l, m, (a >> l.shift) & ((1 << l.nb) - 1), false);
    base -= (size_t)S << l.shift;
    phi = base + (size_t)(a & ((1 << l.shift) - 1)) * S;
  }
}

// ------------------------------------------------------ FP64 contraction --
// Items of 32 rows x a run of columns, 256 threads, 32 x 32 tiles: psi = sum_a L_a R_a
// (2 x 2 per thread), lambda = E psi into shared memory, G += lambda x the column
// table.  The FP64 pipe bounds it (about 2 multiply-adds per clock and SM): 2 D per
// amplitude and contraction against 6 (reps + 1) n of the gate-by-gate sweeps.
constexpr int C64 = CUT_TILE64, C64LD = C64 + 1;

template <bool GRAD>
__global__ void __launch_bounds__(256) k_cut_contract64(const CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  int job, h, idx;
  if (A.items) {
    const int4 it = A.items[blockIdx.x];
    job = it.x;
    h = it.y;
    idx = it.z;
  } else {  // the vectors of one item next to each other: they read the same part of E
    job = blockIdx.x % A.njobs;
    idx = blockIdx.x / A.njobs;
    h = idx >= A.blk0;
    if (h) idx -= A.blk0;
  }
  const CutJob J = cut_job(A, job);
  const int D = J.desc->D, m0 = J.desc->half[0].m;
  const int mr = J.desc->half[h].m, mc = J.desc->half[1 - h].m;
  const int ns = J.lay.ns[h], split = idx % ns, row0 = (idx / ns) * C64;
  const long long Sr = 1LL << mr, Sc = 1LL << mc;
  const int cols = (int)(Sc / ns), col0 = split * cols;
  const double *rt = reinterpret_cast<const double *>(J.ws + J.lay.tab[h]);
  const double *ct = reinterpret_cast<const double *>(J.ws + J.lay.tab[1 - h]);
  const double *E = reinterpret_cast<const double *>(J.table);
  double *sR = reinterpret_cast<double *>(cut_smem), *sC = sR + D * C64LD, *sL = sC + D * C64LD;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int i = tid; i < D * C64; i += 256) sR[(i >> 5) * C64LD + (i & 31)] = rt[(i >> 5) * Sr + row0 + (i & 31)];
  double acc[8], e = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.0;
  const int gi = tid & 31, ga = tid >> 5;  // G: row gi, terms ga + 8 k
  for (int c0 = col0; c0 < col0 + cols; c0 += C64) {
    __syncthreads();
    for (int i = tid; i < D * C64; i += 256) sC[(i >> 5) * C64LD + (i & 31)] = ct[(i >> 5) * Sc + c0 + (i & 31)];
    double t[2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const long long i = row0 + tx + 16 * p, j = c0 + ty + 16 * q;
        t[p][q] = E[h ? ((i << m0) | j) : ((j << m0) | i)];
      }
    __syncthreads();
    double s[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    for (int a = 0; a < D; ++a) {
      const double r0 = sR[a * C64LD + tx], r1 = sR[a * C64LD + tx + 16];
      const double q0 = sC[a * C64LD + ty], q1 = sC[a * C64LD + ty + 16];
      s[0][0] = fma(r0, q0, s[0][0]);
      s[0][1] = fma(r0, q1, s[0][1]);
      s[1][0] = fma(r1, q0, s[1][0]);
      s[1][1] = fma(r1, q1, s[1][1]);
    }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double lam = t[p][q] * s[p][q];
        e = fma(lam, s[p][q], e);
        if (GRAD) sL[(ty + 16 * q) * C64LD + tx + 16 * p] = lam;
      }
    if constexpr (GRAD) {
      __syncthreads();
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int a = ga + 8 * k;
        if (a < D) {
          double g0 = 0.0, g1 = 0.0;
#pragma unroll 8
          for (int j = 0; j < C64; j += 2) {
            g0 = fma(sL[j * C64LD + gi], sC[a * C64LD + j], g0);
            g1 = fma(sL[(j + 1) * C64LD + gi], sC[a * C64LD + j + 1], g1);
          }
          acc[k] += g0 + g1;
        }
      }
    }
  }
  if constexpr (GRAD) {
    double *g = reinterpret_cast<double *>(J.ws + J.lay.g[h]) + (size_t)split * D * Sr;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (ga + 8 * k < D) g[(ga + 8 * k) * Sr + row0 + gi] = acc[k];
  }
  if (h == 0) {
    __shared__ double es[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0) es[tid >> 5] = e;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < 8; ++w) s += es[w];
      double *ep = reinterpret_cast<double *>(J.ws + J.lay.ep) + 2 * idx;
      ep[0] = s;
      ep[1] = 0.0;
    }
  }
}

// ------------------------------------------------------------ final sums --
// One CTA per job: E and, per parameter, the sum over the path values in a fixed
// order.  The FP32 contraction also sums psi^2: E and the gradients are divided by that
// norm, which takes the rounding of cos, sin and of the tensor cores' accumulation out
// of the results to first order (it is 1 up to that rounding).
__global__ void __launch_bounds__(256) k_cut_reduce(const CutArgs A, int prec, int grad) {
  const CutJob J = cut_job(A, blockIdx.x);
  const int tid = threadIdx.x;
  __shared__ double sh[2][256];
  const double *ep = reinterpret_cast<const double *>(J.ws + J.lay.ep);
  const int ni = J.lay.rb[0] * J.lay.ns[0];
  double e = 0.0, z = 0.0;
  for (int i = tid; i < ni; i += 256) {
    e += ep[2 * i];
    z += ep[2 * i + 1];
  }
  sh[0][tid] = e;
  sh[1][tid] = z;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (tid < o) {
      sh[0][tid] += sh[0][tid + o];
      sh[1][tid] += sh[1][tid + o];
    }
    __syncthreads();
  }
  const double inv = prec ? 1.0 : 1.0 / sh[1][0];
  if (tid == 0) *J.E = sh[0][0] * inv;
  if (!grad) return;
  const int n = J.desc->n, reps = J.desc->reps, D = J.desc->D, m0 = J.desc->half[0].m;
  const double *gp = reinterpret_cast<const double *>(J.ws + J.lay.gp);
  for (int p = tid; p < n * (reps + 1); p += 256) {
    const int r = p / n, q = p % n, h = q >= m0;
    const double *src = gp + (size_t)h * D * (reps + 1) * 16 + r * 16 + (h ? q - m0 : q);
    double s = 0.0;
    for (int a = 0; a < D; ++a) s += src[(size_t)a * (reps + 1) * 16];
    J.grad[p] = (J.mask && !J.mask[p]) ? 0.0 : s * inv;
  }
}

__global__ void __launch_bounds__(256) k_transpose(const TransposeJob t0, const TransposeJob *jobs) {
  __shared__ float t[32][33];
  const TransposeJob T = jobs ? jobs[blockIdx.y] : t0;
  if (blockIdx.x >> (T.m0 + T.m1 - 10)) return;
  const int c0 = (blockIdx.x & ((1 << (T.m0 - 5)) - 1)) * 32, r0 = (blockIdx.x >> (T.m0 - 5)) * 32;  // x_lo, x_hi
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int k = y; k < 32; k += 8) t[k][x] = T.src[((long long)(r0 + k) << T.m0) + c0 + x];
  __syncthreads();
  for (int k = y; k < 32; k += 8) T.dst[((long long)(c0 + k) << T.m1) + r0 + x] = t[x][k];
}

cudaError_t launch_transpose_table(const TransposeJob &t, cudaStream_t s) {
  k_transpose<<<1u << (t.m0 + t.m1 - 10), 256, 0, s>>>(t, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_transpose_tables(const TransposeJob *jobs, int njobs, int nmax, cudaStream_t s) {
  for (int j = 0; j < njobs; j += 32768) {  // the grid's second dimension ends at 65535
    k_transpose<<<dim3(1u << (nmax - 10), (unsigned)(njobs - j < 32768 ? njobs - j : 32768)), 256, 0, s>>>(
        TransposeJob{}, jobs + j);
  }
  return cudaGetLastError();
}

// The same limit for every launch of a kernel, so that threads do not race on it: the
// largest half state (2^14 FP64, 2^15 FP32 amplitudes and their padding)
constexpr int CUT_SMEM_MAX = 17 * 8192;
template <typename K>
static cudaError_t set_smem(K k) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, CUT_SMEM_MAX);
}

// 16 amplitudes a thread where the half allows it
int cut_threads(int m0) { return m0 >= 14 ? 1024 : m0 <= 10 ? 64 : 1 << (m0 - 4); }

cudaError_t launch_cut(int prec, const CutArgs &A0, const CutGrid &g, bool grad, cudaStream_t s, int *launches) {
  CutArgs A = A0;
  const int es = prec ? 8 : 4, nt = cut_threads(g.m0);
  const size_t half_smem = (size_t)es * ((1 << g.m0) + (1 << (g.m0 - (prec ? 4 : 5))));
  const CutLayout &l = A.job0.lay;
  const int half_blocks = g.half_items ? g.half_blocks : A.njobs * 2 * g.D;
  cudaError_t e;
#define CUT_CHECK(x) \
  if ((e = (x)) != cudaSuccess) return e
  A.blk0 = g.D;
  A.items = g.half_items;
  if (prec) {
    auto k = grad ? k_cut_fwd<double, true> : k_cut_fwd<double, false>;
    CUT_CHECK(set_smem(k));
    k<<<half_blocks, nt, half_smem, s>>>(A);
  } else {
    auto k = grad ? k_cut_fwd<float, true> : k_cut_fwd<float, false>;
    CUT_CHECK(set_smem(k));
    k<<<half_blocks, nt, half_smem, s>>>(A);
  }
  CUT_CHECK(cudaGetLastError());
  A.blk0 = l.rb[0] * l.ns[0];
  A.nblk = g.con_items ? g.con_blocks : A.njobs * (A.blk0 + (grad ? l.rb[1] * l.ns[1] : 0));
  A.items = g.con_items;
  if (prec) {
    auto k = grad ? k_cut_contract64<true> : k_cut_contract64<false>;
    const size_t sm = (size_t)8 * C64LD * (2 * g.D + (grad ? C64 : 0));
    CUT_CHECK(set_smem(k));
    k<<<A.nblk, 256, sm, s>>>(A);
    CUT_CHECK(cudaGetLastError());
  } else {
    CUT_CHECK(launch_cut_tc(A, cut_k(g.D), grad, s));
  }
  *launches += 3;
  if (grad) {
    A.blk0 = g.D;
    A.items = g.half_items;
    if (prec) {
      CUT_CHECK(set_smem(k_cut_bwd<double>));
      k_cut_bwd<double><<<half_blocks, nt, half_smem, s>>>(A);
    } else {
      CUT_CHECK(set_smem(k_cut_bwd<float>));
      k_cut_bwd<float><<<half_blocks, nt, half_smem, s>>>(A);
    }
    CUT_CHECK(cudaGetLastError());
    *launches += 1;
  }
  k_cut_reduce<<<A.njobs, 256, 0, s>>>(A, prec, grad ? 1 : 0);
#undef CUT_CHECK
  return cudaGetLastError();
}

}  // namespace gvqe
