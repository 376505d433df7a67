// gvqe_cut_half.cu -- the circuits of the two halves (gvqe_cut.cuh), forward and adjoint;
// compiled once per amplitude type (GVQE_INST_T).
//
// One CTA runs one half's circuit for one value a of the path bits, its 2^M amplitudes
// in shared memory and 2^E per thread in registers (32 from M = 10).  A layer is a gather
// through the layer's affine map straight into the registers of the top E bits, RY on
// those, and more register rounds: the bits between (MID) and the lowest (LOW, runs of
// consecutive amplitudes in 16-byte accesses).  16 bytes of padding per 128 keep runs,
// rows and columns apart in the banks.  M is a template argument, so that every shared-
// memory access is a base and an immediate; FP32 rotations run as packed f32x2.
// One CTA per SM at M = 15 (147 KB, 1024 threads of 64 registers), one warp up to M = 10.
// Bound by shared-memory wavefronts and issue: about 200 and 700 per warp and layer.
#include "gvqe_cut.cuh"

namespace gvqe {

// FP64: four warps where the half allows it, one per FP64 pipe of the SM.
template <typename T>
__host__ __device__ constexpr int half_e(int M) {
  return sizeof(T) == 4 ? (M >= 10 ? 5 : M == 9 ? 4 : M >= 7 ? 3 : 2) : (M >= 12 ? 5 : M == 11 ? 4 : M == 10 ? 3 : 2);
}
template <typename T, int M>
struct HalfCfg {
  static constexpr int E = half_e<T>(M);      // register bits
  static constexpr int LT = M - E;            // log2 of the working threads
  static constexpr int G0 = LT < E ? LT : E;  // LOW bits; the other LT - G0 are MID's, at most E at a time
  static constexpr int NT = LT < 5 ? 32 : 1 << LT;
  static_assert(G0 >= 2, "runs of 16 bytes");
};

template <typename T>
struct CutT;
template <>
struct CutT<float> {
  using T2 = float2;
  using V = float4;  // 16 bytes
  static constexpr int ROW = 5, VN = 4;
};
template <>
struct CutT<double> {
  using T2 = double2;
  using V = double2;
  static constexpr int ROW = 4, VN = 2;
};

// place of amplitude i; pad(i | j) = pad(i) + pad(j) for disjoint bits
template <typename T>
__host__ __device__ __forceinline__ constexpr int pad(int i) {
  return i + ((i >> CutT<T>::ROW) << (sizeof(T) == 4 ? 2 : 1));
}

using f2 = unsigned long long;  // two packed floats
__device__ __forceinline__ f2 pk2(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpk2(f2 v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// RY (sg = 1) or its inverse (sg = -1) on register bits 0 .. G-1 of the 2^G values v
template <int G, typename T>
__device__ __forceinline__ void rotate(T *v, const typename CutT<T>::T2 *cs, T sg) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const T c = cs[k].x, s = cs[k].y * sg;
#pragma unroll
      for (int i = 0; i < (1 << G); ++i)
        if (!((i >> k) & 1)) {
          const T a = v[i], b = v[i | (1 << k)];
          v[i] = c * a - s * b;
          v[i | (1 << k)] = s * a + c * b;
        }
    }
  } else {
    {  // bit 0: within the pairs
      const float c = cs[0].x, s = cs[0].y * sg;
#pragma unroll
      for (int i = 0; i < (1 << G); i += 2) {
        const float a = v[i], b = v[i + 1];
        v[i] = c * a - s * b;
        v[i + 1] = s * a + c * b;
      }
    }
    if constexpr (G > 1) {
      constexpr int H = 1 << (G - 1);
      f2 p[H];
#pragma unroll
      for (int i = 0; i < H; ++i) p[i] = pk2(v[2 * i], v[2 * i + 1]);
#pragma unroll
      for (int k = 1; k < G; ++k) {
        const float cc = cs[k].x, ss = cs[k].y * sg;
        const f2 c = pk2(cc, cc), s = pk2(ss, ss), ns = pk2(-ss, -ss);
#pragma unroll
        for (int i = 0; i < H; ++i)
          if (!((i >> (k - 1)) & 1)) {
            const f2 a = p[i], b = p[i | (1 << (k - 1))];
            p[i] = fma2(c, a, mul2(ns, b));
            p[i | (1 << (k - 1))] = fma2(s, a, mul2(c, b));
          }
      }
#pragma unroll
      for (int i = 0; i < H; ++i) unpk2(p[i], v[2 * i], v[2 * i + 1]);
    }
  }
}

// acc[k] += sum of G1 phi0 - G0 phi1 over register bit k; phi(i) loads pairs i, i + 1
template <int G, typename T, typename F>
__device__ __forceinline__ void grads(const T *v, F phi, T *acc) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int i = 0; i < (1 << G); i += 2) {
      T p[2];
      phi(i, p);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < G; ++k) {
          const T g = v[(i + j) ^ (1 << k)];
          acc[k] = (((i + j) >> k) & 1) ? acc[k] - g * p[j] : acc[k] + g * p[j];
        }
    }
  } else {
    f2 a2[G];
#pragma unroll
    for (int k = 1; k < G; ++k) a2[k] = 0;
    const f2 neg1 = pk2(-1.f, -1.f);
#pragma unroll
    for (int i = 0; i < (1 << G); i += 2) {
      float p[2];
      phi(i, p);
      acc[0] += v[i + 1] * p[0];
      acc[0] -= v[i] * p[1];
      const f2 pp = pk2(p[0], p[1]), pn = mul2(pp, neg1);
#pragma unroll
      for (int k = 1; k < G; ++k) {
        const int o = i ^ (1 << k);
        a2[k] = fma2(pk2(v[o], v[o + 1]), ((i >> k) & 1) ? pn : pp, a2[k]);
      }
    }
#pragma unroll
    for (int k = 1; k < G; ++k) {
      float x, y;
      unpk2(a2[k], x, y);
      acc[k] += x + y;
    }
  }
}

template <int I>
struct Int {
  static constexpr int value = I;
};

// One half circuit of 2^M amplitudes: this thread's share of its state in shared memory.
template <typename T, int M>
struct Half {
  using C = HalfCfg<T, M>;
  using T2 = typename CutT<T>::T2;
  using V = typename CutT<T>::V;
  static constexpr int N = 1 << C::E, VN = CutT<T>::VN;
  T *st;
  int tid;
  bool on;  // a working thread (fewer than a warp below M = 8)

  __device__ __forceinline__ void sync() const {
    if constexpr (C::NT == 32)
      __syncwarp();
    else
      __syncthreads();
  }
  // TOP: value s is amplitude tid + (s << LT)
  __device__ __forceinline__ void top_load(T *v) const {
    const T *p = st + pad<T>(tid);
    if (on)
#pragma unroll
      for (int s = 0; s < N; ++s) v[s] = p[pad<T>(s << C::LT)];
  }
  __device__ __forceinline__ void top_store(const T *v) const {
    T *p = st + pad<T>(tid);
    if (on)
#pragma unroll
      for (int s = 0; s < N; ++s) p[pad<T>(s << C::LT)] = v[s];
  }
  // v = the state gathered through an affine map, in TOP order
  __device__ __forceinline__ void gather(T *v, const uint32_t *col, uint32_t off) const {
    uint32_t x = off;
#pragma unroll
    for (int q = 0; q < C::LT; ++q)
      if ((tid >> q) & 1) x ^= col[q];
#pragma unroll
    for (int e = 0; e < N; ++e) {  // places in Gray order: one column per step
      if (e > 0) x ^= col[C::LT + (e & 1 ? 0 : e & 2 ? 1 : e & 4 ? 2 : e & 8 ? 3 : 4)];
      T a = (T)0;
      if (on && (x >> 16) == 0) a = st[pad<T>((int)x)];
      v[e ^ (e >> 1)] = a;
    }
  }
  // LOW: item it holds amplitudes (it << G0) + [0, 2^G0); MID: bits [G0, G0 + GM) of item it
  template <typename F>
  __device__ __forceinline__ void low_round(F f) const {
    if (on)
#pragma unroll
      for (int q = 0; q < (1 << (C::E - C::G0)); ++q) {
        const int it = tid + (q << C::LT);
        T *p = st + pad<T>(it << C::G0);  // (a run of 32 FP64 amplitudes spans two padded rows)
        alignas(16) T v[1 << C::G0];
#pragma unroll
        for (int j = 0; j < (1 << C::G0); j += VN)
          *reinterpret_cast<V *>(v + j) = *reinterpret_cast<const V *>(p + pad<T>(j));
        if (f(it, v))
#pragma unroll
          for (int j = 0; j < (1 << C::G0); j += VN)
            *reinterpret_cast<V *>(p + pad<T>(j)) = *reinterpret_cast<const V *>(v + j);
      }
  }
  // f(LO, G): every group of MID bits [LO, LO + G)
  template <int LO, typename F>
  __device__ __forceinline__ void mid_groups(F f) const {
    if constexpr (LO < C::LT) {
      constexpr int G = C::LT - LO < C::E ? C::LT - LO : C::E;
      f(Int<LO>{}, Int<G>{});
      mid_groups<LO + G>(f);
    }
  }
  template <int LO, int G, typename F>
  __device__ __forceinline__ void mid_round(F f) const {
    if (on)
#pragma unroll
      for (int q = 0; q < (1 << (C::E - G)); ++q) {
        const int it = tid + (q << C::LT);
        const int base = (it & ((1 << LO) - 1)) | ((it >> LO) << (LO + G));
        T *p = st + pad<T>(base);
        T v[1 << G];
#pragma unroll
        for (int s = 0; s < (1 << G); ++s) v[s] = p[pad<T>(s << LO)];
        if (f(base, v))
#pragma unroll
          for (int s = 0; s < (1 << G); ++s) p[pad<T>(s << LO)] = v[s];
      }
  }
  // a state kept for the backward sweep: natural order, and item it of the LOW round in runs of
  // 16 bytes, [j][it]
  __device__ __forceinline__ void keep_natural(T *dst) const {
    T v[N];
    top_load(v);
    if (on)
#pragma unroll
      for (int s = 0; s < N; ++s) dst[tid + (s << C::LT)] = v[s];
  }
  static constexpr int ITEMS = 1 << (M - C::G0);
  __device__ __forceinline__ void keep_run(T *dst, int it, const T *v) const {
#pragma unroll
    for (int j = 0; j < (1 << C::G0) / VN; ++j)
      reinterpret_cast<V *>(dst)[j * ITEMS + it] = reinterpret_cast<const V *>(v)[j];
  }
};

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

// the circuit of one half as its kernels hold it
template <typename T>
struct HalfShared {
  typename CutT<T>::T2 cs[(CUT_MAX_LAYERS + 1) * CUT_MAX_M];
  CutHalf H;
  T red[32 * 16];
};

template <typename T>
__device__ __forceinline__ void half_setup(HalfShared<T> &sh, const CutView &J, int h, int M) {
  for (int i = threadIdx.x; i < (int)(sizeof(CutHalf) / 4); i += blockDim.x)
    reinterpret_cast<int *>(&sh.H)[i] = reinterpret_cast<const int *>(&J.desc->half[h])[i];
  const int n = J.desc->n, q0 = h ? J.desc->half[0].m : 0, np = (J.desc->reps + 1) * M;
  for (int i = threadIdx.x; i < np; i += blockDim.x)
    sh.cs[i] = reinterpret_cast<const typename CutT<T>::T2 *>(J.cs)[(i / M) * n + q0 + i % M];
  __syncthreads();
}

template <typename T, int M, bool GRAD>
__device__ __forceinline__ void half_fwd(const CutView &J, int h, int a, T *st, HalfShared<T> &sh) {
  using HF = Half<T, M>;
  using C = typename HF::C;
  const HF S{st, (int)threadIdx.x, (int)threadIdx.x < (1 << C::LT)};
  const int reps = J.desc->reps;
  constexpr long long SZ = 1LL << M;
  T v[HF::N];
  {  // layer 0: the product state, in TOP order
    T b = (T)1;
#pragma unroll
    for (int q = 0; q < C::LT; ++q) b *= ((S.tid >> q) & 1) ? sh.cs[q].y : sh.cs[q].x;
    v[0] = b;
#pragma unroll
    for (int j = 0; j < C::E; ++j)
#pragma unroll
      for (int s = 0; s < (1 << j); ++s) {
        v[s | (1 << j)] = v[s] * sh.cs[C::LT + j].y;
        v[s] *= sh.cs[C::LT + j].x;
      }
  }
  S.top_store(v);
  S.sync();
  T *phi = reinterpret_cast<T *>(J.ws + J.lay->phi[h]);
  if (GRAD && a == 0) {
    S.keep_natural(phi);
    S.low_round([&](int it, T *u) {
      S.keep_run(phi + SZ, it, u);
      return false;
    });
  }
  for (int r = 1; r <= reps; ++r) {
    const CutLayer &l = sh.H.L[r - 1];
    const typename HF::T2 *cs = sh.cs + r * M;
    S.gather(v, l.ic, l.io[(a >> l.shift) & ((1 << l.nb) - 1)]);
    rotate<C::E>(v, cs + C::LT, (T)1);
    S.sync();
    S.top_store(v);
    S.sync();
    S.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      S.template mid_round<LO, G>([&](int, T *u) {
        rotate<G>(u, cs + LO, (T)1);
        return true;
      });
      S.sync();
    });
    // the state after layer r < reps depends on the path bits so far only: kept once
    T *nat, *run;
    bool keep;
    if (r < reps) {
      phi += 2 * (SZ << l.shift);
      const int bits = l.shift + l.nb;
      nat = phi + (size_t)2 * a * SZ;
      run = nat + SZ;
      keep = GRAD && (a >> bits) == 0;
    } else {
      T *tab = reinterpret_cast<T *>(J.ws + J.lay->tab[h]);
      nat = tab + (size_t)a * SZ;
      run = tab + (size_t)(J.desc->D + a) * SZ;
      keep = true;
    }
    S.low_round([&](int it, T *u) {
      rotate<C::G0>(u, cs, (T)1);
      if (GRAD && keep) S.keep_run(run, it, u);
      return true;
    });
    S.sync();
    if (keep) S.keep_natural(nat);
  }
}

// The adjoint sweep of one half's circuit for one path value, from G_a (the sum of its
// column splits): per layer the RY gradients of all its qubits against the stored state,
// RY(-theta), and the transposed map.
template <typename T, int M>
__device__ __forceinline__ void half_bwd(const CutView &J, int h, int a, T *st, HalfShared<T> &sh) {
  using HF = Half<T, M>;
  using C = typename HF::C;
  using V = typename HF::V;
  const HF S{st, (int)threadIdx.x, (int)threadIdx.x < (1 << C::LT)};
  const int reps = J.desc->reps, D = J.desc->D, lane = S.tid & 31, w = S.tid >> 5;
  constexpr long long SZ = 1LL << M;
  T v[HF::N];
  {
    const T *g = reinterpret_cast<const T *>(J.ws + J.lay->g[h]) + (size_t)a * SZ + S.tid;
    const int ns = J.lay->ns[h];
#pragma unroll
    for (int s = 0; s < HF::N; ++s) v[s] = S.on ? g[s << C::LT] : (T)0;
    for (int k = 1; k < ns; ++k) {
      g += (size_t)D * SZ;
#pragma unroll
      for (int s = 0; s < HF::N; ++s)
        if (S.on) v[s] += g[s << C::LT];
    }
  }
  S.top_store(v);
  double *gp = reinterpret_cast<double *>(J.ws + J.lay->gp) + ((size_t)h * D + a) * (reps + 1) * 16;
  const T *tab = reinterpret_cast<const T *>(J.ws + J.lay->tab[h]);
  const T *nat = tab + (size_t)a * SZ, *run = tab + (size_t)(D + a) * SZ;
  const T *phi = reinterpret_cast<const T *>(J.ws + J.lay->phi[h]);
  for (int r = 0; r < reps; ++r) phi += 2 * (SZ << sh.H.L[r].shift);
  for (int r = reps;; --r) {
    const typename HF::T2 *cs = sh.cs + r * M;
    T acc[M];
#pragma unroll
    for (int q = 0; q < M; ++q) acc[q] = (T)0;
    if (S.on)
      grads<C::E>(v, [&](int i, T *p) {
        p[0] = nat[S.tid + (i << C::LT)];
        p[1] = nat[S.tid + ((i + 1) << C::LT)];
      }, acc + C::LT);
    S.sync();
    // every gradient before any rotation, but for the last round's own bits
    constexpr bool MID = C::LT > C::G0;
    S.low_round([&](int it, T *u) {
      V x;
      grads<C::G0>(u, [&](int i, T *p) {
        if (i % HF::VN == 0) x = reinterpret_cast<const V *>(run)[(i / HF::VN) * HF::ITEMS + it];
        const T *xs = reinterpret_cast<const T *>(&x);
        p[0] = xs[i % HF::VN];
        p[1] = xs[i % HF::VN + 1];
      }, acc);
      if (MID || r == 0) return false;
      rotate<C::G0>(u, cs, (T)-1);
      return true;
    });
    S.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      if (LO + G == C::LT) S.sync();  // the last group: its writes come after all reads
      S.template mid_round<LO, G>([&](int base, T *u) {
        grads<G>(u, [&](int i, T *p) {
          p[0] = nat[base + (i << LO)];
          p[1] = nat[base + ((i + 1) << LO)];
        }, acc + LO);
        if (LO + G < C::LT || r == 0) return false;
        rotate<G>(u, cs + LO, (T)-1);
        return true;
      });
    });
    // this layer's gradients: lanes, then warps in FP64
#pragma unroll
    for (int q = 0; q < M; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    }
    if constexpr (C::NT == 32) {
#pragma unroll
      for (int q = 0; q < M; ++q)
        if (lane == q) gp[r * 16 + q] = (double)acc[q];
    } else {
      if (lane == 0)
#pragma unroll
        for (int q = 0; q < M; ++q) sh.red[w * 16 + q] = acc[q];
      __syncthreads();
      if (S.tid < M) {
        double s = 0.0;
        for (int k = 0; k < C::NT / 32; ++k) s += (double)sh.red[k * 16 + S.tid];
        gp[r * 16 + S.tid] = s;
      }
    }
    if (r == 0) break;
    if constexpr (MID) {
      if constexpr (C::NT == 32) S.sync();
      S.template mid_groups<C::G0>([&](auto lo, auto g) {
        constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
        if constexpr (LO + G < C::LT) {
          S.template mid_round<LO, G>([&](int, T *u) {
            rotate<G>(u, cs + LO, (T)-1);
            return true;
          });
          S.sync();
        }
      });
      S.low_round([&](int, T *u) {
        rotate<C::G0>(u, cs, (T)-1);
        return true;
      });
    }
    S.sync();
    S.top_load(v);
    rotate<C::E>(v, cs + C::LT, (T)-1);
    S.top_store(v);
    S.sync();
    const CutLayer &l = sh.H.L[r - 1];
    S.gather(v, l.fc, l.fo[(a >> l.shift) & ((1 << l.nb) - 1)]);
    S.sync();
    S.top_store(v);
    phi -= 2 * (SZ << l.shift);
    nat = phi + (size_t)2 * (a & ((1 << l.shift) - 1)) * SZ;
    run = nat + SZ;
  }
}

// MODE 0: forward, 1: forward keeping what the backward reads, 2: backward.  One kernel for
// all sizes that run in one warp (mixed in a batch), and one per size M above, which also
// takes the other half of an odd register, a qubit smaller, with some threads idle.
template <typename T, int MODE, int M>
__device__ __forceinline__ void half_run(const CutView &J, int h, int a, T *st, HalfShared<T> &sh) {
  half_setup(sh, J, h, M);
  if (HalfCfg<T, M>::NT == 32 && threadIdx.x >= 32) return;
  if constexpr (MODE == 2)
    half_bwd<T, M>(J, h, a, st, sh);
  else
    half_fwd<T, M, MODE == 1>(J, h, a, st, sh);
}
constexpr int WARP_M = HALF_WARP_M(sizeof(GVQE_INST_T) == 8);
template <typename T, int MODE, int M>
__global__ void __launch_bounds__(HalfCfg<T, M>::NT) k_half(const __grid_constant__ CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  __shared__ HalfShared<T> sh;
  const int3 it = cut_half_item(A);
  const CutView J = cut_view(A, it.x);
  T *st = reinterpret_cast<T *>(cut_smem);
  const int m = J.desc->half[it.y].m;
  if constexpr (M > WARP_M) {
    if (m == M)
      half_run<T, MODE, M>(J, it.y, it.z, st, sh);
    else
      half_run<T, MODE, M - 1>(J, it.y, it.z, st, sh);
  } else {
    if constexpr (sizeof(T) == 8) {
      if (m == 5) half_run<T, MODE, 5>(J, it.y, it.z, st, sh);
      if (m == 6) half_run<T, MODE, 6>(J, it.y, it.z, st, sh);
      if (m == 7) half_run<T, MODE, 7>(J, it.y, it.z, st, sh);
    } else {
      if (m == 7) half_run<T, MODE, 7>(J, it.y, it.z, st, sh);
      if (m == 8) half_run<T, MODE, 8>(J, it.y, it.z, st, sh);
      if (m == 9) half_run<T, MODE, 9>(J, it.y, it.z, st, sh);
      if (m == 10) half_run<T, MODE, 10>(J, it.y, it.z, st, sh);
    }
  }
}

template <typename T, int MODE, int M>
static cudaError_t launch_half_m(const CutArgs &A, int blocks, cudaStream_t s) {
  constexpr size_t sm = (size_t)pad<T>(1 << M) * sizeof(T);
  static SmemLimit limit;
  if (const cudaError_t e = limit.set(k_half<T, MODE, M>, sm)) return e;
  k_half<T, MODE, M><<<blocks, HalfCfg<T, M>::NT, sm, s>>>(A);
  return cudaGetLastError();
}

template <typename T, int MODE>
static cudaError_t launch_half_mode(const CutArgs &A, int m, int blocks, cudaStream_t s) {
  switch (m) {
    case WARP_M: return launch_half_m<T, MODE, WARP_M>(A, blocks, s);
    case WARP_M + 1: return launch_half_m<T, MODE, WARP_M + 1>(A, blocks, s);
    case WARP_M + 2: return launch_half_m<T, MODE, WARP_M + 2>(A, blocks, s);
    case WARP_M + 3: return launch_half_m<T, MODE, WARP_M + 3>(A, blocks, s);
    case WARP_M + 4: return launch_half_m<T, MODE, WARP_M + 4>(A, blocks, s);
    case WARP_M + 5: return launch_half_m<T, MODE, WARP_M + 5>(A, blocks, s);
  }
  if constexpr (WARP_M + 7 == 14) {  // FP64: 14 is the largest half, FP32: 15
    if (m == 13) return launch_half_m<T, MODE, 13>(A, blocks, s);
    if (m == 14) return launch_half_m<T, MODE, 14>(A, blocks, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_half<GVQE_INST_T>(const CutArgs &A, int m, int mode, int blocks, cudaStream_t s) {
  if (mode == 0) return launch_half_mode<GVQE_INST_T, 0>(A, m, blocks, s);
  if (mode == 1) return launch_half_mode<GVQE_INST_T, 1>(A, m, blocks, s);
  return launch_half_mode<GVQE_INST_T, 2>(A, m, blocks, s);
}

}  // namespace gvqe
