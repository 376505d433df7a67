// gvqe_cut_half.cuh -- device parts shared by the real and the complex half circuits of the
// two-half evaluation (gvqe_cut_half.cu, gvqe_cut_halfc.cu).
//
// One CTA runs one half's circuit for one value a of the path bits, its 2^M amplitudes
// in shared memory and 2^E per thread in registers (32 from M = 11).  A layer is a gather
// through the layer's affine map straight into the registers of the top E bits, RY on
// those, and more register rounds: the bits between (MID) and the lowest (LOW, runs of
// consecutive amplitudes in 16-byte accesses).  16 bytes of padding per 128 keep runs,
// rows and columns apart in the banks.  M is a template argument, so that every shared-
// memory access is a base and an immediate; FP32 rotations run as packed f32x2.
// One CTA per SM at M = 15 (147 KB, 1024 threads of 64 registers).
// Bound by shared-memory wavefronts and issue: about 200 and 700 per warp and layer.
#pragma once
#include "gvqe_cut.cuh"

namespace gvqe {

// FP64: four warps where the half allows it, one per FP64 pipe of the SM.  FP32 to 10 qubits: four
// warps too, a chain of 700 instructions per layer and warp otherwise (64 terms, 19 qubits, one
// vector, forward and backward: 47 and 25 us with one warp, 19 and 14 with four).  From 11 qubits 32
// amplitudes a thread save shared-memory rounds (backward, 24 qubits: 37 us, 50 with 16).
template <typename T>
__host__ __device__ constexpr int half_e(int M) {
  return sizeof(T) == 4 ? (M >= 11 ? 5 : M >= 7 ? 3 : 2) : (M >= 12 ? 5 : M == 11 ? 4 : M == 10 ? 3 : 2);
}
template <typename T, int M, int EB = half_e<T>(M)>
struct HalfCfg {
  static constexpr int E = EB;                // register bits
  static constexpr int LT = M - E;            // log2 of the working threads
  static constexpr int G0 = LT < E ? LT : E;  // LOW bits; the other LT - G0 are MID's, at most E at a time
  static constexpr int NT = LT < 5 ? 32 : 1 << LT;
  static_assert(G0 >= 2, "runs of 16 bytes");
};
// threads of a kernel that takes halves of M and of M - 1 qubits
template <typename T, int M>
constexpr int half_nt() {
  return HalfCfg<T, M>::NT > HalfCfg<T, M - 1>::NT ? HalfCfg<T, M>::NT : HalfCfg<T, M - 1>::NT;
}

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

// RY (sg = 1) or its inverse (sg = -1) on register bits 0 .. G-1 of the 2^G values v (CH: bit
// 0 is the re/im channel and has none)
template <int G, bool CH = false, typename T>
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
    if constexpr (!CH) {  // bit 0: within the pairs
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

// acc[k] += sum of G1 phi0 - G0 phi1 over register bit k (CH: not bit 0); phi(i) loads pairs i, i + 1
template <int G, bool CH = false, typename T, typename F>
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
      if constexpr (!CH) {
        acc[0] += v[i + 1] * p[0];
        acc[0] -= v[i] * p[1];
      }
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
template <typename T, int M, int EB = half_e<T>(M)>
struct Half {
  using C = HalfCfg<T, M, EB>;
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
  {
    const double2 c = reinterpret_cast<const double2 *>(J.cs)[(i / M) * n + q0 + i % M];
    sh.cs[i].x = (T)c.x;
    sh.cs[i].y = (T)c.y;
  }
  __syncthreads();
}

}  // namespace gvqe
