// gvqe_cut_half.cu -- the circuits of the two halves (gvqe_cut.cuh), forward and adjoint;
// compiled once per amplitude type (GVQE_INST_T).
#include "gvqe_cut_half.cuh"

namespace gvqe {

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
      phi += 2 * (SZ << l.shift);  // (forward: FP64 only)
      const int bits = l.shift + l.nb;
      nat = phi + (size_t)2 * a * SZ;
      run = nat + SZ;
      keep = GRAD && (a >> bits) == 0;
    } else {
      T *tab = reinterpret_cast<T *>(J.ws + J.lay->tab[h]);
      nat = tab + (size_t)2 * a * SZ;
      run = nat + SZ;
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
    const int ns = J.lay->gs[h];
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
  constexpr int SR = sizeof(T) == 4 ? 3 : 2;  // numbers kept per amplitude
  const T *nat = reinterpret_cast<const T *>(J.ws + J.lay->tab[h]) + (size_t)SR * a * SZ, *run = nat + SZ;
  const T *phi = reinterpret_cast<const T *>(J.ws + J.lay->phi[h]);
  for (int r = 0; r < reps; ++r) phi += SR * (SZ << sh.H.L[r].shift);
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
    phi -= SR * (SZ << l.shift);
    nat = phi + (size_t)SR * (a & ((1 << l.shift) - 1)) * SZ;
    run = nat + SZ;
  }
}

// MODE 0: forward, 1: forward keeping what the backward reads, 2: backward.  One kernel for
// all small sizes (mixed in a batch), and one per size M above, which also
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
constexpr int SMALL_M = HALF_SMALL_M(sizeof(GVQE_INST_T) == 8);
template <typename T, int MODE, int M>
__global__ void __launch_bounds__(half_nt<T, M>()) k_half(const __grid_constant__ CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  __shared__ HalfShared<T> sh;
  const int3 it = cut_half_item(A);
  const CutView J = cut_view(A, it.x);
  T *st = reinterpret_cast<T *>(cut_smem);
  const int m = J.desc->half[it.y].m;
  if constexpr (M > SMALL_M) {
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
  k_half<T, MODE, M><<<blocks, half_nt<T, M>(), sm, s>>>(A);
  return cudaGetLastError();
}

template <typename T, int MODE>
static cudaError_t launch_half_mode(const CutArgs &A, int m, int blocks, cudaStream_t s) {
  switch (m) {
    case SMALL_M: return launch_half_m<T, MODE, SMALL_M>(A, blocks, s);
    case SMALL_M + 1: return launch_half_m<T, MODE, SMALL_M + 1>(A, blocks, s);
    case SMALL_M + 2: return launch_half_m<T, MODE, SMALL_M + 2>(A, blocks, s);
    case SMALL_M + 3: return launch_half_m<T, MODE, SMALL_M + 3>(A, blocks, s);
    case SMALL_M + 4: return launch_half_m<T, MODE, SMALL_M + 4>(A, blocks, s);
    case SMALL_M + 5: return launch_half_m<T, MODE, SMALL_M + 5>(A, blocks, s);
  }
  if constexpr (SMALL_M + 7 == 14) {  // FP64: 14 is the largest half, FP32: 15
    if (m == 13) return launch_half_m<T, MODE, 13>(A, blocks, s);
    if (m == 14) return launch_half_m<T, MODE, 14>(A, blocks, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_half<GVQE_INST_T>(const CutArgs &A, int m, int mode, int blocks, cudaStream_t s) {
  if constexpr (sizeof(GVQE_INST_T) == 8) {
    if (mode == 0) return launch_half_mode<GVQE_INST_T, 0>(A, m, blocks, s);
    if (mode == 1) return launch_half_mode<GVQE_INST_T, 1>(A, m, blocks, s);
  }
  return launch_half_mode<GVQE_INST_T, 2>(A, m, blocks, s);
}

}  // namespace gvqe
