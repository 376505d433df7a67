// gvqe_cut_halfc.cu -- the circuits of the two halves with full EfficientSU2 layers (RY then
// RZ on every qubit; FP32): a half of M qubits is 2^(M+1) floats with the re/im channel as
// index bit 0, run by the register rounds of gvqe_cut_half.cuh.  RY acts on both channels
// alike; a layer's RZ gates are one diagonal phase, applied in a LOW round of their own after
// the state before them has been kept (the adjoint sweep takes the phase off G first, so that
// both vectors sit between RY and RZ: there the RY gradients are the real ones over both
// channels and the RZ gradients sum +-Im(conj(G) phi)).
#include "gvqe_cut_half.cuh"

namespace gvqe {
namespace {

constexpr int MAX_M = 14;  // qubits of a half: 2^15 floats of shared memory

struct SharedC {
  float2 cs[(CUT_MAX_LAYERS + 1) * 2 * MAX_M];  // per layer: RY of the half's qubits, then RZ
  uint32_t col[CUT_MAX_LAYERS][2][MAX_M + 1];   // A^-1 and A over the index bits (channel kept)
  uint32_t off[CUT_MAX_LAYERS][2][4];
  int shift[CUT_MAX_LAYERS], nb[CUT_MAX_LAYERS];
  float red[32 * 32];
};

__device__ __forceinline__ uint32_t up1(uint32_t c) { return ((c & 0x7fffu) << 1) | (c & 0x30000u); }

__device__ __forceinline__ void setup(SharedC &sh, const CutView &J, int h, int M) {
  const CutHalf &H = J.desc->half[h];
  const int n = J.desc->n, reps = J.desc->reps, tid = threadIdx.x, NT = blockDim.x;
  for (int i = tid; i < (reps + 1) * 2 * M; i += NT) {
    const int r = i / (2 * M), z = (i / M) & 1, q = i % M;
    const double2 c = reinterpret_cast<const double2 *>(J.cs)[r * 2 * n + z * n + H.q0 + q];
    sh.cs[i] = make_float2((float)c.x, (float)c.y);
  }
  for (int i = tid; i < reps * 2 * (M + 1); i += NT) {
    const int r = i / (2 * (M + 1)), d = (i / (M + 1)) & 1, q = i % (M + 1);
    sh.col[r][d][q] = q == 0 ? 1u : up1(d ? H.L[r].fc[q - 1] : H.L[r].ic[q - 1]);
  }
  for (int i = tid; i < reps * 8; i += NT) {
    const int r = i >> 3, d = (i >> 2) & 1, b = i & 3;
    sh.off[r][d][b] = up1(d ? H.L[r].fo[b] : H.L[r].io[b]);
  }
  for (int r = tid; r < reps; r += NT) {
    sh.shift[r] = H.L[r].shift;
    sh.nb[r] = H.L[r].nb;
  }
  __syncthreads();
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
// the factor of one qubit: exp(-i t/2) at bit 0, exp(+i t/2) at bit 1 (sg = -1: conjugate)
__device__ __forceinline__ float2 zfac(float2 c, int bit, float sg) { return {c.x, bit ? sg * c.y : -sg * c.y}; }

// u (2^(G0-1) complex values of LOW item it) times the layer's phase; z: its RZ (cos, sin)
template <int M, int G0>
__device__ __forceinline__ void phase(float *u, int it, const float2 *z, float sg) {
  constexpr int QL = G0 - 1, QA = QL / 2, QB = QL - QA;  // low qubits, in two tables
  float2 ph = {1.f, 0.f};
#pragma unroll
  for (int q = QL; q < M; ++q) ph = cmul(ph, zfac(z[q], (it >> (q - QL)) & 1, sg));
  float2 ta[1 << QA], tb[1 << QB];
  ta[0] = {1.f, 0.f};
#pragma unroll
  for (int q = 0; q < QA; ++q)
#pragma unroll
    for (int s = 0; s < (1 << q); ++s) {
      ta[s | (1 << q)] = cmul(ta[s], zfac(z[q], 1, sg));
      ta[s] = cmul(ta[s], zfac(z[q], 0, sg));
    }
  tb[0] = ph;
#pragma unroll
  for (int q = 0; q < QB; ++q)
#pragma unroll
    for (int s = 0; s < (1 << q); ++s) {
      tb[s | (1 << q)] = cmul(tb[s], zfac(z[QA + q], 1, sg));
      tb[s] = cmul(tb[s], zfac(z[QA + q], 0, sg));
    }
#pragma unroll
  for (int b = 0; b < (1 << QB); ++b)
#pragma unroll
    for (int a = 0; a < (1 << QA); ++a) {
      const float2 w = cmul(ta[a], tb[b]);
      float *p = u + 2 * (a | (b << QA));
      const float2 x = cmul({p[0], p[1]}, w);
      p[0] = x.x;
      p[1] = x.y;
    }
}

template <int MB, bool GRAD>
__device__ __forceinline__ void fwd(const CutView &J, int h, int a, float *st, SharedC &sh) {
  using HF = Half<float, MB>;
  using C = typename HF::C;
  constexpr int M = MB - 1;
  constexpr long long SZ = 1LL << MB;
  const HF S{st, (int)threadIdx.x, (int)threadIdx.x < (1 << C::LT)};
  const int reps = J.desc->reps;
  float v[HF::N];
  {  // layer 0: the real product state, in TOP order
    float b = (S.tid & 1) ? 0.f : 1.f;
#pragma unroll
    for (int q = 1; q < C::LT; ++q) b *= ((S.tid >> q) & 1) ? sh.cs[q - 1].y : sh.cs[q - 1].x;
    v[0] = b;
#pragma unroll
    for (int j = 0; j < C::E; ++j)
#pragma unroll
      for (int s = 0; s < (1 << j); ++s) {
        v[s | (1 << j)] = v[s] * sh.cs[C::LT - 1 + j].y;
        v[s] *= sh.cs[C::LT - 1 + j].x;
      }
  }
  S.top_store(v);
  S.sync();
  float *phi = reinterpret_cast<float *>(J.ws + J.lay->phi[h]);
  float *tab = reinterpret_cast<float *>(J.ws + J.lay->tab[h]) + (size_t)a * SZ;
  for (int r = 0;; ++r) {
    const float2 *cs = sh.cs + r * 2 * M - 1;  // RY of index bit b at cs[b]
    // the state before this layer's RZ, once per value of the path bits so far
    const int bits = r < reps ? sh.shift[r] : J.desc->kappa;
    float *nat = phi + (size_t)2 * a * SZ, *run = nat + SZ;
    const bool keep = GRAD && (a >> bits) == 0;
    S.low_round([&](int it, float *u) {
      if (r > 0) rotate<C::G0, true>(u, cs, 1.f);
      if (keep) S.keep_run(run, it, u);
      return r > 0;
    });
    S.sync();
    if (keep) S.keep_natural(nat);
    S.sync();
    S.low_round([&](int it, float *u) {
      phase<M, C::G0>(u, it, sh.cs + r * 2 * M + M, 1.f);
      return true;
    });
    S.sync();
    if (r == reps) break;
    phi += 2 * (SZ << bits);
    cs = sh.cs + (r + 1) * 2 * M - 1;
    S.gather(v, sh.col[r][0], sh.off[r][0][(a >> sh.shift[r]) & ((1 << sh.nb[r]) - 1)]);
    rotate<C::E>(v, cs + C::LT, 1.f);
    S.sync();
    S.top_store(v);
    S.sync();
    S.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      S.template mid_round<LO, G>([&](int, float *u) {
        rotate<G>(u, cs + LO, 1.f);
        return true;
      });
      S.sync();
    });
  }
  S.keep_natural(tab);
}

template <int MB>
__device__ __forceinline__ void bwd(const CutView &J, int h, int a, float *st, SharedC &sh) {
  using HF = Half<float, MB>;
  using C = typename HF::C;
  constexpr int M = MB - 1, QL = C::G0 - 1;
  constexpr long long SZ = 1LL << MB;
  const HF S{st, (int)threadIdx.x, (int)threadIdx.x < (1 << C::LT)};
  const int reps = J.desc->reps, D = J.desc->D, lane = S.tid & 31, w = S.tid >> 5;
  float v[HF::N];
  {  // G of term a: row (x, channel) of the real contraction's terms 2a and 2a + 1
    const float *g = reinterpret_cast<const float *>(J.ws + J.lay->g[h]) + (size_t)2 * a * SZ;
    const float sg = (S.tid & 1) ? -1.f : 1.f;
#pragma unroll
    for (int s = 0; s < HF::N; ++s) v[s] = 0.f;
    for (int k = 0; k < J.lay->gs[h]; ++k, g += (size_t)2 * D * SZ)
#pragma unroll
      for (int s = 0; s < HF::N; ++s)
        if (S.on) {
          const int y = S.tid + (s << C::LT);
          v[s] += g[y] + sg * g[SZ + (y ^ 1)];
        }
  }
  S.top_store(v);
  S.sync();
  double *gp = reinterpret_cast<double *>(J.ws + J.lay->gp) + ((size_t)h * D + a) * (reps + 1) * 32;
  const float *phi = reinterpret_cast<const float *>(J.ws + J.lay->phi[h]);
  for (int r = 0; r < reps; ++r) phi += 2 * (SZ << sh.shift[r]);
  for (int r = reps;; --r) {
    const int bits = r < reps ? sh.shift[r] : J.desc->kappa;
    const float *nat = phi + (size_t)2 * (a & ((1 << bits) - 1)) * SZ, *run = nat + SZ;
    const float2 *cs = sh.cs + r * 2 * M - 1;
    float acc[MB], az[M];
#pragma unroll
    for (int q = 0; q < MB; ++q) acc[q] = 0.f;
#pragma unroll
    for (int q = 0; q < M; ++q) az[q] = 0.f;
    // take the layer's phase off G; RZ gradients of every qubit, RY gradients of the low ones
    S.low_round([&](int it, float *u) {
      phase<M, C::G0>(u, it, sh.cs + r * 2 * M + M, -1.f);
      float4 x;
      float tot = 0.f;
      grads<C::G0, true>(u, [&](int i, float *p) {
        if (i % 4 == 0) x = reinterpret_cast<const float4 *>(run)[(i / 4) * HF::ITEMS + it];
        p[0] = (i & 2) ? x.z : x.x;
        p[1] = (i & 2) ? x.w : x.y;
        const float im = u[i] * p[1] - u[i + 1] * p[0];
        tot += im;
#pragma unroll
        for (int q = 0; q < QL; ++q) az[q] += ((i >> (q + 1)) & 1) ? -im : im;
      }, acc);
#pragma unroll
      for (int q = QL; q < M; ++q) az[q] += ((it >> (q - QL)) & 1) ? -tot : tot;
      return true;
    });
    S.sync();
    S.top_load(v);
    if (S.on)
      grads<C::E>(v, [&](int i, float *p) {
        p[0] = nat[S.tid + (i << C::LT)];
        p[1] = nat[S.tid + ((i + 1) << C::LT)];
      }, acc + C::LT);
    S.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      S.template mid_round<LO, G>([&](int base, float *u) {
        grads<G>(u, [&](int i, float *p) {
          p[0] = nat[base + (i << LO)];
          p[1] = nat[base + ((i + 1) << LO)];
        }, acc + LO);
        return false;
      });
    });
    // this layer's gradients: lanes, then warps in FP64
#pragma unroll
    for (int q = 0; q < M; ++q)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        acc[q + 1] += __shfl_xor_sync(0xffffffffu, acc[q + 1], o);
        az[q] += __shfl_xor_sync(0xffffffffu, az[q], o);
      }
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < M; ++q) {
        sh.red[w * 32 + q] = acc[q + 1];
        sh.red[w * 32 + 16 + q] = az[q];
      }
    S.sync();
    if (S.tid < 32 && (S.tid & 15) < M) {
      double s = 0.0;
      for (int k = 0; k < C::NT / 32; ++k) s += (double)sh.red[k * 32 + S.tid];
      gp[r * 32 + S.tid] = s;
    }
    if (r == 0) break;
    S.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      S.template mid_round<LO, G>([&](int, float *u) {
        rotate<G>(u, cs + LO, -1.f);
        return true;
      });
      S.sync();
    });
    S.low_round([&](int, float *u) {
      rotate<C::G0, true>(u, cs, -1.f);
      return true;
    });
    S.sync();
    S.top_load(v);
    rotate<C::E>(v, cs + C::LT, -1.f);
    S.top_store(v);
    S.sync();
    S.gather(v, sh.col[r - 1][1], sh.off[r - 1][1][(a >> sh.shift[r - 1]) & ((1 << sh.nb[r - 1]) - 1)]);
    S.sync();
    S.top_store(v);
    S.sync();
    phi -= 2 * (SZ << sh.shift[r - 1]);
  }
}

template <int MODE, int MB>
__device__ __forceinline__ void run_c(const CutView &J, int h, int a, float *st, SharedC &sh) {
  setup(sh, J, h, MB - 1);
  if (HalfCfg<float, MB>::NT == 32 && threadIdx.x >= 32) return;
  if constexpr (MODE == 2)
    bwd<MB>(J, h, a, st, sh);
  else
    fwd<MB, MODE == 1>(J, h, a, st, sh);
}

// MB: index bits of the larger half; the other may have one less
template <int MODE, int MB>
__global__ void __launch_bounds__(half_nt<float, MB>()) k_halfc(const __grid_constant__ CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  __shared__ SharedC sh;
  const int3 it = cut_half_item(A);
  const CutView J = cut_view(A, it.x);
  float *st = reinterpret_cast<float *>(cut_smem);
  if (J.desc->half[it.y].m + 1 == MB)
    run_c<MODE, MB>(J, it.y, it.z, st, sh);
  else
    run_c<MODE, MB - 1>(J, it.y, it.z, st, sh);
}

template <int MODE, int MB>
cudaError_t launch_mb(const CutArgs &A, int blocks, cudaStream_t s) {
  constexpr size_t sm = (size_t)pad<float>(1 << MB) * sizeof(float);
  static SmemLimit limit;
  if (const cudaError_t e = limit.set(k_halfc<MODE, MB>, sm)) return e;
  k_halfc<MODE, MB><<<blocks, half_nt<float, MB>(), sm, s>>>(A);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_mode(const CutArgs &A, int m, int blocks, cudaStream_t s) {
  switch (m) {
    case 7: return launch_mb<MODE, 8>(A, blocks, s);
    case 8: return launch_mb<MODE, 9>(A, blocks, s);
    case 9: return launch_mb<MODE, 10>(A, blocks, s);
    case 10: return launch_mb<MODE, 11>(A, blocks, s);
    case 11: return launch_mb<MODE, 12>(A, blocks, s);
    case 12: return launch_mb<MODE, 13>(A, blocks, s);
    case 13: return launch_mb<MODE, 14>(A, blocks, s);
    case 14: return launch_mb<MODE, 15>(A, blocks, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_halfc(const CutArgs &A, int m, int mode, int blocks, cudaStream_t s) {
  if (mode == 0) return launch_mode<0>(A, m, blocks, s);
  if (mode == 1) return launch_mode<1>(A, m, blocks, s);
  return launch_mode<2>(A, m, blocks, s);
}

}  // namespace gvqe
