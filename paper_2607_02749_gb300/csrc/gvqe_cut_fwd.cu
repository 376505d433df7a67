// gvqe_cut_fwd.cu -- the forward half circuits in FP32 (RY layers) with about 45 bits.
//
// Every error of a half's table meets all 2^(n/2) columns of the other half, so the energy
// does not average it away as it does the rounding of a 2^n state.  In plain FP32 the tables still leave
// no more than a stored state does (RMS error of E per sum |c|, RY+RZ layers, whose halves are plain FP32, 20 to
// 25 qubits: 2.7e-10 to 5.7e-10; stored states 6.6e-10 to 1.0e-9); rounded once, a small part of it (RY
// layers, 14 to 26 qubits: 0.5e-10 to 7e-10; stored states 0.8e-9 to 2.9e-9).  So amplitudes are carried as
// unevaluated sums hi + lo of two floats, cos and sin too, and the tables are rounded once, into
// the tensor cores' hi and lo parts.  13 FP32 operations per rotated amplitude, a tenth of
// the FP64 pipe's time.
//
// From 11 qubits a half runs layer by layer, one launch each: a state after layer r depends on
// the path bits so far only, so the layers together do 2 D states instead of (reps + 1) D.
// A CTA computes one state or, at 15 qubits, half of one (2^14 amplitudes; the top qubit's
// rotation is taken while gathering): two parts of 2^14 run 30 qubits' tables, 6 layers, in 200 us,
// four of 2^13 in 247.  Gather from the previous layer's state in L2, TOP, MID and LOW register
// rounds (gvqe_cut_half.cuh).  Up to 10 qubits one CTA of four warps runs the whole
// circuit of one path value.  Bound by the chain of layers (one vector) and by issue: 26 FP32
// operations per pair and rotation.
#include "gvqe_cut_half.cuh"

namespace gvqe {
namespace {

__device__ __forceinline__ float mulv(float a, float b) { return a * b; }
__device__ __forceinline__ float fmav(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float addv(float a, float b) { return a + b; }
__device__ __forceinline__ float subv(float a, float b) { return a - b; }
__device__ __forceinline__ float negv(float a) { return -a; }
__device__ __forceinline__ f2 mulv(f2 a, f2 b) { return mul2(a, b); }
__device__ __forceinline__ f2 fmav(f2 a, f2 b, f2 c) { return fma2(a, b, c); }
__device__ __forceinline__ f2 addv(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 negv(f2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2 subv(f2 a, f2 b) { return fma2(b, pk2(-1.f, -1.f), a); }

template <typename V>
struct Df {  // hi + lo
  V h, l;
};
// c a + s b, c and s with their own low parts: r = c a + s b rounded, its exact error e1 + e2 +
// (p2 - (r - d)), and the low parts' products; lo is not folded into hi (norm).  13 operations.
template <typename V>
__device__ __forceinline__ Df<V> combine(V ch, V cl, V sh, V sl, Df<V> a, Df<V> b) {
  const V p2 = mulv(sh, b.h), r = fmav(ch, a.h, p2);
  const V e2 = fmav(sh, b.h, negv(p2)), d = subv(r, p2);
  V lo = fmav(ch, a.h, negv(d));
  lo = fmav(ch, a.l, lo);
  lo = fmav(cl, a.h, lo);
  lo = fmav(sh, b.l, lo);
  lo = fmav(sl, b.h, lo);
  return {r, addv(addv(lo, e2), subv(p2, subv(r, d)))};
}
__device__ __forceinline__ void norm(float &h, float &l) {
  const float s = h + l;
  l = l - (s - h);
  h = s;
}
__device__ __forceinline__ Df<float> mul_df(Df<float> a, Df<float> b) {
  float p = a.h * b.h, e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  norm(p, e);
  return {p, e};
}

// RY on register bits 0 .. G-1 of the 2^G values h + l; cs: (cos hi, cos lo, sin hi, sin lo)
template <int G>
__device__ __forceinline__ void rotate_df(float *h, float *l, const float4 *cs) {
  {
    const float4 w = cs[0];
#pragma unroll
    for (int i = 0; i < (1 << G); i += 2) {
      const Df<float> a{h[i], l[i]}, b{h[i + 1], l[i + 1]};
      const Df<float> x = combine(w.x, w.y, -w.z, -w.w, a, b), y = combine(w.z, w.w, w.x, w.y, a, b);
      h[i] = x.h;
      l[i] = x.l;
      h[i + 1] = y.h;
      l[i + 1] = y.l;
    }
  }
  if constexpr (G > 1) {
    constexpr int H = 1 << (G - 1);
    Df<f2> p[H];
#pragma unroll
    for (int i = 0; i < H; ++i) p[i] = {pk2(h[2 * i], h[2 * i + 1]), pk2(l[2 * i], l[2 * i + 1])};
#pragma unroll
    for (int k = 1; k < G; ++k) {
      const float4 w = cs[k];
      const f2 ch = pk2(w.x, w.x), cl = pk2(w.y, w.y), sh = pk2(w.z, w.z), sl = pk2(w.w, w.w);
#pragma unroll
      for (int i = 0; i < H; ++i)
        if (!((i >> (k - 1)) & 1)) {
          const int o = i | (1 << (k - 1));
          const Df<f2> a = p[i], b = p[o];
          p[i] = combine(ch, cl, negv(sh), negv(sl), a, b);
          p[o] = combine(sh, sl, ch, cl, a, b);
        }
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
      unpk2(p[i].h, h[2 * i], h[2 * i + 1]);
      unpk2(p[i].l, l[2 * i], l[2 * i + 1]);
    }
  }
#pragma unroll
  for (int i = 0; i < (1 << G); ++i) norm(h[i], l[i]);
}

__device__ __forceinline__ float4 split_cs(double2 c) {
  const float ch = (float)c.x, sh = (float)c.y;
  return make_float4(ch, (float)(c.x - ch), sh, (float)(c.y - sh));
}

// Register bits of the rounds here, twice the registers of the plain FP32 ones: 11 to 13 qubits take
// 16 amplitudes a thread (24 qubits, 16 terms, 4 layers: 53 us, 65 with 32, 57 with 8).
__host__ __device__ constexpr int fwd_e(int M) { return M >= 14 ? 5 : M >= 11 ? 4 : half_e<float>(M); }

// A state in shared memory (hi and lo parts) and its register rounds.
template <int M>
struct State {
  using HF = Half<float, M, fwd_e(M)>;
  using C = typename HF::C;
  static constexpr int N = HF::N;
  HF H, L;
  __device__ __forceinline__ State(float *st, int tid)
      : H{st, tid, tid < (1 << C::LT)}, L{st + pad<float>(1 << M), tid, tid < (1 << C::LT)} {}
  __device__ __forceinline__ void sync() const { H.sync(); }
  __device__ __forceinline__ void top_store(const float *h, const float *l) const {
    H.top_store(h);
    L.top_store(l);
  }
  // RY on the MID bits, then on the LOW bits; keep(it, u): the LOW items' hi parts as they are stored
  template <typename F>
  __device__ __forceinline__ void rest(const float4 *cs, F keep) const {
    H.template mid_groups<C::G0>([&](auto lo, auto g) {
      constexpr int LO = decltype(lo)::value, G = decltype(g)::value;
      if (H.on)
#pragma unroll
        for (int q = 0; q < (1 << (C::E - G)); ++q) {
          const int it = H.tid + (q << C::LT);
          const int base = pad<float>((it & ((1 << LO) - 1)) | ((it >> LO) << (LO + G)));
          float u[1 << G], v[1 << G];
#pragma unroll
          for (int s = 0; s < (1 << G); ++s) {
            u[s] = H.st[base + pad<float>(s << LO)];
            v[s] = L.st[base + pad<float>(s << LO)];
          }
          rotate_df<G>(u, v, cs + LO);
#pragma unroll
          for (int s = 0; s < (1 << G); ++s) {
            H.st[base + pad<float>(s << LO)] = u[s];
            L.st[base + pad<float>(s << LO)] = v[s];
          }
        }
      sync();
    });
    if (H.on)
#pragma unroll
      for (int q = 0; q < (1 << (C::E - C::G0)); ++q) {
        const int it = H.tid + (q << C::LT);
        float4 *p = reinterpret_cast<float4 *>(H.st + pad<float>(it << C::G0));
        float4 *r = reinterpret_cast<float4 *>(L.st + pad<float>(it << C::G0));
        alignas(16) float u[1 << C::G0], v[1 << C::G0];
#pragma unroll
        for (int j = 0; j < (1 << C::G0) / 4; ++j) {
          reinterpret_cast<float4 *>(u)[j] = p[j];
          reinterpret_cast<float4 *>(v)[j] = r[j];
        }
        rotate_df<C::G0>(u, v, cs);
        keep(it, u);
#pragma unroll
        for (int j = 0; j < (1 << C::G0) / 4; ++j) {
          p[j] = reinterpret_cast<float4 *>(u)[j];
          r[j] = reinterpret_cast<float4 *>(v)[j];
        }
      }
    sync();
  }
};

// layer 0, the product state, of amplitude i's low LT bits and, by slot, its E bits above
template <int E, int LT>
__device__ __forceinline__ void product(float *h, float *l, int low, const float4 *cs) {
  Df<float> b{1.f, 0.f};
#pragma unroll
  for (int q = 0; q < LT; ++q) {
    const float4 w = cs[q];
    b = mul_df(b, ((low >> q) & 1) ? Df<float>{w.z, w.w} : Df<float>{w.x, w.y});
  }
  h[0] = b.h;
  l[0] = b.l;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const float4 w = cs[LT + j];
#pragma unroll
    for (int s = 0; s < (1 << j); ++s) {
      const Df<float> x = mul_df({h[s], l[s]}, {w.z, w.w}), y = mul_df({h[s], l[s]}, {w.x, w.y});
      h[s | (1 << j)] = x.h;
      l[s | (1 << j)] = x.l;
      h[s] = y.h;
      l[s] = y.l;
    }
  }
}

// ------------------------------------------------- up to 10 qubits: one launch --
struct SmallShared {
  float4 cs[(CUT_MAX_LAYERS + 1) * 10];
  CutHalf H;
};

template <int M, bool GRAD>
__device__ __forceinline__ void small_fwd(const CutView &J, int h, int a, float *st, SmallShared &sh) {
  using S_ = State<M>;
  using C = typename S_::C;
  const S_ S(st, threadIdx.x);
  if (C::NT == 32 && threadIdx.x >= 32) return;
  const int nt = C::NT == 32 ? 32 : blockDim.x;
  constexpr long long SZ = 1LL << M;
  const int reps = J.desc->reps, n = J.desc->n;
  for (int i = threadIdx.x; i < (int)(sizeof(CutHalf) / 4); i += nt)
    reinterpret_cast<int *>(&sh.H)[i] = reinterpret_cast<const int *>(&J.desc->half[h])[i];
  S.sync();
  for (int i = threadIdx.x; i < (reps + 1) * M; i += nt)
    sh.cs[i] = split_cs(reinterpret_cast<const double2 *>(J.cs)[(i / M) * n + sh.H.q0 + i % M]);
  S.sync();
  float u[S_::N], v[S_::N];
  product<C::E, C::LT>(u, v, S.H.tid & ((1 << C::LT) - 1), sh.cs);
  S.top_store(u, v);
  S.sync();
  float *phi = reinterpret_cast<float *>(J.ws + J.lay->phi[h]);
  if (GRAD && a == 0) {
    S.H.keep_natural(phi);
    S.H.low_round([&](int it, float *x) {
      S.H.keep_run(phi + SZ, it, x);
      return false;
    });
  }
  for (int r = 1; r <= reps; ++r) {
    const CutLayer &l = sh.H.L[r - 1];
    const uint32_t off = l.io[(a >> l.shift) & ((1 << l.nb) - 1)];
    S.H.gather(u, l.ic, off);
    S.L.gather(v, l.ic, off);
    rotate_df<C::E>(u, v, sh.cs + r * M + C::LT);
    S.sync();
    S.top_store(u, v);
    S.sync();
    phi += 3 * (SZ << l.shift);
    float *nat = r < reps ? phi + (size_t)3 * a * SZ : reinterpret_cast<float *>(J.ws + J.lay->tab[h]) + (size_t)3 * a * SZ;
    const bool keep = r == reps || (GRAD && (a >> (l.shift + l.nb)) == 0);
    S.rest(sh.cs + r * M, [&](int it, const float *x) {
      if (GRAD && keep) S.H.keep_run(nat + SZ, it, x);
    });
    if (keep) S.H.keep_natural(nat);
    if (r == reps) S.L.keep_natural(nat + 2 * SZ);
  }
}

template <bool GRAD>
__global__ void __launch_bounds__(HalfCfg<float, 10>::NT) k_fwd_small(const __grid_constant__ CutArgs A) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  __shared__ SmallShared sh;
  const int3 it = cut_half_item(A);
  const CutView J = cut_view(A, it.x);
  float *st = reinterpret_cast<float *>(cut_smem);
  switch (J.desc->half[it.y].m) {
    case 7: small_fwd<7, GRAD>(J, it.y, it.z, st, sh); break;
    case 8: small_fwd<8, GRAD>(J, it.y, it.z, st, sh); break;
    case 9: small_fwd<9, GRAD>(J, it.y, it.z, st, sh); break;
    case 10: small_fwd<10, GRAD>(J, it.y, it.z, st, sh); break;
  }
}

// ------------------------------------- from 11 qubits: one launch per layer --
struct LayerShared {
  float4 cs[CUT_MAX_M];
  uint32_t col[CUT_MAX_M];
};

// the state after layer r for the path bits a so far: chunk b of 2^SB, CH bits each
template <int CH, int SB, bool GRAD>
__device__ __forceinline__ void layer(const CutView &J, int h, int r, int a, int b, float *st, LayerShared &sh) {
  using S_ = State<CH>;
  using C = typename S_::C;
  constexpr int M = CH + SB;
  constexpr long long SZ = 1LL << M;
  const S_ S(st, threadIdx.x);
  const int tid = threadIdx.x, reps = J.desc->reps, n = J.desc->n;
  const CutHalf &H = J.desc->half[h];
  if (tid < M) {
    sh.cs[tid] = split_cs(reinterpret_cast<const double2 *>(J.cs)[r * n + H.q0 + tid]);
    sh.col[tid] = r > 0 ? H.L[r - 1].ic[tid] : 0;
  }
  // where this layer's states are, and the previous one's
  float *base = reinterpret_cast<float *>(J.ws + J.lay->phi[h]);
  const float *prev = base;
  for (int k = 0; k < r; ++k) {
    prev = base;
    base += 3 * (SZ << H.L[k].shift);
  }
  if (r == reps) base = reinterpret_cast<float *>(J.ws + J.lay->tab[h]);
  float *nat = base + (size_t)3 * a * SZ;
  __syncthreads();
  float u[S_::N], v[S_::N];
  if (r == 0) {
    product<C::E, C::LT>(u, v, tid & ((1 << C::LT) - 1), sh.cs);
#pragma unroll
    for (int k = 0; k < SB; ++k) {
      const float4 w = sh.cs[CH + k];
      const Df<float> f = ((b >> k) & 1) ? Df<float>{w.z, w.w} : Df<float>{w.x, w.y};
#pragma unroll
      for (int s = 0; s < S_::N; ++s) {
        const Df<float> x = mul_df({u[s], v[s]}, f);
        u[s] = x.h;
        v[s] = x.l;
      }
    }
  } else {
    const int shift = H.L[r - 1].shift;
    const float *ph = prev + (size_t)3 * (a & ((1 << shift) - 1)) * SZ, *pl = ph + 2 * SZ;
    uint32_t x = H.L[r - 1].io[a >> shift];
#pragma unroll
    for (int q = 0; q < C::LT; ++q)
      if ((tid >> q) & 1) x ^= sh.col[q];
#pragma unroll
    for (int e = 0; e < S_::N; ++e) {  // places in Gray order: one column per step
      if (e > 0) x ^= sh.col[C::LT + (e & 1 ? 0 : e & 2 ? 1 : e & 4 ? 2 : e & 8 ? 3 : 4)];
      const int s = e ^ (e >> 1);
      Df<float> t[1 << SB];
#pragma unroll
      for (int k = 0; k < (1 << SB); ++k) {  // the amplitudes of every chunk at this place
        uint32_t y = x;
#pragma unroll
        for (int j = 0; j < SB; ++j)
          if ((k >> j) & 1) y ^= sh.col[CH + j];
        t[k] = {0.f, 0.f};
        if (S.H.on && (y >> 16) == 0) t[k] = {__ldcg(ph + y), __ldcg(pl + y)};
      }
#pragma unroll
      for (int j = SB - 1; j >= 0; --j) {  // the top qubits' rotations, this chunk's side of each pair
        const float4 w = sh.cs[CH + j];
        const bool one = (b >> j) & 1;
        const float ch = one ? w.z : w.x, cl = one ? w.w : w.y, zh = one ? w.x : -w.z, zl = one ? w.y : -w.w;
#pragma unroll
        for (int k = 0; k < (1 << j); ++k) {
          t[k] = combine(ch, cl, zh, zl, t[k], t[k | (1 << j)]);
          norm(t[k].h, t[k].l);
        }
      }
      u[s] = t[0].h;
      v[s] = t[0].l;
    }
    rotate_df<C::E>(u, v, sh.cs + C::LT);
  }
  S.top_store(u, v);
  S.sync();
  float *run = nat + SZ;
  const long long c0 = (long long)b << CH;
  auto keep = [&](int it, const float *x) {  // in the backward sweep's runs
    if constexpr (GRAD) {
      constexpr int GB = HalfCfg<float, M>::G0 - 2;
      const int g = (it + (b << (CH - C::G0))) << (C::G0 - 2);
#pragma unroll
      for (int j = 0; j < (1 << C::G0) / 4; ++j)
        reinterpret_cast<float4 *>(run)[(((g + j) & ((1 << GB) - 1)) << (M - 2 - GB)) + ((g + j) >> GB)] =
            reinterpret_cast<const float4 *>(x)[j];
    }
  };
  if (r > 0)
    S.rest(sh.cs, keep);
  else if (GRAD)
    S.H.low_round([&](int it, float *x) {
      keep(it, x);
      return false;
    });
  S.H.keep_natural(nat + c0);
  S.L.keep_natural(nat + 2 * SZ + c0);
}

// halves of M and M - 1 qubits
template <int M, int CH, bool GRAD>
__global__ void __launch_bounds__(HalfCfg<float, CH, fwd_e(CH)>::NT) k_fwd_layer(const __grid_constant__ CutArgs A, int r) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  __shared__ LayerShared sh;
  constexpr int SB = M - CH;
  // block -> (job, half, path bits so far, chunk); with items (job, half, path value), those of all layers
  int job, h, a, idx = blockIdx.x >> SB;
  const int b = blockIdx.x & ((1 << SB) - 1);
  if (A.items) {
    const int4 it = A.items[idx];
    job = it.x;
    h = it.y;
    a = it.z;
  } else {
    const int per = A.blk0;  // states of a half after this layer
    a = idx % per;
    h = (idx / per) & 1;
    job = idx / (2 * per);
  }
  const CutView J = cut_view(A, job);
  if (r > J.desc->reps) return;
  const int bits = r == 0 ? 0 : J.desc->half[h].L[r - 1].shift + J.desc->half[h].L[r - 1].nb;
  if (a >> bits) return;
  float *st = reinterpret_cast<float *>(cut_smem);
  if (J.desc->half[h].m == M)
    layer<CH, SB, GRAD>(J, h, r, a, b, st, sh);
  else if constexpr (SB == 0)
    layer<CH - 1, 0, GRAD>(J, h, r, a, 0, st, sh);
  else if (b < (1 << (SB - 1)))
    layer<CH, SB - 1, GRAD>(J, h, r, a, b, st, sh);
}

template <int M, int CH, bool GRAD>
cudaError_t launch_layers(const CutArgs &A0, const CutGrid &g, cudaStream_t s, int *launches) {
  constexpr size_t sm = (size_t)2 * pad<float>(1 << CH) * sizeof(float);
  static_assert(HalfCfg<float, CH, fwd_e(CH)>::NT >= HalfCfg<float, CH - 1, fwd_e(CH - 1)>::NT, "threads for both halves");
  static SmemLimit limit;
  if (const cudaError_t e = limit.set(k_fwd_layer<M, CH, GRAD>, sm)) return e;
  CutArgs A = A0;
  for (int r = 0; r <= g.reps; ++r) {
    A.blk0 = 1 << g.bits[r];
    const int states = A.items ? g.half_blocks : A.njobs * 2 * A.blk0;
    k_fwd_layer<M, CH, GRAD><<<states << (M - CH), HalfCfg<float, CH, fwd_e(CH)>::NT, sm, s>>>(A, r);
    *launches += 1;
  }
  return cudaGetLastError();
}

template <bool GRAD>
cudaError_t launch_fwd_g(const CutArgs &A, const CutGrid &g, cudaStream_t s, int *launches) {
  switch (g.m0) {
    case 11: return launch_layers<11, 11, GRAD>(A, g, s, launches);
    case 12: return launch_layers<12, 12, GRAD>(A, g, s, launches);
    case 13: return launch_layers<13, 13, GRAD>(A, g, s, launches);
    case 14: return launch_layers<14, 14, GRAD>(A, g, s, launches);
    case 15: return launch_layers<15, 14, GRAD>(A, g, s, launches);
  }
  const int blocks = A.items ? g.half_blocks : A.njobs * 2 * g.D;
  constexpr size_t sm = (size_t)2 * pad<float>(1 << 10) * sizeof(float);
  k_fwd_small<GRAD><<<blocks, HalfCfg<float, 10>::NT, sm, s>>>(A);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cut_fwd32(const CutArgs &A, const CutGrid &g, bool grad, cudaStream_t s, int *launches) {
  return grad ? launch_fwd_g<true>(A, g, s, launches) : launch_fwd_g<false>(A, g, s, launches);
}

}  // namespace gvqe
