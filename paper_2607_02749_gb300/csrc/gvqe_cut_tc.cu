// gvqe_cut_tc.cu -- the FP32 contraction of the two half tables on the tensor cores.
//
// An item is 128 rows of one half (i) against a run of the other half's columns (j), in
// tiles of 64 columns.  Per tile, with K terms (16, 32 or 64):
//   S(i, j) = sum_a A(i, a) B(j, a)            128 x K by K x 64
//   lambda = E(i, j) S                         on the FP32 pipe, S read from tensor memory
//   G(i, a) += sum_j lambda(i, j) B(j, a)      128 x 64 by 64 x K
// as tcgen05.mma kind::tf32 with FP32 accumulators.  Every operand is split into two
// TF32 parts (x_hi and x_lo = x - x_hi exactly, its last bits cut by the tensor core:
// about 2^-22 of x), and each product is x_lo y_hi + x_hi y_lo + x_hi y_hi, the small parts
// first so that they meet a small accumulator.  S takes two accumulators, the second half of
// the full-size steps in one of its own: they round toward zero at every step, and what that
// does to E shows where E is near zero.  The tables' x_hi is rounded to nearest, so
// that x_lo has no sign of its own and the dropped x_lo y_lo averages out; lambda's x_hi is
// cut (one instruction).  For the same reason G is taken out after every tile (8 full-size
// steps) and summed on the FP32 pipe.
// What rounding toward zero takes away has a known mean, since it depends on the last bit's size
// alone: TRUNC of the partial sum per step, k / N of the whole at step k of N; and of lambda the
// bits below its 22, on average 0.875 units of its last one.  The sums are scaled back by it once, at
// their end.  Without that every gradient came out short: by 2.0e-7 (20 qubits, 32 terms) to 4.0e-7
// (25 qubits, 2 terms) of itself, as much as its other errors; with it 0 to 1.8e-7.  (Rounding lambda's x_hi to nearest
// instead takes its 7.5e-8 away too, for 1 to 3% of the time.)
//
// Both A operands (the rows, and lambda) sit in tensor memory: lambda never touches shared
// memory, its parts overwrite the two of S in place, and the MMAs read only B from shared
// memory (64 bytes per clock of its 128).  B comes in ready-made operand images
// (k_cut_pack) by bulk copies, E in tile order (k_tile_table).  Warps 0-3 and 4-7 take
// alternate tiles, a row per thread; warps 8 and 11 copy, 9 and 10 issue the MMAs.
// E is loaded straight into registers two tiles ahead (16 coalesced 16-byte loads a thread; warps
// 8-11 hand their registers over) up to 32 terms, and copied into shared memory at 64 terms,
// where the sums of G take the registers: one vector of 30 qubits, 64 terms, 2.20 ms with loads and
// 2.03 ms with copies; 24 qubits, 16 terms, 0.303 and 0.369 ms (each tile then waits
// for a second barrier).
// Nothing is full (24 qubits, 16 vectors: L2 30%, tensor pipe 29%, issue 37%): the chain of a tile,
// S's MMAs, two waits, lambda, G's MMAs, over 2 or 3 buffers of S.  A third group of row warps does not
// help (312 us for 296), nor does a tile shared by both groups (399 us: twice the waits).
#include "gvqe_cut.cuh"

namespace gvqe {
namespace {

constexpr int NT = 384;
constexpr int COLS = 64;

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// K-major operand in shared memory, no swizzle: core matrices of 8 rows x 16 bytes, 128
// bytes apart along K, sbo bytes apart along the rows.  The descriptor's low word is the
// address and the K step, the high word the row step and the version.
__device__ __forceinline__ uint32_t op_lo(uint32_t addr) { return (addr >> 4) | ((128u >> 4) << 16); }
__host__ __device__ constexpr uint32_t op_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }
// FP32 accumulator, TF32 operands, K-major, M = 128
__host__ __device__ constexpr uint32_t idesc(int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}
template <uint32_t HI, uint32_t ID, bool ACC>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t blo) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 b;\n mov.b64 b, {%2, %3};\n setp.ne.b32 p, %5, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], b, %4, p;\n}\n" ::"r"(d),
      "r"(a), "r"(blo), "n"(HI), "n"(ID), "n"(ACC ? 1 : 0)
      : "memory");
}
// one product over N8 steps of 8 along K
template <uint32_t HI, uint32_t ID, bool FIRST, int N8>
__device__ __forceinline__ void mmas(uint32_t d, uint32_t a, uint32_t blo) {
  mma<HI, ID, !FIRST>(d, a, blo);
#pragma unroll
  for (int k = 1; k < N8; ++k) mma<HI, ID, true>(d, a + 8 * k, blo + 16 * k);
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void ld16(uint32_t ta, float *v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(ta)
      : "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void st16(uint32_t ta, const float *v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          ta),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}
__device__ __forceinline__ void st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// A wait that gives up: after its limit, or once another wait of this CTA has given up
// (every MMA and copy completes, so neither is expected).
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, volatile int *bad) {
  uint32_t done = 0;
  for (int it = 0; it < (1 << 16) && !done; ++it) {  // (each sleeps up to 20 us in hardware: about a second)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, 20000;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (!done && *bad) return false;
  }
  if (!done) *bad = 1;
  return done != 0;
}

// The same for a whole warp, all of it leaving together.  (All lanes ask: one lane asking and a
// shuffle of its answer took longer; 24 qubits, 16 vectors 321 us so, 296 with all.)
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int *bad) {
  for (int it = 0; it < (1 << 16); ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, 20000;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (__all_sync(0xffffffffu, done)) return true;
    if (__any_sync(0xffffffffu, *bad)) return false;
  }
  *bad = 1;
  return false;
}

__device__ __forceinline__ void two_sum(float &hi, float &lo, float x) {
  const float s = hi + x, b = s - hi;
  lo += (hi - (s - b)) + (x - b);
  hi = s;
}

struct Yes {
  static constexpr bool value = true;
};
struct No {
  static constexpr bool value = false;
};

using f2 = unsigned long long;  // two packed floats
__device__ __forceinline__ f2 pk2(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpk2(f2 v, float &x, float &y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
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
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

constexpr double TRUNC = 0.36 / (1 << 23);  // mean loss of a sum cut to 24 bits: half of its last bit, 0.72 x 2^-23
constexpr double LOST_LAMBDA = 0.875 * 0.72 / (1 << 23);
// k / N summed over the steps k = 1 .. N
constexpr double steps(int n) { return 0.5 * (n + 1); }

template <int K>
struct Cfg {
  static constexpr int BUFS = K <= 16 ? 3 : 2;   // S / lambda buffers
  static constexpr int GBUFS = K <= 32 ? 4 : 2;  // G buffers: two per warp group where they fit
  // stages of the copies: the row-form and column-form halves of B (freed by S and by G), and E
  static constexpr int RS = K <= 32 ? 4 : 2, CS = K <= 32 ? 4 : 2, ES = K <= 32 ? 0 : 3;
  // Full barriers of S and of E: a barrier's tiles all belong to one group of row warps, which so sees
  // every phase of it.  With one per stage and an odd number of stages a group skips the other's
  // phases, and cannot tell "mine is here" from "the one before the other group's is not yet here".
  static constexpr int SB = BUFS % 2 ? 2 * BUFS : BUFS, EB = ES % 2 ? 2 * ES : ES;
  // tensor-memory columns
  static constexpr int A_HI = 0, A_LO = K, S0 = 2 * K, G0 = S0 + 128 * BUFS;
  static_assert(G0 + GBUFS * K <= 512, "tensor memory");
  static constexpr int PARTS = 64 * K;  // floats of one operand image part
};

// CUT_STATE: S is the result, stored row by row (a warp's 32 rows of a column are 128 bytes);
// bound by the stores, and by S's MMAs at 64 terms.
template <int K, CutUse USE>
__global__ void __launch_bounds__(NT, 1) k_cut_contract_tc(const __grid_constant__ CutArgs A) {
  using C = Cfg<K>;
  constexpr bool GRAD = USE == CUT_GRAD, STATE = USE == CUT_STATE;
  constexpr int HALF = 2 * C::PARTS;  // floats of one half of B: its hi and lo parts
  constexpr int ETILE = 128 * COLS;   // floats of a tile of E (complex: half of them used)
  constexpr int ES = STATE ? 0 : C::ES, EB = STATE ? 0 : C::EB;
  extern __shared__ __align__(128) float dyn[];
  float *sR = dyn, *sE = dyn + C::RS * HALF, *sC = sE + ES * ETILE;
  __shared__ __align__(8) unsigned long long bars[2 * (C::RS + C::CS) + EB + ES + C::SB + C::BUFS + C::GBUFS + 2];
  __shared__ uint32_t tslot;
  __shared__ int bad_s;
  __shared__ double es[2][8];
  volatile int *bad = &bad_s;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
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
  const CutView J = cut_view(A, job);
  // complex: rows (x, channel), two real terms per term, one value of E for both channels
  const int cx = J.desc->cx;
  const int mr = J.desc->half[h].m + cx, mc = J.desc->half[1 - h].m, D = J.desc->D << cx;
  const int ns = J.lay->ns[h], split = idx % ns, row0 = (idx / ns) * 128;
  const int nt = (1 << (mc - 6)) / ns, t0 = split * nt;
  const float *ap = reinterpret_cast<const float *>(J.ws + (cx ? J.lay->packr[h] : J.lay->pack[h]));
  const int ap_ld = (cx ? 128 : 256) * K;  // floats per 64 rows
  const float *bp = reinterpret_cast<const float *>(J.ws + J.lay->pack[1 - h]);
  const float *E = reinterpret_cast<const float *>(h ? J.table_t : J.table);  // in tile order
  const uint32_t bar0 = smem_addr(bars);
  // full barriers, then the empty ones
  auto rfull = [&](int s) { return bar0 + 8 * s; };
  auto rempty = [&](int s) { return rfull(C::RS + s); };
  auto cfull = [&](int s) { return rfull(2 * C::RS + s); };
  auto cempty = [&](int s) { return cfull(C::CS + s); };
  auto efull = [&](int s) { return cfull(2 * C::CS + s); };
  auto eempty = [&](int s) { return efull(EB + s); };
  auto sbar = [&](int b) { return eempty(ES + b); };
  auto lbar = [&](int b) { return sbar(C::SB + b); };
  auto gbar = [&](int b) { return lbar(C::BUFS + b); };
  auto last = [&](int i) { return gbar(C::GBUFS + i); };  // an issuer's MMAs, when it has given up
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(&tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 256) {
    bad_s = 0;
    auto init = [](uint32_t bar, int count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
    };
    for (int s = 0; s < 2 * (C::RS + C::CS) + EB; ++s) init(bar0 + 8 * s, 1);
    for (int s = 0; s < ES; ++s) init(eempty(s), 4);
    for (int b = 0; b < C::SB; ++b) init(sbar(b), 1);
    for (int b = 0; b < C::BUFS; ++b) init(lbar(b), 4);
    for (int b = 0; b < C::GBUFS; ++b) init(gbar(b), 1);
    for (int i = 0; i < 2; ++i) init(last(i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tslot;
  const int r = 32 * (w & 3) + lane;                       // this thread's row (warps 0-7)
  const uint32_t tw = tmem + ((uint32_t)(32 * (w & 3)) << 16);  // ... and lane quarter
  if (w < 4) {
    // the rows' operand: hi and lo parts into tensor memory
    const float *src = ap + (size_t)((row0 + r) >> 6) * ap_ld + ((r & 63) >> 3) * (K * 8) + (r & 7) * 4;
#pragma unroll
    for (int c = 0; c < 2 * K; c += 16) {
      const float *p = src + (c < K ? 0 : C::PARTS) + ((c % K) >> 2) * 32;
      float v[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 x = *reinterpret_cast<const float4 *>(p + 32 * k);
        v[4 * k] = x.x;
        v[4 * k + 1] = x.y;
        v[4 * k + 2] = x.z;
        v[4 * k + 3] = x.w;
      }
      st16(tw + C::A_HI + c, v);
    }
    st_wait();
  }
  fence_before();
  __syncthreads();
  fence_after();

  if constexpr (!ES) {
    if (w < 8)
      asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    else
      asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
  }
  if (w < 8) {
    // ------------------------------------------------------------ rows --
    float acc[K];
    const int g = w >> 2;
    float e_hi = 0.f, e_lo = 0.f, z_hi = 0.f, z_lo = 0.f;
    const int erow = 128 >> cx;  // rows of a tile of E: [j / 4][row][j % 4]
    const float *Ei = E + ((((size_t)(row0 >> 7) << (mc - 6)) + t0)) * (erow * COLS) + (r >> cx) * 4;
    f2 ev[ES ? 1 : COLS / 2];
    auto load = [&](int t) {
      const float *p = Ei + (size_t)t * (erow * COLS);
#pragma unroll
      for (int j = 0; j < COLS / 4; ++j)  // volatile: issued here, not where the values are used
        asm volatile("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(ev[2 * j]), "=l"(ev[2 * j + 1]) : "l"(p + 4 * erow * j));
    };
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.f;
    auto drain = [&](int t) {  // G of tile t
      if (!wait_warp(gbar(t % C::GBUFS), (t / C::GBUFS) & 1, bad)) return false;
      fence_after();
#pragma unroll
      for (int c = 0; c < K; c += 16) {
        float v[16];
        ld16(tw + C::G0 + K * (t % C::GBUFS) + c, v);
        ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[c + j] += v[j];
      }
      fence_before();
      return true;
    };
    constexpr int AHEAD = C::GBUFS == 4 ? 2 : 0;  // tiles between a tile's lambda and its G
    const f2 neg1 = pk2(-1.f, -1.f);
    int t = g;
    if constexpr (!ES && !STATE) load(t);  // (2 tiles at least)
    for (; t < nt; t += 2) {
      const int b = t % C::BUFS, ee = ES ? t % (ES + !ES) : 0;
      if constexpr (ES > 0)
        if (!wait_warp(efull(t % EB), (t / EB) & 1, bad)) break;
      if (!wait_warp(sbar(t % C::SB), (t / C::SB) & 1, bad)) break;
      fence_after();
      const uint32_t ts = tw + C::S0 + 128 * b;
      const float4 *et = reinterpret_cast<const float4 *>(sE + ee * ETILE) + (r >> cx);
      f2 e0 = 0, e1 = 0, z0 = 0, z1 = 0;
      float *out = nullptr;
      if constexpr (STATE)
        out = A.state + (size_t)job * A.state_stride + ((size_t)(t0 + t) << (mr + 6)) + row0 + r;
      auto tile = [&](auto energy) {
#pragma unroll(ES ? 1 : COLS / 16)
        for (int c = 0; c < COLS; c += 16) {
          float v[16], l[16];
          f2 tv[8];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if constexpr (ES > 0) {
              const float4 x = et[(c / 4 + k) * erow];
              tv[2 * k] = pk2(x.x, x.y);
              tv[2 * k + 1] = pk2(x.z, x.w);
            } else {
              tv[2 * k] = ev[c / 2 + 2 * k];
              tv[2 * k + 1] = ev[c / 2 + 2 * k + 1];
            }
          }
          ld16(ts + c, v);
          ld16(ts + 64 + c, l);
          ld_wait();
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const f2 s = add2(pk2(v[j], v[j + 1]), pk2(l[j], l[j + 1]));
            if constexpr (STATE) {
              float x, y;
              unpk2(s, x, y);
              out[(size_t)(c + j) << mr] = x;
              out[(size_t)(c + j + 1) << mr] = y;
              continue;
            }
            const f2 lam = mul2(s, tv[j / 2]);
            if constexpr (decltype(energy)::value) {
              f2 &e = (j & 2) ? e1 : e0, &z = (j & 2) ? z1 : z0;
              e = fma2(lam, s, e);
              z = fma2(s, s, z);
            }
            if constexpr (GRAD) {
              const f2 hi = lam & 0xFFFFE000FFFFE000ull;
              const f2 lo = fma2(hi, neg1, lam);  // exact
              unpk2(hi, v[j], v[j + 1]);
              unpk2(lo, l[j], l[j + 1]);
            }
          }
          if constexpr (GRAD) {
            st16(ts + c, v);
            st16(ts + 64 + c, l);
          }
        }
      };
      if (h == 0 && !STATE)
        tile(Yes{});
      else
        tile(No{});
      if constexpr (GRAD) st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) {
        arrive(lbar(b));
        if constexpr (ES > 0) arrive(eempty(ee));
      }
      if constexpr (!ES && !STATE)
        if (t + 2 < nt) load(t + 2);
      if (h == 0 && !STATE) {
        float x, y;
        unpk2(add2(e0, e1), x, y);
        two_sum(e_hi, e_lo, x + y);
        unpk2(add2(z0, z1), x, y);
        two_sum(z_hi, z_lo, x + y);
      }
      if constexpr (GRAD)
        if (t >= AHEAD && !drain(t - AHEAD)) break;
    }
    if constexpr (GRAD && AHEAD > 0)
      if (t >= 2 && !__any_sync(0xffffffffu, *bad)) drain(t - 2);
    if (h == 0 && !STATE) {
      double e = (double)e_hi + e_lo, z = (double)z_hi + z_lo;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
      }
      if (lane == 0) {
        es[0][w] = e;
        es[1][w] = z;
      }
    }
    // the two warp groups' sums of each row, through shared memory: every G is out, so every
    // MMA and every copy it waited for is complete
    float *x = dyn;
    if (GRAD && w >= 4) {
#pragma unroll
      for (int k = 0; k < K; ++k) x[k * 128 + r] = acc[k];
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const bool good = *bad == 0;  // else a wait gave up: NaN out
    if (GRAD && w < 4) {
      float *gout = reinterpret_cast<float *>(J.ws + J.lay->g[h]) + ((size_t)split * D << mr) + row0 + r;
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (k < D) {
          constexpr float up = (float)(TRUNC * (steps(COLS / 8) + steps(K / 16)) + LOST_LAMBDA);  // G's, S's and lambda's
          const float sum = acc[k] + x[k * 128 + r];
          gout[(size_t)k << mr] = good ? fmaf(sum, up, sum) : __int_as_float(0x7fc00000);
        }
    }
    // (in this item's own first column: the rows' column 0 is another split's to write)
    if (STATE && !good && w < 4)
      A.state[(size_t)job * A.state_stride + ((size_t)t0 << (mr + 6)) + row0 + r] = __int_as_float(0x7fc00000);
    if (h == 0 && tid == 0 && !STATE) {
      double e = 0.0, z = 0.0;
      for (int k = 0; k < 8; ++k) {
        e += es[0][k];
        z += es[1][k];
      }
      constexpr double up = 1.0 + 2.0 * TRUNC * steps(K / 16);  // (of E / z none is left: for X/Y strings' energies)
      e *= up;
      z *= up;
      double *ep = reinterpret_cast<double *>(J.ws + J.lay->ep) + 2 * idx;
      ep[0] = good ? e : __longlong_as_double(0x7ff8000000000000ll);
      ep[1] = good ? z : 1.0;
    }
  } else if (w == 8 || w == 11) {
    // ---------------------------------------------------------- copies --
    if (lane == 0) {
      auto copy = [&](float *dst, const float *src, uint32_t bytes, uint32_t bar) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_addr(dst)),
                     "l"(src), "r"(bytes), "r"(bar)
                     : "memory");
      };
      const float *bt = bp + (size_t)t0 * (256 * K);
      const int et = ETILE >> cx;
      const float *Ei = E + ((((size_t)(row0 >> 7) << (mc - 6)) + t0)) * et;
      if (w == 8) {
        for (int t = 0; t < nt; ++t) {
          const int s = t % C::RS;
          if (t >= C::RS && !wait_bounded(rempty(s), (t / C::RS - 1) & 1, bad)) break;
          copy(sR + s * HALF, bt + (size_t)t * (256 * K), HALF * 4, rfull(s));
          if constexpr (ES > 0) {
            const int e = t % ES;
            if (t >= ES && !wait_bounded(eempty(e), (t / ES - 1) & 1, bad)) break;
            copy(sE + e * ETILE, Ei + (size_t)t * et, et * 4, efull(t % EB));
          }
        }
        // the last commits have arrived before the CTA leaves
        for (int t = nt > C::RS ? nt - C::RS : 0; t < nt; ++t) wait_bounded(rempty(t % C::RS), (t / C::RS) & 1, bad);
      } else if (GRAD) {
        for (int t = 0; t < nt; ++t) {
          const int s = t % C::CS;
          if (t >= C::CS && !wait_bounded(cempty(s), (t / C::CS - 1) & 1, bad)) break;
          copy(sC + s * HALF, bt + (size_t)t * (256 * K) + HALF, HALF * 4, cfull(s));
        }
        for (int t = nt > C::CS ? nt - C::CS : 0; t < nt; ++t) wait_bounded(cempty(t % C::CS), (t / C::CS) & 1, bad);
      }
    }
  } else if (w == 9 || w == 10) {
    // ------------------------------------------------------------ MMAs --
    // Warp 9 issues S, warp 10 G: a warp's barrier polls queue behind its own MMAs (about
    // 250 clocks), so with one warp the pipe ran dry at every change.  One elected lane runs
    // each loop: from a branch on elect.sync an MMA takes 11 clocks to issue, from one on
    // the lane number 45, more than a 128 x 64 x 8 MMA runs.
    uint32_t el;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(el));
    const uint32_t tu = __shfl_sync(0xffffffffu, tmem, 0);
    if (el && w == 9) {
      for (int t = 0; t < nt; ++t) {
        const int s = t % C::RS, b = t % C::BUFS, u = t - C::BUFS;
        if (!wait_bounded(rfull(s), (t / C::RS) & 1, bad)) break;
        // the buffer's previous tile: its lambda has been contracted (or, energies only, read)
        if (u >= 0 && !(GRAD ? wait_bounded(gbar(u % C::GBUFS), (u / C::GBUFS) & 1, bad)
                             : wait_bounded(lbar(b), (u / C::BUFS) & 1, bad)))
          break;
        fence_after();
        const uint32_t bs = smem_addr(sR) + s * (HALF * 4), d = tu + C::S0 + 128 * b;
        const uint32_t bh = op_lo(bs), bl = op_lo(bs + C::PARTS * 4);
        constexpr uint32_t HI = op_hi(K * 32), ID = idesc(COLS);
        mmas<HI, ID, true, K / 8>(d, tu + C::A_LO, bh);
        mmas<HI, ID, false, K / 8>(d, tu + C::A_HI, bl);
        mmas<HI, ID, false, K / 16>(d, tu + C::A_HI, bh);
        mmas<HI, ID, true, K / 16>(d + 64, tu + C::A_HI + K / 2, bh + K);  // (16 per step of 8)
        commit(sbar(t % C::SB));
        commit(rempty(s));
      }
    } else if (GRAD && el && w == 10) {
      for (int t = 0; t < nt; ++t) {
        const int s = t % C::CS, b = t % C::BUFS;
        if (!wait_bounded(cfull(s), (t / C::CS) & 1, bad) || !wait_bounded(lbar(b), (t / C::BUFS) & 1, bad)) break;
        fence_after();
        const uint32_t bs = smem_addr(sC) + s * (HALF * 4);
        const uint32_t lh = tu + C::S0 + 128 * b, ll = lh + 64, d = tu + C::G0 + K * (t % C::GBUFS);
        const uint32_t bh = op_lo(bs), bl = op_lo(bs + C::PARTS * 4);
        constexpr uint32_t HI = op_hi(2048), ID = idesc(K);
        mmas<HI, ID, true, COLS / 8>(d, ll, bh);
        mmas<HI, ID, false, COLS / 8>(d, lh, bl);
        mmas<HI, ID, false, COLS / 8>(d, lh, bh);
        commit(gbar(t % C::GBUFS));
        commit(cempty(s));
      }
    }
    if (el && *bad && (w == 9 || (GRAD && w == 10))) {  // the MMAs in flight end before the CTA does
      int none = 0;
      commit(last(w - 9));
      wait_bounded(last(w - 9), 0, &none);
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  fence_after();
  // unless a wait gave up, every stage copied has been read; if one did, the copies in
  // flight are waited for before leaving
  if (bad_s && tid == 256) {
    int none = 0;
    for (int s = 0; s < C::RS; ++s)
      for (int p = 0; p < 2; ++p) wait_bounded(rfull(s), p, &none);
    for (int s = 0; s < EB; ++s)
      for (int p = 0; p < 2; ++p) wait_bounded(efull(s), p, &none);
    for (int s = 0; GRAD && s < C::CS; ++s)
      for (int p = 0; p < 2; ++p) wait_bounded(cfull(s), p, &none);
  }
  __syncthreads();
  if (w == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

template <int K, CutUse USE>
cudaError_t launch_k(const CutArgs &A, cudaStream_t s) {
  using C = Cfg<K>;
  // (the copies' stages, then reused for the rows' sums: K x 128 floats)
  const size_t need = (size_t)4 * ((C::RS + (USE == CUT_GRAD ? C::CS : 0)) * 2 * C::PARTS +
                                   (USE == CUT_STATE ? 0 : C::ES) * 128 * COLS);
  auto k = k_cut_contract_tc<K, USE>;
  static SmemLimit limit;
  if (const cudaError_t e = limit.set(k, need)) return e;
  k<<<A.nblk, NT, need, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

template <int K>
static cudaError_t launch_use(const CutArgs &A, CutUse use, cudaStream_t s) {
  return use == CUT_GRAD ? launch_k<K, CUT_GRAD>(A, s) : use == CUT_STATE ? launch_k<K, CUT_STATE>(A, s) : launch_k<K, CUT_ENERGY>(A, s);
}
cudaError_t launch_cut_tc(const CutArgs &A, int K, CutUse use, cudaStream_t s) {
  return K == 16 ? launch_use<16>(A, use, s) : K == 32 ? launch_use<32>(A, use, s) : launch_use<64>(A, use, s);
}

}  // namespace gvqe
