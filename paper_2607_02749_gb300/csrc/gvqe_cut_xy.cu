// gvqe_cut_xy.cu -- strings with X/Y letters in the two-half evaluation (FP32).
//
// A string is a signed product of a part on either half, c Q_lo (x) Q_hi with
// Q|u> = (-1)^popcount(u & z) |u ^ x>, and psi = sum_a L_a (x) R_a (gvqe_cut.cuh), so
//   <psi|c Q_lo Q_hi|psi> = c sum_ab M_lo(a, b) M_hi(a, b),   M(a, b) = <T_a|Q|T_b>,
//   G_L(x, a) += c sum_b (Q_lo L_b)(x) M_hi(a, b)             and the same for R.
// Many strings share a part: the work is one D x D matrix M per distinct part (k_xy_m), one
// combination N = sum c M_other per part over its strings (k_xy_n, with the energy), and
// one product of the part's table with N (k_xy_g): 2 D^2 2^m multiply-adds per part and
// half, instead of one pass over 2^n amplitudes per group of strings.
#include "gvqe_cut.cuh"

namespace gvqe {
namespace {

// [a][x] -> [x][a], terms from D to DP zero: 64 rows per CTA
template <int DP>
__global__ void __launch_bounds__(256) k_xy_rows(const __grid_constant__ CutArgs A) {
  __shared__ float s[DP][65];
  const int job = blockIdx.y, h = blockIdx.z;
  const CutView J = cut_view(A, job);
  const int D = J.desc->D, m = J.desc->half[h].m, x0 = blockIdx.x * 64;
  if (x0 >> m) return;
  const float *tab = reinterpret_cast<const float *>(J.ws + J.lay->tab[h]);
  for (int i = threadIdx.x; i < DP * 64; i += 256) {
    const int a = i >> 6, x = i & 63;
    s[a][x] = a < D ? tab[((size_t)3 * a << m) + x0 + x] : 0.f;
  }
  __syncthreads();
  float *rows = reinterpret_cast<float *>(J.ws + J.lay->rows[h]) + (size_t)x0 * DP;
  for (int i = threadIdx.x; i < DP * 64; i += 256) rows[i] = s[i % DP][i / DP];
}

// M(a, b) = sum_y T_a(y) s(y ^ xm) T_b(y ^ xm) over a run of y, for the parts of one CTA: 8 x 8
// outputs per thread, (DP / 8)^2 threads per part.  Both rows come straight from L1 / L2
// (6 wavefronts against 64 multiply-adds per warp and y).  Sums of 64 products in registers,
// 64-sums added in shared memory, runs in FP64 (k_xy_sum): the energy is a sum of many small
// terms, and sums of 256 in one register were ten times less exact.
template <int DP>
__global__ void __launch_bounds__(256) k_xy_m(const __grid_constant__ CutArgs A) {
  constexpr int TPU = (DP / 8) * (DP / 8), UPB = 256 / TPU;
  extern __shared__ float sums[];  // [64][256]
  const int job = blockIdx.z, tid = threadIdx.x;
  const CutView J = cut_view(A, job);
  const int h = blockIdx.y, m = J.desc->half[h].m;
  const CutXy &X = *A.xy;
  const int nu = (X.U[h] + UPB - 1) / UPB, run = J.lay->xrun[h];
  const int sl = blockIdx.x / nu, u = (blockIdx.x % nu) * UPB + tid / TPU;
  if (sl >= (1 << m) / run) return;
  const bool on = u < X.U[h];
  const uint32_t xm = on ? X.xm[h][u] : 0, zm = on ? X.zm[h][u] : 0;
  const int i0 = (tid % TPU) / (DP / 8) * 8, j0 = (tid % TPU) % (DP / 8) * 8;
  const float *rows = reinterpret_cast<const float *>(J.ws + J.lay->rows[h]);
#pragma unroll
  for (int k = 0; k < 64; ++k) sums[k * 256 + tid] = 0.f;
  for (int y0 = sl * run; y0 < (sl + 1) * run; y0 += 64) {
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 2
    for (int y = y0; y < y0 + 64; ++y) {
      const uint32_t v = (uint32_t)y ^ xm;
      const float4 *pa = reinterpret_cast<const float4 *>(rows + (size_t)y * DP + i0);
      const float4 *pb = reinterpret_cast<const float4 *>(rows + (size_t)v * DP + j0);
      const float4 a0 = __ldg(pa), a1 = __ldg(pa + 1), b0 = __ldg(pb), b1 = __ldg(pb + 1);
      const uint32_t sg = (uint32_t)__popc(v & zm) << 31;
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) b[j] = __uint_as_float(__float_as_uint(b[j]) ^ sg);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) sums[(8 * i + j) * 256 + tid] += acc[i][j];
  }
  if (!on) return;
  float *out = reinterpret_cast<float *>(J.ws + J.lay->mpart[h]) + ((size_t)sl * X.U[h] + u) * (DP * DP);
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) out[(i0 + i) * DP + j0 + j] = sums[(8 * i + j) * 256 + tid];
}

// M = sum of its runs in FP64
__global__ void __launch_bounds__(256) k_xy_sum(const __grid_constant__ CutArgs A, int dd) {
  const int job = blockIdx.z, h = blockIdx.y;
  const CutView J = cut_view(A, job);
  const long long cnt = (long long)A.xy->U[h] * dd, i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= cnt) return;
  const float *p = reinterpret_cast<const float *>(J.ws + J.lay->mpart[h]) + i;
  const int ns = (1 << J.desc->half[h].m) / J.lay->xrun[h];
  double s = 0.0;
  for (int k = 0; k < ns; ++k) s += (double)p[(size_t)k * cnt];
  reinterpret_cast<double *>(J.ws + J.lay->mm[h])[i] = s;
}

// N(b, a) = sum over the part's strings of c M_other(a, b); on half 0 also the energy of the
// part's strings, sum_ab M(a, b) N(a, b), in FP64.  One CTA per part.
__global__ void __launch_bounds__(256) k_xy_n(const __grid_constant__ CutArgs A, int dp) {
  const int job = blockIdx.z, h = blockIdx.y, u = blockIdx.x, tid = threadIdx.x;
  const CutXy &X = *A.xy;
  if (u >= X.U[h]) return;
  const CutView J = cut_view(A, job);
  const int dd = dp * dp, t0 = X.start[h][u], t1 = X.start[h][u + 1];
  const double *mo = reinterpret_cast<const double *>(J.ws + J.lay->mm[1 - h]);
  const double *mine = reinterpret_cast<const double *>(J.ws + J.lay->mm[h]) + (size_t)u * dd;
  float *out = J.lay->nn[h] >= 0 ? reinterpret_cast<float *>(J.ws + J.lay->nn[h]) + (size_t)u * dd : nullptr;
  double e = 0.0;
  for (int i = tid; i < dd; i += 256) {
    double s = 0.0;
    for (int t = t0; t < t1; ++t) s = fma(X.coef[h][t], mo[(size_t)X.other[h][t] * dd + i], s);
    if (out) out[(i % dp) * dp + i / dp] = (float)s;
    e = fma(mine[i], s, e);
  }
  if (h) return;
  __shared__ double es[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((tid & 31) == 0) es[tid >> 5] = e;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += es[w];
    reinterpret_cast<double *>(J.ws + J.lay->exy)[u] = s;
  }
}

// G(x, a) = sum over the parts of sum_b s(v) T_b(v) N(b, a), v = x ^ xm, for ROWS rows x: the parts
// with one x mask in turn read the same rows v (one block, transposed in shared memory) and
// add to one accumulator per row v, 8 rows by 4 terms a thread; it goes to rows v ^ xm of the
// sums in shared memory once per mask.  5 shared wavefronts per 32 multiply-adds of a warp.
template <int DP>
struct GCfg {
  static constexpr int ROWS = 64;
  static constexpr int NT = (ROWS / 8) * (DP / 4);
  static constexpr int LD = ROWS + 4;
};
template <int DP>
__global__ void __launch_bounds__(GCfg<DP>::NT) k_xy_g(const __grid_constant__ CutArgs A) {
  using C = GCfg<DP>;
  extern __shared__ __align__(16) float sm[];
  float *sT = sm;                    // [b][v], LD per b
  float *sG = sT + DP * C::LD;       // [a][x], LD per a
  float *sN = sG + DP * C::LD;       // [2][b][a]
  const int job = blockIdx.z, h = blockIdx.y, tid = threadIdx.x;
  const CutView J = cut_view(A, job);
  const int m = J.desc->half[h].m, x0 = blockIdx.x * C::ROWS, D = J.desc->D;
  if (x0 >> m) return;
  const CutXy &X = *A.xy;
  const float *rows = reinterpret_cast<const float *>(J.ws + J.lay->rows[h]);
  const float *nn = reinterpret_cast<const float *>(J.ws + J.lay->nn[h]);
  const int v0 = (tid % (C::ROWS / 8)) * 8, a0 = (tid / (C::ROWS / 8)) * 4;
  for (int i = tid; i < DP * C::LD; i += C::NT) sG[i] = 0.f;
  for (int g = 0; g < X.ng[h]; ++g) {
    const int u0 = X.gstart[h][g], u1 = X.gstart[h][g + 1];
    const uint32_t xm = X.xm[h][u0];
    const int base = x0 ^ (int)(xm & ~(uint32_t)(C::ROWS - 1));  // rows v: the block of x0 ^ xm
    for (int i = tid; i < C::ROWS * DP; i += C::NT)
      sT[(i % DP) * C::LD + i / DP] = rows[(size_t)base * DP + i];
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int u = u0; u < u1; ++u) {
      float *n = sN + (u & 1) * (DP * DP);
      for (int i = tid; i < DP * DP / 4; i += C::NT)
        reinterpret_cast<float4 *>(n)[i] = __ldg(reinterpret_cast<const float4 *>(nn + (size_t)u * (DP * DP)) + i);
      __syncthreads();
      float t[8][4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) t[i][j] = 0.f;
#pragma unroll 4
      for (int b = 0; b < DP; ++b) {
        const float4 p = *reinterpret_cast<const float4 *>(sT + b * C::LD + v0);
        const float4 q = *reinterpret_cast<const float4 *>(sT + b * C::LD + v0 + 4);
        const float4 w = *reinterpret_cast<const float4 *>(n + b * DP + a0);
        const float tv[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) t[i][j] = fmaf(tv[i], wv[j], t[i][j]);
      }
      const uint32_t zm = X.zm[h][u];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float s = (__popc((uint32_t)(base + v0 + i) & zm) & 1) ? -1.f : 1.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(s, t[i][j], acc[i][j]);
      }
    }
    const int xl = (int)(xm & (uint32_t)(C::ROWS - 1));
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sG[(a0 + j) * C::LD + ((v0 + i) ^ xl)] += acc[i][j];
    __syncthreads();  // sT and sG: the next mask's turn
  }
  float *gout = reinterpret_cast<float *>(J.ws + J.lay->g[h]) + (((size_t)J.lay->ns[h] * D) << m) + x0;
  for (int i = tid; i < D * C::ROWS; i += C::NT)
    gout[((size_t)(i / C::ROWS) << m) + i % C::ROWS] = sG[(i / C::ROWS) * C::LD + i % C::ROWS];
}

template <int DP>
cudaError_t launch_dp(const CutArgs &A, const CutGrid &g, const CutXyDims &x, bool grad, cudaStream_t s, int *launches) {
  const unsigned jobs = (unsigned)A.njobs;
  const int U = x.U[0] > x.U[1] ? x.U[0] : x.U[1];
  k_xy_rows<DP><<<dim3(1u << (g.m0 - 6), jobs, 2), 256, 0, s>>>(A);
  constexpr int UPB = 256 / ((DP / 8) * (DP / 8));
  const int run = A.job0.lay.xrun[0];
  static SmemLimit lm, lg;
  cudaError_t e = lm.set(k_xy_m<DP>, 64 * 256 * 4);
  if (e != cudaSuccess) return e;
  k_xy_m<DP><<<dim3((unsigned)((U + UPB - 1) / UPB * ((1 << g.m0) / run)), 2, jobs), 256, 64 * 256 * 4, s>>>(A);
  k_xy_sum<<<dim3((unsigned)(((long long)U * DP * DP + 255) / 256), 2, jobs), 256, 0, s>>>(A, DP * DP);
  k_xy_n<<<dim3((unsigned)U, grad ? 2 : 1, jobs), 256, 0, s>>>(A, DP);
  *launches += 4;
  if (grad) {
    constexpr size_t sm = (size_t)(2 * DP * GCfg<DP>::LD + 2 * DP * DP) * 4;
    e = lg.set(k_xy_g<DP>, sm);
    if (e != cudaSuccess) return e;
    k_xy_g<DP><<<dim3(1u << (g.m0 - 6), 2, jobs), GCfg<DP>::NT, sm, s>>>(A);
    *launches += 1;
  }
  return cudaGetLastError();
}

}  // namespace

int cut_xy_dp(int D) { return D < 8 ? 8 : D; }

cudaError_t launch_cut_xy(const CutArgs &A, const CutGrid &g, const CutXyDims &x, bool grad, cudaStream_t s, int *launches) {
  switch (cut_xy_dp(g.D)) {
    case 8: return launch_dp<8>(A, g, x, grad, s, launches);
    case 16: return launch_dp<16>(A, g, x, grad, s, launches);
    case 32: return launch_dp<32>(A, g, x, grad, s, launches);
    default: return launch_dp<64>(A, g, x, grad, s, launches);
  }
}

}  // namespace gvqe
