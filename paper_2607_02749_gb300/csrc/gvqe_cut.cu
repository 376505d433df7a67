// gvqe_cut.cu -- evaluation of a circuit from its two halves: plan, operand images, the
// FP64 contraction and the final sums (the half circuits are gvqe_cut_half.cu, the FP32
// contraction gvqe_cut_tc.cu).
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

bool cut_build(int n, int reps, int ent, int prec, int gates, CutDesc *d) {
  memset(d, 0, sizeof(*d));
  const int h = (n + 1) / 2;
  // FP32: 128-row and 64-column tiles in the contraction; FP64: 32 x 32 tiles, and a half's
  // state (with its padding) in one CTA's shared memory
  if (reps < 1 || reps > CUT_MAX_LAYERS || n - h < (prec ? 5 : 7) || h > (prec || gates == 2 ? CUT_MAX_M - 1 : CUT_MAX_M))
    return false;
  if (gates == 2 && prec) return false;
  d->cx = gates == 2;
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
    uint32_t pm[2][2] = {{0, 0}, {0, 0}}, pb[2][2] = {{0, 0}, {0, 0}};  // projections: parity(x & pm) == parity(b & pb)
    int np[2] = {0, 0}, nb = 0;
    for (const auto &g : cnot_list(ent, n, r)) {
      const int sc = g.first >= h, st = g.second >= h;
      const int c = g.first - lo[sc], t = g.second - lo[st];
      if (sc == st) {
        xm[st][t] ^= xm[sc][c];
        bm[st][t] ^= bm[sc][c];
        continue;
      }
      if (nb == 2 || np[sc] == 2) return false;
      pm[sc][np[sc]] = xm[sc][c];
      pb[sc][np[sc]++] = bm[sc][c] ^ (1u << nb);
      bm[st][t] ^= 1u << nb;
      ++nb;
    }
    for (int s = 0; s < 2; ++s) {
      const int m = d->half[s].m;
      CutLayer &l = *L[s];
      l.shift = kappa;
      l.nb = nb;
      uint32_t rows[CUT_MAX_M], inv[CUT_MAX_M];
      for (int q = 0; q < m; ++q) {
        rows[q] = xm[s][q];
        inv[q] = 1u << q;
        for (int i = 0; i < m; ++i)
          if ((xm[s][q] >> i) & 1u) l.fc[i] |= 1u << q;
        for (uint32_t b = 0; b < 4; ++b) l.fo[b] |= (uint32_t)parity32(bm[s][q] & b) << q;
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
          if ((inv[q] >> i) & 1u) l.ic[i] |= 1u << q;
      for (uint32_t b = 0; b < 4; ++b) {
        uint32_t x = 0;
        for (int i = 0; i < m; ++i)
          if ((l.fo[b] >> i) & 1u) x ^= l.ic[i];
        l.io[b] = x;
      }
      for (int k = 0; k < np[s]; ++k) {  // the projections test x: the source of a gather, or the place
        const uint32_t bit = 1u << (16 + k);
        for (int i = 0; i < m; ++i) {
          if (parity32(l.ic[i] & 0x7fffu & pm[s][k])) l.ic[i] |= bit;
          if ((pm[s][k] >> i) & 1u) l.fc[i] |= bit;
        }
        for (uint32_t b = 0; b < 4; ++b) {
          if (parity32(l.io[b] & 0x7fffu & pm[s][k]) ^ parity32(pb[s][k] & b)) l.io[b] |= bit;
          if (parity32(pb[s][k] & b)) l.fo[b] |= bit;
        }
      }
    }
    kappa += nb;
    // FP64 above 64 terms: the row form alone (k_cut_rows64); complex: two real terms per term
    if (kappa > (prec && h <= 8 ? CUT_MAX_PATH64 : CUT_MAX_PATH) - d->cx) return false;
  }
  d->kappa = kappa;
  d->D = 1 << kappa;
  return true;
}

// Terms of the tensor-core operands: at least 16 (the smallest N of its MMAs).
int cut_k(int D) { return D < 16 ? 16 : D; }

constexpr int CUT_ROWS32 = 128, CUT_COLS32 = 64;  // FP32 contraction tile
constexpr int CUT_TILE64 = 32;                    // FP64 contraction tile (square)

// FP64 contraction with a CTA per row (k_cut_rows64)
static bool cut_by_rows(int m0, int D) { return m0 <= 8 && D >= 64; }
static bool cut_by_rows(const CutDesc &d) { return cut_by_rows(d.half[0].m, d.D); }

CutLayout cut_layout(const CutDesc &d, int prec, bool grad, const CutXyDims *xy) {
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
    const long long S = 1LL << (d.half[s].m + d.cx), T = (long long)d.D << d.cx;  // rows (with the channel), real terms
    const int mo = d.half[1 - s].m;
    l.rb[s] = (int)(S / (prec ? (cut_by_rows(d) ? 1 : CUT_TILE64) : CUT_ROWS32));
    const long long tiles = (1LL << mo) / (prec ? CUT_TILE64 : CUT_COLS32);
    // enough items for 152 SMs on a single vector, but runs long enough that an item's
    // set-up (its rows into tensor memory, the first tiles) stays small
    const long long per = prec ? 8 : 32;
    l.ns[s] = prec && cut_by_rows(d) ? 1 : (int)(tiles / per < 1 ? 1 : tiles / per > 4 ? 4 : tiles / per);
    const int sr = prec || d.cx ? 2 : 3;  // numbers kept per amplitude
    l.tab[s] = take(d.D * S * es * (d.cx ? 1 : sr));
    if (!prec) l.pack[s] = take((S >> d.cx) * cut_k(T) * 16);
    if (d.cx) l.packr[s] = take(S * cut_k(T) * 8);
    if (grad || (!prec && !d.cx && d.half[0].m > HALF_SMALL_M(0))) {  // FP32 goes layer by layer through them
      long long states = 0;
      for (int r = 0; r < d.reps; ++r) states += 1LL << d.half[s].L[r].shift;
      if (d.cx) states += d.D;  // the last layer's too, before its RZ
      l.phi[s] = take(sr * states * S * es);
    }
    if (grad) {
      l.g[s] = take((l.ns[s] + (xy ? 1 : 0)) * T * S * es);
    }
  }
  for (int s = 0; s < 2; ++s) l.gs[s] = l.ns[s] + (xy ? 1 : 0);
  if (xy) {
    const long long dp = cut_xy_dp(d.D);
    for (int s = 0; s < 2; ++s) {
      const long long S = 1LL << d.half[s].m;
      // runs of one length for both halves: long enough to pay for their sums, 16 at most
      l.xrun[s] = (int)(S / 16 < 128 ? 128 : S / 16 > 1024 ? 1024 : S / 16);
      if (s == 1 && l.xrun[1] > l.xrun[0]) l.xrun[1] = l.xrun[0];
    }
    l.xrun[0] = l.xrun[1] = l.xrun[0] < l.xrun[1] ? l.xrun[0] : l.xrun[1];
    for (int s = 0; s < 2; ++s) {
      const long long S = 1LL << d.half[s].m;
      l.rows[s] = take(S * dp * 4);
      l.mpart[s] = take(S / l.xrun[s] * xy->U[s] * dp * dp * 4);
      l.mm[s] = take((long long)xy->U[s] * dp * dp * 8);
      l.nn[s] = grad ? take((long long)xy->U[s] * dp * dp * 4) : -1;
    }
    l.nexy = xy->U[0];
    l.exy = take((long long)xy->U[0] * 8);
  }
  if (grad) l.gp = take(2LL * d.D * (d.reps + 1) * (16 << d.cx) * 8);
  l.ep = take((long long)l.rb[0] * l.ns[0] * 16);
  l.total = off;
  return l;
}

// The tensor-core operand images of both tables of a job: per 64 rows x the blocks
// [hi | lo] of the row form (K-major over a) and [hi | lo] of the column form (rows a,
// K-major over x), core matrices of 8 rows x 16 bytes; terms beyond the table's are zero.
// One CTA per 64 rows, through shared memory; 16-byte stores.  A complex table T gives the
// columns (Re T_a, Im T_a) of real terms 2a, 2a + 1 over x, and in row form alone the rows
// (x, 0): (Re T_a, -Im T_a) and (x, 1): (Im T_a, Re T_a).
template <bool LOW>
__device__ __forceinline__ void pack_form(const float *s, float4 *out, int K, bool row) {
  for (int i = threadIdx.x; i < K * 16; i += 256) {
    const int r = row ? (i & 7) + 8 * (i / (2 * K)) : 4 * ((i >> 3) & 15);  // [r / 8][a / 4][r % 8]
    const int a = row ? 4 * ((i >> 3) % (K / 4)) : (i & 7) + 8 * (i >> 7);  // [a / 8][r / 4][a % 8]
    float hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int at = row ? (a + k) * 65 + r : a * 65 + r + k;
      const float x = s[at];
      asm("cvt.rna.tf32.f32 %0, %1;" : "=f"(hi[k]) : "f"(x));
      lo[k] = x - hi[k];
      if (LOW) {  // the table's own low part, and the rounding to the tensor cores' 11 bits to nearest
        const float y = lo[k] + s[K * 65 + at];
        asm("cvt.rna.tf32.f32 %0, %1;" : "=f"(lo[k]) : "f"(y));
      }
    }
    out[i] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    out[16 * K + i] = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
}
template <bool CX>
__global__ void __launch_bounds__(256) k_cut_pack(const __grid_constant__ CutArgs A, int K) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  float *s = reinterpret_cast<float *>(cut_smem);  // [term][65]
  int job, h, tile;
  if (A.items) {
    const int4 it = A.items[blockIdx.x];
    job = it.x;
    h = it.y;
    tile = it.z;
  } else {
    const int per = A.nblk;  // tiles of both halves
    job = blockIdx.x / per;
    tile = blockIdx.x % per;
    h = tile >= A.blk0;
    if (h) tile -= A.blk0;
  }
  const CutView J = cut_view(A, job);
  const int D = J.desc->D, m = J.desc->half[h].m;
  const float *tab = reinterpret_cast<const float *>(J.ws + J.lay->tab[h]);
  float4 *out = reinterpret_cast<float4 *>(J.ws + J.lay->pack[h]) + (size_t)tile * (64 * K);
  for (int i = threadIdx.x; i < K * 64; i += 256) {
    const int a = i >> 6, x = tile * 64 + (i & 63);
    float v = 0.f, low = 0.f;
    if constexpr (CX) {
      if (a < 2 * D) v = tab[((size_t)(a >> 1) << (m + 1)) + 2 * x + (a & 1)];
    } else if (a < D) {
      const float *p = tab + ((size_t)3 * a << m) + x;
      v = p[0];
      low = p[(size_t)2 << m];
    }
    s[a * 65 + (i & 63)] = v;
    if constexpr (!CX) s[(K + a) * 65 + (i & 63)] = low;
  }
  __syncthreads();
  pack_form<!CX>(s, out, K, true);
  pack_form<!CX>(s, out + 32 * K, K, false);
  if constexpr (CX) {  // the two 64-row blocks (x, channel) of these 64 x
    float4 *rows = reinterpret_cast<float4 *>(J.ws + J.lay->packr[h]) + (size_t)tile * (64 * K);
    for (int b = 0; b < 2; ++b) {
      __syncthreads();
      for (int i = threadIdx.x; i < K * 64; i += 256) {
        const int a = i >> 6, r = i & 63, x = tile * 64 + b * 32 + (r >> 1), ch = r & 1;
        float v = 0.f;
        if (a < 2 * D) v = tab[((size_t)(a >> 1) << (m + 1)) + 2 * x + (ch ^ (a & 1))];
        s[a * 65 + r] = (a & 1) && !ch ? -v : v;
      }
      __syncthreads();
      pack_form<false>(s, rows + b * 32 * K, K, true);
    }
  }
}

// ------------------------------------------------------ FP64 contraction --
// Items of 32 rows x a run of columns, 256 threads, 32 x 32 tiles: psi = sum_a L_a R_a
// (2 x 2 per thread), lambda = E psi into shared memory, G += lambda x the column
// table.  The FP64 pipe bounds it (about 2 multiply-adds per clock and SM): 2 D per
// amplitude and contraction against 6 (reps + 1) n of the gate-by-gate sweeps.
constexpr int C64 = CUT_TILE64, C64LD = C64 + 1;

constexpr int NA = 8;  // terms per thread of G: 64 in all (more are taken by rows, on registers of up to 16 qubits)
template <bool GRAD>
__global__ void __launch_bounds__(256) k_cut_contract64(const __grid_constant__ CutArgs A) {
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
  const CutView J = cut_view(A, job);
  const int D = J.desc->D, m0 = J.desc->half[0].m;
  const int mr = J.desc->half[h].m, mc = J.desc->half[1 - h].m;
  const int ns = J.lay->ns[h], split = idx % ns, row0 = (idx / ns) * C64;
  const long long Sr = 1LL << mr, Sc = 1LL << mc;
  const int cols = (int)(Sc / ns), col0 = split * cols;
  const double *rt = reinterpret_cast<const double *>(J.ws + J.lay->tab[h]);
  const double *ct = reinterpret_cast<const double *>(J.ws + J.lay->tab[1 - h]);
  const double *E = reinterpret_cast<const double *>(J.table);
  double *sR = reinterpret_cast<double *>(cut_smem), *sC = sR + D * C64LD, *sL = sC + D * C64LD;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int i = tid; i < D * C64; i += 256) sR[(i >> 5) * C64LD + (i & 31)] = rt[(i >> 5) * 2 * Sr + row0 + (i & 31)];
  double acc[NA], e = 0.0;
#pragma unroll
  for (int k = 0; k < NA; ++k) acc[k] = 0.0;
  const int gi = tid & 31, ga = tid >> 5;  // G: row gi, terms ga + 8 k
  for (int c0 = col0; c0 < col0 + cols; c0 += C64) {
    __syncthreads();
    for (int i = tid; i < D * C64; i += 256) sC[(i >> 5) * C64LD + (i & 31)] = ct[(i >> 5) * 2 * Sc + c0 + (i & 31)];
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
      for (int k = 0; k < NA; ++k) {
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
    double *g = reinterpret_cast<double *>(J.ws + J.lay->g[h]) + (size_t)split * D * Sr;
#pragma unroll
    for (int k = 0; k < NA; ++k)
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
      double *ep = reinterpret_cast<double *>(J.ws + J.lay->ep) + 2 * idx;
      ep[0] = s;
      ep[1] = 0.0;
    }
  }
}

// Small registers with many terms (halves of at most 8 qubits): one CTA per row, so that the
// FP64 pipes of many SMs share the work (n = 10, 256 terms: 64 CTAs where 32-row items
// give 2).  psi of the row's columns with the terms split over the threads, then G with a
// thread per term; the column table comes from L2 and stays in L1.
template <bool GRAD>
__global__ void __launch_bounds__(256) k_cut_rows64(const __grid_constant__ CutArgs A) {
  __shared__ double row[256], lam[256], part[256], es[8];
  int job, h, idx;
  if (A.items) {
    const int4 it = A.items[blockIdx.x];
    job = it.x;
    h = it.y;
    idx = it.z;
  } else {
    job = blockIdx.x % A.njobs;
    idx = blockIdx.x / A.njobs;
    h = idx >= A.blk0;
    if (h) idx -= A.blk0;
  }
  const CutView J = cut_view(A, job);
  const int D = J.desc->D, m0 = J.desc->half[0].m, mr = J.desc->half[h].m, mc = J.desc->half[1 - h].m;
  const int tid = threadIdx.x, cols = 1 << mc, j = tid & (cols - 1), np = 256 >> mc;
  const double *rt = reinterpret_cast<const double *>(J.ws + J.lay->tab[h]);
  const double *ct = reinterpret_cast<const double *>(J.ws + J.lay->tab[1 - h]);
  if (tid < D) row[tid] = rt[((size_t)2 * tid << mr) + idx];
  __syncthreads();
  double s0 = 0.0, s1 = 0.0;
  for (int a = tid >> mc; a < D; a += 2 * np) {
    s0 = fma(row[a], ct[((size_t)2 * a << mc) + j], s0);
    if (a + np < D) s1 = fma(row[a + np], ct[((size_t)2 * (a + np) << mc) + j], s1);
  }
  part[tid] = s0 + s1;
  __syncthreads();
  double e = 0.0;
  if (tid < cols) {
    double s = part[tid];
    for (int k = 1; k < np; ++k) s += part[k * cols + tid];
    const long long i = idx, x = h ? ((i << m0) | tid) : (((long long)tid << m0) | i);
    const double l = reinterpret_cast<const double *>(J.table)[x] * s;
    e = l * s;
    lam[tid] = l;
  }
  __syncthreads();
  if constexpr (GRAD)
    if (tid < D) {
      const double2 *c = reinterpret_cast<const double2 *>(ct + ((size_t)2 * tid << mc));
      double g0 = 0.0, g1 = 0.0;
#pragma unroll 8
      for (int k = 0; k < cols / 2; ++k) {
        const double2 x = c[k];
        g0 = fma(lam[2 * k], x.x, g0);
        g1 = fma(lam[2 * k + 1], x.y, g1);
      }
      reinterpret_cast<double *>(J.ws + J.lay->g[h])[((size_t)tid << mr) + idx] = g0 + g1;
    }
  if (h == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0) es[tid >> 5] = e;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < 8; ++w) s += es[w];
      double *ep = reinterpret_cast<double *>(J.ws + J.lay->ep) + 2 * idx;
      ep[0] = s;
      ep[1] = 0.0;
    }
  }
}

// ------------------------------------------------------------ final sums --
// One warp sums the energy's parts (the FP64 adds of a sum over all warps, by all of them, took
// longer than the rest), all of them the parameters' path values: a few lanes for a parameter, in
// an order that depends on the number of terms alone, the parameters next to each other along
// the lanes as in memory.  8 CTAs for a job where there are few jobs (8 x 19 = 152 SMs), each a share of the
// parameters.  The FP32 contraction also sums psi^2: E and the gradients are divided by
// that norm, which takes the rounding of cos, sin and of the tensor cores' accumulation out
// of the results to first order (it is 1 up to that rounding).
constexpr int RED_NT = 256;
__global__ void __launch_bounds__(RED_NT) k_cut_reduce(const __grid_constant__ CutArgs A, int prec, int grad) {
  const CutView J = cut_view(A, blockIdx.x);
  const CutOut O = cut_out(A, blockIdx.x);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ double inv_s;
  if (w == 0) {
    const double *ep = reinterpret_cast<const double *>(J.ws + J.lay->ep);
    const double *ex = reinterpret_cast<const double *>(J.ws + J.lay->exy);  // the X/Y strings', part by part
    const int ni = J.lay->rb[0] * J.lay->ns[0];
    double e = 0.0, z = 0.0;
#pragma unroll 8
    for (int i = lane; i < ni; i += 32) {
      e += ep[2 * i];
      z += ep[2 * i + 1];
    }
    for (int i = lane; i < J.lay->nexy; i += 32) e += ex[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    const double inv = prec ? 1.0 : 1.0 / z;
    if (lane == 0 && blockIdx.y == 0) *O.E = e * inv;
    if (lane == 0) inv_s = inv;
  }
  if (!grad) return;
  __syncthreads();
  const double inv = inv_s;
  const int n = J.desc->n, reps = J.desc->reps, D = J.desc->D, m0 = J.desc->half[0].m, cx = J.desc->cx;
  const int row = 16 << cx, per = n << cx;  // complex: RY then RZ of a layer
  const double *gp = reinterpret_cast<const double *>(J.ws + J.lay->gp);
  const int W = D >= 256 ? 32 : D >= 64 ? 8 : D >= 4 ? 4 : D, G = 32 / W;
  for (int p0 = (w + RED_NT / 32 * blockIdx.y) * G; p0 < per * (reps + 1); p0 += RED_NT / 32 * gridDim.y * G) {
    const int p = p0 + lane % G;
    const bool on = p < per * (reps + 1);
    const int r = p / per, zr = p % per >= n, q = p % per - zr * n, h = q >= m0;
    const double *src = gp + (size_t)h * D * (reps + 1) * row + r * row + 16 * zr + (h ? q - m0 : q);
    double s = 0.0;
#pragma unroll 8
    for (int a = lane / G; a < D; a += W)
      if (on) s += src[(size_t)a * (reps + 1) * row];
    for (int o = G; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (on && lane < G) O.grad[p] = (O.mask && !O.mask[p]) ? 0.0 : s * inv;
  }
}

// One CTA: 128 x_lo by 128 x_hi, read along x_lo, rounded once, and written as two tiles
// of either order (16-byte stores, consecutive threads).  16 bytes per entry: HBM.
constexpr int TT_LD = 129;
__global__ void __launch_bounds__(512) k_tile_table(const TableJob t0, const TableJob *jobs) {
  extern __shared__ __align__(16) unsigned char cut_smem[];
  float *t = reinterpret_cast<float *>(cut_smem);  // [x_hi][x_lo]
  const TableJob T = jobs ? jobs[blockIdx.y] : t0;
  if (blockIdx.x >> (T.m0 + T.m1 - 14)) return;
  const int bl = blockIdx.x & ((1 << (T.m0 - 7)) - 1), bh = blockIdx.x >> (T.m0 - 7);
  const double *src = T.src + ((long long)bh << (T.m0 + 7)) + bl * 128;
  for (int i = threadIdx.x; i < 128 * 128; i += 512)
    t[(i >> 7) * TT_LD + (i & 127)] = (float)src[((long long)(i >> 7) << T.m0) + (i & 127)];
  __syncthreads();
  const int rb = 7 - T.cx, rm = (1 << rb) - 1;  // rows of a tile
  float4 *d0 = reinterpret_cast<float4 *>(T.d0);
  for (int i = threadIdx.x; i < 4096; i += 512) {  // ((row block * 2 + tile) * 16 + j / 4) * rows + row
    const int row = i & rm, j = 4 * ((i >> rb) & 15), tile = (i >> (rb + 4)) & 1, blk = i >> (rb + 5);
    const float *q = t + (64 * tile + j) * TT_LD + (blk << rb) + row;
    const long long at = ((((long long)(bl << T.cx) + blk) << (T.m1 - 6)) + 2 * bh + tile) * (16 << rb) + (i & ((16 << rb) - 1));
    d0[at] = make_float4(q[0], q[TT_LD], q[2 * TT_LD], q[3 * TT_LD]);
  }
  if (!T.d1) return;
  float4 *d1 = reinterpret_cast<float4 *>(T.d1);
  for (int i = threadIdx.x; i < 4096; i += 512) {
    const int row = i & rm, j = 4 * ((i >> rb) & 15), tile = (i >> (rb + 4)) & 1, blk = i >> (rb + 5);
    const float *q = t + ((blk << rb) + row) * TT_LD + 64 * tile + j;
    const long long at = ((((long long)(bh << T.cx) + blk) << (T.m0 - 6)) + 2 * bl + tile) * (16 << rb) + (i & ((16 << rb) - 1));
    d1[at] = make_float4(q[0], q[1], q[2], q[3]);
  }
}
constexpr int TT_SMEM = 128 * TT_LD * 4;

cudaError_t launch_tile_table(const TableJob &t, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_tile_table, cudaFuncAttributeMaxDynamicSharedMemorySize, TT_SMEM);
  if (e != cudaSuccess) return e;
  k_tile_table<<<1u << (t.m0 + t.m1 - 14), 512, TT_SMEM, s>>>(t, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_tile_tables(const TableJob *jobs, int njobs, int nmax, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_tile_table, cudaFuncAttributeMaxDynamicSharedMemorySize, TT_SMEM);
  if (e != cudaSuccess) return e;
  for (int j = 0; j < njobs; j += 32768)  // the grid's second dimension ends at 65535
    k_tile_table<<<dim3(1u << (nmax - 14), (unsigned)(njobs - j < 32768 ? njobs - j : 32768)), 512, TT_SMEM, s>>>(
        TableJob{}, jobs + j);
  return cudaGetLastError();
}

// Problems whose larger halves have the same class share the kernels of their half
// circuits: one class for every small size, one per size above.
int cut_class(int prec, int m) { return m <= HALF_SMALL_M(prec) ? HALF_SMALL_M(prec) : m; }

static cudaError_t launch_pack(CutArgs A, const CutGrid &g, int K, cudaStream_t s) {
  A.items = g.pack_items;
  A.blk0 = 1 << (g.m0 - 6);
  A.nblk = A.blk0 + (1 << (g.m1 - 6));
  auto k = g.cx ? k_cut_pack<true> : k_cut_pack<false>;
  k<<<g.pack_items ? g.pack_blocks : A.njobs * A.nblk, 256, K * 65 * (g.cx ? 4 : 8), s>>>(A, K);
  return cudaGetLastError();
}

cudaError_t launch_cut_halves(const CutArgs &A0, const CutGrid &g, cudaStream_t s, int *launches) {
  CutArgs A = A0;
  A.blk0 = g.D;
  const cudaError_t e = launch_cut_fwd32(A, g, false, s, launches);
  *launches += 1;
  return e == cudaSuccess ? launch_pack(A, g, cut_k(g.D), s) : e;
}

cudaError_t launch_cut_state(const CutArgs &A0, const CutGrid &g, cudaStream_t s, int *launches) {
  CutArgs A = A0;
  A.blk0 = A.job0.lay.rb[0] * A.job0.lay.ns[0];
  A.nblk = A.njobs * A.blk0;
  *launches += 1;
  return launch_cut_tc(A, cut_k(g.D), CUT_STATE, s);
}

cudaError_t launch_cut(int prec, const CutArgs &A0, const CutGrid &g, bool grad, cudaStream_t s, int *launches,
                       const CutXyDims *xy, CutMark *mark) {
  CutArgs A = A0;
  const CutLayout &l = A.job0.lay;
  const int half_blocks = g.half_items ? g.half_blocks : A.njobs * 2 * g.D;
  const int K = cut_k(g.D << g.cx);
  cudaError_t e;
#define CUT_CHECK(x) \
  if ((e = (x)) != cudaSuccess) return e
  A.blk0 = g.D;
  A.items = g.half_items;
  if (prec) {
    CUT_CHECK(launch_half<double>(A, cut_class(1, g.m0), grad ? 1 : 0, half_blocks, s));
  } else {
    CUT_CHECK(g.cx ? launch_halfc(A, g.m0, grad ? 1 : 0, half_blocks, s) : launch_cut_fwd32(A, g, grad, s, launches));
    CUT_CHECK(launch_pack(A, g, K, s));
    *launches += 1;
  }
  A.blk0 = l.rb[0] * l.ns[0];
  A.nblk = g.con_items ? g.con_blocks : A.njobs * (A.blk0 + (grad ? l.rb[1] * l.ns[1] : 0));
  A.items = g.con_items;
  if (mark) mark->mark(true);
  if (prec && cut_by_rows(g.m0, g.D)) {
    auto k = grad ? k_cut_rows64<true> : k_cut_rows64<false>;
    k<<<A.nblk, 256, 0, s>>>(A);
    CUT_CHECK(cudaGetLastError());
  } else if (prec) {
    const size_t sm = (size_t)8 * C64LD * (2 * g.D + (grad ? C64 : 0));  // (64 terms at most: 42 KB)
    auto k = grad ? k_cut_contract64<true> : k_cut_contract64<false>;
    k<<<A.nblk, 256, sm, s>>>(A);
    CUT_CHECK(cudaGetLastError());
  } else {
    CUT_CHECK(launch_cut_tc(A, K, grad ? CUT_GRAD : CUT_ENERGY, s));
  }
  if (mark) mark->mark(false);
  *launches += 3;
  if (xy) CUT_CHECK(launch_cut_xy(A, g, *xy, grad, s, launches));
  if (grad) {
    A.blk0 = g.D;
    A.items = g.half_items;
    CUT_CHECK(prec ? launch_half<double>(A, cut_class(1, g.m0), 2, half_blocks, s)
              : g.cx ? launch_halfc(A, g.m0, 2, half_blocks, s)
                   : launch_half<float>(A, cut_class(0, g.m0), 2, half_blocks, s));
    *launches += 1;
  }
  k_cut_reduce<<<dim3((unsigned)A.njobs, grad && A.njobs <= 19 ? 8 : 1), grad ? RED_NT : 32, 0, s>>>(A, prec, grad ? 1 : 0);
#undef CUT_CHECK
  return cudaGetLastError();
}

}  // namespace gvqe
