// gvqe_readout.cu -- readout of a prepared state (Section IV-F, Section V-A):
// probabilities p(x) = |psi(x)|^2, the most probable bitstring, inverse-CDF
// shot sampling, and the CVaR-alpha of the outcome energy E(x) (Section III).
//
// Everything is summed in FP64 in fixed orders.  The CVaR search narrows the
// alpha-quantile of E with histograms whose bin masses are integer (p scaled
// by 2^60), so they do not depend on the order of the atomic adds.
#include <cstring>

#include "gvqe_engine.cuh"

namespace gvqe {
namespace {

constexpr int RO_NT = 256;

template <typename T>
__device__ __forceinline__ double prob(const T *psi, long long x) {
  const double v = (double)__ldcg(psi + x);
  return v * v;  // exact for an FP32 amplitude
}

// Order-preserving map of a double (given by its bits) onto an unsigned 64-bit
// key: comparisons of table energies run as integer compares (FP64 arithmetic
// is slow on this GPU).
__device__ __forceinline__ unsigned long long key_of_bits(unsigned long long b) {
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
// Keys (and bits) of the table entries 2i and 2i+1 (one 16-byte load).
__device__ __forceinline__ void key_pair(const double *E, long long i, unsigned long long &k0, unsigned long long &k1,
                                         unsigned long long &b0, unsigned long long &b1) {
  const longlong2 b = __ldcg(reinterpret_cast<const longlong2 *>(E) + i);
  b0 = (unsigned long long)b.x;
  b1 = (unsigned long long)b.y;
  k0 = key_of_bits(b0);
  k1 = key_of_bits(b1);
}
template <typename T>
__device__ __forceinline__ void amp_pair(const T *psi, long long i, T &v0, T &v1);
template <>
__device__ __forceinline__ void amp_pair<float>(const float *psi, long long i, float &v0, float &v1) {
  const float2 v = __ldcg(reinterpret_cast<const float2 *>(psi) + i);
  v0 = v.x;
  v1 = v.y;
}
template <>
__device__ __forceinline__ void amp_pair<double>(const double *psi, long long i, double &v0, double &v1) {
  const double2 v = __ldcg(reinterpret_cast<const double2 *>(psi) + i);
  v0 = v.x;
  v1 = v.y;
}

// Histogram mass of one amplitude, floor(p * 2^60): FP32 amplitudes square in
// FP32 and convert through the exponent and mantissa bits (integer work only);
// FP64 amplitudes square and convert in FP64.
__device__ __forceinline__ unsigned long long qmass(float v) {
  const float p = v * v;
  const unsigned b = __float_as_uint(p);
  const int ex = (int)((b >> 23) & 0xFF);
  const unsigned long long m = (b & 0x7FFFFFu) | (ex ? 0x800000u : 0u);
  const int sh = (ex ? ex : 1) - 90;  // p = m 2^(ex - 150); q = m 2^(ex - 90)
  return sh >= 0 ? (m << sh) : (sh > -64 ? (m >> -sh) : 0ull);
}
__device__ __forceinline__ unsigned long long qmass(double v) { return __double2ull_rz(v * v * 0x1p60); }

// Per chunk of 2^cb amplitudes: the sum of p (fixed tree order) and the first
// index of the chunk's largest p.
// A thread sums its (at most 32) p in the amplitude precision and compares
// |psi| (monotone in p, exact); the chunk sums above the thread are FP64.
template <typename T>
__global__ void __launch_bounds__(RO_NT) k_ro_chunks(const T *psi, int cb, double *csum, double *cmax,
                                                     long long *cidx) {
  __shared__ double ss[RO_NT], sm[RO_NT];
  __shared__ long long si[RO_NT];
  const long long c = blockIdx.x;
  const int tid = threadIdx.x;
  const long long base = c << cb;
  const int len = 1 << cb;
  T s = T(0), m = T(-1);
  long long mi = base;
#pragma unroll 16
  for (int i = tid; i < len; i += RO_NT) {
    const T v = __ldcg(psi + base + i);
    const T av = v < T(0) ? -v : v;
    s += v * v;
    if (av > m) {
      m = av;
      mi = base + i;
    }
  }
  ss[tid] = (double)s;
  sm[tid] = m < T(0) ? -1.0 : (double)m * (double)m;
  si[tid] = mi;
  __syncthreads();
  for (int w = RO_NT / 2; w > 0; w >>= 1) {
    if (tid < w) {
      ss[tid] += ss[tid + w];
      const double m2 = sm[tid + w];
      const long long i2 = si[tid + w];
      if (m2 > sm[tid] || (m2 == sm[tid] && i2 < si[tid])) {
        sm[tid] = m2;
        si[tid] = i2;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    csum[c] = ss[0];
    cmax[c] = sm[0];
    cidx[c] = si[0];
  }
}

// cdf[0] = 0, cdf[c + 1] = sum of chunks 0..c (block scans in a fixed order, then their totals one
// after the other), the overall maximum (smallest index on ties) and the total.
// A CTA scans 1024 chunks: 10 FP64 adds each, on an SM's few FP64 lanes 5 us, so that the blocks
// run side by side and a second kernel adds what lies before them (8192 chunks: 45 us in one CTA,
// 9 so).  A block's total, maximum and index stay in its first places of csum, cmax and cidx.
__device__ __forceinline__ void ro_larger(double &m, long long &i, double m2, long long i2) {
  if (m2 > m || (m2 == m && i2 < i)) {
    m = m2;
    i = i2;
  }
}
__global__ void __launch_bounds__(1024) k_ro_scan(double *csum, double *cmax, long long *cidx, long long nch,
                                                  double *cdf, double *stats, long long *argmax) {
  __shared__ double buf[1024];
  __shared__ double bm[1024];
  __shared__ long long bi[1024];
  const int tid = threadIdx.x;
  const long long b0 = (long long)blockIdx.x << 10, i = b0 + tid;
  double v = 0.0, m = -1.0;
  long long mi = 0;
  if (i < nch) {
    v = csum[i];
    ro_larger(m, mi, cmax[i], cidx[i]);
  }
  buf[tid] = v;
  bm[tid] = m;
  bi[tid] = mi;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const double add = tid >= off ? buf[tid - off] : 0.0;
    __syncthreads();
    if (tid >= off) buf[tid] += add;
    __syncthreads();
  }
  for (int w = 512; w > 0; w >>= 1) {
    if (tid < w) ro_larger(bm[tid], bi[tid], bm[tid + w], bi[tid + w]);
    __syncthreads();
  }
  if (i < nch) cdf[i + 1] = buf[tid];
  if (tid != 0) return;
  if (blockIdx.x == 0) cdf[0] = 0.0;
  if (gridDim.x == 1) {
    stats[0] = bm[0];
    stats[2] = buf[1023];
    argmax[0] = bi[0];
  } else {
    csum[b0] = buf[1023];
    cmax[b0] = bm[0];
    cidx[b0] = bi[0];
  }
}
__global__ void __launch_bounds__(1024) k_ro_carry(const double *csum, const double *cmax, const long long *cidx,
                                                   long long nch, double *cdf, double *stats, long long *argmax) {
  __shared__ double before;
  const long long i = ((long long)blockIdx.x << 10) + threadIdx.x;
  if (threadIdx.x == 0) {
    double carry = 0.0;
    for (unsigned b = 0; b < blockIdx.x; ++b) carry += csum[(long long)b << 10];
    before = carry;
    if (blockIdx.x == gridDim.x - 1) {
      double m = -1.0;
      long long mi = 0;
      for (unsigned b = 0; b < gridDim.x; ++b) ro_larger(m, mi, cmax[(long long)b << 10], cidx[(long long)b << 10]);
      stats[0] = m;
      stats[2] = carry + csum[(long long)blockIdx.x << 10];
      argmax[0] = mi;
    }
  }
  __syncthreads();
  if (blockIdx.x > 0 && i < nch) cdf[i + 1] = before + cdf[i + 1];
}

// p * 2^60 of one amplitude, cut to an integer: for FP32 from the exact square of the mantissa
// (integer work only), for FP64 from the rounded square.  Below 2^64 for |v| < 2.
__device__ __forceinline__ unsigned long long qsquare(float v) {
  const unsigned b = __float_as_uint(v);
  const int ex = (int)((b >> 23) & 0xFF), e = ex ? ex : 1;
  const unsigned m = (b & 0x7FFFFFu) | (ex ? 0x800000u : 0u);
  const unsigned long long m2 = (unsigned long long)m * m;  // p = m2 2^(2 e - 300)
  const int sh = 2 * e - 240;
  return sh >= 0 ? (m2 << sh) : (sh > -64 ? (m2 >> -sh) : 0ull);
}
__device__ __forceinline__ unsigned long long qsquare(double v) { return __double2ull_rz(v * v * 0x1p60); }
// four consecutive amplitudes
__device__ __forceinline__ unsigned long long qsquare4(const float *p) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  return qsquare(v.x) + qsquare(v.y) + qsquare(v.z) + qsquare(v.w);
}
__device__ __forceinline__ unsigned long long qsquare4(const double *p) {
  const double2 v = reinterpret_cast<const double2 *>(p)[0], w = reinterpret_cast<const double2 *>(p)[1];
  return qsquare(v.x) + qsquare(v.y) + qsquare(w.x) + qsquare(w.y);
}
// inclusive scan over the warp
__device__ __forceinline__ unsigned long long scan_u64(unsigned long long x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += v;
  }
  return x;
}

// The sample as it is defined: a warp scan through the chunk, 32 amplitudes at a time in FP64, for the first x whose
// cumulative probability exceeds t.  Where rounding leaves t past the chunk's
// own running sum, the chunk's last x with p > 0 is taken.
template <typename T>
__device__ __noinline__ long long ro_scan_chunk(const T *psi, long long base, int len, double run, double t, int lane) {
  long long found = -1, lastnz = -1;
  for (int i0 = 0; i0 < len; i0 += 32) {
    const int i = i0 + lane;
    const double p = i < len ? prob(psi, base + i) : 0.0;
    double incl = p;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, p > 0.0 && run + incl > t);
    const unsigned nz = __ballot_sync(0xffffffffu, p > 0.0);
    if (nz) lastnz = base + i0 + 31 - __clz(nz);
    if (hit) {
      found = base + i0 + __ffs(hit) - 1;
      break;
    }
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  return found >= 0 ? found : lastnz >= 0 ? lastnz : base;
}

// The same in integers, or -1 where they cannot tell.  F, the sum of the cut p * 2^60, is within
// 2^13 of the sum; the FP64 scan's rounding (at most 262 adds of values below 2), that of t - run
// and the cuts come to less than 2^17.  So the first x with F > t - run - 2^18 is the scan's if
// F > t - run + 2^18 there: the scan takes no x before it, and takes it.
constexpr int RO_SEG = 2048;
template <typename T>
__device__ __forceinline__ long long ro_find_chunk(const T *psi, long long base, int len, double run, double t, int lane) {
  const long long d = __double2ll_rz((t - run) * 0x1p60), lo = d - (1 << 18), hi = d + (1 << 18);
  const T *p = psi + base;
  unsigned long long f = 0;
  int seg = 0;
  for (; seg < len; seg += RO_SEG) {
    unsigned long long s = 0;
#pragma unroll
    for (int k = 0; k < RO_SEG / 128; ++k) s += qsquare4(p + seg + 128 * k + 4 * lane);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((long long)(f + s) > lo) break;
    f += s;
  }
  if (seg >= len) return -1;
  // 64 amplitudes a lane, then 2
  unsigned long long s = 0;
#pragma unroll
  for (int k = 0; k < RO_SEG / 128; ++k) s += qsquare4(p + seg + (RO_SEG / 32) * lane + 4 * k);
  unsigned long long incl = scan_u64(s, lane);
  int l = __ffs(__ballot_sync(0xffffffffu, (long long)(f + incl) > lo)) - 1;
  f += __shfl_sync(0xffffffffu, incl - s, l);
  const T *r = p + seg + (RO_SEG / 32) * l;
  const unsigned long long q0 = qsquare(r[2 * lane]), q1 = qsquare(r[2 * lane + 1]);
  incl = scan_u64(q0 + q1, lane);
  l = __ffs(__ballot_sync(0xffffffffu, (long long)(f + incl) > lo)) - 1;
  const long long f1 = (long long)(f + incl), f0 = f1 - (long long)q1;
  const bool first = f0 > lo;
  const long long x = (first ? f0 : f1) > hi ? (r - psi) + 2 * lane + !first : -1;
  return __shfl_sync(0xffffffffu, x, l);
}

// One warp per shot: t = u * total; the chunk whose cumulative range holds t
// (binary search), then the first x of that chunk whose cumulative probability exceeds t.  Summed
// in integers, off the few FP64 lanes, with the FP64 scan only where t is within 2e-13 of a
// step; 26 qubits, 8192 shots: 1010 us with FP64 scans, 87 so.
template <typename T>
__global__ void __launch_bounds__(RO_NT) k_ro_sample(const T *psi, int cb, long long nch, const double *cdf,
                                                     const double *u, int nshots, long long *shots) {
  const int lane = threadIdx.x & 31;
  const long long k = (blockIdx.x * (long long)RO_NT + threadIdx.x) >> 5;
  if (k >= nshots) return;  // the whole warp
  const double total = cdf[nch];
  double t = u[k] * total;
  if (!(t < total)) t = nextafter(total, 0.0);
  long long lo = 0, hi = nch - 1;  // first chunk c with cdf[c + 1] > t
  while (lo < hi) {
    const long long mid = (lo + hi) >> 1;
    if (cdf[mid + 1] > t)
      hi = mid;
    else
      lo = mid + 1;
  }
  const long long base = lo << cb;
  const int len = 1 << cb;
  const double run = cdf[lo];
  long long x = -1;
  if (len >= RO_SEG && total < 2.0 && run <= t) x = ro_find_chunk(psi, base, len, run, t, lane);
  if (x < 0) x = ro_scan_chunk(psi, base, len, run, t, lane);
  if (lane == 0) shots[k] = x;
}

// Keys of the smallest and largest E over all x: ext[1] (min), ext[2] (max).
__global__ void __launch_bounds__(RO_NT) k_ro_minmax(const double *E, long long N, unsigned long long *ext) {
  __shared__ unsigned long long smin, smax;
  if (threadIdx.x == 0) {
    smin = ~0ull;
    smax = 0ull;
  }
  __syncthreads();
  unsigned long long kmin = ~0ull, kmax = 0ull;
  const long long N2 = N >> 1, st = (long long)gridDim.x * RO_NT;
  for (long long i = blockIdx.x * (long long)RO_NT + threadIdx.x; i < N2; i += 2 * st) {
    unsigned long long k[4], raw[4];
    key_pair(E, i, k[0], k[1], raw[0], raw[1]);
    if (i + st < N2)
      key_pair(E, i + st, k[2], k[3], raw[2], raw[3]);
    else
      k[2] = k[3] = k[0];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      kmin = k[j] < kmin ? k[j] : kmin;
      kmax = k[j] > kmax ? k[j] : kmax;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    kmin = min(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
    kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&smin, kmin);
    atomicMax(&smax, kmax);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicMin(&ext[1], smin);
    atomicMax(&ext[2], smax);
  }
}

// One pass of the quantile search over the keys [edges[0], edges[RO_BINS]):
// the integer mass (p * 2^60) of every bin [edges[b], edges[b+1]) and the keys
// of the smallest and largest E inside the range (ext[1], ext[2]).  The edges
// are the keys of evenly spaced energies.  With `below` set, the masses under
// and above the range are summed too (ext[0], ext[3]); otherwise only x inside
// the range read their amplitude (the mass below is known from earlier passes).
//
// Bound by HBM: 26 qubits 178 us with `below` (0.8 GB; 515 with two loads in flight, a branch
// for every warp that met the range and atomics from every thread), 88 without (0.5 GB).
//
// A key's bin: the range is cut into RO_LUT equal key intervals, lut[j] holds
// the bin of interval j's first key, so a key of interval j lies in a bin of
// [lut[j], lut[j+1]], found by a binary search over that (usually one- or
// two-bin) span instead of over all RO_BINS edges.
constexpr int RO_LUT_BITS = 11;
constexpr int RO_LUT = 1 << RO_LUT_BITS;
__device__ __forceinline__ int ro_bin_search(const unsigned long long *se, unsigned long long k, int b0, int b1) {
  while (b0 < b1) {  // largest b in [b0, b1] with se[b] <= k (se[b0] <= k holds)
    const int mid = (b0 + b1 + 1) >> 1;
    if (se[mid] <= k)
      b0 = mid;
    else
      b1 = mid - 1;
  }
  return b0;
}
template <typename T>
__global__ void __launch_bounds__(RO_NT) k_ro_hist(const T *psi, const double *E, long long N,
                                                   const unsigned long long *edges, unsigned long long *gmass,
                                                   unsigned long long *ext, int below) {
  __shared__ unsigned long long se[RO_BINS + 1];
  __shared__ unsigned long long sm[RO_BINS];
  __shared__ unsigned short lut[RO_LUT + 1];
  __shared__ unsigned long long queue[2][RO_NT / 32][64];
  __shared__ unsigned long long smin, smax, sbelow, sabove;
  for (int i = threadIdx.x; i <= RO_BINS; i += RO_NT) {
    se[i] = edges[i];
    if (i < RO_BINS) sm[i] = 0ull;
  }
  if (threadIdx.x == 0) {
    smin = ~0ull;
    smax = sbelow = sabove = 0ull;
  }
  __syncthreads();
  const unsigned long long lo = se[0], hi = se[RO_BINS];
  const unsigned long long span = hi - lo;
  const int lsh = (span == 0ull) ? 0 : max(0, 64 - __clzll((long long)span) - RO_LUT_BITS);
  for (int j = threadIdx.x; j <= RO_LUT; j += RO_NT) {
    const unsigned long long kj = lo + ((unsigned long long)j << lsh);
    lut[j] = (unsigned short)((j == RO_LUT || kj >= hi || kj < lo) ? RO_BINS - 1 : ro_bin_search(se, kj, 0, RO_BINS - 1));
  }
  __syncthreads();
  const unsigned long long lo_read = below ? 0ull : lo;   // keys in [lo_read, hi_read) read psi
  const unsigned long long hi_read = below ? ~0ull : hi;
  unsigned long long kmin = ~0ull, kmax = 0ull, qbelow = 0ull, qabove = 0ull;
  auto drop = [&](unsigned long long k, unsigned long long q) {
    const int j = (int)((k - lo) >> lsh);  // < RO_LUT
    const int b = ro_bin_search(se, k, lut[j], lut[j + 1]);  // largest b with edges[b] <= k
    if (q) atomicAdd(&sm[b], q);
    kmin = k < kmin ? k : kmin;
    kmax = k > kmax ? k : kmax;
  };
  auto add = [&](unsigned long long k, T v) {
    if (k < lo) {
      qbelow += qmass(v);
      return;
    }
    if (k >= hi) {
      qabove += qmass(v);
      return;
    }
    drop(k, qmass(v));
  };
  const long long N2 = N >> 1, st = (long long)gridDim.x * RO_NT;
  long long i = blockIdx.x * (long long)RO_NT + threadIdx.x;
  if (below) {
    // Every amplitude is read: all loads at once.  The few keys inside the range (a few per warp, so
    // that most warps would take that branch for them) queue up in shared memory until there are 32.
    // (i and N2 - 3 st are multiples of 32 across a warp: the loop is the same for all of it.)
    const int lane = threadIdx.x & 31;
    unsigned long long *qk = queue[0][threadIdx.x >> 5], *qq = queue[1][threadIdx.x >> 5];
    int cnt = 0;
    for (; i + 3 * st < N2; i += 4 * st) {
      unsigned long long k[8], r0, r1;
      T v[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        key_pair(E, i + j * st, k[2 * j], k[2 * j + 1], r0, r1);
        amp_pair(psi, i + j * st, v[2 * j], v[2 * j + 1]);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const unsigned long long q = qmass(v[j]);
        const bool in = k[j] >= lo && k[j] < hi;
        if (k[j] < lo)
          qbelow += q;
        else if (!in)
          qabove += q;
        const unsigned mask = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int at = cnt + __popc(mask & ((1u << lane) - 1));
          qk[at] = k[j];
          qq[at] = q;
        }
        cnt += __popc(mask);
        if (cnt >= 32) {
          __syncwarp();
          drop(qk[lane], qq[lane]);
          cnt -= 32;
          const unsigned long long a = qk[32 + lane], b = qq[32 + lane];
          __syncwarp();
          if (lane < cnt) {
            qk[lane] = a;
            qq[lane] = b;
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (lane < cnt) drop(qk[lane], qq[lane]);
  } else {
    for (; i + 7 * st < N2; i += 8 * st) {
      unsigned long long k[16], r0, r1;
#pragma unroll
      for (int j = 0; j < 8; ++j) key_pair(E, i + j * st, k[2 * j], k[2 * j + 1], r0, r1);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const bool in0 = k[2 * j] >= lo && k[2 * j] < hi, in1 = k[2 * j + 1] >= lo && k[2 * j + 1] < hi;
        if (in0 || in1) {
          T v0, v1;
          amp_pair(psi, i + j * st, v0, v1);
          if (in0) add(k[2 * j], v0);
          if (in1) add(k[2 * j + 1], v1);
        }
      }
    }
  }
  for (; i < N2; i += 2 * st) {
    unsigned long long k[4], raw[4];
    key_pair(E, i, k[0], k[1], raw[0], raw[1]);
    const bool two = i + st < N2;
    if (two) key_pair(E, i + st, k[2], k[3], raw[2], raw[3]);
    const bool in0 = k[0] >= lo_read && k[0] < hi_read, in1 = k[1] >= lo_read && k[1] < hi_read;
    const bool in2 = two && k[2] >= lo_read && k[2] < hi_read, in3 = two && k[3] >= lo_read && k[3] < hi_read;
    if (in0 || in1) {
      T v0, v1;
      amp_pair(psi, i, v0, v1);
      if (in0) add(k[0], v0);
      if (in1) add(k[1], v1);
    }
    if (in2 || in3) {
      T v2, v3;
      amp_pair(psi, i + st, v2, v3);
      if (in2) add(k[2], v2);
      if (in3) add(k[3], v3);
    }
  }
  // one atomic per warp and CTA: with two from every thread, all on the same two words of L2, they took
  // 150 of this pass's 330 us (26 qubits)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    kmin = min(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
    kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    qbelow += __shfl_xor_sync(0xffffffffu, qbelow, o);
    qabove += __shfl_xor_sync(0xffffffffu, qabove, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&smin, kmin);
    atomicMax(&smax, kmax);
    if (qbelow) atomicAdd(&sbelow, qbelow);  // integer: order-independent
    if (qabove) atomicAdd(&sabove, qabove);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < RO_BINS; i += RO_NT)
    if (sm[i]) atomicAdd(&gmass[i], sm[i]);
  if (threadIdx.x == 0) {
    atomicMin(&ext[1], smin);
    atomicMax(&ext[2], smax);
    if (sbelow) atomicAdd(&ext[0], sbelow);
    if (sabove) atomicAdd(&ext[3], sabove);
  }
}

// Energies at the shots, out[k] = E[shots[k]].
__global__ void k_ro_gather(const double *E, const long long *shots, int nshots, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nshots) out[k] = E[shots[k]];
}

// The energies of rank r0 (CTA 0) and r1 (CTA 1) among the shots', out[0..1]: their keys' bytes from the top,
// counted in shared memory among the shots that share the bytes before.  Equal bytes of a warp
// are counted once (the top bytes are nearly all the same).  8192 shots: 21 us; copying and
// sorting them on the host took 290.
constexpr int RANK_NT = 1024;
__global__ void __launch_bounds__(RANK_NT) k_ro_rank(const double *es, int n, int r0, int r1, double *out) {
  __shared__ int count[256], digit_s, rank_s;
  const int tid = threadIdx.x, lane = tid & 31;
  int rank = blockIdx.x ? r1 : r0;
  unsigned long long prefix = 0ull;
  for (int sh = 56; sh >= 0; sh -= 8) {
    if (tid < 256) count[tid] = 0;
    __syncthreads();
    const unsigned long long above = sh == 56 ? 0ull : ~0ull << (sh + 8);
    for (int i0 = 0; i0 < n; i0 += RANK_NT) {
      const int i = i0 + tid;
      int d = -1;
      if (i < n) {
        const unsigned long long k = key_of_bits((unsigned long long)__double_as_longlong(es[i]));
        if ((k & above) == prefix) d = (int)(k >> sh) & 255;
      }
      const unsigned same = __match_any_sync(0xffffffffu, d);
      if (d >= 0 && lane == __ffs(same) - 1) atomicAdd(&count[d], __popc(same));
    }
    __syncthreads();
    if (tid < 32) {  // 8 digits a lane: the first whose running count passes the rank
      int c[8], s = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) s += c[j] = count[8 * lane + j];
      int incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int l = __ffs(__ballot_sync(0xffffffffu, incl > rank)) - 1;
      if (lane == l) {
        int left = rank - (incl - s), d = 0;
        while (d < 7 && left >= c[d]) left -= c[d++];
        digit_s = 8 * lane + d;
        rank_s = left;
      }
    }
    __syncthreads();
    rank = rank_s;
    prefix |= (unsigned long long)digit_s << sh;
  }
  if (tid == 0) out[blockIdx.x] = __longlong_as_double((long long)((prefix >> 63) ? prefix & 0x7fffffffffffffffull : ~prefix));
}

// Tail sums for the CVaR: per CTA sum of p*E and p over E < tau, and of p over
// E == tau (fixed per-thread order, fixed tree).
// Compensated (Kahan) running sum in the amplitude precision: FP32 amplitudes
// keep the tail sums off the (slow) FP64 pipe; FP64 amplitudes sum in FP64.
template <typename T>
struct KSum {
  T s = T(0), c = T(0);
  __device__ __forceinline__ void add(T x) {
    const T y = x - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
  }
};

// Bound by HBM: 26 qubits 163 us (0.8 GB), 208 with two loads in flight instead of eight.
template <typename T>
__global__ void __launch_bounds__(RO_NT) k_ro_tail(const T *psi, const double *E, long long N,
                                                   unsigned long long ktau, double *part) {
  __shared__ double r[3][RO_NT];
  KSum<T> ksb, kpb, kpa;
  auto add = [&](unsigned long long k, T v, unsigned long long bits) {
    const T p = v * v;
    if (k < ktau) {
      ksb.add(p * (T)__longlong_as_double((long long)bits));
      kpb.add(p);
    } else {
      kpa.add(p);
    }
  };
  const long long N2 = N >> 1, st = (long long)gridDim.x * RO_NT;
  long long i = blockIdx.x * (long long)RO_NT + threadIdx.x;
  for (; i + 7 * st < N2; i += 8 * st) {  // eight loads at once, the sums in the same order
    unsigned long long k[16], raw[16];
    T v[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) key_pair(E, i + j * st, k[2 * j], k[2 * j + 1], raw[2 * j], raw[2 * j + 1]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[2 * j] = v[2 * j + 1] = T(0);
      if (k[2 * j] <= ktau || k[2 * j + 1] <= ktau) amp_pair(psi, i + j * st, v[2 * j], v[2 * j + 1]);
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (k[j] <= ktau) add(k[j], v[j], raw[j]);
  }
  for (; i < N2; i += 2 * st) {
    unsigned long long k[4], raw[4];
    key_pair(E, i, k[0], k[1], raw[0], raw[1]);
    const bool two = i + st < N2;
    if (two) key_pair(E, i + st, k[2], k[3], raw[2], raw[3]);
    if (k[0] <= ktau || k[1] <= ktau) {
      T v0, v1;
      amp_pair(psi, i, v0, v1);
      if (k[0] <= ktau) add(k[0], v0, raw[0]);
      if (k[1] <= ktau) add(k[1], v1, raw[1]);
    }
    if (two && (k[2] <= ktau || k[3] <= ktau)) {
      T v2, v3;
      amp_pair(psi, i + st, v2, v3);
      if (k[2] <= ktau) add(k[2], v2, raw[2]);
      if (k[3] <= ktau) add(k[3], v3, raw[3]);
    }
  }
  const int tid = threadIdx.x;
  r[0][tid] = (double)ksb.s - (double)ksb.c;
  r[1][tid] = (double)kpb.s - (double)kpb.c;
  r[2][tid] = (double)kpa.s - (double)kpa.c;
  __syncthreads();
  for (int w = RO_NT / 2; w > 0; w >>= 1) {
    if (tid < w)
      for (int j = 0; j < 3; ++j) r[j][tid] += r[j][tid + w];
    __syncthreads();
  }
  if (tid < 3) part[3 * (long long)blockIdx.x + tid] = r[tid][0];
}

// CVaR_alpha = (S + clamp(alpha T - P, 0, Pa) tau) / (alpha T), T = stats[2]:
// the lowest-energy alpha fraction of the outcomes, the outcomes at E == tau
// counted for the remainder.
// Three threads add the parts, one sum each, from shared memory: 29 us for 608 parts, the latency of the
// FP64 adds in their order (88 with one thread reading them from L2).
__global__ void __launch_bounds__(256) k_ro_cvar(const double *part, int nparts, double alpha, double tau, double *stats) {
  extern __shared__ double sp[];
  __shared__ double sums[3];
  for (int i = threadIdx.x; i < 3 * nparts; i += blockDim.x) sp[i] = part[i];
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
#pragma unroll 8
    for (int i = 0; i < nparts; ++i) s += sp[3 * i + threadIdx.x];
    sums[threadIdx.x] = s;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double S = sums[0], P = sums[1], Pa = sums[2];
  const double aT = alpha * stats[2];
  double rest = aT - P;
  rest = rest < 0.0 ? 0.0 : (rest > Pa ? Pa : rest);
  stats[1] = (S + rest * tau) / aT;
}

inline int ro_grid() { return num_sms_cached() * 4; }

}  // namespace

int readout_chunk_bits(int n) { return n < 13 ? n : 13; }
int readout_tail_parts() { return ro_grid(); }

// Complex path: out[x] = |psi(x)| from interleaved (re, im) amplitudes.
template <typename T>
__global__ void k_ro_modulus(const T *__restrict__ psi, long long N, T *__restrict__ out) {
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < N; x += (long long)gridDim.x * blockDim.x) {
    const T re = __ldcg(psi + 2 * x), im = __ldcg(psi + 2 * x + 1);
    out[x] = sqrt(re * re + im * im);
  }
}

cudaError_t launch_ro_modulus(int prec, const void *psi, int n, void *out, cudaStream_t s) {
  const long long N = 1LL << n;
  const long long blocks = (N + RO_NT - 1) / RO_NT;
  const unsigned g = (unsigned)(blocks < 65536 ? blocks : 65536);
  if (prec)
    k_ro_modulus<double><<<g, RO_NT, 0, s>>>((const double *)psi, N, (double *)out);
  else
    k_ro_modulus<float><<<g, RO_NT, 0, s>>>((const float *)psi, N, (float *)out);
  return cudaGetLastError();
}

cudaError_t launch_ro_prob(int prec, const void *psi, int n, double *csum, double *cmax, long long *cidx,
                           double *cdf, double *stats, long long *argmax, cudaStream_t s) {
  const int cb = readout_chunk_bits(n);
  const long long nch = 1LL << (n - cb);
  if (prec)
    k_ro_chunks<double><<<(unsigned)nch, RO_NT, 0, s>>>((const double *)psi, cb, csum, cmax, cidx);
  else
    k_ro_chunks<float><<<(unsigned)nch, RO_NT, 0, s>>>((const float *)psi, cb, csum, cmax, cidx);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned nb = (unsigned)((nch + 1023) / 1024);
  k_ro_scan<<<nb, 1024, 0, s>>>(csum, cmax, cidx, nch, cdf, stats, argmax);
  if (nb > 1) k_ro_carry<<<nb, 1024, 0, s>>>(csum, cmax, cidx, nch, cdf, stats, argmax);
  return cudaGetLastError();
}

cudaError_t launch_ro_sample(int prec, const void *psi, int n, const double *cdf, const double *u, int nshots,
                             long long *shots, cudaStream_t s) {
  if (nshots <= 0) return cudaSuccess;
  const int cb = readout_chunk_bits(n);
  const long long nch = 1LL << (n - cb);
  const unsigned grid = (unsigned)(((long long)nshots * 32 + RO_NT - 1) / RO_NT);
  if (prec)
    k_ro_sample<double><<<grid, RO_NT, 0, s>>>((const double *)psi, cb, nch, cdf, u, nshots, shots);
  else
    k_ro_sample<float><<<grid, RO_NT, 0, s>>>((const float *)psi, cb, nch, cdf, u, nshots, shots);
  return cudaGetLastError();
}

cudaError_t launch_ro_minmax(const double *E, int n, unsigned long long *ext, cudaStream_t s) {
  k_ro_minmax<<<ro_grid(), RO_NT, 0, s>>>(E, 1LL << n, ext);
  return cudaGetLastError();
}

cudaError_t launch_ro_hist(int prec, const void *psi, const double *E, int n, const unsigned long long *edges,
                           unsigned long long *gmass, unsigned long long *ext, int below, cudaStream_t s) {
  if (prec)
    k_ro_hist<double><<<ro_grid(), RO_NT, 0, s>>>((const double *)psi, E, 1LL << n, edges, gmass, ext, below);
  else
    k_ro_hist<float><<<ro_grid(), RO_NT, 0, s>>>((const float *)psi, E, 1LL << n, edges, gmass, ext, below);
  return cudaGetLastError();
}

cudaError_t launch_ro_gather(const double *E, const long long *shots, int nshots, double *out, cudaStream_t s) {
  if (nshots <= 0) return cudaSuccess;
  k_ro_gather<<<(nshots + 255) / 256, 256, 0, s>>>(E, shots, nshots, out);
  return cudaGetLastError();
}

cudaError_t launch_ro_rank(const double *es, int nshots, int r0, int r1, double *out, cudaStream_t s) {
  k_ro_rank<<<2, RANK_NT, 0, s>>>(es, nshots, r0, r1, out);
  return cudaGetLastError();
}

cudaError_t launch_ro_cvar(int prec, const void *psi, const double *E, int n, double alpha, double tau,
                           double *part, double *stats, cudaStream_t s) {
  const int g = ro_grid();
  unsigned long long kt;
  memcpy(&kt, &tau, sizeof(kt));
  kt = (kt >> 63) ? ~kt : (kt | 0x8000000000000000ull);
  if (prec)
    k_ro_tail<double><<<g, RO_NT, 0, s>>>((const double *)psi, E, 1LL << n, kt, part);
  else
    k_ro_tail<float><<<g, RO_NT, 0, s>>>((const float *)psi, E, 1LL << n, kt, part);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_ro_cvar<<<1, 256, 24 * (size_t)g, s>>>(part, g, alpha, tau, stats);
  return cudaGetLastError();
}

}  // namespace gvqe
