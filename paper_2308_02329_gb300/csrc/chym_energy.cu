// chym_energy.cu -- Ising readout, Ising energy and ground-state statistics.
//
// Readout s_p = sign(x_{p,0}) (ties to +1) and E = -sum_{p,q} J_pq s_p s_q
// (Eq. 3 with Ising spins); for +-1/0 couplings the sum is exact in integers.
// The statistics kernel counts ground-state hits per pump value (P_Ising(h)),
// bins the energy histogram H_E and finds the best run, i.e. the inputs of the
// figures of merit (i)-(iii) that follow Fig. 3 of arXiv 2308.02329.
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "chym_internal.cuh"

namespace chym {
namespace {

constexpr int kEnergyThreads = 256;

// Deterministic block sum (fixed shuffle tree, then warp 0 over the partials).
template <typename V>
__device__ V block_sum(V v, V* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  V t = V(0);
  if (w == 0) {
    t = (lane < (int)(blockDim.x >> 5)) ? red[lane] : V(0);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
  }
  return t;  // valid in thread 0
}

constexpr int kMaxSpinWords = 64;  // N <= 4096

// Spin words of the CTA's nr runs into sw[r][w] (bit q of word w: s_{64 w + q} = +1), one
// warp per (run, word) with the signs collected by ballot; bad(r, q) is called for a spin
// that is not finite.  Ends with a barrier.
template <typename T, typename Bad>
__device__ __forceinline__ void read_spins(const T* __restrict__ X, int run0, int nr, int N, int D,
                                           uint64_t (*sw)[kMaxSpinWords], Bad bad) {
  const int words = (N + 63) / 64, lane = threadIdx.x & 31;
#pragma unroll 2
  for (int t = threadIdx.x >> 5; t < nr * words; t += blockDim.x >> 5) {
    const int r = t / words, w = t % words;
    uint32_t half[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int q = 64 * w + 32 * i + lane;
      bool up = false, finite = true;
      if (q < N) {
        const T* x = X + ((size_t)(run0 + r) * N + q) * D;
        up = x[0] >= T(0);
#pragma unroll 4
        for (int mu = 0; mu < D; ++mu) finite &= isfinite(x[mu]) != 0;  // no short cut: independent loads
      }
      if (!finite) bad(r, q);
      half[i] = __ballot_sync(0xffffffffu, up);
    }
    if (lane == 0) sw[r][w] = (uint64_t)half[0] | ((uint64_t)half[1] << 32);
  }
  __syncthreads();
}

// Energies of RB consecutive runs per CTA, so that a row of couplings is read once for RB
// runs; thread = row p.
//
// +-1 J: bit planes of J, plane[w][p] = the bits of row p's columns 64 w .. 64 w + 63
// where J = +1 (Jpos) or -1 (Jneg), word-major so that consecutive rows are coalesced.
// With d_p = the spins that differ from s_p (one xor of the spin words),
//   sum_q J_pq s_p s_q = deg_p - 2 (popc(Jpos_p & d_p) - popc(Jneg_p & d_p)),
// deg_p = (#J = +1) - (#J = -1) in row p: an exact integer from N/64 words a row.
//
// kSplit: block (x, y) takes the y-th share of the rows and adds its part to E (zeroed
// before; integers, so the order does not matter): a few dozen runs of a large N would
// otherwise leave most SMs idle (64 runs, N = 1000: 42 us).
template <typename T, int RB, bool kSplit>
__global__ void __launch_bounds__(kEnergyThreads) energy_pm1_kernel(
    const T* __restrict__ X, int N, int D, int n_runs, const uint64_t* __restrict__ Jpos,
    const uint64_t* __restrict__ Jneg, const int32_t* __restrict__ deg, double* __restrict__ E,
    uint64_t* __restrict__ spins) {
  __shared__ uint64_t sw[RB][kMaxSpinWords];
  __shared__ int bad[RB], sum[RB];
  const int run0 = blockIdx.x * RB, nr = min(RB, n_runs - run0), tid = threadIdx.x;
  const int words = (N + 63) / 64;
  if (tid < RB) bad[tid] = sum[tid] = 0;
  __syncthreads();
  read_spins<T>(X, run0, nr, N, D, sw, [&](int r, int) { bad[r] = 1; });
  if (spins && (!kSplit || blockIdx.y == 0))
    for (int t = tid; t < nr * words; t += blockDim.x) spins[(size_t)run0 * words + t] = sw[t / words][t % words];
  int acc[RB];  // at most N^2 <= 2^24 in magnitude
#pragma unroll
  for (int r = 0; r < RB; ++r) acc[r] = 0;
  const int p_begin = kSplit ? (int)((long long)N * blockIdx.y / gridDim.y) : 0;
  const int p_end = kSplit ? (int)((long long)N * (blockIdx.y + 1) / gridDim.y) : N;
  for (int p = p_begin + tid; p < p_end; p += blockDim.x) {
    uint64_t flip[RB];  // d = spins unlike s_p (padding bits meet no J)
    int c[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      flip[r] = (r < nr && ((sw[r][p >> 6] >> (p & 63)) & 1u)) ? ~0ull : 0ull;
      c[r] = 0;
    }
    for (int w = 0; w < words; ++w) {
      const uint64_t jp = __ldg(Jpos + (size_t)w * N + p), jn = __ldg(Jneg + (size_t)w * N + p);
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const uint64_t d = sw[r][w] ^ flip[r];
        c[r] += __popcll(jp & d) - __popcll(jn & d);
      }
    }
    const int dg = deg[p];
#pragma unroll
    for (int r = 0; r < RB; ++r) acc[r] += dg - 2 * c[r];
  }
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    const int t = __reduce_add_sync(0xffffffffu, acc[r]);
    if ((tid & 31) == 0) atomicAdd(&sum[r], t);
  }
  __syncthreads();
  if (tid >= nr) return;
  const double part = bad[tid] ? (double)NAN : -(double)sum[tid];
  if (kSplit) atomicAdd(E + run0 + tid, part);
  else E[run0 + tid] = part;
}

// Real J in fixed point on the tensor cores.  Row p of J times 2^e_p is rounded to integers,
// e_p such that the row's absolute sum stays below 2^60, and split into kDigits signed
// digits of 11 bits, each exact in FP16.  The products of a digit plane with the spins
// (+-1) then add up exactly in FP32 (at most 2^10 N <= 2^22), so the local field is exact
// but for the entries' rounding, which is below 2^-60 of the row's absolute sum and below
// the rounding of an FP64 sum.  J is symmetric: of the 16 x 16 tiles only those on and
// above the diagonal are read, E = -sum_p s_p (sum_{q in p's tile} + 2 sum_{later tiles}),
// summed over p in FP64.  m16n8k16 products with the digits stored as ready A fragments:
// N = 1000, 8192 runs took 30.1 ms with FP64 products (2 lanes per clock and SM) and one
// run a block, and 2.53 ms with 64-bit integer adds.
constexpr int kDigits = 6, kDigitBits = 11;

// Place of tile (i, j), i <= j, among those on and above the diagonal, row by row.
__host__ __device__ inline size_t digit_tile(int i, int j, int tiles) {
  return (size_t)i * tiles - (size_t)i * (i - 1) / 2 + (j - i);
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// NT x 8 consecutive runs per CTA; warp w takes the row tiles w, w + warps, ...  Fragment
// coordinates of lane l: g = l / 4, t = l % 4; A rows g and g + 8, columns 2t, 2t + 1 and
// 2t + 8, 2t + 9; B the same columns of run g; C rows g and g + 8 of runs 2t and 2t + 1.
template <typename T, int NT>
__global__ void __launch_bounds__(kEnergyThreads) energy_real_kernel(
    const T* __restrict__ X, int N, int D, int n_runs, const uint4* __restrict__ Jd,
    const int32_t* __restrict__ e_row, double* __restrict__ E, uint64_t* __restrict__ spins) {
  constexpr int RB = 8 * NT, kWarps = kEnergyThreads / 32;
  __shared__ uint64_t sw[RB][kMaxSpinWords];
  __shared__ int bad[RB];
  __shared__ double red[kWarps][RB];
  const int run0 = blockIdx.x * RB, nr = min(RB, n_runs - run0), tid = threadIdx.x;
  const int words = (N + 63) / 64, tiles = (N + 15) / 16;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  if (tid < RB) bad[tid] = 0;
  for (int i = tid; i < RB * kMaxSpinWords; i += blockDim.x) (&sw[0][0])[i] = 0ull;  // unused runs
  __syncthreads();
  read_spins<T>(X, run0, nr, N, D, sw, [&](int r, int) { bad[r] = 1; });
  if (spins)
    for (int t = tid; t < nr * words; t += blockDim.x) spins[(size_t)run0 * words + t] = sw[t / words][t % words];
  double acc[NT][2];
#pragma unroll
  for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = 0.0;
  for (int i = warp; i < tiles; i += kWarps) {
    const uint4* a = Jd + digit_tile(i, i, tiles) * (kDigits * 32) + lane;
    float c[NT][kDigits][4];
    auto clear = [&]() {
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int d = 0; d < kDigits; ++d)
#pragma unroll
          for (int v = 0; v < 4; ++v) c[n][d][v] = 0.f;
    };
    long long f[NT][4];  // local fields of the tile's rows
    auto field = [&](int n, int v) {
      long long x = 0;
#pragma unroll
      for (int d = kDigits - 1; d >= 0; --d) x = (x << kDigitBits) + (long long)(int)c[n][d][v];
      return x;
    };
    clear();
    for (int j = i; j < tiles; ++j, a += kDigits * 32) {
      uint4 av[kDigits];
#pragma unroll
      for (int d = 0; d < kDigits; ++d) av[d] = __ldg(a + d * 32);
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        // FP16 +-1 of two columns: 0x3C00 with the sign bit where the spin is down
        const uint32_t dn = ~(uint32_t)reinterpret_cast<const uint16_t*>(sw[8 * n + g])[j] >> t2;
        const uint32_t b0 = 0x3C003C00u | (dn & 1u) << 15 | (dn & 2u) << 30;
        const uint32_t b1 = 0x3C003C00u | (dn & 0x100u) << 7 | (dn & 0x200u) << 22;
#pragma unroll
        for (int d = 0; d < kDigits; ++d) mma_f16(c[n][d], av[d], b0, b1);
      }
      if (j == i) {  // the diagonal tile counts once, the later ones twice
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int v = 0; v < 4; ++v) f[n][v] = field(n, v);
        clear();
      }
    }
    const int p0 = 16 * i + g;
    const int e0 = p0 < N ? e_row[p0] : 0, e1 = p0 + 8 < N ? e_row[p0 + 8] : 0;  // rows past N hold zeros
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int p = p0 + (v >= 2 ? 8 : 0), r = 8 * n + t2 + (v & 1);
        const bool up = (sw[r][(p >> 6) & (kMaxSpinWords - 1)] >> (p & 63)) & 1u;
        const double x = ldexp((double)(f[n][v] + 2 * field(n, v)), v >= 2 ? -e1 : -e0);
        acc[n][v & 1] += up ? x : -x;
      }
  }
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      double x = acc[n][v];
      for (int o = 16; o >= 4; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (g == 0) red[warp][8 * n + t2 + v] = x;
    }
  __syncthreads();
  if (tid < nr) {
    double t = 0.0;
    for (int w = 0; w < kWarps; ++w) t += red[w][tid];
    E[run0 + tid] = bad[tid] ? (double)NAN : -t;
  }
}

// Row exponents of energy_real_kernel, one warp per row.
__global__ void row_exponents_kernel(const double* __restrict__ J, int N, int32_t* __restrict__ e_row) {
  const int lane = threadIdx.x & 31;
  for (int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < N; p += gridDim.x * (blockDim.x >> 5)) {
    double top = 0.0;
    for (int q = lane; q < N; q += 32) top = fmax(top, fabs(J[(size_t)p * N + q]));
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    int x = 0, n = 0;
    frexp(top, &x);    // |J| < 2^x
    double sum = 0.0;  // of |J| 2^-x: at most N, rounded by at most N 2^-53 of itself
    for (int q = lane; q < N; q += 32) sum += ldexp(fabs(J[(size_t)p * N + q]), -x);
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    frexp(sum * 1.000001, &n);  // sum < 2^n
    if (lane == 0) e_row[p] = top > 0.0 ? 60 - x - n : 0;
  }
}

// Digit planes as A fragments: Jd[digit_tile][digit][lane], four FP16 pairs of columns
// (2t, 2t+1): rows g, g + 8 at columns 2t, then at 2t + 8.  Zero past N.
__global__ void digits_kernel(const double* __restrict__ J, int N, const int32_t* __restrict__ e_row,
                              uint4* __restrict__ Jd) {
  const int tiles = (N + 15) / 16;
  const size_t total = (size_t)tiles * tiles * 32;
  for (size_t s = blockIdx.x * (size_t)blockDim.x + threadIdx.x; s < total; s += (size_t)gridDim.x * blockDim.x) {
    const int lane = (int)(s & 31), g = lane >> 2, t2 = 2 * (lane & 3);
    const int i = (int)(s / 32 / tiles), j = (int)(s / 32 % tiles);
    if (j < i) continue;
    uint32_t out[kDigits][4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int p = 16 * i + g + (v & 1) * 8, q = 16 * j + t2 + (v >> 1) * 8;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        long long x = p < N && q + h < N ? llrint(ldexp(J[(size_t)p * N + q + h], e_row[p])) : 0ll;
#pragma unroll
        for (int d = 0; d < kDigits; ++d) {
          constexpr long long half = 1ll << (kDigitBits - 1);
          const long long dig = ((x + half) & (2 * half - 1)) - half;  // in [-1024, 1023]
          x = (x - dig) >> kDigitBits;
          const uint32_t bits = __half_as_ushort(__int2half_rn((int)dig));
          out[d][v] = h ? out[d][v] | bits << 16 : bits;
        }
      }
    }
#pragma unroll
    for (int d = 0; d < kDigits; ++d)
      Jd[digit_tile(i, j, tiles) * (kDigits * 32) + d * 32 + lane] = make_uint4(out[d][0], out[d][1], out[d][2], out[d][3]);
  }
}

// Energies of the spin segments of RB runs, E_i = -sum_{p,q in i} J_pq s_p s_q (the
// energies of the graphs of a block-diagonal packing), +-1 J, by the bit planes masked to
// the segment of row p; NaN when a state value of the segment is not finite.  One CTA for
// all segments of its runs, so that short segments share its threads: 672 runs of up to 128
// packed spins take 6.0 us (9.7 us with one CTA per run and segment and int8 products).
template <typename T, int RB>
__global__ void __launch_bounds__(kEnergyThreads) energy_segments_pm1_kernel(
    const T* __restrict__ X, int N, int D, int n_runs, const uint64_t* __restrict__ Jpos,
    const uint64_t* __restrict__ Jneg, SegTable t, double* __restrict__ E) {
  extern __shared__ uint8_t seg_of[];  // N
  __shared__ uint64_t sw[RB][kMaxSpinWords];
  __shared__ int sum[RB][kMaxSegments], bad[RB][kMaxSegments];
  const int run0 = blockIdx.x * RB, nr = min(RB, n_runs - run0), tid = threadIdx.x;
  for (int i = tid; i < RB * kMaxSegments; i += blockDim.x) (&sum[0][0])[i] = (&bad[0][0])[i] = 0;
  for (int p = tid; p < N; p += blockDim.x) {
    int lo = 0, hi = t.n;  // begin[lo] <= p < begin[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (t.begin[mid] <= p) lo = mid;
      else hi = mid;
    }
    seg_of[p] = (uint8_t)lo;
  }
  __syncthreads();
  read_spins<T>(X, run0, nr, N, D, sw, [&](int r, int q) { bad[r][seg_of[q]] = 1; });
  for (int p = tid; p < N; p += blockDim.x) {
    const int sg = seg_of[p], b = t.begin[sg], e = t.begin[sg + 1];
    int v[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) v[r] = 0;
    for (int w = b >> 6; w <= (e - 1) >> 6; ++w) {
      // bits of word w inside [b, e)
      uint64_t mask = ~0ull;
      if (b > 64 * w) mask &= ~0ull << (b - 64 * w);
      if (e < 64 * w + 64) mask &= ~0ull >> (64 * w + 64 - e);
      const uint64_t jp = __ldg(Jpos + (size_t)w * N + p) & mask, jn = __ldg(Jneg + (size_t)w * N + p) & mask;
      const int dg = __popcll(jp) - __popcll(jn);
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const uint64_t d = sw[r][w] ^ (((sw[r][p >> 6] >> (p & 63)) & 1u) ? ~0ull : 0ull);
        v[r] += dg - 2 * (__popcll(jp & d) - __popcll(jn & d));
      }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) atomicAdd(&sum[r][sg], v[r]);
  }
  __syncthreads();
  for (int i = tid; i < nr * t.n; i += blockDim.x) {
    const int r = i / t.n, sg = i % t.n;
    E[(size_t)run0 * t.n + i] = bad[r][sg] ? (double)NAN : -(double)sum[r][sg];
  }
}

// Real J: one CTA per (run, segment), FP64.
template <typename T>
__global__ void __launch_bounds__(kEnergyThreads) energy_segments_real_kernel(
    const T* __restrict__ X, int N, int D, const double* __restrict__ J64, SegTable t, double* __restrict__ E) {
  extern __shared__ int8_t s[];
  __shared__ int bad;
  __shared__ double red_d[32];
  const int run = blockIdx.x, seg = blockIdx.y, tid = threadIdx.x;
  const int b = t.begin[seg], n = t.begin[seg + 1] - b;
  if (tid == 0) bad = 0;
  __syncthreads();
  const T* x = X + ((size_t)run * N + b) * D;
  int my_bad = 0;
  for (int p = tid; p < n; p += blockDim.x) {
    s[p] = (x[(size_t)p * D] >= T(0)) ? 1 : -1;
    for (int mu = 0; mu < D; ++mu) my_bad |= !isfinite((double)x[(size_t)p * D + mu]);
  }
  if (my_bad) atomicOr(&bad, 1);
  __syncthreads();
  double* out = E + (size_t)run * t.n + seg;
  double acc = 0.0;
  for (int p = tid; p < n; p += blockDim.x) {
    double f = 0.0;
    for (int q = 0; q < n; ++q) f += J64[(size_t)(b + q) * N + b + p] * (double)s[q];
    acc += (double)s[p] * f;
  }
  const double tot = block_sum<double>(acc, red_d);
  if (tid == 0) *out = bad ? (double)NAN : -tot;
}

// Single CTA, deterministic: per-h hits, histogram, best run, finite count,
// sum of (E - E_gs) over finite runs.  out layout (see StatsOut).
struct StatsOut {
  double sum_dE;
  double best_E;
  long long best_run;
  long long n_finite;
  long long n_hits;
  long long pad[3];
  // followed by hits[n_h] and hist[n_bins] (long long)
};

constexpr int kStatsThreads = 1024;

__global__ void __launch_bounds__(kStatsThreads) stats_kernel(const double* __restrict__ E,
                                                              const int32_t* __restrict__ hidx,
                                                              int n_runs, int replicas, int n_h,
                                                              double E_gs, double tol,
                                                              double bin_w, int n_bins,
                                                              StatsOut* out) {
  extern __shared__ unsigned long long sh_hits[];  // n_h counters
  __shared__ double red_d[32];
  __shared__ long long red_i[32];
  __shared__ double best_e[kStatsThreads / 32];
  __shared__ long long best_r[kStatsThreads / 32];
  long long* hits_out = reinterpret_cast<long long*>(out + 1);
  unsigned long long* hist_out = reinterpret_cast<unsigned long long*>(hits_out + n_h);
  const int tid = threadIdx.x;
  for (int i = tid; i < n_h; i += blockDim.x) sh_hits[i] = 0ull;
  for (int i = tid; i < n_bins; i += blockDim.x) hist_out[i] = 0ull;
  __syncthreads();
  double sum = 0.0, be = INFINITY;
  long long br = -1, nf = 0, nh = 0;
  for (int r = tid; r < n_runs; r += blockDim.x) {
    const double e = E[r];
    if (!isfinite(e)) continue;
    ++nf;
    sum += e - E_gs;
    const bool hit = fabs(e - E_gs) <= tol;
    if (hit) {
      atomicAdd(&sh_hits[hidx ? hidx[r] : r / replicas], 1ull);
      ++nh;
    }
    if (e < be || (e == be && r < br)) { be = e; br = r; }
    if (n_bins > 0) {
      double b = floor((e - E_gs) / bin_w + 0.5);
      int bi = b < 0.0 ? 0 : (b >= (double)n_bins ? n_bins - 1 : (int)b);
      atomicAdd(&hist_out[bi], 1ull);
    }
  }
  const double tsum = block_sum<double>(sum, red_d);
  __syncthreads();
  const long long tnf = block_sum<long long>(nf, red_i);
  __syncthreads();
  const long long tnh = block_sum<long long>(nh, red_i);
  // best (E, run): warp argmin then block argmin, ties to the lowest run
  for (int o = 16; o > 0; o >>= 1) {
    const double oe = __shfl_down_sync(0xffffffffu, be, o);
    const long long orr = __shfl_down_sync(0xffffffffu, br, o);
    if (orr >= 0 && (oe < be || (oe == be && (br < 0 || orr < br)))) { be = oe; br = orr; }
  }
  if ((tid & 31) == 0) { best_e[tid >> 5] = be; best_r[tid >> 5] = br; }
  __syncthreads();
  if (tid == 0) {
    double e0 = INFINITY;
    long long r0 = -1;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
      if (best_r[w] >= 0 && (best_e[w] < e0 || (best_e[w] == e0 && best_r[w] < r0))) {
        e0 = best_e[w];
        r0 = best_r[w];
      }
    out->sum_dE = tsum;
    out->best_E = e0;
    out->best_run = r0;
    out->n_finite = tnf;
    out->n_hits = tnh;
  }
  for (int i = tid; i < n_h; i += blockDim.x) hits_out[i] = (long long)sh_hits[i];
}

// Runs per CTA: several runs share one read of the couplings; with fewer runs than one such
// CTA per SM, one run (+-1 J) or one eight-run tile (real J) a CTA spreads the work.
constexpr int kEnergyRuns = 8, kEnergyRealTiles = 4;
bool many_runs(const chym_ctx* c, int rb) { return c->n_runs >= rb * 152; }
int energy_threads(int rows) { return rows <= 128 ? 128 : kEnergyThreads; }

template <typename T>
cudaError_t launch_energy_typed(chym_ctx* c, double* d_E, uint64_t* d_spins, cudaStream_t st) {
  const T* X = (const T*)c->d_X;
  const int N = c->N, R = c->n_runs;
  if (N > 64 * kMaxSpinWords) return cudaErrorInvalidValue;
  const int W = (N + 63) / 64;
  if (c->kind == CHYM_J_PM1) {
    const uint64_t *jp = c->d_Jbits, *jn = c->d_Jbits + (size_t)W * N;
    const int groups = (R + kEnergyRuns - 1) / kEnergyRuns;
    if (many_runs(c, kEnergyRuns)) {
      energy_pm1_kernel<T, kEnergyRuns, false>
          <<<groups, energy_threads(N), 0, st>>>(X, N, c->D, R, jp, jn, c->d_jdeg, d_E, d_spins);
    } else if (N >= 2 * kEnergyThreads) {
      // shares of at least one row a thread, up to four blocks per SM
      const int shares = std::max(1, std::min(N / kEnergyThreads, 4 * 152 / R));
      cudaError_t e = cudaMemsetAsync(d_E, 0, sizeof(double) * (size_t)R, st);
      if (e != cudaSuccess) return e;
      energy_pm1_kernel<T, 1, true><<<dim3((unsigned)R, (unsigned)shares), kEnergyThreads, 0, st>>>(
          X, N, c->D, R, jp, jn, c->d_jdeg, d_E, d_spins);
    } else {
      energy_pm1_kernel<T, 1, false><<<R, energy_threads(N), 0, st>>>(X, N, c->D, R, jp, jn, c->d_jdeg, d_E, d_spins);
    }
  } else if (many_runs(c, 8 * kEnergyRealTiles)) {
    energy_real_kernel<T, kEnergyRealTiles>
        <<<(R + 8 * kEnergyRealTiles - 1) / (8 * kEnergyRealTiles), kEnergyThreads, 0, st>>>(
            X, N, c->D, R, (const uint4*)c->d_Jdig, c->d_Jexp, d_E, d_spins);
  } else {
    energy_real_kernel<T, 1><<<(R + 7) / 8, kEnergyThreads, 0, st>>>(X, N, c->D, R, (const uint4*)c->d_Jdig,
                                                                    c->d_Jexp, d_E, d_spins);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_segments_typed(chym_ctx* c, const SegTable& t, double* d_E, cudaStream_t st) {
  const T* X = (const T*)c->d_X;
  const int N = c->N, R = c->n_runs, W = (N + 63) / 64;
  if (N > 64 * kMaxSpinWords) return cudaErrorInvalidValue;
  if (c->kind == CHYM_J_PM1) {
    const uint64_t *jp = c->d_Jbits, *jn = c->d_Jbits + (size_t)W * N;
    if (many_runs(c, kEnergyRuns))
      energy_segments_pm1_kernel<T, kEnergyRuns><<<(R + kEnergyRuns - 1) / kEnergyRuns, energy_threads(N), (size_t)N, st>>>(
          X, N, c->D, R, jp, jn, t, d_E);
    else
      energy_segments_pm1_kernel<T, 1><<<R, energy_threads(N), (size_t)N, st>>>(X, N, c->D, R, jp, jn, t, d_E);
    return cudaGetLastError();
  }
  int longest = 0;
  for (int i = 0; i < t.n; ++i) longest = std::max(longest, t.begin[i + 1] - t.begin[i]);
  energy_segments_real_kernel<T><<<dim3((unsigned)R, (unsigned)t.n), kEnergyThreads, (size_t)longest, st>>>(
      X, N, c->D, c->d_J64, t, d_E);
  return cudaGetLastError();
}

}  // namespace

// Digit planes and row exponents of a context with real couplings, from its FP64 copy.
cudaError_t prepare_energy_digits(chym_ctx* c) {
  const int tiles = (c->N + 15) / 16;
  cudaError_t e = cudaMalloc((void**)&c->d_Jexp, sizeof(int32_t) * c->N);
  if (e == cudaSuccess) e = cudaMalloc(&c->d_Jdig, digit_tile(tiles, tiles, tiles) * kDigits * 32 * sizeof(uint4));
  if (e != cudaSuccess) return e;
  row_exponents_kernel<<<152 * 2, 256>>>(c->d_J64, c->N, c->d_Jexp);
  digits_kernel<<<152 * 8, 256>>>(c->d_J64, c->N, c->d_Jexp, (uint4*)c->d_Jdig);
  e = cudaGetLastError();
  return e == cudaSuccess ? cudaStreamSynchronize(cudaStreamLegacy) : e;
}

cudaError_t launch_energy(chym_ctx* c, double* d_E, uint64_t* d_spins, cudaStream_t st) {
  if (c->n_runs <= 0) return cudaSuccess;
  if (c->prec == CHYM_PREC_FP64) return launch_energy_typed<double>(c, d_E, d_spins, st);
  return launch_energy_typed<float>(c, d_E, d_spins, st);
}

cudaError_t launch_energy_segments(chym_ctx* c, const SegTable& t, double* d_E, cudaStream_t st) {
  if (c->n_runs <= 0) return cudaSuccess;
  if (c->prec == CHYM_PREC_FP64) return launch_segments_typed<double>(c, t, d_E, st);
  return launch_segments_typed<float>(c, t, d_E, st);
}

size_t stats_out_bytes(int n_h, int n_bins) {
  return sizeof(StatsOut) + sizeof(long long) * ((size_t)n_h + (size_t)n_bins);
}

cudaError_t launch_stats(chym_ctx* c, const double* d_E, double E_gs, double tol, double bin_w,
                         int n_bins, void* d_out, cudaStream_t st) {
  const size_t smem = sizeof(unsigned long long) * (size_t)c->n_h;
  auto kern = stats_kernel;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<1, kStatsThreads, smem, st>>>(d_E, c->d_hidx, c->n_runs, c->n_runs / c->n_h, c->n_h, E_gs, tol,
                                       bin_w, n_bins, (StatsOut*)d_out);
  return cudaGetLastError();
}



// ---------------------------------------------------------------------------
// Allocation-free statistics.
//
// Some callers cannot allocate device memory when they need the statistics:
// code running under a memory manager that owns the whole device pool, callers
// that must not trigger the device-wide synchronisation cudaMalloc/cudaFree can
// imply, or real-time loops with a fixed memory budget.  For them the statistics
// kernel writes its result block into this file-scope device array instead of a
// context buffer.  Every GPU that loads the library holds the array until exit.
// ---------------------------------------------------------------------------
namespace {
constexpr int kNoAllocMaxH = 4096;      // pump values
constexpr int kNoAllocMaxBins = 65536;  // histogram bins
constexpr size_t kNoAllocBytes =
    sizeof(StatsOut) + sizeof(long long) * ((size_t)kNoAllocMaxH + kNoAllocMaxBins);
static __device__ __align__(256) unsigned char g_stats_noalloc_scratch[kNoAllocBytes];

// Device address of the array on each device, looked up once per device with that
// device current (host code must not pass the array's name to a kernel).
constexpr int kMaxDevices = 64;
void* g_noalloc_addr[kMaxDevices] = {};
std::mutex g_noalloc_mutex;

cudaError_t noalloc_scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_stats_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return cudaSuccess;
}
}  // namespace

}  // namespace chym

extern "C" CHYM_API chym_status chym_stats_noalloc(const double* d_E, int n_runs, int n_h,
                                                   chym_jkind kind, double E_gs,
                                                   chym_stats_t* out, int64_t* hits_per_h,
                                                   int64_t* hist, int n_bins,
                                                   void* cuda_stream) {
  using namespace chym;
  if (!d_E || !out) return fail(CHYM_EINVAL, "NULL argument");
  if (n_h < 1 || n_runs < 1 || n_runs % n_h)
    return fail(CHYM_EINVAL, "n_runs must be a positive multiple of n_h");
  if (n_h > kNoAllocMaxH)
    return fail(CHYM_EINVAL, "chym_stats_noalloc: n_h exceeds the fixed limit of 4096");
  if (n_bins < 0 || n_bins > kNoAllocMaxBins || (hist && n_bins < 1))
    return fail(CHYM_EINVAL, "chym_stats_noalloc: n_bins must be in [1, 65536] with a histogram");
  if (kind != CHYM_J_PM1 && kind != CHYM_J_REAL) return fail(CHYM_EINVAL, "unknown J kind");
  if (!isfinite(E_gs)) return fail(CHYM_EINVAL, "E_gs must be finite");
  if (!hist) n_bins = 0;
  void* scratch = nullptr;
  cudaError_t e = noalloc_scratch_address(&scratch);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(stats scratch)");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const bool pm1 = kind == CHYM_J_PM1;
  const double tol = pm1 ? 0.0 : 1e-9 * fabs(E_gs);
  double bin_w = pm1 ? 4.0 : 1e-3 * fabs(E_gs);
  if (!(bin_w > 0.0)) bin_w = 1.0;
  // the kernel initialises every word it reports (hits, bins, totals), so the
  // previous call's contents never leak into this one
  stats_kernel<<<1, kStatsThreads, sizeof(unsigned long long) * (size_t)n_h, st>>>(
      d_E, nullptr, n_runs, n_runs / n_h, n_h, E_gs, tol, bin_w, n_bins, (StatsOut*)scratch);
  CHYM_CUDA_TRY(cudaGetLastError());
  StatsOut head;
  CHYM_CUDA_TRY(cudaMemcpyAsync(&head, scratch, sizeof(head), cudaMemcpyDeviceToHost, st));
  const long long* d_hits = reinterpret_cast<const long long*>((const StatsOut*)scratch + 1);
  // per-pump counts are needed for P_max and W; without a caller buffer they go to a
  // fixed per-thread host array of the maximum size.  Every copy is ordered on st and
  // one synchronisation of st ends the call, so no other stream is waited for.
  static thread_local long long hits_tmp[kNoAllocMaxH];
  long long* hits = hits_per_h ? reinterpret_cast<long long*>(hits_per_h) : hits_tmp;
  CHYM_CUDA_TRY(cudaMemcpyAsync(hits, d_hits, sizeof(long long) * n_h, cudaMemcpyDeviceToHost, st));
  if (hist && n_bins)
    CHYM_CUDA_TRY(cudaMemcpyAsync(hist, d_hits + n_h, sizeof(long long) * n_bins,
                                  cudaMemcpyDeviceToHost, st));
  CHYM_CUDA_TRY(cudaStreamSynchronize(st));
  const int reps = n_runs / n_h;
  double pmax = 0.0, psum = 0.0;
  int nz = 0;
  for (int i = 0; i < n_h; ++i) {
    const double P = (double)hits[i] / reps;
    pmax = std::max(pmax, P);
    psum += P;
    if (hits[i] > 0) ++nz;
  }
  out->P_max = pmax;
  out->W_range = nz ? psum / nz : 0.0;
  out->W_scan = psum / n_h;
  out->dE_mean = head.n_finite ? head.sum_dE / (double)head.n_finite : NAN;
  out->best_E = head.best_E;
  out->best_run = head.best_run;
  out->n_finite = head.n_finite;
  out->n_hits = head.n_hits;
  return CHYM_OK;
}

