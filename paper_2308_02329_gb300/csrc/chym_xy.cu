// chym_xy.cu -- readout of XY (D = 2) runs by best-axis rounding.
//
// The XY machine (D = 2 without annealing, text after Fig. 2) leaves every
// hyperspin as a planar vector; reading only its first component, as the Ising
// readout does, fixes the axis arbitrarily.  Best-axis rounding tries every axis
// u = (cos phi, sin phi): the pattern s_p = sign(x_p . u) changes only where u is
// perpendicular to a spin, at phi_p = theta_p + pi/2 (mod pi), so sweeping phi
// over [0, pi) flips one spin per critical angle.  Per run:
//   1. critical angles (FP64 atan2, so that their order matches the oracle) and
//      the pattern of an axis inside the interval that wraps through pi;
//   2. bitonic sort of (angle, spin) in shared memory;
//   3. local fields h_q = sum_p J_qp s_p (N^2 multiply-adds) and E = -sum s h;
//   4. the sweep: per critical angle, E += 4 s_p h_p, s_p = -s_p and every h_q
//      moves by 2 J_qp s_p; after the last spin of a group of equal angles the
//      energy is a candidate; the lowest one (first in sweep order) wins;
//   5. the winning pattern is rebuilt and bit-packed.
// +-1 couplings: integers throughout, one warp per run up to N = 256 (one block above), so
// that the sweep's hand-overs are warp barriers: N = 100, 1024 runs take 60 us (513 us with one
// block per run and FP64 fields).  Real couplings: one block per run, FP64.
// A run whose state holds a non-finite value (a diverged run) gets E = NaN, as in
// the Ising readout, and no sweep; its spins are then unspecified.
#include <math.h>

#include "chym_internal.cuh"

namespace chym {
namespace {

constexpr int kXyThreads = 256;
constexpr int kXyMaxN = 4096;

// Critical angle of a spin (a, b) != 0 in [0, pi): theta + pi/2 (mod pi).
__device__ __forceinline__ double critical_angle(double a, double b) {
  constexpr double pi = 3.14159265358979323846;
  double k = atan2(b, a) + 0.5 * pi;  // in [-pi/2, 3 pi/2]
  if (k >= pi) k -= pi;               // exact
  else if (k < 0.0) k += pi;
  return k + 0.0;  // no negative zero: the keys compare as integers
}

constexpr int kXyWarpMaxN = 256;  // one warp per run up to here
constexpr int kXyAhead = 8;       // couplings of the next flipped spin's row held ahead, per thread

__host__ __device__ inline size_t xy_run_bytes(int N, int P2) {  // keys, indices, fields, spin words
  return ((size_t)P2 * 10 + (size_t)N * 4 + 7) / 8 * 8 + (size_t)((N + 63) / 64) * 8;
}

// NW warps per run (1 or 8), 8 / NW runs per block.
template <typename T, int NW>
__global__ void __launch_bounds__(kXyThreads) round_xy_pm1_kernel(const T* __restrict__ X, int N, int P2, int n_runs,
                                                                  const int8_t* __restrict__ J8,
                                                                  const uint64_t* __restrict__ Jpos,
                                                                  const uint64_t* __restrict__ Jneg,
                                                                  const int32_t* __restrict__ deg,
                                                                  double* __restrict__ E_out,
                                                                  uint64_t* __restrict__ spins_out) {
  constexpr int kT = 32 * NW, kRuns = kXyThreads / kT;
  extern __shared__ __align__(16) unsigned char xy_smem[];
  __shared__ int red[kRuns][NW];
  __shared__ int s_bad[kRuns];
  const int slot = threadIdx.x / kT, tid = threadIdx.x % kT, lane = threadIdx.x & 31;
  const int run = blockIdx.x * kRuns + slot, words = (N + 63) / 64;
  unsigned char* base = xy_smem + (size_t)slot * xy_run_bytes(N, P2);
  unsigned long long* key = reinterpret_cast<unsigned long long*>(base);  // bits of angles >= 0: ordered as integers
  int* h = reinterpret_cast<int*>(key + P2);
  uint16_t* idx = reinterpret_cast<uint16_t*>(h + N);
  uint64_t* up = reinterpret_cast<uint64_t*>(base + ((size_t)P2 * 10 + (size_t)N * 4 + 7) / 8 * 8);
  auto sync = [&]() {
    if constexpr (NW == 1) __syncwarp();
    else __syncthreads();
  };
  if (NW == 1 && run >= n_runs) return;
  const double pi = 3.14159265358979323846;
  const unsigned long long never = 0x7FF0000000000000ull;  // +inf: spins of zero length never flip
  if (tid == 0) s_bad[slot] = 0;
  sync();
  const T* x = X + (size_t)run * N * 2;
  // 1. critical angles
  for (int i = tid; i < P2; i += kT) {
    unsigned long long k = never;
    if (i < N) {
      const double a = (double)x[2 * i], b = (double)x[2 * i + 1];
      if (!isfinite(a) || !isfinite(b)) s_bad[slot] = 1;
      else if (a != 0.0 || b != 0.0) k = (unsigned long long)__double_as_longlong(critical_angle(a, b));
    }
    key[i] = k;
    idx[i] = (uint16_t)i;
  }
  sync();
  // 2. bitonic sort by angle (ties by spin index)
  for (int kk = 2; kk <= P2; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < P2 / 2; t += kT) {
        const int i = (t / j) * 2 * j + t % j, l = i + j;
        const unsigned long long a = key[i], b = key[l];
        const uint16_t ia = idx[i], ib = idx[l];
        const bool gt = a > b || (a == b && ia > ib);
        if (gt == ((i & kk) == 0)) {
          key[i] = b;
          key[l] = a;
          idx[i] = ib;
          idx[l] = ia;
        }
      }
      sync();
    }
  const bool bad = s_bad[slot] != 0;
  int live = 0;  // spins that flip: the keys before the first `never`
  for (int hi = N; live < hi;) {
    const int mid = (live + hi) / 2;
    if (key[mid] < never) live = mid + 1;
    else hi = mid;
  }
  if (bad) live = 0;
  // an axis inside the interval that wraps from the last critical angle through pi
  const double phi0 =
      live > 0 ? 0.5 * (__longlong_as_double((long long)key[live - 1]) + __longlong_as_double((long long)key[0]) + pi) : 0.0;
  const double u0 = cos(phi0), u1 = sin(phi0);
  for (int w = tid / 32; w < 2 * words; w += NW) {
    const int p = 32 * w + lane;
    const bool plus = p < N && (double)x[2 * p] * u0 + (double)x[2 * p + 1] * u1 >= 0.0;
    const unsigned bits = __ballot_sync(0xffffffffu, plus);
    if (lane == 0) reinterpret_cast<unsigned*>(up)[w] = bits;
  }
  sync();
  auto spin = [&](int p) { return ((up[p >> 6] >> (p & 63)) & 1u) ? 1 : -1; };
  // 3. local fields and the energy of the starting pattern
  int part = 0;
  for (int q = tid; q < N; q += kT) {
    int c = 0;
    for (int w = 0; w < words; ++w) {
      const uint64_t dn = ~up[w];  // (padding bits meet no J)
      c += __popcll(__ldg(Jpos + (size_t)w * N + q) & dn) - __popcll(__ldg(Jneg + (size_t)w * N + q) & dn);
    }
    const int f = deg[q] - 2 * c;
    h[q] = f;
    part += spin(q) * f;
  }
  part = __reduce_add_sync(0xffffffffu, part);
  if (lane == 0) red[slot][tid / 32] = part;
  sync();
  int E = 0;
  for (int w = 0; w < NW; ++w) E -= red[slot][w];
  // 4. the sweep (every thread keeps the same E); a spin flips once, from its starting sign
  int best = E, best_i = -1;
  int8_t jn[kXyAhead];
  auto fetch = [&](int i) {
    const int8_t* row = J8 + (size_t)idx[i] * N;  // J symmetric: its column
#pragma unroll
    for (int v = 0; v < kXyAhead; ++v) jn[v] = tid + v * kT < N ? __ldg(row + tid + v * kT) : (int8_t)0;
  };
  if (live > 0) fetch(0);
  for (int i = 0; i < live; ++i) {
    const int p = idx[i], sp = spin(p);
    E += 4 * sp * h[p];
    int8_t jc[kXyAhead];
#pragma unroll
    for (int v = 0; v < kXyAhead; ++v) jc[v] = jn[v];
    if (i + 1 < live) fetch(i + 1);
    sync();  // every thread has read h[p]
#pragma unroll
    for (int v = 0; v < kXyAhead; ++v)
      if (tid + v * kT < N) h[tid + v * kT] -= 2 * sp * jc[v];
    for (int q = tid + kXyAhead * kT; q < N; q += kT) h[q] -= 2 * sp * __ldg(J8 + (size_t)p * N + q);
    sync();
    if ((i + 1 == live || key[i + 1] != key[i]) && E < best) {
      best = E;
      best_i = i;
    }
  }
  // 5. the winning pattern: the starting one with the first best_i + 1 spins flipped
  if (tid == 0) E_out[run] = bad ? (double)NAN : (double)best;
  if (spins_out) {
    for (int i = tid; i <= best_i; i += kT)
      atomicXor(reinterpret_cast<unsigned long long*>(up) + (idx[i] >> 6), 1ull << (idx[i] & 63));
    sync();
    for (int w = tid; w < words; w += kT) spins_out[(size_t)run * words + w] = up[w];
  }
}

// Real couplings.
template <typename T>
__global__ void __launch_bounds__(kXyThreads) round_xy_kernel(const T* __restrict__ X, int N, int P2,
                                                              const double* __restrict__ J64,
                                                              double* __restrict__ E_out,
                                                              uint64_t* __restrict__ spins_out) {
  extern __shared__ __align__(16) unsigned char xy_smem[];
  double* key = reinterpret_cast<double*>(xy_smem);         // P2 critical angles
  double* h = key + P2;                                      // N local fields
  int* idx = reinterpret_cast<int*>(h + N);                  // P2 spin indices
  int8_t* s = reinterpret_cast<int8_t*>(idx + P2);           // N spins
  __shared__ double red[kXyThreads / 32];
  __shared__ double s_phi0;
  __shared__ int s_live, s_bad;
  const int run = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) s_bad = 0;
  __syncthreads();
  const T* x = X + (size_t)run * N * 2;
  const double pi = 3.14159265358979323846;
  // 1. critical angles; spins of zero length never flip (key +inf)
  for (int i = tid; i < P2; i += blockDim.x) {
    double k = INFINITY;
    if (i < N) {
      const double a = (double)x[2 * (size_t)i], b = (double)x[2 * (size_t)i + 1];
      if (!isfinite(a) || !isfinite(b)) s_bad = 1;
      else if (a != 0.0 || b != 0.0) k = critical_angle(a, b);
    }
    key[i] = k;
    idx[i] = i;
  }
  __syncthreads();
  // 2. bitonic sort by angle (ties by spin index)
  for (int kk = 2; kk <= P2; kk <<= 1)
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < P2; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i) {
          const double a = key[i], b = key[l];
          const int ia = idx[i], ib = idx[l];
          const bool gt = a > b || (a == b && ia > ib);
          const bool up = (i & kk) == 0;
          if (gt == up) {
            key[i] = b;
            key[l] = a;
            idx[i] = ib;
            idx[l] = ia;
          }
        }
      }
      __syncthreads();
    }
  if (tid == 0) {
    int live = 0;
    while (live < N && key[live] < INFINITY) ++live;
    if (s_bad) live = 0;
    s_live = live;
    // an axis inside the interval that wraps from the last critical angle through pi
    s_phi0 = live > 0 ? 0.5 * (key[live - 1] + key[0] + pi) : 0.0;
  }
  __syncthreads();
  const int live = s_live;
  const double u0 = cos(s_phi0), u1 = sin(s_phi0);
  for (int p = tid; p < N; p += blockDim.x)
    s[p] = ((double)x[2 * (size_t)p] * u0 + (double)x[2 * (size_t)p + 1] * u1 >= 0.0) ? 1 : -1;
  __syncthreads();
  // 3. local fields and the energy of the starting pattern
  double part = 0.0;
  for (int q = tid; q < N; q += blockDim.x) {
    double f = 0.0;
    for (int p = 0; p < N; ++p) f += J64[(size_t)p * N + q] * (double)s[p];  // J symmetric
    h[q] = f;
    part += (double)s[q] * f;
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((tid & 31) == 0) red[tid >> 5] = part;
  __syncthreads();
  double E = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) E -= red[w];
  // 4. the sweep over the critical angles (every thread keeps the same E)
  double best = E;
  int best_i = -1;
  for (int i = 0; i < live; ++i) {
    const int p = idx[i];
    const double sp = (double)s[p];
    E += 4.0 * sp * h[p];
    __syncthreads();  // every thread has read h[p] and s[p]
    const double ns = -sp;
    if (tid == 0) s[p] = (int8_t)ns;
    for (int q = tid; q < N; q += blockDim.x)
      h[q] += 2.0 * ns * J64[(size_t)p * N + q];
    __syncthreads();
    if ((i + 1 == live || key[i + 1] != key[i]) && E < best) {
      best = E;
      best_i = i;
    }
  }
  // 5. the winning pattern: the starting one with the first best_i + 1 spins flipped
  for (int p = tid; p < N; p += blockDim.x)
    s[p] = ((double)x[2 * (size_t)p] * u0 + (double)x[2 * (size_t)p + 1] * u1 >= 0.0) ? 1 : -1;
  __syncthreads();
  for (int i = tid; i <= best_i; i += blockDim.x) s[idx[i]] = (int8_t)(-s[idx[i]]);
  __syncthreads();
  if (tid == 0) E_out[run] = s_bad ? (double)NAN : best;
  if (spins_out) {
    const int words = (N + 63) / 64;
    for (int wd = tid; wd < words; wd += blockDim.x) {
      uint64_t bits = 0;
      for (int b = 0; b < 64 && wd * 64 + b < N; ++b)
        if (s[wd * 64 + b] > 0) bits |= (uint64_t)1 << b;
      spins_out[(size_t)run * words + wd] = bits;
    }
  }
}

template <typename T>
cudaError_t launch_round_xy_typed(chym_ctx* c, double* d_E, uint64_t* d_spins, cudaStream_t st) {
  int P2 = 1;
  while (P2 < c->N) P2 <<= 1;
  const int R = c->n_runs, W = (c->N + 63) / 64;
  const T* X = (const T*)c->d_X;
  auto go = [&](auto kern, int grid, size_t smem, auto... args) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, kXyThreads, smem, st>>>(args...);
    return cudaGetLastError();
  };
  if (c->kind != CHYM_J_PM1)
    return go(round_xy_kernel<T>, R, (size_t)P2 * (sizeof(double) + sizeof(int)) + (size_t)c->N * (sizeof(double) + 1), X,
              c->N, P2, (const double*)c->d_J64, d_E, d_spins);
  const uint64_t *jp = c->d_Jbits, *jn = c->d_Jbits + (size_t)W * c->N;
  if (c->N <= kXyWarpMaxN)
    return go(round_xy_pm1_kernel<T, 1>, (R + 7) / 8, 8 * xy_run_bytes(c->N, P2), X, c->N, P2, R, (const int8_t*)c->d_J8,
              jp, jn, (const int32_t*)c->d_jdeg, d_E, d_spins);
  return go(round_xy_pm1_kernel<T, 8>, R, xy_run_bytes(c->N, P2), X, c->N, P2, R, (const int8_t*)c->d_J8, jp, jn,
            (const int32_t*)c->d_jdeg, d_E, d_spins);
}

cudaError_t launch_round_xy(chym_ctx* c, double* d_E, uint64_t* d_spins, cudaStream_t st) {
  if (c->n_runs <= 0) return cudaSuccess;
  if (c->prec == CHYM_PREC_FP64) return launch_round_xy_typed<double>(c, d_E, d_spins, st);
  return launch_round_xy_typed<float>(c, d_E, d_spins, st);
}

chym_status check_xy(const chym_ctx* c) {
  if (c->D != 2) return fail(CHYM_EINVAL, "best-axis rounding needs D = 2");
  if (c->N > kXyMaxN) return fail(CHYM_EINVAL, "best-axis rounding supports N <= 4096");
  if (c->prec < 0) return fail(CHYM_ESTATE, "no state: call chym_run first");
  return CHYM_OK;
}

}  // namespace
}  // namespace chym

using namespace chym;

extern "C" {

CHYM_API chym_status chym_readout_xy_device(chym_ctx* c, double* d_E, uint64_t* d_spins, void* stream) {
  chym::TraceRange trace_("chym_readout_xy_device");
  if (!c || !d_E) return fail(CHYM_EINVAL, "NULL argument");
  const chym_status ok = check_xy(c);
  if (ok != CHYM_OK) return ok;
  CHYM_CUDA_TRY(launch_round_xy(c, d_E, d_spins, (cudaStream_t)stream));
  return CHYM_OK;
}

CHYM_API chym_status chym_readout_xy(chym_ctx* c, double* E_out, uint64_t* spins_out, void* stream) {
  chym::TraceRange trace_("chym_readout_xy");
  if (!c || !E_out) return fail(CHYM_EINVAL, "NULL argument");
  const chym_status ok = check_xy(c);
  if (ok != CHYM_OK) return ok;
  cudaStream_t st = (cudaStream_t)stream;
  // the context's energy buffers hold the result; the cached Ising energies are gone
  CHYM_CUDA_TRY(launch_round_xy(c, c->d_E, c->d_spins, st));
  c->have_energy = false;
  CHYM_CUDA_TRY(cudaMemcpyAsync(E_out, c->d_E, sizeof(double) * c->n_runs, cudaMemcpyDeviceToHost, st));
  if (spins_out) {
    const size_t words = (size_t)(c->N + 63) / 64;
    CHYM_CUDA_TRY(cudaMemcpyAsync(spins_out, c->d_spins, sizeof(uint64_t) * c->n_runs * words,
                                  cudaMemcpyDeviceToHost, st));
  }
  CHYM_CUDA_TRY(cudaStreamSynchronize(st));
  return CHYM_OK;
}

}  // extern "C"
