// chym_simt.cu -- SIMT step kernels (FP64 oracle-comparison mode and the plain
// FP32 form) and the initial-state kernel.
//
// Every step kernel owns RC runs per CTA for the whole launch and keeps their state
// in shared memory across all steps.  A sparse J (at most N^2 / 16 nonzeros) is read
// as compressed rows, so the product costs 2 nnz D flops per run and step rather
// than 2 N^2 D.  Per step:
//   phase A  y_{p,mu} = sum_q J_pq x_{q,mu}  (C = J_N (x) 1_D, Eq. 1);
//   phase B  x <- x + dt [(h-1) x - kappa x^3 - gamma x |x_p|^2 + eps alpha_mu y]
//            + sigma sqrt(dt) xi  with xi from Philox4x32-10 + Box-Muller.
// FP32 runs on the register-tiled kernel (step_simt_tiled_kernel, below), whose
// threads each own 4 spins x RB runs through both phases, or, for a sparse J whose run
// groups do not fit it, on step_csr_kernel; FP64 runs on step_f64_kernel, with the noise
// drawn ahead by warps of its own.  A dense FP32 J and FP64 runs whose buffers do not fit
// these run on the per-spin kernel (step_simt_kernel), whose
// threads each take one (spin, run group) in phase A and one (spin, run) in phase B,
// with J staged in shared memory when it fits and read through L1/L2 otherwise.
#include <algorithm>

#include "chym_internal.cuh"

namespace chym {
namespace {

template <typename T>
struct SimtTraits;
template <>
struct SimtTraits<double> {
  static constexpr int RB = 1;
};
template <>
struct SimtTraits<float> {
  static constexpr int RB = 4;
};

// Normal numbers of spin p for components 0..D-1 at step k (tag 0 or 1).
// For D <= 2 the 4/D spins with the same p / (4/D) share one Philox block: spin p
// takes the normals (p % (4/D)) * D .. + D - 1 of it (one Box-Muller pair).
template <typename T, int D>
__device__ __forceinline__ void spin_normals(uint64_t seed, uint32_t tag, uint64_t k, int p,
                                             T scale, T z[D]) {
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  if constexpr (D <= 2) {
    constexpr uint32_t per = 4u / D;
    const uint4 w = philox4x32_10(noise_counter((uint32_t)p / per, 0u, tag, k), k0, k1);
    const uint32_t j0 = ((uint32_t)p % per) * D;  // first normal of this spin in the block
    const uint32_t wr = j0 >= 2u ? w.z : w.x, wa = j0 >= 2u ? w.w : w.y;
    T c, sn;
    if constexpr (sizeof(T) == 8) {
      double d0, d1;
      box_muller_f64(wr, wa, d0, d1);
      c = (T)(d0 * (double)scale);
      sn = (T)(d1 * (double)scale);
    } else {
      box_muller_f32(wr, wa, (float)scale, c, sn);
    }
    z[0] = (j0 & 1u) ? sn : c;
    if constexpr (D == 2) z[1] = sn;
  } else {
#pragma unroll
  for (int blk = 0; blk < (D + 3) / 4; ++blk) {
    const uint4 w = philox4x32_10(noise_counter((uint32_t)p, (uint32_t)blk, tag, k), k0, k1);
    T zz[4];
    if constexpr (sizeof(T) == 8) {
      double d[4];
      box_muller_f64(w.x, w.y, d[0], d[1]);
      if (D - 4 * blk > 2) box_muller_f64(w.z, w.w, d[2], d[3]);
      else d[2] = d[3] = 0.0;
#pragma unroll
      for (int j = 0; j < 4; ++j) zz[j] = (T)(d[j] * (double)scale);
    } else {
      box_muller_f32(w.x, w.y, (float)scale, zz[0], zz[1]);
      if (D - 4 * blk > 2) box_muller_f32(w.z, w.w, (float)scale, zz[2], zz[3]);
      else zz[2] = zz[3] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (4 * blk + j < D) z[4 * blk + j] = zz[j];
  }
  }
}

// FP32 Box-Muller on the SFU approximations with denormals flushed (no argument or
// result of the transform is denormal): u = (w + 1/2) 2^-32, r = scale sqrt(-2 ln u_r),
// angle 2 pi u_a - pi, and the pair negated back (cos t = -cos(t - pi), likewise sin).
__device__ __forceinline__ void box_muller_sfu(uint32_t wr, uint32_t wa, float scale, float& z0,
                                               float& z1) {
  const float ur = __fmaf_rn((float)wr, 2.3283064365386963e-10f, 1.1641532182693481e-10f);
  const float ua = __fmaf_rn((float)wa, 2.3283064365386963e-10f, 1.1641532182693481e-10f);
  float l2, r, s, c;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l2) : "f"(ur));
  const float r2 = l2 * (-1.3862943611198906f * scale * scale);  // -2 ln 2 scale^2 log2 u
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(r2));
  const float t = __fmaf_rn(ua, 6.2831853071795865f, -3.1415926535897932f);
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(t));
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(t));
  z0 = -r * c;
  z1 = -r * s;
}

// Philox4x32-10 with the ten round keys precomputed (two rounds per uint4).
__device__ __forceinline__ uint4 philox_rounds(uint4 c, const uint4* rk) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const uint4 kk = rk[i];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t k0 = h ? kk.z : kk.x, k1 = h ? kk.w : kk.y;
      const uint64_t p0 = (uint64_t)kPhiloxM0 * c.x, p1 = (uint64_t)kPhiloxM1 * c.z;
      c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k0, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k1, (uint32_t)p0);
    }
  }
  return c;
}

template <typename T, int D>
__global__ void init_kernel(T* __restrict__ X, const uint64_t* __restrict__ seeds, int N,
                            int n_runs, T init_std) {
  const int64_t pairs = (int64_t)N * n_runs;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < pairs;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int run = (int)(s / N), p = (int)(s % N);
    T z[D];
    spin_normals<T, D>(seeds[run], 1u, 0ull, p, init_std, z);
#pragma unroll
    for (int mu = 0; mu < D; ++mu) X[s * D + mu] = z[mu];
  }
}

// Compressed rows of a sparse J: row p holds the nonzeros rp[p] .. rp[p + 1] - 1.
template <typename T>
struct CsrRows {
  const int32_t* rp;
  const int32_t* ci;
  const T* cv;
};

template <typename T, int D, bool J_SMEM, bool CSR>
__global__ void __launch_bounds__(512) step_simt_kernel(const T* __restrict__ Jg,
                                                        T* __restrict__ Xg,
                                                        const double* __restrict__ hg,
                                                        const uint64_t* __restrict__ seeds,
                                                        StepConsts sc, int RC, CsrRows<T> csr) {
  constexpr int RB = CSR ? 1 : SimtTraits<T>::RB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = sc.N;
  T* Js = reinterpret_cast<T*>(smem_raw);
  T* Xs = J_SMEM ? Js + (size_t)N * N : Js;
  T* Ys = Xs + (size_t)RC * N * D;
  const int run0 = blockIdx.x * RC;
  const int nr = min(RC, sc.n_runs - run0);
  const int tid = threadIdx.x, nt = blockDim.x;

  if (J_SMEM)
    for (int i = tid; i < N * N; i += nt) Js[i] = Jg[i];
  for (int i = tid; i < RC * N * D; i += nt)
    Xs[i] = (i < nr * N * D) ? Xg[(size_t)run0 * N * D + i] : T(0);
  __syncthreads();
  const T* Jsrc = J_SMEM ? Js : Jg;

  const T dt = (T)sc.dt, gamma = (T)sc.gamma, kappa = (T)sc.kappa;
  const T inv_ramp = sc.sched_kind == 1 ? T(1) / (T)(sc.k_total - sc.k_anneal) : T(0);
  const int n_groups = RC / RB;
  for (int64_t k = sc.k0; k < sc.k0 + sc.steps; ++k) {
    // ---- phase A: coupling product, RB runs per thread ----
    for (int slot = tid; slot < N * n_groups; slot += nt) {
      const int p = slot % N, g = slot / N;
      T acc[RB][D];
#pragma unroll
      for (int b = 0; b < RB; ++b)
#pragma unroll
        for (int mu = 0; mu < D; ++mu) acc[b][mu] = T(0);
      const T* xg = Xs + (size_t)(g * RB) * N * D;
      if constexpr (CSR) {
        const int e1 = __ldg(csr.rp + p + 1);
        for (int e = __ldg(csr.rp + p); e < e1; ++e) {
          const T j = __ldg(csr.cv + e);
          const int q = __ldg(csr.ci + e);
#pragma unroll
          for (int b = 0; b < RB; ++b)
#pragma unroll
            for (int mu = 0; mu < D; ++mu) acc[b][mu] = fma(j, xg[((size_t)b * N + q) * D + mu], acc[b][mu]);
        }
      } else {
        for (int q = 0; q < N; ++q) {
          const T j = J_SMEM ? Jsrc[q * N + p] : __ldg(Jsrc + (size_t)q * N + p);
#pragma unroll
          for (int b = 0; b < RB; ++b)
#pragma unroll
            for (int mu = 0; mu < D; ++mu) acc[b][mu] = fma(j, xg[((size_t)b * N + q) * D + mu], acc[b][mu]);
        }
      }
#pragma unroll
      for (int b = 0; b < RB; ++b)
#pragma unroll
        for (int mu = 0; mu < D; ++mu) Ys[((size_t)(g * RB + b) * N + p) * D + mu] = acc[b][mu];
    }
    __syncthreads();
    // ---- phase B: local drift, annealing and noise (at each run's local step) ----
    for (int s = tid; s < nr * N; s += nt) {
      const int rl = s / N, p = s % N, run = run0 + rl;
      const int64_t kl = k - sc.koff[run];
      T ramp = T(1);  // alpha_mu(kl) for mu >= 1; mu = 0 keeps alpha = 1
      if (sc.sched_kind == 1 && kl >= sc.k_anneal)
        ramp = kl >= sc.k_total ? T(0) : T(1) - (T)(kl - sc.k_anneal) * inv_ramp;
      const T wp = sc.w ? (T)sc.w[p] : T(1);  // this spin's coupling weight
      T ea[D];
#pragma unroll
      for (int mu = 0; mu < D; ++mu) ea[mu] = (T)sc.eps * wp * (mu == 0 ? T(1) : ramp);
      const T hm1 = (T)(hg[sc.hidx[run]] - 1.0);
      T* x = Xs + (size_t)s * D;
      const T* y = Ys + (size_t)s * D;
      T n2 = T(0);
#pragma unroll
      for (int mu = 0; mu < D; ++mu) n2 = fma(x[mu], x[mu], n2);
      T z[D];
      spin_normals<T, D>(seeds[run], 0u, (uint64_t)kl, p, (T)sc.noise_scale, z);
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        const T xm = x[mu];
        const T f = hm1 * xm - kappa * xm * xm * xm - gamma * xm * n2 + ea[mu] * y[mu];
        x[mu] = xm + dt * f + z[mu];
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < nr * N * D; i += nt) Xg[(size_t)run0 * N * D + i] = Xs[i];
}

// ---------------------------------------------------------------------------
// FP64 form.  The FP64 units take 16 cycles for a warp's instruction, so what counts is full
// warps and several of them under way: the state's warps take one (run, spin, component)
// per thread, and the noise's warps draw the next step's Box-Muller pairs, one per thread,
// at the same time.  State and noise are double buffered, one barrier a step.  N = 20, D = 3,
// 256 runs: 3.9 us a step (8.9 with one thread per (run, spin) through product, noise and
// update, 20 of 64 threads busy).  Every value is formed by the same operations as there.
template <int D, bool J_SMEM, bool CSR>
__global__ void __launch_bounds__(512) step_f64_kernel(const double* __restrict__ Jg, double* __restrict__ Xg,
                                                       const double* __restrict__ hg,
                                                       const uint64_t* __restrict__ seeds, StepConsts sc, int RC,
                                                       int state_warps, CsrRows<double> csr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = sc.N, size = RC * N * D;
  double* Js = reinterpret_cast<double*>(smem_raw);
  double* Xs = J_SMEM ? Js + (size_t)N * N : Js;  // two state buffers, two noise buffers
  double* Zs = Xs + 2 * (size_t)size;
  const int run0 = blockIdx.x * RC;
  const int nr = min(RC, sc.n_runs - run0), used = nr * N * D;
  const int tid = threadIdx.x, nt = blockDim.x, ns = 32 * state_warps;
  if (J_SMEM)
    for (int i = tid; i < N * N; i += nt) Js[i] = Jg[i];
  for (int i = tid; i < used; i += nt) Xs[i] = Xg[(size_t)run0 * N * D + i];
  const double* Jsrc = J_SMEM ? Js : Jg;
  // the pairs of a run: a spin's pairs (D >= 3: ceil(D / 2)), or for D <= 2 the pairs of the
  // blocks that 4 / D spins share
  constexpr int kPairs = (D + 1) / 2;  // per spin, D >= 3
  const int pairs = D >= 3 ? N * kPairs : (N * D + 1) / 2;
  auto draw = [&](int64_t k, double* Z, int first, int stride) {
    for (int t = first; t < nr * pairs; t += stride) {
      const int r = t / pairs, j = t % pairs, run = run0 + r;
      const uint64_t kl = (uint64_t)(k - sc.koff[run]), seed = seeds[run];
      uint32_t ctr, blk;
      int half, at;  // half: pair of the block; at: first value in the run's N D
      if constexpr (D >= 3) {
        const int p = j / kPairs, m = j % kPairs;
        ctr = (uint32_t)p;
        blk = (uint32_t)(m / 2);
        half = m % 2;
        at = p * D + 2 * m;
      } else {
        ctr = (uint32_t)(j / 2);
        blk = 0u;
        half = j % 2;
        at = 2 * j;
      }
      const uint4 w = philox4x32_10(noise_counter(ctr, blk, 0u, kl), (uint32_t)seed, (uint32_t)(seed >> 32));
      double z0, z1;
      box_muller_f64(half ? w.z : w.x, half ? w.w : w.y, z0, z1);
      double* z = Z + (size_t)r * N * D + at;
      z[0] = z0 * sc.noise_scale;
      if (D >= 3 ? at % D + 1 < D : at + 1 < N * D) z[1] = z1 * sc.noise_scale;
    }
  };
  draw(sc.k0, Zs, tid, nt);
  __syncthreads();
  const double dt = sc.dt, gamma = sc.gamma, kappa = sc.kappa;
  const double inv_ramp = sc.sched_kind == 1 ? 1.0 / (double)(sc.k_total - sc.k_anneal) : 0.0;
  int cur = 0;
  for (int64_t k = sc.k0; k < sc.k0 + sc.steps; ++k, cur ^= 1) {
    const double* X = Xs + (size_t)cur * size;
    const double* Z = Zs + (size_t)cur * size;
    if (tid >= ns) {
      if (k + 1 < sc.k0 + sc.steps) draw(k + 1, Zs + (size_t)(cur ^ 1) * size, tid - ns, nt - ns);
    } else {
      double* Xn = Xs + (size_t)(cur ^ 1) * size;
      for (int i = tid; i < used; i += ns) {
        const int mu = i % D, p = i / D % N, r = i / (N * D), run = run0 + r;
        const double* xr = X + (size_t)r * N * D;
        double y = 0.0;
        if constexpr (CSR) {
          const int e1 = __ldg(csr.rp + p + 1);
          for (int e = __ldg(csr.rp + p); e < e1; ++e) y = fma(__ldg(csr.cv + e), xr[__ldg(csr.ci + e) * D + mu], y);
        } else {
#pragma unroll 4
          for (int q = 0; q < N; ++q) y = fma(J_SMEM ? Jsrc[q * N + p] : __ldg(Jsrc + (size_t)q * N + p), xr[q * D + mu], y);
        }
        const int64_t kl = k - sc.koff[run];
        double ramp = 1.0;  // alpha_mu(kl) for mu >= 1; mu = 0 keeps alpha = 1
        if (mu > 0 && sc.sched_kind == 1 && kl >= sc.k_anneal)
          ramp = kl >= sc.k_total ? 0.0 : 1.0 - (double)(kl - sc.k_anneal) * inv_ramp;
        const double wp = sc.w ? sc.w[p] : 1.0;  // this spin's coupling weight
        const double hm1 = hg[sc.hidx[run]] - 1.0;
        double n2 = 0.0;
#pragma unroll
        for (int m = 0; m < D; ++m) n2 = fma(xr[p * D + m], xr[p * D + m], n2);
        const double xm = xr[p * D + mu];
        const double f = hm1 * xm - kappa * xm * xm * xm - gamma * xm * n2 + sc.eps * wp * ramp * y;
        Xn[i] = xm + dt * f + Z[i];
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < used; i += nt) Xg[(size_t)run0 * N * D + i] = Xs[(size_t)cur * size + i];
}

// Launch of the FP64 form; InvalidConfiguration when a run's buffers do not fit its shared
// memory (the caller then takes the per-spin kernel, which holds half as much).
template <int D>
cudaError_t launch_f64(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  const int N = c->N;
  const bool csr = c->sparse;
  const size_t j_bytes = (size_t)N * N * sizeof(double), per_run = (size_t)4 * N * D * sizeof(double);
  const bool j_smem = !csr && j_bytes <= kSimtSmemBudget / 2;
  const size_t avail = kSimtSmemBudget - (j_smem ? j_bytes : 0);
  if (per_run > avail) return cudaErrorInvalidConfiguration;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  // as many runs a CTA as give every SM one, within shared memory and one state value a thread
  // of 512 where that suffices
  const int fit = (int)std::min<size_t>(avail / per_run, 64);
  int RC = std::max(1, std::min(fit, (sc.n_runs + sms - 1) / sms));
  while (RC > 1 && RC * N * D > 512) --RC;
  // warps in proportion to the FP64 work: a state value costs a row of J and about 12
  // operations, a pair of normals about 70 (logarithm, square root, sine and cosine)
  const double row = csr ? (double)c->nnz / N : (double)N;
  const int values = RC * N * D, pairs = RC * (D >= 3 ? N * ((D + 1) / 2) : (N * D + 1) / 2);
  const double ws = values * (row + 12.0), wn = pairs * 70.0;
  const int want_s = (values + 31) / 32, want_n = (pairs + 31) / 32;
  int state_warps = want_s, noise_warps = want_n;
  if (want_s + want_n > 16) {
    state_warps = std::min(want_s, std::max(1, std::min(15, (int)(16.0 * ws / (ws + wn) + 0.5))));
    noise_warps = std::min(want_n, 16 - state_warps);
  }
  const size_t smem = (j_smem ? j_bytes : 0) + (size_t)RC * per_run;
  const CsrRows<double> rows{c->d_rp, c->d_ci, c->d_cv64};
  auto kern = csr ? step_f64_kernel<D, false, true> : j_smem ? step_f64_kernel<D, true, false> : step_f64_kernel<D, false, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(sc.n_runs + RC - 1) / RC, 32 * (state_warps + noise_warps), smem, st>>>(
      c->d_J64, (double*)c->d_X, c->d_h, c->d_seeds, sc, RC, state_warps, rows);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Register-tiled FP32 form (the plain FP32 form: dense J, or the nonzeros of a sparse J).
// The CTA keeps its RC runs in shared memory as Xs[q][r][DP] (spin-major, the runs of
// one spin contiguous, components padded to DP).  Thread (tp, rg) owns the tile of
// spins 4 tp .. 4 tp + 3 and runs RB rg .. RB rg + RB - 1.  Dense J: per q it loads the
// four couplings J_{q, 4tp..4tp+3} (J symmetric, rows zero padded to NP; one 16-byte
// read-only load that stays in L1) and the RB x DP state values of its runs (16-byte
// shared loads) for 4 RB D FMAs.  Sparse J: per nonzero J_pq of each of its spins the
// same RB x DP state values for RB D FMAs.  The thread then updates its own tile, so the
// coupling product never leaves registers, and its noise follows the counter layout of
// the other kernels; a tile of four spins holds whole Philox blocks for D <= 2.
// (J in shared memory instead of L1 measured slower: it leaves fewer CTAs per SM.)
// RB shrinks (by SH halvings) while the threads would not fill the SMs: the work per thread is
// a long chain, and 4096 runs of N = 100, D = 4 at RB = 4 left 5 warps on an SM.
template <int D, int SH>
struct TileCfg {
  static constexpr int DP = D == 3 ? 4 : (D > 4 ? 8 : D);
  static constexpr int RB = (D == 1 ? 8 : D <= 4 ? 4 : 2) >> SH;
  static_assert(RB * DP <= 2 || (RB * DP) % 4 == 0, "state loads are 4, 8 or 16k bytes");
};
constexpr int tile_halvings(int D) { return D <= 4 ? 2 : 1; }

// The n = RB DP consecutive state values of one spin and run group (n = 1, 2 or 4k).
template <int n>
__device__ __forceinline__ void load_x(const float* src, float (&xv)[n]) {
  if constexpr (n == 1) {
    xv[0] = src[0];
  } else if constexpr (n == 2) {
    const float2 t = *reinterpret_cast<const float2*>(src);
    xv[0] = t.x;
    xv[1] = t.y;
  } else {
#pragma unroll
    for (int v = 0; v < n / 4; ++v) {
      const float4 t = reinterpret_cast<const float4*>(src)[v];
      xv[4 * v] = t.x;
      xv[4 * v + 1] = t.y;
      xv[4 * v + 2] = t.z;
      xv[4 * v + 3] = t.w;
    }
  }
}

template <int D, bool CSR, int SH>
__global__ void __launch_bounds__(512) step_simt_tiled_kernel(const float* __restrict__ Jp,
                                                              float* __restrict__ Xg,
                                                              const double* __restrict__ hg,
                                                              const uint64_t* __restrict__ seeds,
                                                              StepConsts sc, int RC, int NP,
                                                              CsrRows<float> csr) {
  using Cfg = TileCfg<D, SH>;
  constexpr int DP = Cfg::DP, RB = Cfg::RB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = sc.N;
  float* Xs = reinterpret_cast<float*>(smem_raw);                     // NP x RC x DP
  uint4* s_rk = reinterpret_cast<uint4*>(Xs + (size_t)NP * RC * DP);  // RC x 5 round keys
  int64_t* s_koff = reinterpret_cast<int64_t*>(s_rk + (size_t)RC * 5);
  float* s_hm1 = reinterpret_cast<float*>(s_koff + RC);
  const int run0 = blockIdx.x * RC;
  const int nr = min(RC, sc.n_runs - run0);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int tiles_p = NP / 4;
  const int tp = tid % tiles_p, rg = tid / tiles_p;
  const int p0 = 4 * tp, r0 = RB * rg;
  const bool active = rg < RC / RB;

  for (int i = tid; i < NP * RC * DP; i += nt) {
    const int mu = i % DP, r = (i / DP) % RC, p = i / (DP * RC);
    Xs[i] = (mu < D && p < N && r < nr) ? Xg[((size_t)(run0 + r) * N + p) * D + mu] : 0.f;
  }
  for (int r = tid; r < RC; r += nt) {
    uint32_t k0 = 0u, k1 = 0u;
    float hm1 = 0.f;
    int64_t ko = 0;
    if (r < nr) {
      const int run = run0 + r;
      k0 = (uint32_t)seeds[run];
      k1 = (uint32_t)(seeds[run] >> 32);
      hm1 = (float)(hg[sc.hidx[run]] - 1.0);
      ko = sc.koff[run];
    }
    for (int i = 0; i < 5; ++i)  // Weyl key schedule: round j uses key + j (W0, W1)
      s_rk[r * 5 + i] = make_uint4(k0 + (2u * i) * kPhiloxW0, k1 + (2u * i) * kPhiloxW1,
                                   k0 + (2u * i + 1u) * kPhiloxW0, k1 + (2u * i + 1u) * kPhiloxW1);
    s_koff[r] = ko;
    s_hm1[r] = hm1;
  }
  __syncthreads();

  const float dt = (float)sc.dt, gamma = (float)sc.gamma, kappa = (float)sc.kappa;
  const float nscale = (float)sc.noise_scale;
  const float inv_ramp = sc.sched_kind == 1 ? 1.f / (float)(sc.k_total - sc.k_anneal) : 0.f;
  float edt[4];  // dt eps w_p of the tile's spins
  int e_beg[4], e_end[4];  // the tile's compressed rows
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int p = p0 + i;
    edt[i] = (float)(sc.dt * sc.eps) * ((sc.w && p < N) ? (float)sc.w[p] : 1.f);
    e_beg[i] = e_end[i] = 0;
    if (CSR && p < N) {
      e_beg[i] = __ldg(csr.rp + p);
      e_end[i] = __ldg(csr.rp + p + 1);
    }
  }
  const float* xcol = Xs + (size_t)r0 * DP;
  for (int64_t k = sc.k0; k < sc.k0 + sc.steps; ++k) {
    float acc[4][RB][D];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int b = 0; b < RB; ++b)
#pragma unroll
        for (int mu = 0; mu < D; ++mu) acc[i][b][mu] = 0.f;
    // ---- coupling product y = (J (x) 1_D) x of the tile, in registers ----
    if (active) {
      if constexpr (CSR) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          for (int e = e_beg[i]; e < e_end[i]; ++e) {
            const float j = __ldg(csr.cv + e);
            float xv[RB * DP];
            load_x<RB * DP>(xcol + (size_t)__ldg(csr.ci + e) * RC * DP, xv);
#pragma unroll
            for (int b = 0; b < RB; ++b)
#pragma unroll
              for (int mu = 0; mu < D; ++mu) acc[i][b][mu] = fmaf(j, xv[b * DP + mu], acc[i][b][mu]);
          }
        }
      } else {
#pragma unroll 2
        for (int q = 0; q < N; ++q) {
          const float4 jv = __ldg(reinterpret_cast<const float4*>(Jp + (size_t)q * NP + p0));
          const float jq[4] = {jv.x, jv.y, jv.z, jv.w};
          float xv[RB * DP];
          load_x<RB * DP>(xcol + (size_t)q * RC * DP, xv);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int b = 0; b < RB; ++b)
#pragma unroll
              for (int mu = 0; mu < D; ++mu) acc[i][b][mu] = fmaf(jq[i], xv[b * DP + mu], acc[i][b][mu]);
        }
      }
    }
    __syncthreads();  // every read of the old state precedes the first update
    // ---- drift, annealing scale and noise of the tile ----
    if (active) {
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        const int r = r0 + b;
        if (r >= nr) continue;
        const int64_t kl = k - s_koff[r];
        float ramp = 1.f;  // alpha_mu(kl) for mu >= 1
        if (sc.sched_kind == 1 && kl >= sc.k_anneal)
          ramp = kl >= sc.k_total ? 0.f : fmaxf(0.f, 1.f - (float)(kl - sc.k_anneal) * inv_ramp);
        const float a1 = 1.f + dt * s_hm1[r];
        const uint4* rk = s_rk + r * 5;
        float z[4][D];
        if constexpr (D == 1) {
          const uint4 w = philox_rounds(noise_counter((uint32_t)tp, 0u, 0u, (uint64_t)kl), rk);
          box_muller_sfu(w.x, w.y, nscale, z[0][0], z[1][0]);
          box_muller_sfu(w.z, w.w, nscale, z[2][0], z[3][0]);
        } else if constexpr (D == 2) {
#pragma unroll
          for (int hb = 0; hb < 2; ++hb) {
            const uint4 w = philox_rounds(noise_counter((uint32_t)(2 * tp + hb), 0u, 0u, (uint64_t)kl), rk);
            box_muller_sfu(w.x, w.y, nscale, z[2 * hb][0], z[2 * hb][1]);
            box_muller_sfu(w.z, w.w, nscale, z[2 * hb + 1][0], z[2 * hb + 1][1]);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int blk = 0; blk < (D + 3) / 4; ++blk) {
              const uint4 w = philox_rounds(noise_counter((uint32_t)(p0 + i), (uint32_t)blk, 0u, (uint64_t)kl), rk);
              float zz[4];
              box_muller_sfu(w.x, w.y, nscale, zz[0], zz[1]);
              if (D - 4 * blk > 2) box_muller_sfu(w.z, w.w, nscale, zz[2], zz[3]);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (4 * blk + j < D) z[i][4 * blk + j] = zz[j];
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int p = p0 + i;
          if (p >= N) continue;
          float* x = Xs + ((size_t)p * RC + r) * DP;
          float xv[D];
          float n2 = 0.f;
#pragma unroll
          for (int mu = 0; mu < D; ++mu) {
            xv[mu] = x[mu];
            n2 = fmaf(xv[mu], xv[mu], n2);
          }
#pragma unroll
          for (int mu = 0; mu < D; ++mu) {
            const float xm = xv[mu];
            // x + dt [(h-1) x - kappa x^3 - gamma x |x_p|^2 + eps w_p alpha_mu y] + noise
            const float lin = a1 - dt * (kappa * xm * xm + gamma * n2);
            const float ea = mu == 0 ? edt[i] : edt[i] * ramp;
            x[mu] = fmaf(xm, lin, fmaf(ea, acc[i][b][mu], z[i][mu]));
          }
        }
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < nr * N * D; i += nt) {
    const int mu = i % D, p = (i / D) % N, r = i / (D * N);
    Xg[(size_t)run0 * N * D + i] = Xs[((size_t)p * RC + r) * DP + mu];
  }
}

template <int D, bool CSR, int SH>
cudaError_t launch_simt_tiles(chym_ctx* c, const StepConsts& sc, int sms, size_t per_run, cudaStream_t st) {
  constexpr int RB = TileCfg<D, SH>::RB;
  const int NP = c->j32p_ld, tiles = NP / 4;
  // Fewer threads than kTileWarps warps an SM: halve the runs per thread.
  constexpr int kTileWarps = 10;
  if constexpr (SH < tile_halvings(D))
    if ((long long)tiles * ((sc.n_runs + RB - 1) / RB) < (long long)sms * 32 * kTileWarps)
      return launch_simt_tiles<D, CSR, SH + 1>(c, sc, sms, per_run, st);
  int RC = (int)std::min<size_t>(kSimtSmemBudget / per_run, (size_t)std::max(1, 512 / tiles) * RB);
  RC = RC / RB * RB;
  if (RC < RB || tiles * (RC / RB) > 512) return cudaErrorInvalidConfiguration;
  // CTAs of equal size: the runs of an SM over as few of them as that takes
  const int share = (sc.n_runs + sms - 1) / sms, per_sm = (share + RC - 1) / RC;
  RC = std::min(RC, ((share + per_sm - 1) / per_sm + RB - 1) / RB * RB);
  const int threads = std::max(32, (tiles * (RC / RB) + 31) / 32 * 32);
  const size_t smem = (size_t)RC * per_run;
  const int grid = (sc.n_runs + RC - 1) / RC;
  const CsrRows<float> rows{c->d_rp, c->d_ci, c->d_cv32};
  auto kern = step_simt_tiled_kernel<D, CSR, SH>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, threads, smem, st>>>(c->d_J32p, (float*)c->d_X, c->d_h, c->d_seeds, sc, RC, NP, rows);
  return cudaGetLastError();
}

// Launch of the tiled FP32 form; InvalidConfiguration when a run group does not fit its
// shared memory (the caller then takes another kernel).
template <int D, bool CSR>
cudaError_t launch_simt_tiled(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  using Cfg = TileCfg<D, 0>;
  const int N = c->N, NP = c->j32p_ld;
  if (!CSR && (!c->d_J32p || NP < N)) return cudaErrorInvalidConfiguration;
  const size_t per_run = (size_t)NP * Cfg::DP * sizeof(float) + 5 * sizeof(uint4) + sizeof(int64_t) + sizeof(float);
  if (Cfg::RB * per_run > kSimtSmemBudget || NP / 4 > 512) return cudaErrorInvalidConfiguration;
  // sparse J with long rows of state (N of about 1000 and more): the compressed-row kernel,
  // whose 1024-thread CTAs measured faster there than CTAs of a few run groups
  if (CSR && kSimtSmemBudget / per_run < (size_t)(4 * Cfg::RB)) return cudaErrorInvalidConfiguration;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  return launch_simt_tiles<D, CSR, 0>(c, sc, sms, per_run, st);
}

// ---------------------------------------------------------------------------
// FP32 form over the compressed rows of a large sparse J (a run group does not fit the tiled
// kernel).  A thread owns its spins for the whole launch, with the first kHeld nonzeros of
// their rows in registers, and takes every run of the CTA through product, noise and update
// in one pass; the state is double buffered, one barrier a step.  What depends on the run
// and step only (the first two Philox rounds as far as they do, round keys, pump, annealing
// scale) is formed once per run and step and read from shared memory.  (Two passes with the
// product through shared memory and all of that per spin: ladder N = 2048, D = 3, 2048 runs,
// 63 us a step.)
struct __align__(16) CsrRun {
  uint4 r12[2];  // per Philox block, see csr_rounds12
  uint4 rk[4];   // keys of rounds 3..10
  float hm1, ramp;
};
// Philox counter (p, blk, k_lo, k_hi), key (k0, k1), k' the round-2 key: what rounds 1 and 2
// leave that does not depend on p:
//   x = k_hi ^ k1, y = lo(M1 k_lo) ^ k0', z = hi(M0 c) ^ k1', w = lo(M0 c) with
//   c = hi(M1 k_lo) ^ blk ^ k0.
__device__ __forceinline__ uint4 csr_rounds12(uint32_t blk, uint64_t k, uint32_t k0, uint32_t k1) {
  const uint64_t p1 = (uint64_t)kPhiloxM1 * (uint32_t)k;
  const uint64_t p0 = (uint64_t)kPhiloxM0 * ((uint32_t)(p1 >> 32) ^ blk ^ k0);
  return make_uint4((uint32_t)(k >> 32) ^ k1, (uint32_t)p1 ^ (k0 + kPhiloxW0), (uint32_t)(p0 >> 32) ^ (k1 + kPhiloxW1),
                    (uint32_t)p0);
}

template <int D>
__global__ void __launch_bounds__(D <= 4 ? 1024 : 512) step_csr_kernel(float* __restrict__ Xg,
                                                                       const double* __restrict__ hg,
                                                                       const uint64_t* __restrict__ seeds,
                                                                       StepConsts sc, int RC, CsrRows<float> csr) {
  constexpr int kHeld = 3, NB = (D + 3) / 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = sc.N, tid = threadIdx.x, nt = blockDim.x;
  CsrRun* s_run = reinterpret_cast<CsrRun*>(smem_raw);  // 2 RC: by step parity
  float* Xs = reinterpret_cast<float*>(s_run + 2 * RC);  // 2 x RC x N x D
  const int run0 = blockIdx.x * RC;
  const int nr = min(RC, sc.n_runs - run0), used = nr * N * D;
  const size_t buf = (size_t)RC * N * D;
  for (int i = tid; i < used; i += nt) Xs[i] = Xg[(size_t)run0 * N * D + i];
  // run r's constants at step k, by thread r (its keys stay in registers)
  uint32_t k0 = 0u, k1 = 0u;
  int64_t koff = 0;
  float hm1 = 0.f;
  if (tid < nr) {
    const uint64_t seed = seeds[run0 + tid];
    k0 = (uint32_t)seed;
    k1 = (uint32_t)(seed >> 32);
    koff = sc.koff[run0 + tid];
    hm1 = (float)(hg[sc.hidx[run0 + tid]] - 1.0);
  }
  const float inv_ramp = sc.sched_kind == 1 ? 1.f / (float)(sc.k_total - sc.k_anneal) : 0.f;
  auto put_run = [&](int64_t k, bool keys) {
    if (tid >= nr) return;
    CsrRun& o = s_run[(k & 1) * RC + tid];
    const int64_t kl = k - koff;
#pragma unroll
    for (int b = 0; b < NB; ++b) o.r12[b] = csr_rounds12((uint32_t)b, (uint64_t)kl, k0, k1);
    float ramp = 1.f;  // alpha_mu(kl) for mu >= 1
    if (sc.sched_kind == 1 && kl >= sc.k_anneal) ramp = kl >= sc.k_total ? 0.f : 1.f - (float)(kl - sc.k_anneal) * inv_ramp;
    o.ramp = ramp;
    if (keys) {
      o.hm1 = hm1;
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {  // Weyl key schedule: round j (0-based) uses key + j (W0, W1)
        const uint32_t j = 2u * i + 2u;
        o.rk[i] = make_uint4(k0 + j * kPhiloxW0, k1 + j * kPhiloxW1, k0 + (j + 1u) * kPhiloxW0, k1 + (j + 1u) * kPhiloxW1);
      }
    }
  };
  put_run(sc.k0, true);
  put_run(sc.k0 + 1, true);
  __syncthreads();
  const float dt = (float)sc.dt, gamma = (float)sc.gamma, kappa = (float)sc.kappa, scale = (float)sc.noise_scale;
  for (int64_t k = sc.k0; k < sc.k0 + sc.steps; ++k) {
    const float* X = Xs + (size_t)((k - sc.k0) & 1) * buf;
    float* Xn = Xs + (size_t)((k - sc.k0 + 1) & 1) * buf;
    const CsrRun* runs = s_run + (k & 1) * RC;
    for (int p = tid; p < N; p += nt) {
      const int e0 = __ldg(csr.rp + p), e1 = __ldg(csr.rp + p + 1);
      float jv[kHeld];
      int jo[kHeld];
#pragma unroll
      for (int t = 0; t < kHeld; ++t) {
        const bool in = e0 + t < e1;
        jv[t] = in ? __ldg(csr.cv + e0 + t) : 0.f;
        jo[t] = in ? __ldg(csr.ci + e0 + t) * D : p * D;
      }
      const float ew = (float)sc.eps * (sc.w ? (float)sc.w[p] : 1.f);
      const uint64_t mp = (uint64_t)kPhiloxM0 * (D <= 2 ? (uint32_t)p / (4u / (D <= 2 ? D : 4)) : (uint32_t)p);
      for (int r = 0; r < nr; ++r) {
        const float* xr = X + (size_t)r * N * D;
        const CsrRun& rc = runs[r];
        float y[D], x[D], z[4 * NB], n2 = 0.f;
#pragma unroll
        for (int mu = 0; mu < D; ++mu) {
          y[mu] = 0.f;
#pragma unroll
          for (int t = 0; t < kHeld; ++t)
            if (e0 + t < e1) y[mu] = fmaf(jv[t], xr[jo[t] + mu], y[mu]);
          x[mu] = xr[p * D + mu];
        }
        for (int e = e0 + kHeld; e < e1; ++e) {
          const float j = __ldg(csr.cv + e);
          const int o = __ldg(csr.ci + e) * D;
#pragma unroll
          for (int mu = 0; mu < D; ++mu) y[mu] = fmaf(j, xr[o + mu], y[mu]);
        }
#pragma unroll
        for (int mu = 0; mu < D; ++mu) n2 = fmaf(x[mu], x[mu], n2);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const uint4 t = rc.r12[b];
          const uint64_t q = (uint64_t)kPhiloxM1 * ((uint32_t)(mp >> 32) ^ t.x);
          uint4 c = make_uint4((uint32_t)(q >> 32) ^ t.y, (uint32_t)q, t.z ^ (uint32_t)mp, t.w);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 kk = rc.rk[i];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint64_t p0 = (uint64_t)kPhiloxM0 * c.x, p1 = (uint64_t)kPhiloxM1 * c.z;
              c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ (h ? kk.z : kk.x), (uint32_t)p1,
                             (uint32_t)(p0 >> 32) ^ c.w ^ (h ? kk.w : kk.y), (uint32_t)p0);
            }
          }
          if constexpr (D <= 2) {  // the spin's pair of a block it shares
            const uint32_t j0 = ((uint32_t)p % (4u / D)) * D;
            float cz, sz;
            box_muller_f32(j0 >= 2u ? c.z : c.x, j0 >= 2u ? c.w : c.y, scale, cz, sz);
            z[0] = (j0 & 1u) ? sz : cz;
            z[1] = sz;
          } else {
            box_muller_f32(c.x, c.y, scale, z[4 * b], z[4 * b + 1]);
            if (D - 4 * b > 2) box_muller_f32(c.z, c.w, scale, z[4 * b + 2], z[4 * b + 3]);
          }
        }
        float* xo = Xn + (size_t)r * N * D + p * D;
#pragma unroll
        for (int mu = 0; mu < D; ++mu) {
          const float xm = x[mu];
          const float f = rc.hm1 * xm - kappa * xm * xm * xm - gamma * xm * n2 + ew * (mu == 0 ? 1.f : rc.ramp) * y[mu];
          xo[mu] = xm + dt * f + z[mu];
        }
      }
    }
    __syncthreads();
    put_run(k + 2, false);  // this step's parity: read next after the barrier of step k + 1
  }
  const float* X = Xs + (size_t)(sc.steps & 1) * buf;
  for (int i = tid; i < used; i += nt) Xg[(size_t)run0 * N * D + i] = X[i];
}

template <int D>
cudaError_t launch_csr(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  const int N = c->N;
  const size_t per_run = (size_t)2 * N * D * sizeof(float);
  const int fit = (int)std::min<size_t>(kSimtSmemBudget / per_run, 32);
  if (fit < 1) return cudaErrorInvalidConfiguration;  // N too large
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  // runs per CTA (one CTA per SM): the fewest run slots over the waves of CTAs, each wave
  // counted half a run more for its barriers and constants (2048 runs, up to 4 a CTA: 7 waves
  // of 2 rather than 4 of 4)
  int RC = 1;
  double best = 0.0;
  for (int rc = 1; rc <= fit; ++rc) {
    const int grid = (sc.n_runs + rc - 1) / rc;
    const double t = (double)((grid + sms - 1) / sms) * (rc + 0.5);
    if (rc == 1 || t < best) {
      best = t;
      RC = rc;
    }
  }
  const int threads = std::min(D <= 4 ? 1024 : 512, std::max(64, (N + 31) / 32 * 32));
  const size_t smem = (size_t)RC * (per_run + 2 * sizeof(CsrRun));
  const CsrRows<float> rows{c->d_rp, c->d_ci, c->d_cv32};
  auto kern = step_csr_kernel<D>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(sc.n_runs + RC - 1) / RC, threads, smem, st>>>((float*)c->d_X, c->d_h, c->d_seeds, sc, RC, rows);
  return cudaGetLastError();
}

// Runs per CTA with which the FP64 per-spin form (step_simt_kernel) fills the SMs in equal
// waves, or 0 where step_f64_kernel is the better one.  A thread with all D components of a spin
// loads J once for D products and shares the drift's factors, so it wins where its warps are
// full: four warps of (run, spin) slots an SM.  us a step, step_f64_kernel -> per spin:
//   one CTA an SM: ladder N = 100, D = 3, 4096 runs 174 -> 142; SK N = 500, D = 3, 64 runs 343 ->
//   213; N = 20, D = 3, 1520 runs 24.4 -> 15.3; below the line, 304 runs 4.2 / 9.2;
//   several: SK N = 100, D = 3, 4096 runs 385 -> 345, 7904 runs 741 -> 663; ladder, 32768 runs 1384
//   -> 1155; N = 64, D = 5, 9728 runs 692 -> 629.
// Fewer slots will do where step_f64_kernel would cut an SM's runs into several CTAs (N = 20,
// D = 8, 608 runs 21.7 -> 20.1).  The waves are those that waste the least, a CTA whose last
// pass of 512 threads leaves most idle counted a tenth longer (SK N = 300, D = 3, 256 runs: 187 in
// CTAs of two runs, 172 of one; N = 20, 4096 runs: 42 of 27, 38 of 14); where a twelfth is wasted
// all the same, step_f64_kernel's smaller CTAs win (SK N = 1000, D = 2, 1024 runs 3687 / 4115).
// D = 1 has nothing to share and draws a pair of normals for one: only long dense rows in one
// full wave outweigh that (N = 500, 64 runs 104 -> 76; N = 300, 7904 runs 1461 / 1532).
int per_spin_f64_runs(const chym_ctx* c, int D, int n_runs) {
  const int N = c->N;
  if (D == 1 && (c->sparse || N < 256)) return 0;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (sms <= 0) return 0;
  const long long share = ((long long)n_runs + sms - 1) / sms, slots = share * N;
  if (slots < 128 && (share == 1 || slots * D <= 512)) return 0;
  const size_t j_bytes = (size_t)N * N * sizeof(double);
  const size_t avail = kSimtSmemBudget - (!c->sparse && j_bytes <= kSimtSmemBudget / 2 ? j_bytes : 0);
  const long long fit = std::min<long long>(64, avail / ((size_t)2 * N * D * sizeof(double)));
  if (fit < 1) return 0;
  const long long fewest = (share + fit - 1) / fit;
  if (D == 1 && fewest > 1) return 0;
  long long RC = 0, least = 0;  // in tenths of a run
  for (long long waves = fewest; waves <= (D == 1 ? 1 : 2 * fewest); ++waves) {
    const long long runs = (share + waves - 1) / waves, passes = (runs * N + 511) / 512;
    const bool full = passes == 1 || runs == 1 || 4 * runs * N >= 3 * 512 * passes;
    if (D == 1 && !full) return 0;
    const long long cost = waves * runs * (full ? 10 : 11);
    if (RC == 0 || cost < least) {
      RC = runs;
      least = cost;
    }
  }
  const long long used = (share + RC - 1) / RC * RC;
  return 12 * used <= 13 * share ? (int)RC : 0;
}

constexpr size_t kSmSharedBytes = 228 * 1024;  // of an SM

template <typename T, int D>
cudaError_t launch_simt_typed(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  const bool csr = c->sparse;  // the SIMT kernels use the compressed rows whenever they exist
  if constexpr (sizeof(T) == 4) {
    const cudaError_t e = csr ? launch_simt_tiled<D, true>(c, sc, st) : launch_simt_tiled<D, false>(c, sc, st);
    if (e != cudaErrorInvalidConfiguration) return e;
    if (csr) return launch_csr<D>(c, sc, st);
  }
  int full = 0;  // runs per CTA of per_spin_f64_runs
  if constexpr (sizeof(T) == 8) {
    full = per_spin_f64_runs(c, D, sc.n_runs);
    if (full == 0) {
      const cudaError_t e = launch_f64<D>(c, sc, st);
      if (e != cudaErrorInvalidConfiguration) return e;
    }
  }
  const int RB = csr ? 1 : SimtTraits<T>::RB;
  const int N = c->N;
  const size_t budget = kSimtSmemBudget;
  const size_t j_bytes = (size_t)N * N * sizeof(T);
  const bool j_smem = !csr && j_bytes <= budget / 2;
  const size_t per_run = (size_t)2 * N * D * sizeof(T);
  const size_t avail = budget - (j_smem ? j_bytes : 0);
  int RC = (int)std::min<size_t>(avail / per_run, 64);
  RC = std::max(RB, RC / RB * RB);
  if ((size_t)RC * per_run > avail) return cudaErrorInvalidConfiguration;  // N too large
  // do not make CTAs larger than needed to fill the GPU
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  while (RC > RB && (int64_t)((sc.n_runs + RC - 1) / RC) < sms) RC -= RB;
  size_t smem_least = 0;
  if (full > 0) {
    RC = full;
    // No more CTAs on an SM than the waves: SMs that come free before others (behind another
    // kernel) would take two where one each was meant (N = 100, D = 3, 1024 runs behind the
    // large-N launch of a batch: 173 us a step on half the SMs, 87 on all)
    const int waves = ((sc.n_runs + sms - 1) / sms + RC - 1) / RC;
    smem_least = kSmSharedBytes / (waves + 1);
  }
  const size_t smem = std::max((j_smem ? j_bytes : 0) + (size_t)RC * per_run, smem_least);
  const int threads = std::min(512, std::max(64, ((N * (RC / RB) + 31) / 32) * 32));
  const int grid = (sc.n_runs + RC - 1) / RC;
  const T* J = sizeof(T) == 8 ? (const T*)c->d_J64 : (const T*)c->d_J32;
  T* X = (T*)c->d_X;
  const CsrRows<T> rows{c->d_rp, c->d_ci, sizeof(T) == 8 ? (const T*)c->d_cv64 : (const T*)c->d_cv32};
  auto kern = j_smem ? step_simt_kernel<T, D, true, false> : step_simt_kernel<T, D, false, false>;
  if constexpr (sizeof(T) == 8)
    if (csr) kern = step_simt_kernel<T, D, false, true>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, threads, smem, st>>>(J, X, c->d_h, c->d_seeds, sc, RC, rows);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_simt_D(chym_ctx* c, const StepConsts& sc, cudaStream_t st) {
  switch (c->D) {
    case 1: return launch_simt_typed<T, 1>(c, sc, st);
    case 2: return launch_simt_typed<T, 2>(c, sc, st);
    case 3: return launch_simt_typed<T, 3>(c, sc, st);
    case 4: return launch_simt_typed<T, 4>(c, sc, st);
    case 5: return launch_simt_typed<T, 5>(c, sc, st);
    case 6: return launch_simt_typed<T, 6>(c, sc, st);
    case 7: return launch_simt_typed<T, 7>(c, sc, st);
    case 8: return launch_simt_typed<T, 8>(c, sc, st);
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_init_typed(chym_ctx* c, cudaStream_t st, double init_std) {
  const int64_t pairs = (int64_t)c->N * c->n_runs;
  const int threads = 256;
  const int grid = (int)std::min<int64_t>((pairs + threads - 1) / threads, 152 * 32);
  T* X = (T*)c->d_X;
  switch (c->D) {
#define CHYM_INIT_CASE(DD) \
  case DD: init_kernel<T, DD><<<grid, threads, 0, st>>>(X, c->d_seeds, c->N, c->n_runs, (T)init_std); break;
    CHYM_INIT_CASE(1) CHYM_INIT_CASE(2) CHYM_INIT_CASE(3) CHYM_INIT_CASE(4)
    CHYM_INIT_CASE(5) CHYM_INIT_CASE(6) CHYM_INIT_CASE(7) CHYM_INIT_CASE(8)
#undef CHYM_INIT_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Reinitialise the listed runs from new seeds at local step 0 (offset = current k).
__global__ void fill_hidx_kernel(int32_t* hidx, int n_runs, int replicas) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n_runs; r += gridDim.x * blockDim.x)
    hidx[r] = r / replicas;
}

template <typename T, int D>
__global__ void reseed_kernel(T* __restrict__ X, uint64_t* __restrict__ seeds, int64_t* __restrict__ koff,
                              int32_t* __restrict__ hidx, const int32_t* __restrict__ runs, int n,
                              const uint64_t* __restrict__ new_seeds, const int32_t* __restrict__ new_hidx,
                              int N, int64_t k_now, T init_std) {
  const int64_t total = (int64_t)n * N;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < total;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(s / N), p = (int)(s % N);
    const int run = runs[i];
    const uint64_t sd = new_seeds[i];
    T z[D];
    spin_normals<T, D>(sd, 1u, 0ull, p, init_std, z);
#pragma unroll
    for (int mu = 0; mu < D; ++mu) X[((int64_t)run * N + p) * D + mu] = z[mu];
    if (p == 0) {
      seeds[run] = sd;
      koff[run] = k_now;
      if (new_hidx) hidx[run] = new_hidx[i];
    }
  }
}

template <typename T>
cudaError_t launch_reseed_typed(chym_ctx* c, const int32_t* runs, int n, const uint64_t* ns,
                                const int32_t* nh, double init_std, cudaStream_t st) {
  const int threads = 256;
  const int grid = (int)std::min<int64_t>(((int64_t)n * c->N + threads - 1) / threads, 152 * 16);
  T* X = (T*)c->d_X;
  switch (c->D) {
#define CHYM_RESEED_CASE(DD)                                                                       \
  case DD:                                                                                        \
    reseed_kernel<T, DD><<<grid, threads, 0, st>>>(X, c->d_seeds, c->d_koff, c->d_hidx, runs, n, ns, nh, \
                                                  c->N, c->k, (T)init_std);                        \
    break;
    CHYM_RESEED_CASE(1) CHYM_RESEED_CASE(2) CHYM_RESEED_CASE(3) CHYM_RESEED_CASE(4)
    CHYM_RESEED_CASE(5) CHYM_RESEED_CASE(6) CHYM_RESEED_CASE(7) CHYM_RESEED_CASE(8)
#undef CHYM_RESEED_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_reseed(chym_ctx* c, const int32_t* d_runs, int n, const uint64_t* d_new_seeds,
                          const int32_t* d_new_hidx, double init_std, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (c->prec == CHYM_PREC_FP64)
    return launch_reseed_typed<double>(c, d_runs, n, d_new_seeds, d_new_hidx, init_std, st);
  return launch_reseed_typed<float>(c, d_runs, n, d_new_seeds, d_new_hidx, init_std, st);
}

cudaError_t launch_fill_hidx(int32_t* hidx, int n_runs, int replicas, cudaStream_t st) {
  if (n_runs <= 0) return cudaSuccess;
  fill_hidx_kernel<<<(n_runs + 255) / 256, 256, 0, st>>>(hidx, n_runs, replicas);
  return cudaGetLastError();
}

cudaError_t launch_step_simt(chym_ctx* c, const StepConsts& sc, int32_t prec, cudaStream_t st) {
  if (sc.steps <= 0 || sc.n_runs <= 0) return cudaSuccess;
  if (prec == CHYM_PREC_FP64) return launch_simt_D<double>(c, sc, st);
  return launch_simt_D<float>(c, sc, st);
}

cudaError_t launch_init(chym_ctx* c, int32_t prec, cudaStream_t st, double init_std) {
  if (c->n_runs <= 0) return cudaSuccess;
  if (prec == CHYM_PREC_FP64) return launch_init_typed<double>(c, st, init_std);
  return launch_init_typed<float>(c, st, init_std);
}

}  // namespace chym
