// solve_small.cu -- a whole solve of a small dense instance in one launch.
//
// For N <= 128 and P * N <= 1024 (and 2 P <= N) one CTA holds one run: J
// (FP32, N x N) and
// f(X) (N x P), and the run's schedule in shared memory, and the state (one
// (spin, replica) element per thread) in registers for all steps.
// Each step: G = J f(X) from shared memory (exact: integer terms), the update of Sec. II A Eqs. 6-7 with the
// wall rule and the threshold of Eq. 8, the ring neighbours by warp shuffle
// (P divides 32, thread t = i * P + k).  At the end the CTA reads out the
// exact int64 energies of its P replicas, the best replica and its spins, and
// writes the final state.  Results equal the per-step path bit for bit.
// Served for integer instances (exact energies in any summation order).
//
// Two forms.  |J_ij| <= 127 (k_solve_small_i8): each thread keeps its row of J
// as packed bytes in registers (N / 4 words, loaded once) and f(X) lies as
// bytes [replica][spin] in shared memory, so a step is N / 16 16-byte loads and
// N / 4 four-way dot products per thread instead of 2 N loads and N FMAs; the
// sums are the same integers.  Larger |J| keeps J in shared memory in FP32.
// A step is a chain of latencies (barrier, loads, dot products, update); SK
// N = 64, P = 8, R = 16, 1000 steps with its results: 1328 us in FP32, 334 in
// bytes.
#include <cfloat>
#include <climits>

#include "step_common.cuh"

namespace sbqa {

__device__ __forceinline__ uint64_t sm64(uint64_t seed, uint64_t ctr) {
  uint64_t z = seed + (ctr + 1ull) * 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ float uni(uint64_t z, float amp) {
  return __fmul_rn(float(int(z >> 40) - 8388608) * 0x1p-23f, amp);
}

template <int P>
__global__ void __launch_bounds__(1024) k_solve_small(SmallArgs a) {
  extern __shared__ float sh[];
  const int N = a.N, S = a.S;
  const int ldj = N + 1;                // padded rows: the four spins of a warp hit four banks
  float *sJ = sh;                       // [N][N + 1]
  float *sF = sJ + N * ldj;             // [2][N][P] f values
  float *sKa = sF + 2 * N * P;          // [S]
  float *sDl = sKa + S;                 // [S + 1]
  float *sKj = sDl + S + 1;             // [S] of this run
  const size_t red_off = (size_t(N * ldj + 2 * N * P + 3 * S + 1) * sizeof(float) + 7) & ~size_t(7);
  double *sRed = reinterpret_cast<double *>(reinterpret_cast<char *>(sh) + red_off);  // [P + 1]
  const int r = blockIdx.x, t = threadIdx.x;
  const int k = t % P, i = t / P;
  const bool live = i < N;
  for (int q = t; q < N * N; q += blockDim.x) sJ[(q / N) * ldj + q % N] = a.J[q];
  for (int q = t; q < S; q += blockDim.x) {
    sKa[q] = a.ka[q];
    sKj[q] = a.kj[size_t(q) * a.R + r];
  }
  for (int q = t; q <= S; q += blockDim.x) sDl[q] = a.dl[q];
  // initial state, same counter layout as k_init
  float x = 0.f, y = 0.f;
  const int c = r * P + k;
  if (live) {
    const uint64_t el = uint64_t(c) * uint64_t(N) + uint64_t(i);
    x = uni(sm64(a.seed, 2ull * el), a.amp);
    y = uni(sm64(a.seed, 2ull * el + 1ull), a.amp);
    sF[i * P + k] = float(int(fcode(x, 0.f)) - 1);
  }
  const float hi = live ? a.h[i] : 0.f;
  __syncthreads();
  const int lane = t & 31;
  const int src_l = (k == 0) ? lane + P - 1 : lane - 1;
  const int src_r = (k == P - 1) ? lane - P + 1 : lane + 1;
  for (int n = 0; n < S; ++n) {
    const float *Fn = sF + (n & 1) * N * P;
    float *Fo = sF + ((n + 1) & 1) * N * P;
    float G = 0.f;
    if (live) {
      // four independent partial sums; every term is a small integer, so the
      // sum is exact and equals the sequential one
      const float *Ji = sJ + i * ldj;
      float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f;
      int j = 0;
      for (; j + 3 < N; j += 4) {
        g0 = fmaf(Ji[j], Fn[j * P + k], g0);
        g1 = fmaf(Ji[j + 1], Fn[(j + 1) * P + k], g1);
        g2 = fmaf(Ji[j + 2], Fn[(j + 2) * P + k], g2);
        g3 = fmaf(Ji[j + 3], Fn[(j + 3) * P + k], g3);
      }
      for (; j < N; ++j) g0 = fmaf(Ji[j], Fn[j * P + k], g0);
      G = (g0 + g1) + (g2 + g3);
    }
    // ring neighbours (P consecutive threads of one spin hold the run's replicas)
    float xm, xp;
    if constexpr (P == 1) {
      xm = xp = x;
    } else {
      xm = __shfl_sync(0xffffffffu, x, src_l);
      xp = __shfl_sync(0xffffffffu, x, src_r);
    }
    if (live) {
      float yn = fmaf(a.kc, G + hi, y);
      yn = fmaf(-sKa[n], x, yn);
      yn = fmaf(sKj[n], xm + xp, yn);
      const float xn = fmaf(a.kx, yn, x);
      const float xc = fminf(fmaxf(xn, -1.f), 1.f);  // wall
      y = (xc != xn) ? 0.f : yn;
      x = xc;
      const float d = sDl[n + 1];
      Fo[i * P + k] = float(int(x > d) - int(x < -d));
    }
    __syncthreads();
  }
  // final state
  if (live) {
    const size_t off = size_t(i) * a.Cp + c;
    a.x[off] = x;
    a.y[off] = y;
    a.Sg[off] = x >= 0.f ? 1 : -1;
  }
  // readout: t_i = sum_j J_ij s_j in integers, then per replica
  // -(1/2) sum_i s_i (t_i + 2 h_i)
  float *sS = sF;  // reuse: spins as floats [N][P]
  if (live) sS[i * P + k] = x >= 0.f ? 1.f : -1.f;
  __syncthreads();
  long long vi = 0;
  if (live) {
    const long long si = x >= 0.f ? 1 : -1;
    long long ti = 0;
    for (int j = 0; j < N; ++j) ti += (long long)a.J_i32[size_t(i) * N + j] * (long long)sS[j * P + k];
    vi = si * (ti + 2 * a.h_i64[i]);
  }
  // fixed-order reduction over i for each replica k: thread k sums i = 0..N-1
  __syncthreads();
  long long *red = reinterpret_cast<long long *>(sJ);  // J no longer needed: [N][P] partials
  if (live) red[i * P + k] = vi;
  __syncthreads();
  if (t < P) {
    long long acc = 0;
    for (int q = 0; q < N; ++q) acc += red[q * P + t];
    const int cc = r * P + t;
    const long long e = -(acc / 2);
    a.e_int[cc] = e;
    a.e_f64[cc] = double(e);
    sRed[t] = double(e);
  }
  __syncthreads();
  if (t == 0) {
    int kb = 0;
    for (int q = 1; q < P; ++q)
      if (sRed[q] < sRed[kb]) kb = q;
    a.best_k[r] = kb;
    a.best_e[r] = sRed[kb];
    a.best_e_int[r] = (long long)sRed[kb];
    a.best_step[r] = S - 1;
    a.have_best[r] = 1;
    sRed[P] = double(kb);
  }
  __syncthreads();
  const int kb = int(sRed[P]);
  if (live && k == kb) a.best_spins[size_t(r) * N + i] = x >= 0.f ? 1 : -1;
}

// NQ: 16-byte pieces of a row, N <= 16 NQ.  The f rows are padded to 16 NQ + 16
// bytes: the eight rows a quarter warp reads start in eight different groups
// of four banks.
template <int P, int NQ>
__global__ void __launch_bounds__(1024) k_solve_small_i8(SmallArgs a) {
  constexpr int kLdf = 16 * NQ + 16;
  extern __shared__ float sh[];
  const int N = a.N, S = a.S;
  int8_t *sF = reinterpret_cast<int8_t *>(sh);              // [2][P][kLdf] f values
  long long *red = reinterpret_cast<long long *>(sh + 2 * P * kLdf / 4);  // [N][P]
  double *sRed = reinterpret_cast<double *>(red + N * P);   // [P + 1]
  float *sKa = reinterpret_cast<float *>(sRed + P + 1);     // [S]
  float *sDl = sKa + S;                                     // [S + 1]
  float *sKj = sDl + S + 1;                                 // [S] of this run
  const int r = blockIdx.x, t = threadIdx.x;
  const int k = t % P, i = t / P;
  const bool live = i < N;
  for (int q = t; q < 2 * P * kLdf / 4; q += blockDim.x) reinterpret_cast<int *>(sF)[q] = 0;
  for (int q = t; q < S; q += blockDim.x) {
    sKa[q] = a.ka[q];
    sKj[q] = a.kj[size_t(q) * a.R + r];
  }
  for (int q = t; q <= S; q += blockDim.x) sDl[q] = a.dl[q];
  int jr[4 * NQ];  // row i of J, four entries a word
#pragma unroll
  for (int w = 0; w < 4 * NQ; ++w) {
    uint32_t v = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = 4 * w + b;
      if (live && j < N) v |= uint32_t(uint8_t(int8_t(a.J_i32[size_t(i) * N + j]))) << (8 * b);
    }
    jr[w] = int(v);
  }
  // initial state, same counter layout as k_init
  float x = 0.f, y = 0.f;
  const int c = r * P + k;
  __syncthreads();  // f cleared
  if (live) {
    const uint64_t el = uint64_t(c) * uint64_t(N) + uint64_t(i);
    x = uni(sm64(a.seed, 2ull * el), a.amp);
    y = uni(sm64(a.seed, 2ull * el + 1ull), a.amp);
    sF[k * kLdf + i] = int8_t(int(fcode(x, 0.f)) - 1);
  }
  const float hi = live ? a.h[i] : 0.f;
  auto dot = [&](const int8_t *F) {  // sum_j J_ij F_j, four independent integer sums
    int g[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int4 f = *reinterpret_cast<const int4 *>(F + k * kLdf + 16 * q);
      g[0] = __dp4a(jr[4 * q], f.x, g[0]);
      g[1] = __dp4a(jr[4 * q + 1], f.y, g[1]);
      g[2] = __dp4a(jr[4 * q + 2], f.z, g[2]);
      g[3] = __dp4a(jr[4 * q + 3], f.w, g[3]);
    }
    return (g[0] + g[1]) + (g[2] + g[3]);
  };
  __syncthreads();
  const int lane = t & 31;
  const int src_l = (k == 0) ? lane + P - 1 : lane - 1;
  const int src_r = (k == P - 1) ? lane - P + 1 : lane + 1;
  for (int n = 0; n < S; ++n) {
    const int8_t *Fn = sF + (n & 1) * P * kLdf;
    int8_t *Fo = sF + ((n + 1) & 1) * P * kLdf;
    const float G = float(dot(Fn));
    float xm, xp;
    if constexpr (P == 1) {
      xm = xp = x;
    } else {
      xm = __shfl_sync(0xffffffffu, x, src_l);
      xp = __shfl_sync(0xffffffffu, x, src_r);
    }
    if (live) {
      float yn = fmaf(a.kc, G + hi, y);
      yn = fmaf(-sKa[n], x, yn);
      yn = fmaf(sKj[n], xm + xp, yn);
      const float xn = fmaf(a.kx, yn, x);
      const float xc = fminf(fmaxf(xn, -1.f), 1.f);  // wall
      y = (xc != xn) ? 0.f : yn;
      x = xc;
      const float d = sDl[n + 1];
      Fo[k * kLdf + i] = int8_t(int(x > d) - int(x < -d));
    }
    __syncthreads();
  }
  // final state, and the spins as bytes
  if (live) {
    const size_t off = size_t(i) * a.Cp + c;
    a.x[off] = x;
    a.y[off] = y;
    a.Sg[off] = x >= 0.f ? 1 : -1;
    sF[k * kLdf + i] = x >= 0.f ? 1 : -1;
  }
  __syncthreads();
  if (live) {  // s_i (sum_j J_ij s_j + 2 h_i)
    const long long v = (long long)dot(sF) + 2 * a.h_i64[i];
    red[i * P + k] = x >= 0.f ? v : -v;
  }
  __syncthreads();
  if (t < P) {
    long long acc = 0;
    for (int q = 0; q < N; ++q) acc += red[q * P + t];
    const int cc = r * P + t;
    const long long e = -(acc / 2);
    a.e_int[cc] = e;
    a.e_f64[cc] = double(e);
    sRed[t] = double(e);
  }
  __syncthreads();
  if (t == 0) {
    int kb = 0;
    for (int q = 1; q < P; ++q)
      if (sRed[q] < sRed[kb]) kb = q;
    a.best_k[r] = kb;
    a.best_e[r] = sRed[kb];
    a.best_e_int[r] = (long long)sRed[kb];
    a.best_step[r] = S - 1;
    a.have_best[r] = 1;
    sRed[P] = double(kb);
  }
  __syncthreads();
  const int kb = int(sRed[P]);
  if (live && k == kb) a.best_spins[size_t(r) * N + i] = x >= 0.f ? 1 : -1;
}

// Shared memory of the byte form: at most 3 KB more than small_smem_bytes (N <
// 28, where its rows are padded most), which small_eligible keeps 27 KB below
// what a block can have.
template <int P, int NQ>
static cudaError_t launch_small_i8(const SmallArgs &a, cudaStream_t st) {
  const size_t smem = size_t(2) * P * (16 * NQ + 16) + size_t(a.N) * P * 8 + 8 * (P + 1) + (3 * size_t(a.S) + 1) * 4;
  static_assert((2 * P * (16 * NQ + 16)) % 8 == 0, "the sums behind the f rows are 8-byte aligned");
  const cudaError_t e = cudaFuncSetAttribute(k_solve_small_i8<P, NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(smem));
  if (e != cudaSuccess) return e;
  k_solve_small_i8<P, NQ><<<a.R, (a.N * P + 31) / 32 * 32, smem, st>>>(a);
  return cudaGetLastError();
}

template <int P>
static cudaError_t launch_small_i8_p(const SmallArgs &a, cudaStream_t st) {
  if (a.N <= 32) return launch_small_i8<P, 2>(a, st);
  if (a.N <= 64) return launch_small_i8<P, 4>(a, st);
  if (a.N <= 96) return launch_small_i8<P, 6>(a, st);
  return launch_small_i8<P, 8>(a, st);
}

size_t small_smem_bytes(int N, int P, int S) {
  return sizeof(float) * (size_t(N) * (N + 1) + 2 * size_t(N) * P + 3 * size_t(S) + 4) + sizeof(double) * (P + 1) + 16;
}

bool small_eligible(int N, int P, int S) {
  return S >= 1 && N <= 128 && N * P <= 1024 && small_smem_bytes(N, P, S) <= 200 * 1024 &&
         size_t(N) * P * sizeof(long long) <= size_t(N) * N * sizeof(float);
}

cudaError_t launch_solve_small(const SmallArgs &a, cudaStream_t st) {
  if (a.max_abs_j <= 127) {
    switch (a.P) {
      case 1: return launch_small_i8_p<1>(a, st);
      case 2: return launch_small_i8_p<2>(a, st);
      case 4: return launch_small_i8_p<4>(a, st);
      case 8: return launch_small_i8_p<8>(a, st);
      case 16: return launch_small_i8_p<16>(a, st);
      case 32: return launch_small_i8_p<32>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
  const size_t smem = small_smem_bytes(a.N, a.P, a.S);
  const int threads = ((a.N * a.P + 31) / 32) * 32;
  cudaError_t e = cudaSuccess;
#define SBQA_SMALL_CASE(PP)                                                                              \
  case PP:                                                                                               \
    e = cudaFuncSetAttribute(k_solve_small<PP>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)); \
    if (e != cudaSuccess) return e;                                                                      \
    k_solve_small<PP><<<a.R, threads, smem, st>>>(a);                                                    \
    break;
  switch (a.P) {
    SBQA_SMALL_CASE(1)
    SBQA_SMALL_CASE(2)
    SBQA_SMALL_CASE(4)
    SBQA_SMALL_CASE(8)
    SBQA_SMALL_CASE(16)
    SBQA_SMALL_CASE(32)
    default: return cudaErrorInvalidValue;
  }
#undef SBQA_SMALL_CASE
  return cudaGetLastError();
}

}  // namespace sbqa
