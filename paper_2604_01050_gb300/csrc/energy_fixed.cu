// energy_fixed.cu -- readout energies of real dense instances on the tensor
// cores, in fixed point.
//
// E_c = -(1/2) sum_i s_ic (t_ic + 2 h_i), t_ic = sum_j J_ij s_jc (Sec. II A,
// Eq. 4 sign; Sec. II B).  An FP64 sum of N^2 Cp terms on the CUDA cores is
// bound by this chip's FP64 rate (two FMAs per SM and clock): 10.7 ms at
// N = 2000, R*P = 1024, as long as 700 steps of the solver.  Here J and h are
// integers X = rint(2^k J), H = rint(2^k h) of 63 bits, with k such that no
// |t_i + 2 h_i| reaches 2^63, and a bfloat16 operand per byte of X (0 .. 255,
// exact; the top byte signed): the tensor cores form the eight exact integer
// sums of a tile (below 2^24 in FP32), which the epilogue joins as
// acc = 256 acc + digit in 64-bit integers.  Rows and then row blocks add as
// integers too (the 64-bit values in two 32-bit halves), so the only roundings
// are those of X and H and one of the result.
//
// One unit 2^-k serves the whole instance, so what is small beside the largest
// row sum is held in few bits, where an FP64 sum would keep it: a spin pinned
// by a large field, say.  The plan is therefore made only where the error is
// no larger than that of the FP64 sums (fx_scale); elsewhere they serve.  For
// Gaussian J of N = 64 .. 2048 the error is 0.36 to 0.46 of theirs (root mean
// square), with fields of up to the size of the row sums 0.55 to 0.61.
// At N = 2000, R*P = 1024 the eight GEMMs (66 GFLOP, operands 64 MB, in L2)
// and the kernels around them take 0.14 ms instead of 10.7; at N = 1000, R*P =
// 256 the readout takes 0.04 ms instead of 1.34.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "dense_tc_common.cuh"

namespace sbqa {

constexpr int kFxDigits = 8;
constexpr int kFxMaxKp = 16384;  // 4.3 GB of digits; larger instances keep the FP64 readout

struct FxPlan {
  CUtensorMap A;  // digits [8 Kp][Kp] bfloat16, most significant plane first
  const int64_t *H;
  int k, Kp;
};

// Per row, for the choice of the scale: A_i = sum_j |J_ij|, and q_i = sum_j
// (N - j) J_ij^2 in units of 2^(2 ilogb(A_i)), to a few per mille: the leading 21 bits
// of each entry, by its exponent field, as a float (no FP64 arithmetic;
// subnormal entries count as 0).
__global__ void __launch_bounds__(256) k_fx_rows(const double *J, int N, double *A, double *q) {
  __shared__ double sm[8];
  __shared__ float sq[8];
  __shared__ int s_e;
  const int i = blockIdx.x;
  const double *row = J + size_t(i) * N;
  double acc = 0.0;
  for (int j = threadIdx.x; j < N; j += 256) acc += fabs(row[j]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) acc += sm[w];
    A[i] = acc;
    s_e = (__double2hiint(acc) >> 20) & 0x7ff;  // not 0x7ff: the host refuses infinite sums whatever q is
  }
  __syncthreads();
  float w2 = 0.f;
  for (int j = threadIdx.x; j < N; j += 256) {
    const int hi = __double2hiint(row[j]), field = (hi >> 20) & 0x7ff, e = field - s_e + 127;
    const float v = field > 0 && e > 0 ? __uint_as_float(uint32_t(e) << 23 | uint32_t(hi & 0xfffff) << 3) : 0.f;
    w2 = fmaf(v * v, float(N - j), w2);
  }
  for (int o = 16; o > 0; o >>= 1) w2 += __shfl_down_sync(0xffffffffu, w2, o);
  if ((threadIdx.x & 31) == 0) sq[threadIdx.x >> 5] = w2;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) w2 += sq[w];
    q[i] = w2;
  }
}

// Bytes of X [N][N] into the planes [8][Kp][Kp], zero padded; H.
__global__ void k_fx_digits(const double *J, const double *h, int N, int Kp, int k, uint16_t *out, int64_t *H) {
  const size_t e = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= size_t(Kp) * Kp) return;
  const int i = int(e / Kp), j = int(e % Kp);
  const long long X = (i < N && j < N) ? __double2ll_rn(scalbn(J[size_t(i) * N + j], k)) : 0ll;
#pragma unroll
  for (int d = 0; d < kFxDigits; ++d) {
    const int byte = int((X >> (8 * (kFxDigits - 1 - d))) & 0xff);
    const float v = d == 0 ? float(int(int8_t(byte))) : float(byte);
    out[size_t(d) * Kp * Kp + e] = uint16_t(__float_as_uint(v) >> 16);  // at most 8 significant bits: exact
  }
  if (j == 0 && i < N) H[i] = __double2ll_rn(scalbn(h[i], k));
}

// Spins S [N][Cp] (+1, -1; 0 past C) -> bfloat16 [Cp][Kp] (zeros for padded
// spins), through 64 x 64 tiles so that both sides are coalesced.
__global__ void __launch_bounds__(256) k_sign_to_ft16(StateView s, uint16_t *FT, int Kp) {
  __shared__ int8_t t[64][68];
  const int i0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  for (int q = threadIdx.x; q < 64 * 16; q += 256) {
    const int r = q >> 4, w = q & 15;
    uint32_t v = 0;
    if (i0 + r < s.N) v = *reinterpret_cast<const uint32_t *>(s.Sg + size_t(i0 + r) * s.Cp + c0 + 4 * w);
    *reinterpret_cast<uint32_t *>(&t[r][4 * w]) = v;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 64 * 32; q += 256) {
    const int c = q >> 5, r = (q & 31) * 2;
    auto code = [](int8_t v) { return v == 0 ? 0u : (v > 0 ? 0x3F80u : 0xBF80u); };
    const uint32_t v = code(t[r][c]) | (code(t[r + 1][c]) << 16);
    *reinterpret_cast<uint32_t *>(FT + size_t(c0 + c) * Kp + i0 + r) = v;
  }
}

// One 128 x 128 tile (spin rows x columns) per block: warps 0-15 the epilogue,
// warp 16 the TMA producer, warp 17 the MMAs.  The K loop runs once per digit,
// most significant first, into one of two TMEM accumulators, while the
// epilogue takes in the digit before from the other.  Six stages of 32 KB.
constexpr int kFxStages = 6, kFxThreads = 18 * 32;
constexpr int kFxSmem = kFxStages * 2 * kTcTile + 4 * kTcBN * 16 + 1024 + 256;
static_assert(16 * 32 * 33 * 8 <= kFxStages * 2 * kTcTile, "row reductions must fit the operand stages");
static_assert(kFxSmem <= 227 * 1024, "shared memory of one block");

__global__ void __launch_bounds__(kFxThreads, 1)
    k_energy_dense_fx(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, StateView s,
                      int Kp, int *err, const int64_t *H, int64_t *part) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sA = smem, *sB = smem + kFxStages * kTcTile;
  int64_t *cols = reinterpret_cast<int64_t *>(smem + kFxStages * 2 * kTcTile);  // [4 quarters][128 columns][hi, lo]
  uint64_t *full = reinterpret_cast<uint64_t *>(cols + 4 * kTcBN * 2);
  uint64_t *empty = full + kFxStages;
  uint64_t *acc_full = empty + kFxStages, *acc_free = acc_full + 2;
  uint64_t *drained = acc_free + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drained + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kTcBM, n0 = blockIdx.x * kTcBN;
  const int KB = Kp / 64, total = KB * kFxDigits;
  if (threadIdx.x == 0) {
    for (int q = 0; q < kFxStages; ++q) {
      tc::mbar_init(&full[q], 1);
      tc::mbar_init(&empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&acc_full[q], 1);
      tc::mbar_init(&acc_free[q], 16);
    }
    tc::mbar_init(drained, 1);
    tc::fence_mbar_init();
    tc::prefetch_tmap(&mapA);
    tc::prefetch_tmap(&mapB);
  }
  if (warp == 0) tc::tmem_alloc(tmem_slot, 256);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  uint64_t acc[32];
  if (warp == 16) {
    if (lane == 0) {
      int g = 0;
      for (; g < total; ++g) {
        const int st = g % kFxStages, use = g / kFxStages, d = g / KB, kb = g % KB;
        if (use > 0 && !tc::mbar_wait(&empty[st], (use - 1) & 1, err, tc::ERR_WAIT_EMPTY)) break;
        tc::mbar_arrive_expect_tx(&full[st], 2 * kTcTile);
        tc::tma_load_2d(sA + st * kTcTile, &mapA, &full[st], kb * 64, d * Kp + m0);
        tc::tma_load_2d(sB + st * kTcTile, &mapB, &full[st], kb * 64, n0);
      }
      // no copy lands once the stages are reused, whether the MMAs took them or a wait ran out
      for (int q = max(0, g - kFxStages); q < g; ++q)
        tc::mbar_wait(&full[q % kFxStages], (q / kFxStages) & 1, err, tc::ERR_WAIT_FULL);
    }
  } else if (warp == 17) {
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16(kTcBM, kTcBN);
      bool ok = true;
      for (int d = 0; d < kFxDigits && ok; ++d) {
        if (d >= 2) ok = tc::mbar_wait(&acc_free[d & 1], (d / 2 - 1) & 1, err, tc::ERR_WAIT_DONE);
        tc::tc_fence_after();
        for (int kb = 0; kb < KB && ok; ++kb) {
          const int g = d * KB + kb, st = g % kFxStages;
          ok = tc::mbar_wait(&full[st], (g / kFxStages) & 1, err, tc::ERR_WAIT_FULL);
          if (!ok) break;
          tc::tc_fence_after();
          const uint32_t a0 = tc::smem_u32(sA + st * kTcTile), b0 = tc::smem_u32(sB + st * kTcTile);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc::mma_bf16(tmem + uint32_t(128 * (d & 1)), tc::smem_desc_sw128(a0 + kk * 32),
                         tc::smem_desc_sw128(b0 + kk * 32), idesc, (kb | kk) != 0 ? 1u : 0u);
          tc::mma_commit(&empty[st]);
        }
        if (ok) tc::mma_commit(&acc_full[d & 1]);
      }
      if (!ok) {  // the epilogue has not waited for these
        tc::mma_commit(drained);
        tc::mbar_wait(drained, 0, err, tc::ERR_WAIT_DONE);
      }
    }
  } else {
    const uint32_t at = tmem + (uint32_t((warp & 3) * 32) << 16) + uint32_t(32 * (warp >> 2));
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0;
    for (int d = 0; d < kFxDigits; ++d) {
      if (!tc::mbar_wait(&acc_full[d & 1], (d / 2) & 1, err, tc::ERR_WAIT_DONE)) break;
      tc::tc_fence_after();
      __syncwarp();
      uint32_t g[32];
      tc::tmem_ld_32x32b_x32(at + uint32_t(128 * (d & 1)), g);
      tc::reg_fence(g);
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&acc_free[d & 1]);
#pragma unroll
      for (int j = 0; j < 32; ++j)
        acc[j] = (acc[j] << 8) + uint64_t(int64_t(__float2int_rn(__uint_as_float(g[j]))));
    }
  }
  // every copy into the stages and every MMA that read them has completed: row reductions reuse them
  __syncthreads();
  if (warp < 16) {
    const int quarter = warp & 3, chunk = warp >> 2;
    const int i = m0 + quarter * 32 + lane, c0 = n0 + 32 * chunk;
    int64_t *red = reinterpret_cast<int64_t *>(smem) + size_t(warp) * 32 * 33;
    uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    uint64_t h2 = 0;
    if (i < s.N) {
      const uint4 *ps = reinterpret_cast<const uint4 *>(s.Sg + size_t(i) * s.Cp + c0);
      const uint4 u0 = ps[0], u1 = ps[1];
      w[0] = u0.x; w[1] = u0.y; w[2] = u0.z; w[3] = u0.w; w[4] = u1.x; w[5] = u1.y; w[6] = u1.z; w[7] = u1.w;
      h2 = 2 * uint64_t(H[i]);
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const int8_t si = int8_t(w[j >> 2] >> (8 * (j & 3)));
      const uint64_t v = acc[j] + h2;
      red[lane * 33 + j] = int64_t(si == 0 ? 0 : (si > 0 ? v : 0 - v));
    }
    __syncwarp();
    int64_t hi = 0, lo = 0;  // the rows of this quarter in 32-bit halves: no sum can wrap
#pragma unroll 8
    for (int r = 0; r < 32; ++r) {
      const int64_t v = red[r * 33 + lane];
      hi += v >> 32;
      lo += int64_t(uint64_t(v) & 0xffffffffu);
    }
    int64_t *o = cols + (quarter * kTcBN + 32 * chunk + lane) * 2;
    o[0] = hi;
    o[1] = lo;
  }
  tc::tc_fence_before();
  __syncthreads();
  if (threadIdx.x < kTcBN) {
    int64_t hi = 0, lo = 0;
    for (int q = 0; q < 4; ++q) {
      hi += cols[(q * kTcBN + threadIdx.x) * 2];
      lo += cols[(q * kTcBN + threadIdx.x) * 2 + 1];
    }
    int64_t *o = part + size_t(blockIdx.y) * 2 * s.Cp + n0 + threadIdx.x;
    o[0] = hi;
    o[s.Cp] = lo;
  }
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 256);
  }
}

// E_c = -2^(-k-1) (sum of the row blocks), one warp per column.
__global__ void k_energy_fx_final(int C, int Cp, int blocks, int k, const int64_t *part, double *e) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= C) return;
  long long hi = 0, lo = 0;
  for (int q = lane; q < blocks; q += 32) {
    hi += part[size_t(q) * 2 * Cp + c];
    lo += part[(size_t(q) * 2 + 1) * Cp + c];
  }
  for (int o = 16; o > 0; o >>= 1) {
    hi += __shfl_down_sync(0xffffffffu, hi, o);
    lo += __shfl_down_sync(0xffffffffu, lo, o);
  }
  if (lane == 0) {
    hi += lo >> 32;  // now 0 <= lo < 2^32 and |hi| < 2^48: both exact in FP64
    lo &= 0xffffffffll;
    e[c] = -scalbn(fma(double(hi), 4294967296.0, double(lo)), -k - 1);
  }
}

static int tc_padded(int N) { return (N + 127) / 128 * 128; }
size_t fx_digit_bytes(int N) { return size_t(kFxDigits) * tc_padded(N) * tc_padded(N) * 2; }
size_t fx_spin_bytes(int N, int Cp) { return size_t(Cp) * tc_padded(N) * 2; }
// From N = 64 on: below, the FP64 sums are short, and the partial sums and the
// spins would not fit the buffers they are given.
bool fx_eligible(int N) { return N >= 64 && tc_padded(N) <= kFxMaxKp; }

// Whether the fixed point serves, and its scale k: row sums |J_i| + 2 |h_i|
// below 2^62 after scaling.  The energies' root mean square errors, for spins
// of random signs: here N^2 / 2 pairs rounded to units u = 2^-k, 0.20 N u; in
// FP64, a rounding of 0.43 2^-53 of each partial sum along a row (variance
// sum_{l <= j} J_il^2 after entry j; halved in the energy) and of each row's
// field, 0.21 2^-53 sqrt(sum_i q_i + 4 sum_i h_i^2).  N counts the rows that are
// not empty, and both sums are taken as N times the median one's, so that a few large rows or fields, which may cancel
// in FP64 and leave the others' sums intact, do not stand for the rest.  The
// line lies where the two are equal, which favours FP64: aligned spins make
// its partial sums larger.  (One row 10^4 times the others at N = 300 and
// fields of N times the couplings at N = 2048, on either side of the line:
// 0.24 and 0.55 of the FP64 error.)
static bool fx_scale(const std::vector<double> &A, const std::vector<double> &q, const double *h, int N, int *k) {
  double most = 0.0, largest = 0.0;
  for (int i = 0; i < N; ++i) {
    largest = std::max(largest, A[i]);
    most = std::max(most, A[i] + (h ? 2.0 * std::fabs(h[i]) : 0.0));
  }
  if (!std::isfinite(most)) return false;
  *k = most > 0.0 ? 61 - std::ilogb(most) : 0;
  if (most == 0.0) return true;
  // in units of 2^e, so that no square leaves the FP64 range
  const int e = std::ilogb(largest > 0.0 ? largest : most);
  auto median = [](std::vector<double> &v) {
    auto mid = v.begin() + v.size() / 2;
    std::nth_element(v.begin(), mid, v.end());
    return *mid;
  };
  std::vector<double> rq, rh;
  for (int i = 0; i < N; ++i) {
    if (A[i] == 0.0 && (!h || h[i] == 0.0)) continue;
    rq.push_back(A[i] > 0.0 ? std::ldexp(q[i], 2 * (std::ilogb(A[i]) - e)) : 0.0);
    rh.push_back(h ? std::fabs(std::ldexp(h[i], -e)) : 0.0);
  }
  const double mq = median(rq), mh = median(rh);
  return std::sqrt(double(rq.size())) * std::ldexp(1.0, -*k - e) <= std::ldexp(std::sqrt(mq + 4.0 * mh * mh), -53);
}

cudaError_t fx_choose(const double *J, const double *h_host, int N, double *scratch, int *k, bool *serves,
                      cudaStream_t st) {
  *serves = false;
  k_fx_rows<<<N, 256, 0, st>>>(J, N, scratch, scratch + N);
  std::vector<double> A(N), q(N);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(A.data(), scratch, N * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(q.data(), scratch + N, N * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) *serves = fx_scale(A, q, h_host, N, k);
  return e;
}

cudaError_t fx_plan_make(void **plan, const double *J, const double *h, int N, int k, void *digits, int64_t *H,
                         cudaStream_t st) {
  const int Kp = tc_padded(N);
  *plan = nullptr;
  cudaError_t e = cudaFuncSetAttribute((const void *)k_energy_dense_fx, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kFxSmem);
  if (e != cudaSuccess) return e;
  auto *p = new FxPlan();
  p->k = k;
  p->H = H;
  p->Kp = Kp;
  const size_t total = size_t(Kp) * Kp;
  k_fx_digits<<<unsigned((total + 255) / 256), 256, 0, st>>>(J, h, N, Kp, k, static_cast<uint16_t *>(digits), H);
  e = cudaGetLastError();
  if (e == cudaSuccess && !tc_make_map(&p->A, digits, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, uint64_t(kFxDigits) * Kp,
                                       uint64_t(Kp), 64, 128, CU_TENSOR_MAP_SWIZZLE_128B))
    e = cudaErrorInvalidValue;
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    delete p;
    return e;
  }
  *plan = p;
  return cudaSuccess;
}

void fx_plan_free(void *plan) { delete static_cast<FxPlan *>(plan); }

cudaError_t launch_energy_partials_fx(const void *fx_plan, const StateView &s, void *spins, int *err,
                                      const BestView &best, cudaStream_t st) {
  const auto *p = static_cast<const FxPlan *>(fx_plan);
  const int Kp = p->Kp;
  CUtensorMap B;
  if (!tc_make_map(&B, spins, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, uint64_t(s.Cp), uint64_t(Kp), 64, 128,
                   CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  k_sign_to_ft16<<<dim3(unsigned(Kp / 64), unsigned(s.Cp / 64)), 256, 0, st>>>(s, static_cast<uint16_t *>(spins), Kp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const dim3 grid(unsigned(s.Cp / kTcBN), unsigned(Kp / kTcBM));
  // the partial sums of 128 rows take 16 bytes, those of the FP64 kernel's 32 rows 8
  int64_t *part = reinterpret_cast<int64_t *>(best.part_f64);
  k_energy_dense_fx<<<grid, kFxThreads, kFxSmem, st>>>(p->A, B, s, Kp, err, p->H, part);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_energy_fx_final<<<unsigned((s.C + 7) / 8), 256, 0, st>>>(s.C, s.Cp, Kp / kTcBM, p->k, part, best.e_f64);
  return cudaGetLastError();
}

}  // namespace sbqa
