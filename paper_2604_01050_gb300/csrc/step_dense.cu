// step_dense.cu -- one SBQA step for dense couplings on the CUDA cores
// (Sec. II A, Eq. 7, G = J f(X) with an N x N matrix), product and update
// fused.  This is the general dense path (any real J in FP32, small-integer J
// exactly) and that of the ballistic form f(x) = x with FP32 positions; the
// tensor-core paths live in step_dense_tc.cu.
//
// Every G_ic is the sequence of fused multiply-adds over j = 0 .. N - 1, so K
// is not split; the FMA rate bounds the step once its operands come from
// shared memory in few enough reads.  A warp owns 8 rows x 32 CW columns, a
// lane 8 rows x CW columns: per spin j it reads one quarter of a 16-byte
// broadcast per row (four j at a time) and CW columns of f, which the stage
// already holds as floats -- 2 + CW shared-memory wavefronts for 8 CW FMAs per
// lane.  (One lane with 4 rows x 4 columns, f decoded at every use and J read
// word by word, took 8 loads and 20 other instructions for 16 FMAs.)
// Four warps take 32 rows.  CW = 2 (64 columns, P <= 64) where 128-column
// tiles would leave SMs idle, else CW = 4.  Stages of 32 spins, two in flight:
// J by cp.async, f codes through registers (decoded on the way), positions by
// cp.async.  N = 1000, R*P = 256: 69 -> 35 us per step.
#include "step_common.cuh"

namespace sbqa {

constexpr int kDenseRows = 32, kDenseK = 32, kDenseThreads = 128;
constexpr int kDenseLdj = kDenseK + 4;  // floats of a J row in a stage: 16-byte aligned, rows in different banks

__device__ __forceinline__ void cp_async4(void *dst, const void *src, bool valid) {
  const uint32_t d = uint32_t(__cvta_generic_to_shared(dst));
  const int n = valid ? 4 : 0;  // the rest of the word is zero-filled
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid) {
  const uint32_t d = uint32_t(__cvta_generic_to_shared(dst));
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

template <int P, int CW, bool BSB>
__global__ void __launch_bounds__(kDenseThreads) k_step_dense(StateView s, DenseView J, StepTables t, int n) {
  constexpr int kCols = 32 * CW;
  struct Stage {
    float j[kDenseRows][kDenseLdj];
    float f[kDenseK][kCols];
  };
  __shared__ __align__(16) Stage st[2];
  const int row0 = blockIdx.y * kDenseRows, col0 = blockIdx.x * kCols;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = s.N;
  const bool vec = N % 4 == 0;  // rows of J on 16-byte boundaries
  const uint8_t *F = BSB ? nullptr : s.f_of(n);
  const float *Fx = BSB ? s.fx_of(n) : nullptr;

  // f codes of a stage in registers: kCols / 4 bytes per thread and pass of 32 spins
  constexpr int kWords = kDenseK * kCols / 4 / kDenseThreads;  // 4-code words per thread
  uint32_t codes[kWords];
  auto load = [&](int k0, Stage &q) {
    if (vec) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int e = tid + u * kDenseThreads, r = e >> 3, k = (e & 7) * 4;
        const bool ok = row0 + r < N && k0 + k < N;
        cp_async16(&q.j[r][k], J.J + (ok ? size_t(row0 + r) * N + k0 + k : 0), ok);
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = tid + u * kDenseThreads, r = e >> 5, k = e & 31;
        const bool ok = row0 + r < N && k0 + k < N;
        cp_async4(&q.j[r][k], J.J + (ok ? size_t(row0 + r) * N + k0 + k : 0), ok);
      }
    }
    if constexpr (BSB) {
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int e = tid + u * kDenseThreads, r = e / (kCols / 4), c = e % (kCols / 4) * 4;
        const bool ok = k0 + r < N;
        cp_async16(&q.f[r][c], Fx + (ok ? size_t(k0 + r) * s.Cp + col0 + c : 0), ok);
      }
    } else {
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int e = tid + u * kDenseThreads, r = e / (kCols / 4), c = e % (kCols / 4) * 4;
        codes[u] = kFZero4;  // f = 0 past the last spin
        if (k0 + r < N) codes[u] = __ldg(reinterpret_cast<const uint32_t *>(F + size_t(k0 + r) * s.Cp + col0 + c));
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto decode = [&](Stage &q) {
    if constexpr (!BSB) {
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int e = tid + u * kDenseThreads, r = e / (kCols / 4), c = e % (kCols / 4) * 4;
        *reinterpret_cast<float4 *>(&q.f[r][c]) =
            make_float4(fdec(codes[u], 0), fdec(codes[u], 1), fdec(codes[u], 2), fdec(codes[u], 3));
      }
    }
  };

  float acc[8][CW];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < CW; ++c) acc[a][c] = 0.f;
  const int stages = (N + kDenseK - 1) / kDenseK;
  load(0, st[0]);
  decode(st[0]);
  for (int q = 0; q < stages; ++q) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // stage q is in shared memory; stage q + 1's buffer has been read
    const bool more = q + 1 < stages;
    if (more) load((q + 1) * kDenseK, st[(q + 1) & 1]);
    const Stage &g = st[q & 1];
#pragma unroll
    for (int k = 0; k < kDenseK; k += 4) {
      float w[8][4];
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const float4 v = *reinterpret_cast<const float4 *>(&g.j[warp * 8 + a][k]);
        w[a][0] = v.x; w[a][1] = v.y; w[a][2] = v.z; w[a][3] = v.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float f[CW];
        if constexpr (CW == 2) {
          const float2 v = *reinterpret_cast<const float2 *>(&g.f[k + u][2 * lane]);
          f[0] = v.x; f[1] = v.y;
        } else {
          const float4 v = *reinterpret_cast<const float4 *>(&g.f[k + u][4 * lane]);
          f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
        }
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int c = 0; c < CW; ++c) acc[a][c] = fmaf(w[a][u], f[c], acc[a][c]);
      }
    }
    if (more) decode(st[(q + 1) & 1]);
  }
  // The update takes 4 consecutive columns per lane: with CW = 2 the sums pass
  // through shared memory (the warp's own rows), two rows per warp at a time.
  __syncthreads();
  float *tile = reinterpret_cast<float *>(st) + warp * 8 * kCols;
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int c = 0; c < CW; ++c) tile[a * kCols + CW * lane + c] = acc[a][c];
  __syncwarp();
  constexpr int kLanes = kCols / 4, kRowsAtOnce = 32 / kLanes;
  const int c4 = col0 + lane % kLanes * 4;
#pragma unroll
  for (int a = 0; a < 8; a += kRowsAtOnce) {
    const int r = a + lane / kLanes, i = row0 + warp * 8 + r;
    const bool ok = i < N;  // a lane past the last row takes part in the ring shuffles only
    const size_t off = size_t(ok ? i : N - 1) * s.Cp + c4;
    const float4 xv = *reinterpret_cast<const float4 *>(s.x + off), yv = *reinterpret_cast<const float4 *>(s.y + off);
    const float4 g = *reinterpret_cast<const float4 *>(&tile[r * kCols + lane % kLanes * 4]);
    const float G[4] = {g.x, g.y, g.z, g.w};
    const float hi = ok ? __ldg(J.h + i) : 0.f;
    const int cu = ok ? c4 : s.C;
    if constexpr (BSB) sb_update4_bsb<P>(s, t, n, i, cu, G, hi, xv, yv, s.fx_of(n + 1));
    else sb_update4<P>(s, t, n, i, cu, G, hi, xv, yv, s.f_of(n + 1));
  }
}

// 128-column tiles when they give every SM at least two blocks (or a run
// spans more than 64 columns), else 64-column ones.
template <int P, bool BSB>
static cudaError_t launch_p(const StateView &s, const DenseView &J, const StepTables &t, int n, cudaStream_t st) {
  const unsigned rows = unsigned((s.N + kDenseRows - 1) / kDenseRows);
  static const int sms = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
  }();
  if constexpr (P <= 64) {
    if (int64_t(rows) * (s.Cp / 128) < 2 * sms) {
      k_step_dense<P, 2, BSB><<<dim3(s.Cp / 64, rows), kDenseThreads, 0, st>>>(s, J, t, n);
      return cudaGetLastError();
    }
  }
  k_step_dense<P, 4, BSB><<<dim3(s.Cp / 128, rows), kDenseThreads, 0, st>>>(s, J, t, n);
  return cudaGetLastError();
}

template <bool BSB>
static cudaError_t launch(const StateView &s, const DenseView &J, const StepTables &t, int n, cudaStream_t st) {
  switch (s.P) {
    case 1: return launch_p<1, BSB>(s, J, t, n, st);
    case 2: return launch_p<2, BSB>(s, J, t, n, st);
    case 4: return launch_p<4, BSB>(s, J, t, n, st);
    case 8: return launch_p<8, BSB>(s, J, t, n, st);
    case 16: return launch_p<16, BSB>(s, J, t, n, st);
    case 32: return launch_p<32, BSB>(s, J, t, n, st);
    case 64: return launch_p<64, BSB>(s, J, t, n, st);
    case 128: return launch_p<128, BSB>(s, J, t, n, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step_dense(const StateView &s, const DenseView &J, const StepTables &t, int n,
                              cudaStream_t st) {
  return launch<false>(s, J, t, n, st);
}

cudaError_t launch_step_dense_bsb(const StateView &s, const DenseView &J, const StepTables &t, int n,
                                  cudaStream_t st) {
  return launch<true>(s, J, t, n, st);
}

}  // namespace sbqa
