// step_dense.cu -- one SBQA step for dense couplings on the CUDA cores
// (Sec. II A, Eq. 7, G = J f(X) with an N x N matrix), product and update
// fused.  This is the general dense path (any real J in FP32, small-integer J
// exactly) and that of the ballistic form f(x) = x with FP32 positions; the
// tensor-core paths live in step_dense_tc.cu.
//
// Every G_ic is the sequence of fused multiply-adds over j = 0 .. N - 1, so K
// is not split.  The FMAs take the packed form (two rows of a column per
// instruction; scalar ones stopped at half the rate), and then two rates bound
// the loop: the FMA pipe, and what shared memory returns to the registers (128
// bytes per clock and SM, a broadcast counting per lane).  A lane owns 2 CW
// rows x CW columns, a warp 2 CW rows x 32 CW columns: per spin j it reads the
// J values of its rows by CW / 2 16-byte broadcasts -- a stage holds J by spin,
// rows side by side, which the symmetric J gives without a transposition -- and
// CW columns of f, which the stage already holds as floats.  A block takes 32
// rows.  CW = 4 (128 columns, 4 warps) is the better tile (FMA pipe 80 % busy
// on the fullest SM); where it gives fewer blocks than SMs, CW = 2 (64 columns,
// 8 warps, P <= 64) fills more of them.  Stages of 32 spins: J and positions by
// cp.async up to two stages ahead, f codes through registers a stage ahead
// (decoded on the way); within a stage the operands of the next four spins are
// read while four are multiplied.  (Codes kept as bytes and decoded after the
// read, 4 x 4 per lane: 23.4 us at N = 1000, R*P = 256, but 239 at N = 2000.)
// us per step with 32 x 128 tiles of 4 x 4 per lane, f decoded at every use,
// and now: N = 1000, R*P = 256 53.7 -> 23.9, R*P = 1024 92.6 -> 57.9; N = 2000,
// R*P = 1024 341 -> 201; N = 200, R*P = 256 14.6 -> 7.1; ballistic N = 1000,
// R*P = 256 54.1 -> 23.7.
#include "step_common.cuh"

namespace sbqa {

constexpr int kDenseRows = 32, kDenseK = 32;
constexpr int kDenseLdj = kDenseRows + 4;  // floats of one spin's J column piece in a stage

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

// A lane's tile is 2 CW rows x CW columns.
constexpr int dense_threads(int CW) { return 32 * kDenseRows / (2 * CW); }

template <int P, int CW, bool BSB>
__global__ void __launch_bounds__(dense_threads(CW)) k_step_dense(StateView s, DenseView J, StepTables t, int n) {
  constexpr int kCols = 32 * CW, kStages = CW == 2 ? 3 : 2, kThreads = dense_threads(CW), RW = 2 * CW;
  struct Stage {
    float j[kDenseK][kDenseLdj];  // [spin][row]: rows of the symmetric J read as its columns
    float f[kDenseK][kCols];
  };
  __shared__ __align__(16) Stage st[kStages];
  const int row0 = blockIdx.y * kDenseRows, col0 = blockIdx.x * kCols;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = s.N;
  const bool vec = N % 4 == 0;  // rows of J on 16-byte boundaries
  const uint8_t *F = BSB ? nullptr : s.f_of(n);
  const float *Fx = BSB ? s.fx_of(n) : nullptr;
  const int stages = (N + kDenseK - 1) / kDenseK;

  // J (and positions) of stage q on their way into its buffer; one group per call, empty past the end
  auto load = [&](int q) {
    if (q < stages) {
      Stage &g = st[q % kStages];
      const int k0 = q * kDenseK;
      if (vec) {
#pragma unroll
        for (int u = 0; u < kDenseRows * kDenseK / 4 / kThreads; ++u) {
          const int e = tid + u * kThreads, k = e >> 3, r = (e & 7) * 4;
          const bool ok = row0 + r < N && k0 + k < N;
          cp_async16(&g.j[k][r], J.J + (ok ? size_t(k0 + k) * N + row0 + r : 0), ok);
        }
      } else {
#pragma unroll
        for (int u = 0; u < kDenseRows * kDenseK / kThreads; ++u) {
          const int e = tid + u * kThreads, k = e >> 5, r = e & 31;
          const bool ok = row0 + r < N && k0 + k < N;
          cp_async4(&g.j[k][r], J.J + (ok ? size_t(k0 + k) * N + row0 + r : 0), ok);
        }
      }
      if constexpr (BSB) {
#pragma unroll
        for (int u = 0; u < kDenseK * kCols / 4 / kThreads; ++u) {
          const int e = tid + u * kThreads, r = e / (kCols / 4), c = e % (kCols / 4) * 4;
          const bool ok = k0 + r < N;
          cp_async16(&g.f[r][c], Fx + (ok ? size_t(k0 + r) * s.Cp + col0 + c : 0), ok);
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // f codes of a stage: into registers, and a stage later as floats into its buffer
  constexpr int kWords = kDenseK * kCols / 4 / kThreads;  // 4-code words per thread
  uint32_t codes[kWords];
  auto load_codes = [&](int q) {
    if constexpr (!BSB) {
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int e = tid + u * kThreads, r = q * kDenseK + e / (kCols / 4), c = e % (kCols / 4) * 4;
        codes[u] = kFZero4;  // f = 0 past the last spin
        if (r < N) codes[u] = __ldg(reinterpret_cast<const uint32_t *>(F + size_t(r) * s.Cp + col0 + c));
      }
    }
  };
  auto decode = [&](int q) {
    if constexpr (!BSB) {
      Stage &g = st[q % kStages];
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int e = tid + u * kThreads, r = e / (kCols / 4), c = e % (kCols / 4) * 4;
        *reinterpret_cast<float4 *>(&g.f[r][c]) =
            make_float4(fdec(codes[u], 0), fdec(codes[u], 1), fdec(codes[u], 2), fdec(codes[u], 3));
      }
    }
  };

  float2 acc[RW / 2][CW];  // rows 2 p and 2 p + 1 of the warp's RW
#pragma unroll
  for (int p = 0; p < RW / 2; ++p)
#pragma unroll
    for (int c = 0; c < CW; ++c) acc[p][c] = make_float2(0.f, 0.f);
  // operands of four spins, read while the four before are multiplied
  float4 w[2][4][RW / 4];
  float f[2][4][CW];
  auto fetch = [&](const Stage &g, int k, float4 (&wv)[4][RW / 4], float (&fv)[4][CW]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int h = 0; h < RW / 4; ++h) wv[u][h] = *reinterpret_cast<const float4 *>(&g.j[k + u][warp * RW + 4 * h]);
      if constexpr (CW == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(&g.f[k + u][2 * lane]);
        fv[u][0] = v.x; fv[u][1] = v.y;
      } else {
        const float4 v = *reinterpret_cast<const float4 *>(&g.f[k + u][4 * lane]);
        fv[u][0] = v.x; fv[u][1] = v.y; fv[u][2] = v.z; fv[u][3] = v.w;
      }
    }
  };
  for (int q = 0; q < kStages - 1; ++q) load(q);
  load_codes(0);
  decode(0);
  load_codes(1);
  for (int q = 0; q < stages; ++q) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // stage q is in shared memory; the buffer of stage q - 1 has been read
    load(q + kStages - 1);
    const Stage &g = st[q % kStages];
    fetch(g, 0, w[0], f[0]);
#pragma unroll
    for (int k = 0; k < kDenseK; k += 4) {
      const int b = (k / 4) & 1;
      if (k + 4 < kDenseK) fetch(g, k + 4, w[b ^ 1], f[b ^ 1]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          const float2 ff = make_float2(f[b][u][c], f[b][u][c]);
#pragma unroll
          for (int h = 0; h < RW / 4; ++h) {
            const float4 v = w[b][u][h];
            acc[2 * h][c] = __ffma2_rn(make_float2(v.x, v.y), ff, acc[2 * h][c]);
            acc[2 * h + 1][c] = __ffma2_rn(make_float2(v.z, v.w), ff, acc[2 * h + 1][c]);
          }
        }
      if (k == kDenseK / 2 && q + 1 < stages) {  // the codes of the next stage have arrived by now
        decode(q + 1);
        load_codes(q + 2);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // The update takes 4 consecutive columns per lane: with CW = 2 the sums pass
  // through shared memory (the warp's own rows), two rows per warp at a time.
  __syncthreads();
  float *tile = reinterpret_cast<float *>(st) + warp * RW * kCols;
#pragma unroll
  for (int p = 0; p < RW / 2; ++p)
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      tile[2 * p * kCols + CW * lane + c] = acc[p][c].x;
      tile[(2 * p + 1) * kCols + CW * lane + c] = acc[p][c].y;
    }
  __syncwarp();
  constexpr int kLanes = kCols / 4, kRowsAtOnce = 32 / kLanes;
  const int c4 = col0 + lane % kLanes * 4;
#pragma unroll
  for (int a = 0; a < RW; a += kRowsAtOnce) {
    const int r = a + lane / kLanes, i = row0 + warp * RW + r;
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

// 128-column tiles when there is one for every SM (or a run spans more than 64
// columns), else 64-column ones (N = 1000, R*P = 1024, 256 wide tiles: 58 us per
// step against 79 with narrow ones).
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
    if (int64_t(rows) * (s.Cp / 128) < sms) {
      k_step_dense<P, 2, BSB><<<dim3(s.Cp / 64, rows), dense_threads(2), 0, st>>>(s, J, t, n);
      return cudaGetLastError();
    }
  }
  k_step_dense<P, 4, BSB><<<dim3(s.Cp / 128, rows), dense_threads(4), 0, st>>>(s, J, t, n);
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
