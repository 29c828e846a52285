// solve_persistent.cu -- all steps of a CSR run batch in one cooperative launch.
//
// For rows of degree <= 32 (+-1, FP32 or BF16 couplings; up to 8 for the
// ballistic form, whose lists and the streaming form's are of 8 slots).  One
// block of kPersistWarps (24) warps per SM; every warp owns fixed work items
// (spin row, 128 or 256 replica columns) for the whole launch.  A pass is what
// the warp works on at a time: one 256-column item, or two 128-column ones on
// its half warps (8 columns per lane either way).
//
// What a launch reads from memory more than once it keeps on the SM:
//   neighbour lists (columns, signs or values, degrees) in shared memory;
//   x and y of a warp's first kTmemPasses (5) passes in tensor memory (the
//   block takes all 512 TMEM columns; the kWarpTmem = 80 of a warp hold 5
//   passes of 8 + 8 values per lane) and of kMaxSlots (1) more in shared
//   memory (2 KB).
// Passes past those keep x and y in global memory, so a launch of any size
// streams only the part of its state that does not fit the chip.  The 3648
// warps of 152 SMs hold 37 MB of state in TMEM and 7.5 MB in shared memory: 6
// of the 9 passes (67 MB) of the L = 16 lattice with R*P = 2048, whose other
// passes stay in L2, and 6 of the 14 (102 MB) of N = 10^5 with R*P = 128.
// Between SMs only the one-byte f codes move, through L2 (relaxed accesses at GPU
// scope: other blocks read and write them).
//
// What bounds a pass then is the ALU pipe (compares, selects, logic, byte
// permutes at half rate: about 150 a pass; busy 69 % of the cycles at L = 16,
// 63 % at degree 20, 75 % in the ballistic form) and the latency of the
// gathers; 24 warps of 80 registers were faster than 32 of 64, which spill much
// more (lattice L = 16 13.3 against 16.1 us per step), and one 2 KB state slot
// per warp faster than more, which take the L1 the gathers pass through (14.5
// with three, 17.4 with four).  At 80 registers the short lists of +-1 and real
// J do not spill for P = 2, 4 and 16 up (P = 1: at most 12 bytes, P = 8: 4 to 36),
// the ballistic form spills 4 to 16 bytes, and the long lists 12 to 60 but for
// those of real J on half warps from P = 16 up, which do not; at P = 8 260 to 460
// bytes: a general and a plain ring stand side by side.
// us per step, before (the streaming form) and with this kernel:
//   lattice L = 16, R*P = 2048     24.0 -> 13.3    random graph N = 10^5,
//   lattice L = 10, R*P = 1024      4.9 ->  3.1    R*P = 128, BF16 46.8 -> 27.8
//   lattice L = 24, R*P = 2048     81.9 -> 70.2    N = 3000 3.0 -> 2.0
//   degree 12 (per-step kernels before), N = 20000, R*P = 128, FP32 13.9 -> 8.5
//   degree 20, N = 3001, R*P = 160 6.1 -> 4.4; N = 60000, R*P = 128 52.8 -> 35.9
//   ballistic L = 16 36.6 -> 32.0, L = 12, R*P = 512 5.6 -> 3.8, N = 10^5 61.8 -> 55.3
//
// Per pass a warp gathers the codes of the (at most 8) neighbours, sums (same
// arithmetic and order as k_step_csr), updates and writes the next codes.
//
// Steps are not separated by a grid barrier: every f code carries one bit of
// its generation, and a warp that gathers a code of the generation before
// reads it again until the new one has arrived.  The f buffers alternate by
// step parity, so a buffer's generation is (steps since the launch began + 1)
// / 2 mod 2, and the bit tells the codes of step n from those of step n - 2
// (0 in the buffer the launch starts from, and in the other one, which the
// launch clears first; the host keeps ballistic states with |x| >= 2, whose
// bit would read as 1, on the per-step kernel).  Overwriting is safe because the couplings are
// symmetric: row i writes f_{n+1} over f_{n-1} only after it has read f_n of
// all its neighbours, and a neighbour wrote its f_n after it had read f_{n-1}
// of row i.  A code is its own message (one byte holds value and bit), so no
// fence orders it behind anything else.  The grid is co-resident
// (cooperative launch), so the lowest step always progresses.  A wait is
// bounded (1 s, or at once when another warp has already failed): a warp that
// gives up records an error and stops stepping, and the launch ends with a
// status the host reads.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "grid_sync.cuh"  // globaltimer_ns and the limits of a bounded wait
#include "step_common.cuh"
#include "tc_common.cuh"

namespace sbqa {

constexpr int kPersistMaxDeg = 8;    // slots of the short lists
constexpr int kPersistWideDeg = 32;  // and of the long ones
constexpr int kWideAtOnce = 12;      // slots of a long list gathered at a time (24 registers of codes; 16 and 24 spill more)
constexpr int kPersistWarps = 24, kPersistThreads = 32 * kPersistWarps;
constexpr int kPersistSmem = 225 * 1024;               // dynamic shared memory of a block
constexpr int kWarpSmem = kPersistSmem / kPersistWarps;  // 9600 bytes per warp
constexpr int kSlotBytes = 2048;                       // x, y of one pass: 16 floats x 32 lanes
constexpr uint32_t kPersistTmem = 512;                 // the block takes all TMEM columns of its SM
constexpr int kMaxSlots = 1;                           // state slots per warp: what shared memory takes, L1 lacks
// Passes per warp; run batches with more take the streaming form (30 passes, L
// = 24: 70 us per step against 82 there; 72, L = 32: 183 there)
constexpr int kMaxPasses = 40;
static_assert(2 * kMaxPasses * 76 + kSlotBytes <= kWarpSmem, "lists and state slots fit a warp's shared memory");
constexpr int kTmemPasses = 5;                         // x, y of 5 passes
constexpr int kWarpTmem = 80;                          // TMEM columns per warp: 6 warps share a lane quarter
static_assert(kPersistWarps / 4 * kWarpTmem <= 512 && 16 * kTmemPasses <= kWarpTmem, "TMEM columns");
static_assert(kWarpSmem % 16 == 0, "warp regions hold 16-byte vectors");

struct PersistArgs {
  StateView s;
  const float *h;
  // ELL form of the couplings (rows of degree <= 8, the CSR kernels' entry order)
  const int32_t *ell_col, *ell_meta;
  const float *ell_val;
  CsrView csr;    // the long lists are filled from the CSR arrays
  int wide;       // slots of a long list (degree rounded up to a multiple of 4)
  StepTables t;
  int n_begin, n_end;
  int *err;       // error flag
  int skip_step;  // test hook: block 0 does not publish the codes of this step (-1: never)
  int degree;     // largest row degree: a pass reads 4, 6 or 8 slots
  int cache_cap;  // items a warp holds at most
  int slots;      // passes (ballistic form: items) whose state is kept in shared memory
  int warp_smem;  // bytes of a warp's shared memory: its slots, then its cache
};

// Bytes of one cached item: 8 columns, 8 values (signs as bytes for +-1), a
// word of the degree and the sum of the signs, and (row, chunk).  Unused
// slots name the row itself with weight 0, so that a pass reads the same
// number of slots for every row without a test per slot.
constexpr int entry_bytes(bool vals) { return 32 + (vals ? 32 : 8) + 4 + 8; }

// A warp's cached neighbour lists, in arrays over its entries.
template <bool VALS>
struct WarpCache {
  int4 *cols;     // [2 cap]
  float4 *vals;   // [2 cap]; +-1: int2 [cap] of signed bytes
  int2 *item;     // [cap] (row, chunk)
  uint32_t *meta;  // [cap] degree | (sum of signs) << 16
  __device__ WarpCache(char *base, int cap) {
    cols = reinterpret_cast<int4 *>(base);
    base += 32 * cap;
    vals = reinterpret_cast<float4 *>(base);
    base += (VALS ? 32 : 8) * cap;
    item = reinterpret_cast<int2 *>(base);
    base += 8 * cap;
    meta = reinterpret_cast<uint32_t *>(base);
  }
  // Fills entry q with row `row` (lanes 0-7 one slot each).
  __device__ __forceinline__ void fill(const PersistArgs &a, int q, int row, int chunk, int lane) const {
    const int2 m = __ldg(reinterpret_cast<const int2 *>(a.ell_meta) + row);  // (degree, +1 count)
    if (lane < kPersistMaxDeg) {
      const bool used = lane < m.x;
      reinterpret_cast<int32_t *>(cols)[8 * q + lane] =
          used ? __ldg(a.ell_col + size_t(row) * kPersistMaxDeg + lane) : row;
      if constexpr (VALS)
        reinterpret_cast<float *>(vals)[8 * q + lane] =
            used ? __ldg(a.ell_val + size_t(row) * kPersistMaxDeg + lane) : 0.f;
      else
        reinterpret_cast<int8_t *>(vals)[8 * q + lane] = used ? (lane < m.y ? 1 : -1) : 0;
    } else if (lane == kPersistMaxDeg) {
      meta[q] = uint32_t(m.x) | (uint32_t(2 * m.y - m.x) << 16);
      item[q] = make_int2(row, chunk);
    }
  }
};

// The same for rows of up to 32 entries: lists of W slots (a multiple of 4),
// filled from the CSR arrays a slot per lane.
constexpr int wide_bytes(int W, bool vals) { return 4 * W + (vals ? 4 * W : W) + 12; }

template <bool VALS>
struct WideCache {
  int4 *cols;      // [cap][W / 4]
  float4 *vals;    // [cap][W / 4]
  int2 *item;      // [cap] (row, chunk)
  uint32_t *meta;  // [cap] degree | (sum of signs) << 16
  uint32_t *signs;  // [cap][W / 4] signed bytes
  int W;
  __device__ WideCache(char *base, int cap, int w) : W(w) {
    cols = reinterpret_cast<int4 *>(base);
    base += 4 * W * cap;
    vals = reinterpret_cast<float4 *>(base);
    if (VALS) base += 4 * W * cap;
    item = reinterpret_cast<int2 *>(base);
    base += 8 * cap;
    meta = reinterpret_cast<uint32_t *>(base);
    signs = meta + cap;
  }
  __device__ __forceinline__ void fill(const PersistArgs &a, int q, int row, int chunk, int lane) const {
    const int e0 = __ldg(a.csr.row_ptr + row), deg = __ldg(a.csr.row_ptr + row + 1) - e0;
    const int pos = VALS ? deg : __ldg(a.csr.npos + row);
    if (lane < W) {
      const bool used = lane < deg;
      reinterpret_cast<int32_t *>(cols)[W * q + lane] = used ? __ldg(a.csr.col + e0 + lane) : row;
      if constexpr (VALS) {
        float v = 0.f;
        if (used)
          v = a.csr.kind == VAL_BF16 ? __bfloat162float(static_cast<const __nv_bfloat16 *>(a.csr.val)[e0 + lane])
                                     : static_cast<const float *>(a.csr.val)[e0 + lane];
        reinterpret_cast<float *>(vals)[W * q + lane] = v;
      } else {
        reinterpret_cast<int8_t *>(signs)[W * q + lane] = used ? (lane < pos ? 1 : -1) : 0;
      }
    }
    if (lane == 0) {
      meta[q] = uint32_t(deg) | (uint32_t(2 * pos - deg) << 16);
      item[q] = make_int2(row, chunk);
    }
  }
};

// f codes (8 bytes) and positions (16 bytes) that other SMs write in this
// launch, through L2; volatile, so that a wait reads them again.
struct Codes8 {
  uint32_t w[2];
  __device__ __forceinline__ void load(const uint8_t *p) {
    asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p) : "memory");
  }
};
__device__ __forceinline__ void publish(uint8_t *p, uint32_t a, uint32_t b) {
  asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}
struct Pos4 {
  uint32_t w[4];
  __device__ __forceinline__ void load(const float *p) {
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "l"(p)
                 : "memory");
  }
};

// 8 consecutive floats, loaded where this stands in the program (a plain load
// may be moved down to its use).
__device__ __forceinline__ void load_row_now(const float *p, float (&v)[8]) {
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p + 4));
}

// Generation bits: the top bit of every code byte; bit 30 of a position
// (|x| <= 1 after an update, so its exponent leaves that bit 0).
constexpr uint32_t kTagCodes = 0x80808080u, kTagPos = 0x40000000u;
// the bit of step n's codes in a launch that began at step n0 (0 for n = n0)
__device__ __forceinline__ uint32_t tag_of(int n, int n0, uint32_t bits) { return ((n - n0 + 1) & 2) ? bits : 0u; }

// Whether the bounded wait that has read its entries `it` times gives up (looked
// at every 16th time; t0 = 0 before); records the error then.
__device__ __forceinline__ bool wait_over(unsigned it, uint64_t &t0, int *err) {
  if ((it & 15) != 15) return false;
  const uint64_t now = globaltimer_ns();
  if (t0 == 0) t0 = now;
  const bool over = now - t0 > kBarrierTimeoutNs || it > kBarrierSpins || *(volatile int *)err != 0;
  if (!__any_sync(0xffffffffu, over)) return false;
  if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, 4);
  return true;
}

// Packed sums of sign * code of four columns a word: per byte 64 + the sum over
// the entries, between 0 and 128 for up to 32 of them.
__device__ __forceinline__ uint32_t packed_start(uint32_t tag, int sum) { return 0x40404040u - tag * uint32_t(sum); }
__device__ __forceinline__ void add_signed(uint32_t (&acc)[2], const Codes8 &f, uint32_t signs, int byte) {
  const uint32_t b = uint32_t(byte);
  uint32_t sign;  // the byte, sign extended
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(sign) : "r"(signs), "r"(b | (0x888u | b * 0x111u) << 4));
  acc[0] += sign * f.w[0];
  acc[1] += sign * f.w[1];
}
__device__ __forceinline__ void packed_finish(const uint32_t (&acc)[2], int sum, float (&G)[8]) {
  const float off = -8388608.f - float(64 + sum);
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    const uint32_t m0 = __byte_perm(acc[c / 4], 0x4B000000u, 0x7540u | uint32_t(c % 4));
    const uint32_t m1 = __byte_perm(acc[c / 4], 0x4B000000u, 0x7540u | uint32_t(c % 4 + 1));
    const float2 g = __fadd2_rn(make_float2(__uint_as_float(m0), __uint_as_float(m1)), make_float2(off, off));
    G[c] = g.x;
    G[c + 1] = g.y;
  }
}
// -(2^23 + 1), and the generation bit of a code read through the low mantissa bits of 2^23
__device__ __forceinline__ float code_offset(uint32_t tag) { return tag ? -8388737.f : -8388609.f; }

// Coupling sums of one pass from the gathered codes of the lane's 8 columns
// (with their generation bits).  +-1: packed sums of sign * code -- integers
// modulo 2^32, so the bits and the offset codes carry are taken out at the
// end, in the low mantissa bits of 2^23 (exact); otherwise FP32 FMAs in entry
// order, as k_step_csr, each code through the low mantissa bits of 2^23.
// The integer multiply-adds and FP32 adds run on the FMA pipes: the ALU pipe,
// which takes every compare, select, logic and byte-permute instruction at
// half rate, is what bounds a pass.
template <int KIND>
__device__ __forceinline__ void sum_codes(const Codes8 (&f)[kPersistMaxDeg], uint32_t tag, const float4 *vals,
                                          uint32_t meta, int slots, float (&G)[8]) {
  if constexpr (KIND == VAL_PM1) {
    const int2 sg = *reinterpret_cast<const int2 *>(vals);
    const int sum = int(meta) >> 16;
    uint32_t acc[2];
    acc[0] = acc[1] = packed_start(tag, sum);
    auto add = [&](int e) { add_signed(acc, f[e], uint32_t(e < 4 ? sg.x : sg.y), e & 3); };
#pragma unroll
    for (int e = 0; e < 4; ++e) add(e);
    if (slots > 4) {
      add(4);
      add(5);
    }
    if (slots > 6) {
      add(6);
      add(7);
    }
    packed_finish(acc, sum, G);
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) G[c] = 0.f;
    const float off = code_offset(tag);
    const float4 v = vals[0];
    acc_codes_off<8>(G, v.x, f[0].w, off);
    acc_codes_off<8>(G, v.y, f[1].w, off);
    acc_codes_off<8>(G, v.z, f[2].w, off);
    acc_codes_off<8>(G, v.w, f[3].w, off);
    if (slots > 4) {
      const float4 u = vals[1];
      acc_codes_off<8>(G, u.x, f[4].w, off);
      acc_codes_off<8>(G, u.y, f[5].w, off);
      if (slots > 6) {
        acc_codes_off<8>(G, u.z, f[6].w, off);
        acc_codes_off<8>(G, u.w, f[7].w, off);
      }
    }
  }
}

// Whether all gathered codes carry the generation bits of tag: the AND (bits
// set) or the OR (bits clear) of their words.
__device__ __forceinline__ bool codes_fresh(const Codes8 (&f)[kPersistMaxDeg], uint32_t tag, int slots) {
  if (tag) {
    uint32_t v = f[0].w[0] & f[0].w[1];
#pragma unroll
    for (int e = 1; e < 4; ++e) v &= f[e].w[0] & f[e].w[1];
    if (slots > 4) v &= f[4].w[0] & f[4].w[1] & f[5].w[0] & f[5].w[1];
    if (slots > 6) v &= f[6].w[0] & f[6].w[1] & f[7].w[0] & f[7].w[1];
    return (v & kTagCodes) == kTagCodes;
  }
  uint32_t v = f[0].w[0] | f[0].w[1];
#pragma unroll
  for (int e = 1; e < 4; ++e) v |= f[e].w[0] | f[e].w[1];
  if (slots > 4) v |= f[4].w[0] | f[4].w[1] | f[5].w[0] | f[5].w[1];
  if (slots > 6) v |= f[6].w[0] | f[6].w[1] | f[7].w[0] | f[7].w[1];
  return (v & kTagCodes) == 0;
}

// LPI = 32: passes of one 256-column item on the whole warp; 16: of two 128-column ones on half warps.
// WIDE: lists of up to 32 slots, gathered and summed 12 at a time.
template <int P, int KIND, int LPI, bool WIDE>
__global__ void __launch_bounds__(kPersistThreads, 1) k_solve_csr_persistent(PersistArgs a) {
  constexpr bool VALS = KIND != VAL_PM1;
  constexpr int IPW = 32 / LPI;  // items per pass
  extern __shared__ __align__(16) char s_raw[];
  __shared__ uint32_t s_tmem;
  const StateView &s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LPI;
  const int chunks = s.Cp / (LPI * 8);
  const int warps_total = gridDim.x * kPersistWarps;
  const int gw = blockIdx.x * kPersistWarps + warp;
  char *mine = s_raw + warp * a.warp_smem;
  float4 *state = reinterpret_cast<float4 *>(mine);  // [slots][x lo, x hi, y lo, y hi][lane]
  const auto cache = [&] {
    if constexpr (WIDE) return WideCache<VALS>(mine + a.slots * kSlotBytes, a.cache_cap, a.wide);
    else return WarpCache<VALS>(mine + a.slots * kSlotBytes, a.cache_cap);
  }();
  if (warp == 0) tc::tmem_alloc(&s_tmem, kPersistTmem);
  int my_count = 0;
  const int n_units = s.N * chunks;
  for (int u = gw; u < n_units && my_count < a.cache_cap; u += warps_total, ++my_count) {
    const int row = u / chunks;
    cache.fill(a, my_count, row, u - row * chunks, lane);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  // TMEM columns of this warp: its 32 lanes of the quarter warp % 4
  const uint32_t tm = s_tmem + (uint32_t(warp & 3) << 21) + uint32_t(warp >> 2) * kWarpTmem;
  const int passes = (my_count + IPW - 1) / IPW;
  const int resident = min(passes, kTmemPasses + a.slots);

  // A pass: the entry, row and first column of this lane; live = false: a half warp without an
  // item, or columns past C.
  struct Pass {
    int e, i, c0;
    bool live;
  };
  auto locate = [&](int p) {
    Pass t;
    t.e = p * IPW + sub;
    t.live = t.e < my_count;
    if (!t.live) t.e = p * IPW;
    const int2 it = cache.item[t.e];
    t.i = it.x;
    t.c0 = it.y * (LPI * 8) + (lane % LPI) * 8;
    t.live = t.live && t.c0 < s.C;
    return t;
  };
  auto put = [&](int p, const float (&xs)[8], const float (&ys)[8]) {
    if (p < kTmemPasses) {
      uint32_t r[16];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        r[j] = __float_as_uint(xs[j]);
        r[8 + j] = __float_as_uint(ys[j]);
      }
      tc::tmem_st_32x32b_x16(tm + uint32_t(p) * 16u, r);
    } else {
      float4 *q = state + (p - kTmemPasses) * 128 + lane;
      q[0] = make_float4(xs[0], xs[1], xs[2], xs[3]);
      q[32] = make_float4(xs[4], xs[5], xs[6], xs[7]);
      q[64] = make_float4(ys[0], ys[1], ys[2], ys[3]);
      q[96] = make_float4(ys[4], ys[5], ys[6], ys[7]);
    }
  };
  auto get = [&](int p, float (&xs)[8], float (&ys)[8]) {
    if (p < kTmemPasses) {
      uint32_t r[16];
      tc::tmem_ld_32x32b_x16_nowait(tm + uint32_t(p) * 16u, r);
      tc::tmem_wait_ld();
      tc::reg_fence_n(r);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        xs[j] = __uint_as_float(r[j]);
        ys[j] = __uint_as_float(r[8 + j]);
      }
    } else {
      const float4 *q = state + (p - kTmemPasses) * 128 + lane;
      const float4 x0 = q[0], x1 = q[32], y0 = q[64], y1 = q[96];
      xs[0] = x0.x; xs[1] = x0.y; xs[2] = x0.z; xs[3] = x0.w; xs[4] = x1.x; xs[5] = x1.y; xs[6] = x1.z; xs[7] = x1.w;
      ys[0] = y0.x; ys[1] = y0.y; ys[2] = y0.z; ys[3] = y0.w; ys[4] = y1.x; ys[5] = y1.y; ys[6] = y1.z; ys[7] = y1.w;
    }
  };
  for (int p = 0; p < resident; ++p) {
    const Pass t = locate(p);
    float xs[8], ys[8];
    load_row<8>(s.x + size_t(t.i) * s.Cp + t.c0, xs);
    load_row<8>(s.y + size_t(t.i) * s.Cp + t.c0, ys);
    put(p, xs, ys);
  }
  // replica counts below the run width take the general ring (one form per launch)
  const bool gen = P > 2 && s.Pr != P;

  // the codes of a row's neighbours at step n
  auto gather = [&](Codes8 (&f)[kPersistMaxDeg], int n, const int4 *cols, int c0) {
    const uint8_t *F = s.f_of(n) + c0;
    const int4 ca = cols[0];
    f[0].load(F + size_t(ca.x) * s.Cp);
    f[1].load(F + size_t(ca.y) * s.Cp);
    f[2].load(F + size_t(ca.z) * s.Cp);
    f[3].load(F + size_t(ca.w) * s.Cp);
    if (a.degree > 4) {
      const int4 cb = cols[1];
      f[4].load(F + size_t(cb.x) * s.Cp);
      f[5].load(F + size_t(cb.y) * s.Cp);
      if (a.degree > 6) {
        f[6].load(F + size_t(cb.z) * s.Cp);
        f[7].load(F + size_t(cb.w) * s.Cp);
      }
    }
  };
  // Gathers until all codes are of step n (lanes that are not live do not wait); false when the
  // warp gave up.
  auto fresh = [&](Codes8 (&f)[kPersistMaxDeg], int n, const int4 *cols, int c0, bool live, uint32_t tag) {
    uint64_t t0 = 0;
    for (unsigned it = 0;; ++it) {
      if (!__any_sync(0xffffffffu, live && !codes_fresh(f, tag, a.degree))) return true;
      if (n == a.n_begin) return true;  // the codes a launch starts from are complete whatever their bits
      if (wait_over(it, t0, a.err)) return false;
      gather(f, n, cols, c0);
    }
  };
  // Coupling sums of a long list; false when the warp gave up.
  auto wide_sums = [&](int n, const Pass &t, uint32_t tag, float (&G)[8]) {
    if constexpr (WIDE) {
      const uint8_t *F = s.f_of(n) + t.c0;
      const int W4 = a.wide / 4, sum = int(cache.meta[t.e]) >> 16;
      uint32_t acc[2];
      acc[0] = acc[1] = packed_start(tag, sum);
#pragma unroll
      for (int c = 0; c < 8; ++c) G[c] = 0.f;
      const float coff = code_offset(tag);
      for (int g0 = 0; g0 < W4; g0 += kWideAtOnce / 4) {
        const int4 *cols = cache.cols + W4 * t.e + g0;
        Codes8 f[kWideAtOnce];
        uint64_t t0 = 0;
        for (unsigned it = 0;; ++it) {  // until every live lane's codes are of step n
#pragma unroll
          for (int g = 0; g < kWideAtOnce / 4; ++g)
            if (g0 + g < W4) {
              const int4 c = cols[g];
              f[4 * g].load(F + size_t(c.x) * s.Cp);
              f[4 * g + 1].load(F + size_t(c.y) * s.Cp);
              f[4 * g + 2].load(F + size_t(c.z) * s.Cp);
              f[4 * g + 3].load(F + size_t(c.w) * s.Cp);
            }
          uint32_t all = ~0u, any = 0u;
#pragma unroll
          for (int g = 0; g < kWideAtOnce / 4; ++g)
            if (g0 + g < W4)
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                if (tag) all &= f[4 * g + u].w[0] & f[4 * g + u].w[1];
                else any |= f[4 * g + u].w[0] | f[4 * g + u].w[1];
              }
          const bool stale = tag ? (all & kTagCodes) != kTagCodes : (any & kTagCodes) != 0;
          if (!__any_sync(0xffffffffu, t.live && stale) || n == a.n_begin) break;
          if (wait_over(it, t0, a.err)) return false;
        }
#pragma unroll
        for (int g = 0; g < kWideAtOnce / 4; ++g)
          if (g0 + g < W4) {
            if constexpr (VALS) {
              const float4 v = cache.vals[W4 * t.e + g0 + g];
              acc_codes_off<8>(G, v.x, f[4 * g].w, coff);
              acc_codes_off<8>(G, v.y, f[4 * g + 1].w, coff);
              acc_codes_off<8>(G, v.z, f[4 * g + 2].w, coff);
              acc_codes_off<8>(G, v.w, f[4 * g + 3].w, coff);
            } else {
              const uint32_t sg = cache.signs[W4 * t.e + g0 + g];
#pragma unroll
              for (int u = 0; u < 4; ++u) add_signed(acc, f[4 * g + u], sg, u);
            }
          }
      }
      if constexpr (!VALS) packed_finish(acc, sum, G);
    }
    return true;
  };
  // Update of one pass from its coupling sums; slot < 0: the state is in xs, ys and goes back to
  // global memory, else it lives on the chip in that slot.
  auto update = [&](int n, const Pass &t, int slot, const float (&G)[8], const float (&kj)[P >= 8 ? 1 : 8 / P],
                    float hi, float ka, float dnext, float (&xs)[8], float (&ys)[8]) {
    const size_t off = size_t(t.i) * s.Cp + t.c0;
    if (slot >= 0) get(slot, xs, ys);
    float xm[8], xp[8];
    if (gen) ring_nb<P, 8, true>(xs, s.Pr, xm, xp);
    else ring_nb<P, 8, false>(xs, s.Pr, xm, xp);
    if (t.live) {
      uint32_t code[2];
      sb_advanceW<P, 8>(s.C, a.t.kc, a.t.kx, ka, dnext, kj, t.c0, G, hi, xm, xp, xs, ys, code);
      // the codes a launch leaves carry no bit
      const uint32_t next = n + 1 < a.n_end ? tag_of(n + 1, a.n_begin, kTagCodes) : 0u;
      if (!(n == a.skip_step && blockIdx.x == 0)) publish(s.f_of(n + 1) + off, code[0] | next, code[1] | next);
      if (slot < 0) {
        store_row<8>(s.x + off, xs);
        store_row<8>(s.y + off, ys);
      }
    }
    __syncwarp();
    if (slot >= 0) put(slot, xs, ys);
  };

  bool ok = true;
  for (int n = a.n_begin; ok && n < a.n_end; ++n) {
    const float ka = __ldg(a.t.ka + n), dnext = __ldg(a.t.dl + n + 1);
    const float *kjn = a.t.kj + size_t(n) * a.t.R;
    const uint32_t tag = tag_of(n, a.n_begin, kTagCodes);
    tc::tmem_wait_st();  // the step before's stores into TMEM are complete
    for (int p = 0; p < passes; ++p) {
      const Pass t = locate(p);
      float xs[8], ys[8], G[8], kj[P >= 8 ? 1 : 8 / P];
      const size_t off = size_t(t.i) * s.Cp + t.c0;
      float hi;
      if constexpr (!WIDE) {
        if (p >= resident) {
          load_row_now(s.x + off, xs);
          load_row_now(s.y + off, ys);
        }
        Codes8 f[kPersistMaxDeg];
        const int4 *cols = cache.cols + 2 * t.e;
        gather(f, n, cols, t.c0);
        load_kj<P, 8>(kjn, s.C, t.c0, kj);
        hi = __ldg(a.h + t.i);
        if (!(ok = fresh(f, n, cols, t.c0, t.live, tag))) break;
        sum_codes<KIND>(f, tag, VALS ? cache.vals + 2 * t.e : reinterpret_cast<const float4 *>(
                                                                  reinterpret_cast<const int2 *>(cache.vals) + t.e),
                        cache.meta[t.e], a.degree, G);
      } else {
        if (!(ok = wide_sums(n, t, tag, G))) break;
        if (p >= resident) {
          load_row_now(s.x + off, xs);
          load_row_now(s.y + off, ys);
        }
        load_kj<P, 8>(kjn, s.C, t.c0, kj);
        hi = __ldg(a.h + t.i);
      }
      update(n, t, p < resident ? p : -1, G, kj, hi, ka, dnext, xs, ys);
    }
  }
  tc::tmem_wait_st();
  for (int p = 0; p < resident; ++p) {  // the resident state back to global memory
    const Pass t = locate(p);
    float xs[8], ys[8];
    get(p, xs, ys);
    if (t.live) {
      store_row<8>(s.x + size_t(t.i) * s.Cp + t.c0, xs);
      store_row<8>(s.y + size_t(t.i) * s.Cp + t.c0, ys);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(s_tmem, kPersistTmem);
  }
}

// The ballistic form f(x) = x (the bSB choice named in Sec. II A): the same
// scheme with items of 128 columns on whole warps (4 columns per lane),
// gathering the neighbours' FP32 positions of the step before (written by
// other blocks: read through L2).  An item's own x is its entry of that f
// buffer, so only y is separate state: it stays in TMEM for a warp's first 20
// items and in shared memory for one more (512 bytes), and x goes
// to the state array once, after the last step.  The sum runs over the row's
// cache slots in order, a zero weight past the degree -- the sequence of
// fused multiply-adds of k_step_csr_bsb -- and the update is sb_advance4_bsb,
// so results equal the per-step kernel bit for bit.
constexpr int kTmemItemsBsb = 20, kSlotBytesBsb = 512;

template <int P, int KIND>
__global__ void __launch_bounds__(kPersistThreads, 1) k_solve_csr_persistent_bsb(PersistArgs a) {
  constexpr bool VALS = KIND != VAL_PM1;
  extern __shared__ __align__(16) char s_raw[];
  __shared__ uint32_t s_tmem;
  const StateView &s = a.s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = s.Cp / kColsPerWarp;
  const int warps_total = gridDim.x * kPersistWarps;
  const int gw = blockIdx.x * kPersistWarps + warp;
  char *mine = s_raw + warp * a.warp_smem;
  float4 *slots = reinterpret_cast<float4 *>(mine);  // [slots][lane] y
  const WarpCache<VALS> cache(mine + a.slots * kSlotBytesBsb, a.cache_cap);
  if (warp == 0) tc::tmem_alloc(&s_tmem, kPersistTmem);
  int my_count = 0;
  const int n_units = s.N * chunks;
  for (int u = gw; u < n_units && my_count < a.cache_cap; u += warps_total, ++my_count) {
    const int row = u / chunks;
    cache.fill(a, my_count, row, u - row * chunks, lane);
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tm = s_tmem + (uint32_t(warp & 3) << 21) + uint32_t(warp >> 2) * kWarpTmem;
  const int resident = min(my_count, kTmemItemsBsb + a.slots);
  auto put = [&](int q, const float (&ys)[4]) {
    if (q < kTmemItemsBsb) {
      const uint32_t r[4] = {__float_as_uint(ys[0]), __float_as_uint(ys[1]), __float_as_uint(ys[2]),
                             __float_as_uint(ys[3])};
      tc::tmem_st_32x32b_x4(tm + uint32_t(q) * 4u, r);
    } else {
      slots[(q - kTmemItemsBsb) * 32 + lane] = make_float4(ys[0], ys[1], ys[2], ys[3]);
    }
  };
  auto get = [&](int q, float (&ys)[4]) {
    if (q < kTmemItemsBsb) {
      uint32_t r[4];
      tc::tmem_ld_32x32b_x4_nowait(tm + uint32_t(q) * 4u, r);
      tc::tmem_wait_ld();
      tc::reg_fence_n(r);
#pragma unroll
      for (int j = 0; j < 4; ++j) ys[j] = __uint_as_float(r[j]);
    } else {
      const float4 v = slots[(q - kTmemItemsBsb) * 32 + lane];
      ys[0] = v.x; ys[1] = v.y; ys[2] = v.z; ys[3] = v.w;
    }
  };
  auto offset = [&](int q) {
    const int2 it = cache.item[q];
    return size_t(it.x) * s.Cp + it.y * kColsPerWarp + lane * 4;
  };
  for (int q = 0; q < resident; ++q) {
    float ys[4];
    load_row<4>(s.y + offset(q), ys);
    put(q, ys);
  }
  bool ok = true;
  for (int n = a.n_begin; ok && n < a.n_end; ++n) {
    const float *Fin = s.fx_of(n);
    float *Fout = s.fx_of(n + 1);
    const bool last = n + 1 == a.n_end;
    const uint32_t tag = tag_of(n, a.n_begin, kTagPos), next = last ? 0u : tag_of(n + 1, a.n_begin, kTagPos);
    tc::tmem_wait_st();
    for (int q = 0; q < my_count; ++q) {
      const int2 it = cache.item[q];
      const int i = it.x, c4 = it.y * kColsPerWarp + lane * 4;
      const size_t off = size_t(i) * s.Cp + c4;
      const bool live = c4 < s.C;
      float xs[4], ys[4];
      if (q >= resident) load_row<4>(s.y + off, ys);
      Pos4 f[kPersistMaxDeg], own;  // own: this lane stored it the step before, or it stood there before this launch
      {
        const float *F = Fin + c4;
        const int4 ca = cache.cols[2 * q], cb = cache.cols[2 * q + 1];
        uint64_t t0 = 0;
        for (unsigned it = 0;; ++it) {  // until every live lane's entries are of step n
          own.load(Fin + off);
          f[0].load(F + size_t(ca.x) * s.Cp);
          f[1].load(F + size_t(ca.y) * s.Cp);
          f[2].load(F + size_t(ca.z) * s.Cp);
          f[3].load(F + size_t(ca.w) * s.Cp);
          if (a.degree > 4) {
            f[4].load(F + size_t(cb.x) * s.Cp);
            f[5].load(F + size_t(cb.y) * s.Cp);
          }
          if (a.degree > 6) {
            f[6].load(F + size_t(cb.z) * s.Cp);
            f[7].load(F + size_t(cb.w) * s.Cp);
          }
          uint32_t all = ~0u, any = 0u;
          auto look = [&](const Pos4 &v) {
            if (tag) all &= v.w[0] & v.w[1] & v.w[2] & v.w[3];
            else any |= v.w[0] | v.w[1] | v.w[2] | v.w[3];
          };
#pragma unroll
          for (int e = 0; e < 4; ++e) look(f[e]);
          if (a.degree > 4) {
            look(f[4]);
            look(f[5]);
          }
          if (a.degree > 6) {
            look(f[6]);
            look(f[7]);
          }
          const bool stale = tag ? (all & kTagPos) == 0 : (any & kTagPos) != 0;
          if (!__any_sync(0xffffffffu, live && stale) || n == a.n_begin) break;
          if (wait_over(it, t0, a.err)) {
            ok = false;
            break;
          }
        }
        if (!ok) break;
      }
      const uint32_t meta = cache.meta[q];
      const int deg = int(meta & 0xffffu), npos = (deg + (int(meta) >> 16)) / 2;
      const float hi = __ldg(a.h + i);
#pragma unroll
      for (int j = 0; j < 4; ++j) xs[j] = __uint_as_float(own.w[j] ^ tag);
      float g[4] = {0.f, 0.f, 0.f, 0.f};
      auto add = [&](int e) {  // a weight of 0 past the degree
        float w;
        if constexpr (VALS) w = reinterpret_cast<const float *>(cache.vals + 2 * q)[e];
        else w = e < npos ? 1.f : (e < deg ? -1.f : 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) g[j] = fmaf(w, __uint_as_float(f[e].w[j] ^ tag), g[j]);
      };
#pragma unroll
      for (int e = 0; e < 4; ++e) add(e);
      if (a.degree > 4) {
        add(4);
        add(5);
      }
      if (a.degree > 6) {
        add(6);
        add(7);
      }
      if (q < resident) get(q, ys);
      sb_advance4_bsb<P>(s, a.t, n, c4, g, hi, xs, ys);
      if (live) {
        if (!(n == a.skip_step && blockIdx.x == 0))
          asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(Fout + off),
                       "r"(__float_as_uint(xs[0]) | next), "r"(__float_as_uint(xs[1]) | next),
                       "r"(__float_as_uint(xs[2]) | next), "r"(__float_as_uint(xs[3]) | next)
                       : "memory");
        if (last) store_row<4>(s.x + off, xs);
      }
      if (q < resident) {
        __syncwarp();
        put(q, ys);
      } else if (live) {
        store_row<4>(s.y + off, ys);
      }
    }
  }
  tc::tmem_wait_st();
  for (int q = 0; q < resident; ++q) {
    float ys[4];
    get(q, ys);
    if (cache.item[q].y * kColsPerWarp + lane * 4 < s.C) store_row<4>(s.y + offset(q), ys);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(s_tmem, kPersistTmem);
  }
}

template <int KIND>
static const void *persistent_bsb_fn_k(int P) {
  switch (P) {
    case 1: return (const void *)k_solve_csr_persistent_bsb<1, KIND>;
    case 2: return (const void *)k_solve_csr_persistent_bsb<2, KIND>;
    case 4: return (const void *)k_solve_csr_persistent_bsb<4, KIND>;
    case 8: return (const void *)k_solve_csr_persistent_bsb<8, KIND>;
    case 16: return (const void *)k_solve_csr_persistent_bsb<16, KIND>;
    case 32: return (const void *)k_solve_csr_persistent_bsb<32, KIND>;
    case 64: return (const void *)k_solve_csr_persistent_bsb<64, KIND>;
    case 128: return (const void *)k_solve_csr_persistent_bsb<128, KIND>;
    default: return nullptr;
  }
}

// BF16 values are FP32 in the ELL form
static const void *persistent_bsb_fn(int P, int kind) {
  return kind == VAL_PM1 ? persistent_bsb_fn_k<VAL_PM1>(P) : persistent_bsb_fn_k<VAL_F32>(P);
}

template <int KIND, int LPI, bool WIDE>
static const void *persistent_fn_p(int P) {
  switch (P) {
    case 1: return (const void *)k_solve_csr_persistent<1, KIND, LPI, WIDE>;
    case 2: return (const void *)k_solve_csr_persistent<2, KIND, LPI, WIDE>;
    case 4: return (const void *)k_solve_csr_persistent<4, KIND, LPI, WIDE>;
    case 8: return (const void *)k_solve_csr_persistent<8, KIND, LPI, WIDE>;
    case 16: return (const void *)k_solve_csr_persistent<16, KIND, LPI, WIDE>;
    case 32: return (const void *)k_solve_csr_persistent<32, KIND, LPI, WIDE>;
    case 64: return (const void *)k_solve_csr_persistent<64, KIND, LPI, WIDE>;
    case 128: return (const void *)k_solve_csr_persistent<128, KIND, LPI, WIDE>;
    default: return nullptr;
  }
}

template <bool WIDE>
static const void *persistent_fn_k(int P, int kind, int lpi) {
  if (kind == VAL_PM1) return lpi == 32 ? persistent_fn_p<VAL_PM1, 32, WIDE>(P) : persistent_fn_p<VAL_PM1, 16, WIDE>(P);
  return lpi == 32 ? persistent_fn_p<VAL_F32, 32, WIDE>(P) : persistent_fn_p<VAL_F32, 16, WIDE>(P);
}

static const void *persistent_fn(int P, int kind, int lpi, bool wide) {
  return wide ? persistent_fn_k<true>(P, kind, lpi) : persistent_fn_k<false>(P, kind, lpi);
}

// Items of 256 columns on whole warps when R * P allows it, else of 128 on half warps.
static int persist_lpi(int Cp) { return Cp % 256 == 0 ? 32 : (Cp % 128 == 0 ? 16 : 0); }

// The test hook of solve_streaming.cu that caps a warp's cache; here it sends
// instances with more items to the streaming form (ballistic: per step).
static int cache_cap_hook() {
  const char *v = std::getenv("SBQA_TEST_PERSIST_CACHE");
  const int k = v ? std::atoi(v) : 0;
  return k > 0 ? k : (1 << 30);
}

// Test hook: SBQA_TEST_PERSIST_PASSES=k sends run batches of more than k passes per warp to the streaming
// form, so that small instances take it (not for production use).
static int max_passes() {
  const char *v = std::getenv("SBQA_TEST_PERSIST_PASSES");
  return v ? std::max(0, std::min(kMaxPasses, std::atoi(v))) : kMaxPasses;
}

// Blocks of the grid: one per SM, as the registers and shared memory of every
// instantiation allow (0 when one does not fit the device, or the streaming
// form's blocks do not).  Also sets their shared-memory limits, which last for
// the context.
int persistent_blocks() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto fits = [](const void *fn) {
    int per_sm = 0;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kPersistSmem) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kPersistThreads, kPersistSmem) == cudaSuccess &&
           per_sm >= 1;
  };
  const int Ps[8] = {1, 2, 4, 8, 16, 32, 64, 128};
  for (int P : Ps)
    for (int kind : {VAL_PM1, VAL_F32}) {
      for (int wide = 0; wide < 2; ++wide)
        if (!fits(persistent_fn(P, kind, 16, wide != 0)) || !fits(persistent_fn(P, kind, 32, wide != 0))) return 0;
      if (!fits(persistent_bsb_fn(P, kind))) return 0;
    }
  return streaming_fits() ? sms : 0;
}

// Lays out a warp's shared memory: its share of `units` items of `eb` bytes,
// and state slots of `slot` bytes for the passes of `per_pass` items beyond
// the `tmem` ones, at most kMaxSlots of them.
static void split_smem(PersistArgs *a, long long units, int warps, int eb, int per_pass, int tmem, int slot) {
  a->cache_cap = int((units + warps - 1) / warps);
  const int cache = (a->cache_cap * eb + 15) / 16 * 16;
  const int passes = (a->cache_cap + per_pass - 1) / per_pass;
  a->slots = std::max(0, std::min({(kWarpSmem - cache) / slot, passes - tmem, kMaxSlots}));
  a->warp_smem = cache + a->slots * slot;
}

// Items of the ballistic form a warp takes at most before the streaming form
// is the faster one (L = 24, R*P = 2048: 61 items, 126 us per step against
// 119).  Below, see persistent_bsb_may_stream.
static bool bsb_resident(int N, int Cp, int blocks) {
  return (long long)N * (Cp / kColsPerWarp) <=
         (long long)blocks * kPersistWarps * std::min(max_passes(), cache_cap_hook());
}

bool persistent_bsb_ok(int N, int Cp, int max_degree, int kind, int blocks) {
  if (blocks <= 0 || max_degree > kPersistMaxDeg || Cp % kColsPerWarp != 0) return false;
  return bsb_resident(N, Cp, blocks) || streaming_bsb_ok(N, Cp, max_degree, kind, blocks * kStreamBlocksPerSm);
}

// Whether the two ballistic forms are close enough for the autotuner to time
// both.  Bound by the ALU pipe, an item takes the on-chip form 0.78 of its time
// in the streaming one (1.83 and 2.35 us at one block per SM), but that has 32
// warps per SM to the 24 here, and the fullest warp sets the step: L = 14, R*P =
// 1024, 7 items against 5: 12.9 us per step and 11.5 streaming; L = 20, R*P =
// 2048, 36 against 27: 67.6 and 63.9; but 18 against 14, L = 16: 32.0 and 36.6.
// Where the on-chip form has less than 5 items for 4, it was the faster one in
// every shape measured (L = 6 .. 20, random graphs of N = 3000 .. 10^5, R*P =
// 128 .. 2048).
bool persistent_bsb_may_stream(int N, int Cp, int max_degree, int kind, int blocks) {
  if (!bsb_resident(N, Cp, blocks) || !streaming_bsb_ok(N, Cp, max_degree, kind, blocks * kStreamBlocksPerSm))
    return false;
  const long long items = (long long)N * (Cp / kColsPerWarp), on_chip = (long long)blocks * kPersistWarps,
                  streaming = (long long)blocks * kStreamBlocksPerSm * 8;
  return 4 * ((items + on_chip - 1) / on_chip) >= 5 * ((items + streaming - 1) / streaming);
}

bool persistent_bsb_streams(int N, int Cp, int max_degree, int kind, int blocks, bool wanted) {
  return !bsb_resident(N, Cp, blocks) ||
         (wanted && streaming_bsb_ok(N, Cp, max_degree, kind, blocks * kStreamBlocksPerSm));
}

static PersistArgs persist_args(const StateView &s, const CsrView &J, const StepTables &t, int n_begin, int n_end,
                                int *err) {
  PersistArgs a;
  a.s = s;
  a.h = J.h;
  a.ell_col = J.ell_col;
  a.ell_meta = J.ell_meta;
  a.ell_val = J.ell_val;
  a.t = t;
  a.n_begin = n_begin;
  a.n_end = n_end;
  a.err = err;
  // test hook for the bounded waits: SBQA_TEST_SKIP_BARRIER_STEP=n makes block 0
  // keep the codes of step n of a launch that runs it (not for production use)
  const char *skip = std::getenv("SBQA_TEST_SKIP_BARRIER_STEP");
  a.skip_step = skip ? std::atoi(skip) : -1;
  a.csr = J;
  a.degree = J.max_degree;
  a.wide = (J.max_degree + 3) / 4 * 4;
  a.cache_cap = a.slots = a.warp_smem = 0;
  return a;
}

// `other`: the f buffer of step n_begin + 1, cleared so that none of its
// generation bits is left from an earlier launch.
static cudaError_t launch_persist(const void *fn, PersistArgs &a, int kind, void *other, size_t bytes, int blocks,
                                  cudaStream_t st) {
  const bool lists = a.degree > kPersistMaxDeg
                         ? a.csr.row_ptr && a.csr.col &&
                               (kind == VAL_PM1 ? a.csr.npos != nullptr : a.csr.val != nullptr)
                         : a.ell_col && a.ell_meta && (kind == VAL_PM1 || a.ell_val);
  if (!fn || !lists) return cudaErrorInvalidValue;
  const cudaError_t e = cudaMemsetAsync(other, 0, bytes, st);
  if (e != cudaSuccess) return e;
  void *args[] = {&a};
  return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kPersistThreads), args,
                                     size_t(a.warp_smem) * kPersistWarps, st);
}

cudaError_t launch_solve_csr_persistent_bsb(const StateView &s, const CsrView &J, const StepTables &t, int n_begin,
                                            int n_end, unsigned *bar, int *err, int blocks, bool streams,
                                            cudaStream_t st) {
  if (persistent_bsb_streams(s.N, s.Cp, J.max_degree, J.kind, blocks, streams))
    return launch_solve_csr_streaming_bsb(s, J, t, n_begin, n_end, bar, err, blocks * kStreamBlocksPerSm, st);
  PersistArgs a = persist_args(s, J, t, n_begin, n_end, err);
  split_smem(&a, (long long)s.N * (s.Cp / kColsPerWarp), blocks * kPersistWarps, entry_bytes(J.kind != VAL_PM1), 1,
             kTmemItemsBsb, kSlotBytesBsb);
  return launch_persist(persistent_bsb_fn(s.P, J.kind), a, J.kind, s.fx_of(n_begin + 1),
                        size_t(s.N) * s.Cp * sizeof(float), blocks, st);
}

int persistent_mode(int N, int Cp, int max_degree, int kind, int blocks, bool force_rows, bool ell) {
  const int lpi = persist_lpi(Cp);
  const bool wide = max_degree > kPersistMaxDeg;
  if (blocks <= 0 || max_degree > kPersistWideDeg || lpi == 0 || (!wide && !ell)) return 0;
  const long long items = (long long)N * (Cp / (8 * lpi)), warps = (long long)blocks * kPersistWarps;
  long long most = std::min<long long>(max_passes() * (32 / lpi), cache_cap_hook());
  if (wide) most = std::min<long long>(most, kWarpSmem / wide_bytes((max_degree + 3) / 4 * 4, kind != VAL_PM1));
  if (!force_rows && items <= warps * most) return kPersistResident;
  return wide ? 0 : streaming_mode(N, Cp, max_degree, kind, blocks * kStreamBlocksPerSm, force_rows, ell);
}

cudaError_t launch_solve_csr_persistent(const StateView &s, const CsrView &J, const StepTables &t, int n_begin,
                                        int n_end, unsigned *bar, int *err, int blocks, int mode, cudaStream_t st) {
  const int lpi = persist_lpi(s.Cp);
  if (mode != kPersistResident)
    return launch_solve_csr_streaming(s, J, t, n_begin, n_end, bar, err, blocks * kStreamBlocksPerSm, mode, st);
  PersistArgs a = persist_args(s, J, t, n_begin, n_end, err);
  const bool vals = J.kind != VAL_PM1, wide = J.max_degree > kPersistMaxDeg;
  split_smem(&a, (long long)s.N * (s.Cp / (8 * lpi)), blocks * kPersistWarps,
             wide ? wide_bytes(a.wide, vals) : entry_bytes(vals), 32 / lpi, kTmemPasses, kSlotBytes);
  return launch_persist(persistent_fn(s.P, J.kind, lpi, wide), a, J.kind, s.f_of(n_begin + 1), size_t(s.N) * s.Cp,
                        blocks, st);
}

}  // namespace sbqa
