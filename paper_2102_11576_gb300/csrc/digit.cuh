// digit.cuh -- FP64-accurate matrix products on the BF16 tensor cores, by
// splitting every operand into short integer digits whose products the FP32
// accumulators hold exactly (the error-free splitting of Ozaki, Ogita, Oishi &
// Rump, 2012; on tensor cores Mukunoki, Ozaki, Ogita & Imamura, 2020).
//
// D = A S with S symmetric (the sine matrix S_n of Section 4.1), so both
// operands are K-major rows.  Each row of A is scaled by a power of two to
// integers of 55 bits (E its largest biased exponent, x_q = round(x
// 2^(1077-E))), S by one power of two, and both are written as eight signed
// digits of seven bits, x_q = sum_i d_i 128^(7-i), -64 <= d_i <= 64: small
// integers, which BF16 holds exactly.  Then
//     x_q S_q = 128^7 sum_s 128^(7-s) g_s + (terms below the kept ones),
//     g_s = sum over i + j = s of sum_k d_i e_j,      s = 0..7,
// thirty-six BF16 products into eight accumulators.  Every g_s (and every
// partial sum of it) is an integer of at most 2^24 in magnitude -- 64 times the
// sum of |e_j| over half a row of S, which the plan checks when it builds S (21 sides
// up to 2048 have no such digits: build_sine) -- so
// the FP32 accumulation is exact in any order.  What is lost: the two
// roundings to 55 bits (2^-56 of the row's largest entry; 2^-55 or 2^-56 of
// S's) and the groups s > 7 (about 2^-54 of the result's root mean square):
// together below the rounding error of an FP64 FFT of the same length.
//
// The eight groups are put together in one 64-bit integer W (the result divided
// by 2^58 2^(E ...), rounded: about 2^-54 of the root mean square again).  The
// intermediate results stay in that form, with the exponent of their row of A:
// the next split only shifts them.  What leaves the chain becomes FP64, by
// integer instructions (GB300 issues one FP64 instruction per warp and 64
// clocks of a scheduler).
//
// Symmetric form (sym_perm, dst_gemm.cuh): the K operand holds the even-j
// entries in [0, hk) and the odd-j entries in [hk, 2 hk); outputs i and n-1-i
// are u + e and u - e with u from the first half and e from the second.
//
// Why tensor cores: GB300 runs an FP64 FFT at 2 multiply-adds per clock and
// SM, and the BF16 pipe 4096, so even 36 products per output and the O(n)
// instead of O(log n) operations of a matrix product are faster up to the
// n <= 2048 that the exactness bound allows (measured at 2048 x 2048 and below;
// figures at digit_gemm_kernel).
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "df.cuh"
#include "umma.cuh"

namespace rsfde {

constexpr int kDgDigits = 8;    // digits of seven bits per operand
constexpr int kDgMaxN = 2048;   // K = n/2 <= 1024 per half: 8 * 64 * 32 * 1024 is 2^24
constexpr int kDgBM = 128, kDgBK = 64;
constexpr int kDgATile = kDgBM * kDgBK * 2;  // one digit of a K slice of A
__host__ __device__ constexpr int dg_btile(int BN) { return BN * kDgBK * 2; }
constexpr int kDgASlots = 6;                 // digit tiles of A, in ring order
__host__ __device__ constexpr int dg_bslice(int BN) { return kDgDigits * dg_btile(BN); }  // double-buffered
__host__ __device__ constexpr int dg_smem(int BN) { return kDgASlots * kDgATile + 2 * dg_bslice(BN) + 1024; }
constexpr int kDgThreads = 512;
constexpr int kDgNone = -(1 << 20);           // exponent of a row of zeros
constexpr int kDgNan = 1 << 20;               // exponent of a row that holds an infinity or NaN

enum DigitEpi {
  DG_FIXED = 0,     // W of out^T, and the largest exponent of every row of out^T
  DG_QUOTIENT = 1,  // the same, with bounds of the exponents of both quotients of Eq. 4.6's tau divides
  DG_STORE = 2,     // out^T in FP64
  DG_COMBINE = 3,   // masked combine of Eq. 4.6 into z (FP64)
  DG_ROWS = 4,      // the operands' roles swapped (A the matrix's pairs, S the rows of z): out = pre - product
  DG_COLS = 5       // out = pre - product^T + (dt/eta) phi z, in FP64
};

struct DigitEpiParams {
  int M, N, n_full;   // rows of A; output pairs (n_full + 1) / 2; transform length
  int hk;             // K extent of each half (a multiple of 16)
  const int* rexp;    // exponent E of each row of A: entries below 2^(E-1022) (kDgNone, kDgNan)
  int kexp;           // result = W 2^(E + kexp)
  int row_b;          // rows m >= row_b are the second channel
  void* out0;         // out^T of channel 0 and 1: out[n * ldo + m], W or FP64
  void* out1;
  int ldo;
  int* oexp;          // exponents of the rows of out^T: [n], and [oexp_b + n] for channel 1 (quotient 1)
  int oexp_b;
  const double* inv0;  // DG_QUOTIENT: 1 / (1 - lx - ly) and 1 / (1 + dt/eta - lx - ly) at [n * M + m]
  const double* inv1;
  const uint8_t* phi;  // DG_COMBINE: out0[n * ldo + x] from channel phi[n * ldo + x]
  const int* kexp_dev; // if set, added to kexp
  const double* pre;   // DG_ROWS, DG_COLS
  const void* z;       // DG_COLS: z (FP32 if z_float)
  int z_float;
  double pen;          // dt/eta
  int early;           // trigger the next kernel of the chain at once (launch_digit)
  long long wait_cycles;
  int* gave_up;        // set when a wait gave up
};

// Digits of x_q (|x_q| <= 2^55): x_q + sum_i 64 128^i has the base-128 digits
// d_i + 64, so each comes out by a shift and a mask (the top one, 0..128,
// unmasked).
constexpr long long kDgBias = 64LL * ((1LL << 56) - 1) / 127;
__device__ __forceinline__ uint32_t dg_digit(unsigned long long biased, int i) {  // d_i + 64, i = 0 the top
  const uint32_t v = (uint32_t)(biased >> (7 * (7 - i)));
  return i == 0 ? v : (v & 127u);
}
// Two digits as a BF16 pair: 128 + (d + 64) has the bits 0x4300 + (d + 64)
// (BF16 holds 8 bits: 128..256 in steps of one), and subtracting 192 is exact.
__device__ __forceinline__ uint32_t dg_pack(uint32_t a, uint32_t b) {
  const uint32_t u = 0x43004300u + (a | (b << 16));
  const __nv_bfloat162 c = __nv_bfloat162(__ushort_as_bfloat16(0x4340), __ushort_as_bfloat16(0x4340));
  __nv_bfloat162 r = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&u), c);
  return *reinterpret_cast<uint32_t*>(&r);
}
// round(x 2^(1077 - E)) for E >= the biased exponent of x (E >= 1), |.| <= 2^55
__device__ __forceinline__ long long dg_quantize(double x, int E) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((unsigned long long)b >> 52) & 0x7FF;
  const long long m = b & 0xFFFFFFFFFFFFFll;
  const long long mag = e ? (m | (1ll << 52)) : m;
  const int sh = E - (e ? e : 1) - 2;
  long long q;
  if (sh <= 0) q = mag << (-sh);
  else q = sh < 60 ? (mag + (1ll << (sh - 1))) >> sh : 0ll;
  return b < 0 ? -q : q;
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}
// 32 lanes x 2 columns of tensor memory (no wait)
__device__ __forceinline__ void tmem_ld2_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// round(sum_s 128^(7-s) g_s / 2^9): the group sums of one output as one integer
// (below 2^63: the sum is below 2^71 as |sum_k x_k S_k| <= max |x| sum_k |S_k|).
__device__ __forceinline__ long long dg_sum(const int* g) {
  const int a = g[0] * 128 + g[1], b = g[2] * 128 + g[3], c = g[4] * 128 + g[5];  // each below 2^31
  const int d = (g[6] + ((g[7] + 256) >> 7)) >> 2;
  return ((long long)a << 33) + (long long)b * (1 << 19) + (long long)c * 32 + d;
}
// The eight accumulators' words of two adjacent columns (no wait), and their sums.
struct DgRaw {
  uint32_t r[kDgDigits][2];
};
template <int BN>
__device__ __forceinline__ void dg_load2(uint32_t taddr, DgRaw& t) {
#pragma unroll
  for (int s = 0; s < kDgDigits; ++s) tmem_ld2_nowait(taddr + (uint32_t)(s * BN), t.r[s]);
}
__device__ __forceinline__ long long dg_sum(const DgRaw& t, int q) {
  int g[kDgDigits];
#pragma unroll
  for (int s = 0; s < kDgDigits; ++s) g[s] = __float2int_rn(__uint_as_float(t.r[s][q]));
  return dg_sum(g);
}
// E with |W 2^k| <= 2^(E - 1022), at least that of a W of 32 bits (which the
// next split takes without loss).
__device__ __forceinline__ int dg_fixed_exponent(long long w, int k) {
  const int h = (int)(w >> 32);
  return 64 - __clz(h ^ (h >> 31)) + k + 1022;
}
__device__ __forceinline__ uint32_t dg_exponent(double x) {
  return (uint32_t)((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FFu;
}

// One CTA per 128 x BN tile of pairs.  Per 64-wide K slice the eight digit
// tiles of A (16 KB each) and of S (stacked to one tile of 8 BN rows) come by
// TMA.  All eight accumulators live at once (8 BN TMEM columns), so a slice is
// loaded once for its 36 products; and as the accumulators of neighbouring
// groups are neighbours too, one MMA multiplies A_i with several stacked digits
// of S: groups 4..7 from S_{4-i} .. S_{7-i} (N = 4 BN), groups 0..3 from S_0 ..
// S_{3-i}.  Twelve MMAs (times four K steps of 16) instead of 36: at BN = 64 A
// is read from shared memory a third as often -- with N = 64 those reads (6 KB
// per 32 clocks of the tensor pipe, at 128 B per clock) bound the loop at 8000
// clocks a slice, now it runs at the pipe's 4608 -- and fewer instructions are
// issued, each costing its thread 75 to 100 clocks.
//
// BN = 64 fills the tensor memory: the even half's accumulators are added up
// (into u, in registers) before the odd half's products start.  BN = 32 and 16
// hold both halves' accumulators and add them up once; they are for grids
// that leave SMs idle (dg_bn).
//
// Roles: warp 0 lane 0 loads (A in a ring of six slots, S double-buffered),
// warps 1 and 2 issue the MMAs of groups 0..3 and 4..7; step[i] counts both
// warps' products with A_i done (the top warp has none for i >= 4 and just
// arrives, once it has seen A_i land).  As the ring has six slots, A_i of the next slice is
// loaded after step i + 2 of this one (i < 6) or step i - 6 of the next: no
// step can complete twice before the loader's wait has seen it, and no slot
// is refilled before both issuing warps have seen what it held, so the waits'
// phase parities are never ambiguous.  All sixteen warps add up and store.
template <int EPI, int BN>
__global__ void __launch_bounds__(kDgThreads, 1)
    digit_gemm_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB,
                      const __grid_constant__ DigitEpiParams ep, int* err, const int* gate) {
  static_assert(BN == 64 || BN == 32 || BN == 16, "tile widths");
  constexpr bool kBoth = BN <= 32;                        // both halves' accumulators at once
  constexpr int kCols = (kBoth ? 2 : 1) * kDgDigits * BN;  // TMEM columns
  constexpr int kBTile = dg_btile(BN), kBSlice = dg_bslice(BN);
  constexpr int CW = BN / 4;  // columns per warp (four warps per lane quarter)
  extern __shared__ __align__(1024) uint8_t dg_smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dg_smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* const smB = smem + kDgASlots * kDgATile;
  __shared__ uint64_t fullA[kDgASlots], fullB[2], step[kDgDigits], done[2], drained;
  __shared__ uint32_t tmem_base;
  // the warp index as a warp-uniform value, so that what the issuing warps compute
  // from it stays in uniform registers (the operands of tcgen05.mma)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDgASlots; ++s) mbar_init(&fullA[s], 1);
    for (int s = 0; s < kDgDigits; ++s) mbar_init(&step[s], 2);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&done[s], 2);
    }
    mbar_init(&drained, kDgThreads / 32);
    mbar_fence_init();
  }
  // everything above touches only this block; what the previous kernel wrote is read below
  pdl_wait();
  if (ep.early) pdl_trigger();
  if (gate && *(volatile const int*)gate == 0) return;
  if (warp == 0) {
    tmem_alloc(&tmem_base, kCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = __shfl_sync(0xffffffffu, tmem_base, 0);
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * kDgBM;
  const int KB = (ep.hk + kDgBK - 1) / kDgBK;  // slices per half
  // loads: A tile q = 8 g + i (slice g, digit i) into slot q mod 6; S of slice g
  // into buffer g mod 2.  Slices KB .. 2 KB - 1 are the odd half's.
  int qnext = 0;      // loader: A tiles issued
  int bnext = 0;      // loader: slices of S issued
  bool stop = false;  // loader or issuer: a wait gave up
  auto load_a = [&](int q) {
    const int g = q / kDgDigits, i = q % kDgDigits, s = q % kDgASlots;
    const int h = g >= KB, kb = g - h * KB;
    mbar_expect_tx(&fullA[s], kDgATile);
    tma_load_3d(smem + s * kDgATile, &mA, h * ep.hk + kb * kDgBK, m0, i, &fullA[s]);
  };
  auto load_b = [&](int g) {
    const int h = g >= KB, kb = g - h * KB;
    mbar_expect_tx(&fullB[g & 1], kBSlice);
    tma_load_3d(smB + (g & 1) * kBSlice, &mB, h * ep.hk + kb * kDgBK, n0, 0, &fullB[g & 1]);
    bnext = g + 1;
  };
  // this thread's outputs: row m, columns c0 .. c0 + CW - 1 of the tile
  const int q4 = warp & 3, c0 = (warp >> 2) * CW;
  const int m = m0 + q4 * 32 + lane;
  const bool mvalid = m < ep.M;
  const uint32_t tb = taddr + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0;
  const bool live = n0 + c0 < ep.N;  // this warp's columns reach into the matrix
  // the row's exponent (DG_ROWS: lane l has column c0 + l's), read ahead of the main loop
  const int E = EPI == DG_ROWS ? (lane < CW && n0 + c0 + lane < ep.N ? __ldg(ep.rexp + n0 + c0 + lane) : kDgNone)
                               : (mvalid ? __ldg(ep.rexp + m) : kDgNone);
  const int kdev = ep.kexp_dev ? __ldg(ep.kexp_dev) : 0;
  bool ok = true;
  long long u[kBoth ? 2 : CW];
  DgRaw raw;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    if (warp == 0 && lane == 0) {
      if (h == 0) load_b(0);
      // BN = 64, even half: its tiles and those of the odd half that its steps make room for
      const int qlast = (h || kBoth) ? 2 * KB * kDgDigits : min(KB * kDgDigits + kDgASlots, 2 * KB * kDgDigits);
      for (; qnext < qlast && !stop; ++qnext) {
        const int f = qnext - kDgASlots;  // the tile that leaves the slot
        if (f >= 0 && !mbar_wait(&step[f % kDgDigits], (f / kDgDigits) & 1, err, ep.wait_cycles)) {
          stop = true;
          break;
        }
        load_a(qnext);
        // S of the next slice: its buffer is free since step 7 of the slice before
        // this one, which this wait (f: that step) has seen
        if (qnext % kDgDigits == kDgASlots - 1 && qnext / kDgDigits + 1 < 2 * KB) load_b(qnext / kDgDigits + 1);
      }
    } else if ((warp == 1 || warp == 2) && elect_one()) {
      const bool top = warp == 1;  // groups 0..3
      if (!kBoth && h) {  // the even half's accumulators have been read
        if (!stop && !mbar_wait(&drained, 0, err)) stop = true;
        tc_fence_after();
      }
      const uint32_t tacc = taddr + (kBoth ? (uint32_t)(h * kDgDigits * BN) : 0u);
      for (int kb = 0; kb < KB && !stop; ++kb) {
        const int g = h * KB + kb;
        const int left = (ep.hk - kb * kDgBK) >> 4, ks = left < 4 ? left : 4;  // K steps of 16 in the slice
        if (!mbar_wait(&fullB[g & 1], (g >> 1) & 1, err, ep.wait_cycles)) {
          stop = true;
          break;
        }
        const uint64_t b0 = umma_desc_sw128(smem_u32(smB) + (g & 1) * kBSlice);
#pragma unroll 1
        for (int i = 0; i < kDgDigits; ++i) {
          const int q = g * kDgDigits + i, sa = q % kDgASlots;
          if (!mbar_wait(&fullA[sa], (q / kDgASlots) & 1, err, ep.wait_cycles)) {
            stop = true;
            break;
          }
          if (top && i >= 4) {  // groups 0..3 end with A_3
            mbar_arrive(&step[i]);
            continue;
          }
          tc_fence_after();
          // groups s0 .. s0 + cnt - 1 from the digits s0 - i .. of S
          const int s0 = top ? i : (i < 4 ? 4 : i), cnt = top ? 4 - i : (i < 4 ? 4 : 8 - i);
          const uint64_t ad = umma_desc_sw128(smem_u32(smem) + sa * kDgATile);
          const uint64_t bd = b0 + (uint64_t)((s0 - i) * (kBTile >> 4));
          const uint32_t idesc = umma_idesc_bf16(kDgBM, 0) | ((uint32_t)(cnt * (BN >> 3)) << 17);
          const uint32_t dd = tacc + (uint32_t)(s0 * BN);
          // every group's first product is A_0's
          umma_bf16(dd, ad, bd, idesc, (kb > 0 || i > 0) ? 1u : 0u);
          if (ks == 4) {
            umma_bf16(dd, ad + 2, bd + 2, idesc, 1u);
            umma_bf16(dd, ad + 4, bd + 4, idesc, 1u);
            umma_bf16(dd, ad + 6, bd + 6, idesc, 1u);
          } else {
            if (ks > 1) umma_bf16(dd, ad + 2, bd + 2, idesc, 1u);
            if (ks > 2) umma_bf16(dd, ad + 4, bd + 4, idesc, 1u);
          }
          umma_commit(&step[i]);
        }
      }
      umma_commit(&done[h]);  // also after a wait gave up: the epilogue waits are never left without it
    }
    if constexpr (!kBoth) {
      __syncwarp();
      ok = mbar_wait(&done[h], 0, err) && ok;
      tc_fence_after();
      if (h == 0) {
        if (live) {
          dg_load2<BN>(tb, raw);
          tmem_ld_wait();
#pragma unroll 1
          for (int c = 0; c < CW; c += 2) {
            DgRaw next;
            dg_load2<BN>(tb + (uint32_t)(c < CW - 2 ? c + 2 : 0), next);  // in flight during these sums
            const long long t0 = dg_sum(raw, 0), t1 = dg_sum(raw, 1);
#pragma unroll
            for (int k = 0; k < CW - 2; ++k) u[k] = u[k + 2];
            u[CW - 2] = t0;
            u[CW - 1] = t1;
            tmem_ld_wait();
            raw = next;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&drained);
      }
    }
  }
  if constexpr (kBoth) {
    __syncwarp();
    ok = mbar_wait(&done[0], 0, err);
    ok = mbar_wait(&done[1], 0, err) && ok;
    tc_fence_after();
  }
  const bool bad = !ok || *(volatile int*)err != 0;  // *err: a wait of this application's launches gave up
  if (bad && lane == 0) atomicExch(ep.gave_up, 1);
  const int kexp = ep.kexp + kdev, kx = E + kexp;
  const bool nan = bad || E == kDgNan;  // an incomplete tile, or a row that held an infinity or NaN
  const bool ch = m >= ep.row_b;
  const int mm = ch ? m - ep.row_b : m;
  // a warp whose rows are all of one channel reduces the exponents once
  const bool mixed = EPI == DG_FIXED &&
                     __shfl_sync(0xffffffffu, (int)ch, 0) != __shfl_sync(0xffffffffu, (int)ch, 31);
  int mx0 = kDgNone, mx1 = kDgNone;  // lane l < CW: column c0 + l; CW <= l < 2 CW: its mirror
  // two columns at a time (BN = 64: u moving down by two): rolled, as the loop
  // written out is more code than the instruction caches hold
  if (!kBoth && live) {
    dg_load2<BN>(tb, raw);
    tmem_ld_wait();
  }
#pragma unroll 1
  for (int c = 0; c < CW && n0 + c0 + c < ep.N; c += 2) {
    // what the outputs read, in flight during the sums
    constexpr bool kPre = EPI == DG_ROWS || EPI == DG_COLS, kPhi = EPI == DG_COLS || EPI == DG_COMBINE;
    double pre[2][2];
    uint8_t phi[2][2];
    uint32_t inv[2][2][2];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int mir = 0; mir < 2; ++mir) {
        const int n = n0 + c0 + c + q;
        if (!mvalid || n >= ep.N) continue;
        const size_t o = EPI == DG_ROWS ? (size_t)n * ep.ldo + (mir ? ep.n_full - 1 - m : m)
                                        : (size_t)(mir ? ep.n_full - 1 - n : n) * ep.ldo + mm;
        if constexpr (kPre) pre[q][mir] = ep.pre[o];
        if constexpr (kPhi) phi[q][mir] = ep.phi[o];
        if constexpr (EPI == DG_QUOTIENT) {  // (ldo = M)
          inv[q][mir][0] = __ldg(reinterpret_cast<const uint32_t*>(ep.inv0 + o) + 1);
          inv[q][mir][1] = __ldg(reinterpret_cast<const uint32_t*>(ep.inv1 + o) + 1);
        }
      }
    DgRaw next;
    if constexpr (kBoth) {
      dg_load2<BN>(tb + (uint32_t)c, raw);
      dg_load2<BN>(tb + (uint32_t)(kDgDigits * BN + c), next);
      tmem_ld_wait();
      u[0] = dg_sum(raw, 0);
      u[1] = dg_sum(raw, 1);
      raw = next;
    } else {
      dg_load2<BN>(tb + (uint32_t)(c < CW - 2 ? c + 2 : 0), next);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = n0 + c0 + c + q;
      if (n >= ep.N) continue;  // uniform over the warp
      const long long e = dg_sum(raw, q);
#pragma unroll
      for (int mir = 0; mir < 2; ++mir) {
        const int nn = mir ? ep.n_full - 1 - n : n;
        const long long w = mir ? u[q] - e : u[q] + e;
        if constexpr (EPI == DG_ROWS) {  // pairs along m, the scale along n
          const int En = __shfl_sync(0xffffffffu, E, c + q);
          if (mvalid) {
            const size_t o = (size_t)n * ep.ldo + (mir ? ep.n_full - 1 - m : m);
            // (the middle pairs with itself: written once)
            if (!(mir && 2 * m + 1 == ep.n_full))
              static_cast<double*>(ep.out0)[o] = (bad || En == kDgNan) ? __longlong_as_double(0x7FF8000000000000ll)
                                                                      : pre[q][mir] - ldexp_i64(w, En + kexp);
          }
          continue;
        }
        if constexpr (EPI == DG_FIXED || EPI == DG_QUOTIENT) {
          long long* __restrict__ out = static_cast<long long*>(ch ? ep.out1 : ep.out0);
          if (mvalid) out[(size_t)nn * ep.ldo + mm] = w;
          int x = nan ? kDgNan : dg_fixed_exponent(w, kx), x0 = kDgNone, x1 = kDgNone;
          if constexpr (EPI == DG_QUOTIENT) {
            if (mvalid) {  // |W inv| < 2^(x - 1022) 2^(e - 1022), e the biased exponent of inv
              x0 = nan ? kDgNan : x + (int)((inv[q][mir][0] >> 20) & 0x7FF) - 1022;
              x1 = nan ? kDgNan : x + (int)((inv[q][mir][1] >> 20) & 0x7FF) - 1022;
            }
            x0 = __reduce_max_sync(0xffffffffu, x0);
            x1 = __reduce_max_sync(0xffffffffu, x1);
          } else {
            if (!mvalid) x = kDgNone;
            x0 = __reduce_max_sync(0xffffffffu, mixed && ch ? kDgNone : x);
            if (mixed) x1 = __reduce_max_sync(0xffffffffu, ch ? x : kDgNone);
          }
          if (lane == mir * CW + c + q) {
            mx0 = x0;
            mx1 = x1;
          }
        } else {
          double* __restrict__ out = static_cast<double*>(ep.out0);
          const size_t o = (size_t)nn * ep.ldo + mm;
          if constexpr (EPI == DG_COLS) {
            if (mvalid && !(mir && nn == n)) {  // (the middle once: out may be z itself)
              double v = pre[q][mir] - ldexp_i64(w, kx);
              if (phi[q][mir])
                v = __fma_rn(ep.pen,
                             ep.z_float ? f64_exact(static_cast<const float*>(ep.z)[o])
                                        : static_cast<const double*>(ep.z)[o],
                             v);
              out[o] = nan ? __longlong_as_double(0x7FF8000000000000ll) : v;
            }
          } else if (mvalid && (EPI == DG_STORE || (phi[q][mir] != 0) == ch))
            out[o] = nan ? __longlong_as_double(0x7FF8000000000000ll) : ldexp_i64(w, kx);
        }
      }
    }
    if constexpr (!kBoth) {
#pragma unroll
      for (int k = 0; k < CW - 2; ++k) u[k] = u[k + 2];
      tmem_ld_wait();
      raw = next;
    }
  }
  if constexpr (EPI == DG_FIXED || EPI == DG_QUOTIENT) {
    const int n = n0 + c0 + (lane & (CW - 1));
    if (n < ep.N && lane < 2 * CW) {
      const int nn = lane < CW ? n : ep.n_full - 1 - n;
      const bool second = EPI == DG_FIXED && !mixed && ch;  // uniform over the warp
      if (mx0 > kDgNone / 2) atomicMax(ep.oexp + (second ? ep.oexp_b : 0) + nn, min(mx0, kDgNan));
      if (mx1 > kDgNone / 2) atomicMax(ep.oexp + ep.oexp_b + nn, min(mx1, kDgNan));
    }
  }
  // every issued load lands before the block exits, also after a wait gave up:
  // the last load of each slot (completed phases return at once)
  if (warp == 0 && lane == 0) {
    for (int q = qnext > kDgASlots ? qnext - kDgASlots : 0; q < qnext; ++q)
      mbar_wait(&fullA[q % kDgASlots], (q / kDgASlots) & 1, err);
    for (int g = bnext > 2 ? bnext - 2 : 0; g < bnext; ++g) mbar_wait(&fullB[g & 1], (g >> 1) & 1, err);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(taddr, kCols);
}

}  // namespace rsfde
