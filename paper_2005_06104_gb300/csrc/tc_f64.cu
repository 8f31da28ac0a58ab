// FP64 complex GEMMs on the BF16 tensor cores (sm_103a, tcgen05 kind::f16), without rounding in
// the tensor core: the splitting of the operands into exact slices of Ozaki, Ogita, Oishi and Rump
// (Numer. Algorithms 59, 2012), with fixed-point slices.
//
// GB300 runs FP64 at 1.1 TFLOP/s and dense BF16 at 1860.  Each row of a real operand (the 4M
// embedding of the complex one) is written as integers of 56 bits under one power of two, cut
// into seven signed 8-bit digits, each exact in BF16:
//   x = 2^(E-55) (d0 2^48 + d1 2^40 + ... + d6) + r,  |x| < 2^E on the whole row,
//   |d_s| <= 128,  |r| <= 2^(E-56).
// Digit products are summed by weight: group g = s + t holds g + 1 digit pairs, and a sum of
// at most 7 x 128 products of magnitude <= 2^14 stays below 2^24, so the FP32 accumulators hold
// integers and nothing rounds.  Groups 0..7 are kept (34 products); the first group left out is
// 2^-64 of the operands' maxima.  The epilogue adds each chunk's group sums into 64-bit integers
// (128-deep chunks; 256 for the groups 0..3, whose sums have room) and converts once at the end.
// The error is the operands' rounding at 2^-56 of their row maxima whatever K is.  Against the product of
// the operands' norms that is below the error of FP64 multiply-adds, which grows with the square root
// of K.  It is not relative to each result: an entry below 2^-3 of its row's maximum keeps fewer than 53
// bits, one below 2^-57 none, and a result is good to 2^-52 K of its row's times its column's maximum (a
// row (1, 1e-12) against a column (0, 1): 1e-5 of the result, where multiply-adds are exact).
// Operands graded against each other along K: as good as multiply-adds over six decades each (1.7e-16 to
// 2.9e-16 of the result's norm against 3.8e-16), up to 8e-14 over fourteen.  The contractions here
// meet no such pairs: an environment or an isometry, one factor of each, is level along K.
// (Groups 0..6 alone, 28 products, leave 2.4e-16 of the norm: more than the split-K CUDA-core product
// has at K near 128.)
// Measured against 113-bit sums, bond operator (two chained products), norm-wise: 1.15e-16 here
// and 3.4e-16 on CUDA cores at 129 x 127, w = 14; 1.4e-16 and 5.2e-16 with rows falling over six
// decades; 1.25e-16 and 2.3e-15 at 512.
// Measured time, H_eff: 512 x 512, w = 14: 53.4 -> 2.4 ms (25 TFLOP/s of FP64, 46 % of the BF16
// peak per digit product); 129 x 127, w = 8: 630 -> 95 us; both environment updates and the bond
// operator at 300 x 277, w = 14: 31.8 -> 1.9 ms.
//
// The eight groups need 8 x 128 TMEM columns and the 64-bit sums two registers per entry and
// set, so one CTA takes one of two passes over its K range: groups 0..3 (slices 0..3, 10
// products) or groups 4..7 (24 products); the partial results, and those of a split K, are added
// in FP64 by k_f64_reduce.
// Bound: the tensor pipe through shared memory (128 x 128 x 16 MMAs read 8 KB in 64 cycles).
//
// Kernel layout (one CTA per 128 x 128 real output tile, three warpgroups): warp 0 TMA, warp 1
// tcgen05.mma, warps 4..11 epilogue (one row, 64 columns each).  The groups of a pass fill one
// after the other, highest first, each with its own full / empty barrier, so group g drains while
// the next ones are multiplied.  All waits are bounded (see tc_ptx.cuh).
#include <cuda_bf16.h>

#include <cstring>

#include "contract.cuh"
#include "tc_ptx.cuh"

namespace tcf {
using namespace tc;

constexpr int NS = 7;                       // digits
constexpr int BM = 128, BN = 128, BK = 32;  // BK real entries per stage (64-byte swizzle)
constexpr int KC = 128, KC_KB = KC / BK;    // entries and k-blocks of a chunk
constexpr int kMaxChunks = 768;          // chunks one CTA lists (16-bit, beside 225 KB of stages)
constexpr int EPI_WARP0 = 4, EPI_WARPS = 8, THREADS = 128 + 32 * EPI_WARPS;
constexpr int REGS_LAUNCH = 168, REGS_LOW = 40, REGS_HIGH = 232;
static_assert(128 * REGS_LOW + 32 * EPI_WARPS * REGS_HIGH <= THREADS * REGS_LAUNCH, "register split");
constexpr int TILE = BM * BK * 2;           // one slice of one operand tile (bytes)
constexpr int TMEM_COLS = 512;
constexpr int EC = 64;                      // output columns per epilogue thread
constexpr int EPI_ROW = EC * 8 + 16;        // bytes of a row of a warp's turned output
constexpr int MAX_STAGES = 3;
constexpr int STAGE_AREA = 2 * 2 * NS * TILE;  // two stages of the 7-slice pass; three of the 4-slice one fit
static_assert(3 * 2 * 4 * TILE <= STAGE_AREA, "stages of the first pass");
constexpr int SMEM_BYTES = STAGE_AREA + 1024 + 256;
static_assert(EPI_WARPS * 32 * EPI_ROW <= STAGE_AREA, "output tile in the stages");
static_assert(SMEM_BYTES + 2 * kMaxChunks + 64 <= 227 * 1024, "shared memory");
constexpr int kBadRow = 1 << 20;            // row exponent of a row with a non-finite entry

// The MMAs of one stage for group G0 + g of a pass (G0 = 0 or 4): all digit pairs with s + t = G0 + g
template <int G0>
__device__ __forceinline__ void mma_group(int g, uint32_t d, uint32_t a0, uint32_t b0, uint32_t hi, uint32_t idesc,
                                          uint32_t cont) {
#pragma unroll
  for (int gg = 0; gg < 4; ++gg) {
    if (gg != g) continue;
    constexpr int KS = 2;  // 16 bf16 along K
    const int sum = G0 + gg, lo = sum > NS - 1 ? sum - (NS - 1) : 0, up = sum < NS - 1 ? sum : NS - 1;
#pragma unroll
    for (int sa = 0; sa < NS; ++sa) {
      if (sa < lo || sa > up) continue;
#pragma unroll
      for (int k = 0; k < BK / 16; ++k) {
        const uint32_t da = a0 + (sa * TILE >> 4) + k * KS, db = b0 + ((sum - sa) * TILE >> 4) + k * KS;
        if (sa == lo && k == 0)
          mma_bf16_first(d, da, db, hi, idesc, cont);
        else
          mma_bf16_acc(d, da, db, hi, idesc);
      }
    }
  }
}

// a 2^e as a double, rounded to nearest even; integer arithmetic (an FP64 conversion and a
// scaling would take 32 cycles of the FP64 pipe per warp and entry)
__device__ __forceinline__ double scaled_int(long long a, int e) {
  const unsigned long long u = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  if (u == 0) return 0.0;
  const int lz = __clzll((long long)u);
  const unsigned long long n = u << lz;
  const int ex = 63 - lz + e + 1023;
  if (ex < 1 || ex > 2045) return ldexp((double)a, e);  // under- or overflow
  unsigned long long m = n >> 11;
  const unsigned rem = (unsigned)n & 0x7ffu;
  m += (rem > 0x400u || (rem == 0x400u && (m & 1))) ? 1 : 0;
  const unsigned long long bits = ((unsigned long long)ex << 52) + (m - (1ull << 52));
  return __longlong_as_double((long long)(bits | ((unsigned long long)a & (1ull << 63))));
}

__global__ void __launch_bounds__(THREADS, 1)
    k_gemm_f64s(const __grid_constant__ CUtensorMap tmA4, const __grid_constant__ CUtensorMap tmB4,
                const __grid_constant__ CUtensorMap tmA7, const __grid_constant__ CUtensorMap tmB7, int M, int N,
                int nkb_total, int splits_hi, int kb_hi, int kb_lo, const int* __restrict__ eA,
                const int* __restrict__ eB, double* __restrict__ out, int* __restrict__ err,
                const unsigned* __restrict__ maskA, const unsigned* __restrict__ maskB, int mwords) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGE_AREA);
  uint64_t* full = bars;
  uint64_t* empty = bars + MAX_STAGES;
  uint64_t* tfull = bars + 2 * MAX_STAGES;
  uint64_t* tempty = bars + 2 * MAX_STAGES + 4;
  uint64_t* done = bars + 2 * MAX_STAGES + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 9);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  // pass: groups g0 .. g0 + ng - 1 of the digit sums, from the first nS slices
  const bool hi = (int)blockIdx.z < splits_hi;
  constexpr int ng = 4;
  const int nS = hi ? 4 : 7, g0 = hi ? 0 : 4, stages = hi ? 3 : 2;
  const int per_drain = hi ? 2 : 1;  // chunks whose sums stay below 2^24
  const int stage_bytes = 2 * nS * TILE;
  const int split = hi ? blockIdx.z : blockIdx.z - splits_hi;
  const int kb_split = hi ? kb_hi : kb_lo;
  const int kb0 = split * kb_split;
  const int nkb = min(nkb_total, kb0 + kb_split) - kb0;
  const int c0 = kb0 / KC_KB;
  const int nchunks = (nkb + KC_KB - 1) / KC_KB;
  // chunks with a nonzero entry in both operand tiles (the others add exact zeros)
  __shared__ unsigned short act[kMaxChunks];
  __shared__ int n_act;
  if (warp == 0) {
    const int n = active_chunks(maskA + (long long)blockIdx.y * mwords, maskB + (long long)blockIdx.x * mwords, c0,
                                nchunks, kMaxChunks, act);
    if (lane == 0) n_act = n;
  }
  if (threadIdx.x == 32) {
    prefetch_map(hi ? &tmA4 : &tmA7);
    prefetch_map(hi ? &tmB4 : &tmB7);
    for (int s = 0; s < MAX_STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 4; ++b) {
      mbar_init(smem_u32(&tfull[b]), 1);
      mbar_init(smem_u32(&tempty[b]), EPI_WARPS);
    }
    mbar_init(smem_u32(done), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const int ndrains = (n_act + per_drain - 1) / per_drain;
  if (warp < EPI_WARP0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LOW));
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer: the nS slices of the A and B tiles of one k-block
      int issued = 0;
      for (int ai = 0; ai < n_act && !*abort_flag; ++ai) {
        const int kb_end = min(nkb, (act[ai] + 1) * KC_KB);
        for (int kb = act[ai] * KC_KB; kb < kb_end; ++kb) {
          const int s = issued % stages, it = issued / stages;
          if (it > 0 && !mbar_wait(smem_u32(&empty[s]), (it - 1) & 1)) *abort_flag = 1;
          if (*abort_flag) break;
          uint8_t* st = smem + s * stage_bytes;
          const uint32_t fb = smem_u32(&full[s]);
          mbar_expect_tx(fb, stage_bytes);
          tma_load_3d(smem_u32(st), hi ? &tmA4 : &tmA7, fb, (kb0 + kb) * BK, m0, 0);
          tma_load_3d(smem_u32(st + nS * TILE), hi ? &tmB4 : &tmB7, fb, (kb0 + kb) * BK, n0, 0);
          ++issued;
        }
      }
      if (*abort_flag)
        for (int q = (issued > stages ? issued - stages : 0); q < issued; ++q)
          (void)mbar_wait(smem_u32(&full[q % stages]), (q / stages) & 1);
    } else if (warp == 1 && lane == 0) {
      // ---------------- MMA issuer
      const uint32_t idesc = idesc_bf16(BM, BN);
      const uint64_t desc = sdesc<64>(smem_u32(smem));
      const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
      int used = 0;
      for (int dr = 0; dr < ndrains && !*abort_flag; ++dr) {
        const int a_end = min(n_act, (dr + 1) * per_drain);
        for (int ai = dr * per_drain; ai < a_end && !*abort_flag; ++ai) {
          const int kb_beg = act[ai] * KC_KB, kb_end = min(nkb, kb_beg + KC_KB);
          for (int kb = kb_beg; kb < kb_end; ++kb) {
            const int s = used % stages, it = used / stages;
            ++used;
            if (!mbar_wait(smem_u32(&full[s]), it & 1)) {
              *abort_flag = 1;
              break;
            }
            fence_after();
            const bool first = ai == dr * per_drain && kb == kb_beg;
            const bool last = ai == a_end - 1 && kb == kb_end - 1;
            const uint32_t a0 = desc_lo + s * (stage_bytes >> 4);
            const uint32_t b0 = a0 + nS * (TILE >> 4);
            const uint32_t cont = first ? 0u : 1u;
#pragma unroll
            for (int g = ng - 1; g >= 0; --g) {
              if (first && dr > 0) {
                if (!mbar_wait(smem_u32(&tempty[g]), (dr - 1) & 1)) {
                  *abort_flag = 1;
                  break;
                }
                fence_after();
              }
              if (hi)
                mma_group<0>(g, tmem + g * BN, a0, b0, desc_hi, idesc, cont);
              else
                mma_group<4>(g, tmem + g * BN, a0, b0, desc_hi, idesc, cont);
              if (last) mma_commit(smem_u32(&tfull[g]));
            }
            mma_commit(smem_u32(&empty[s]));
            if (*abort_flag) break;
          }
        }
      }
      mma_commit(smem_u32(done));
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_HIGH));
    // ---------------- epilogue: group sums into 64-bit integers
    const int q = warp & 3;
    const int half = (warp - EPI_WARP0) >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const int nb = n0 + half * EC;
    long long acc[EC];
#pragma unroll
    for (int j = 0; j < EC; ++j) acc[j] = 0;
    bool ok = true;
    for (int dr = 0; dr < ndrains && ok; ++dr) {
      for (int g = ng - 1; g >= 0; --g) {
        const bool got = mbar_wait(smem_u32(&tfull[g]), dr & 1);
        if (!got) *abort_flag = 1;
        ok = __all_sync(0xffffffffu, got && !*abort_flag);
        if (!ok) break;
        fence_after();
        const int mult = 1 << (8 * (ng - 1 - g));
#pragma unroll
        for (int j0 = 0; j0 < EC; j0 += 16) {
          uint32_t v[16];
          const uint32_t col = tmem + lane_base + (uint32_t)(g * BN + half * EC + j0);
          tmem_ld16(v, col);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j)
            acc[j0 + j] += (long long)__float2int_rn(__uint_as_float(v[j])) * mult;
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tempty[g]));
      }
    }
    if (ok) {
      // the warp turns its 32 x 64 sums through the stages and stores whole rows (see tc_bf16.cu)
      uint8_t* reg = smem + (warp - EPI_WARP0) * 32 * EPI_ROW;
#pragma unroll
      for (int j = 0; j < EC; j += 2)
        *reinterpret_cast<longlong2*>(reg + lane * EPI_ROW + j * 8) = make_longlong2(acc[j], acc[j + 1]);
      __syncwarp();
      const int col = nb + 2 * lane;  // N is even
      const int eb = col < N ? eB[col] : 0;  // the rows (n, re) and (n, im) of B share their exponent
      const int rows = min(32, M - (m0 + q * 32));
      for (int r = 0; r < rows; ++r) {
        const longlong2 a = *reinterpret_cast<const longlong2*>(reg + r * EPI_ROW + lane * 16);
        const int row = m0 + q * 32 + r, ea = eA[row];
        // d_s d_t weighs 2^(96 - 8 (s + t)) of 2^(EA + EB - 110); the unit of acc is the last group's
        const int e = ea + eb + (hi ? 72 - 110 : 40 - 110);
        double2 v = make_double2(scaled_int(a.x, e), scaled_int(a.y, e));
        if (ea == kBadRow || eb == kBadRow) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
        if (col < N) *reinterpret_cast<double2*>(out + ((long long)blockIdx.z * M + row) * N + col) = v;
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    (void)mbar_wait(smem_u32(done), 0);
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(err, 1);
}

// C = alpha sum_z P[z] + beta C over complex entries (P: the real partials, (re, im) interleaved)
__global__ void k_f64_reduce(const cplx* __restrict__ P, int nz, int M, int N, cplx alpha, cplx beta,
                             cplx* __restrict__ C, long long ldc) {
  const long long per = (long long)M * N;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < per; e += (long long)gridDim.x * blockDim.x) {
    cplx acc = P[(long long)(nz - 1) * per + e];  // the small partials first
    for (int z = nz - 2; z >= 0; --z) acc = cadd(acc, P[z * per + e]);
    cplx* c = C + e / N * ldc + e % N;
    if (alpha.x != 1.0 || alpha.y != 0.0) acc = cmul(alpha, acc);
    if (beta.x != 0.0 || beta.y != 0.0) acc = cadd(acc, cmul(beta, *c));
    *c = acc;
  }
}

// ---------------------------------------------------------------- digits
// Row exponent from the largest high word of |x|: |x| < 2^E; kBadRow for a NaN or infinity.
__device__ __forceinline__ int row_exponent(unsigned hi) {
  const int ex = (int)(hi >> 20);
  return ex == 0x7ff ? kBadRow : max(ex, 1) - 1022;
}
__device__ __forceinline__ unsigned high_word(cplx z) {
  return max((unsigned)__double2hiint(z.x) & 0x7fffffffu, (unsigned)__double2hiint(z.y) & 0x7fffffffu);
}
// x as an integer of units 2^(E-55), rounded to nearest: |X| <= 2^55; digit s is byte 6 - s of X
// plus 128 in every lower byte, less 128
__device__ __forceinline__ unsigned long long biased_digits(double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  long long X = 0;
  const unsigned long long m53 = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = max(ex, 1) - 1020 - E;  // <= 2
  if (E != kBadRow && sh > -55) {
    X = sh >= 0 ? (long long)(m53 << sh) : (long long)((m53 + (1ull << (-sh - 1))) >> -sh);
    if (b >> 63) X = -X;
  }
  return (unsigned long long)(X + 0x0000808080808080ll);
}
// digit s as the BF16 bits in the upper half of a float's pattern
__device__ __forceinline__ unsigned digit_bits(unsigned long long y, int s) {
  if (s == 0) {  // the signed top
    const int t = (int)((long long)y >> 48);
    return __float_as_uint(__fadd_rn(__int_as_float(0x4B400000 + t), -12582912.0f));
  }
  const unsigned byte = (unsigned)(y >> (48 - 8 * s)) & 0xffu;
  return __float_as_uint(__fadd_rn(__int_as_float((int)(0x4B000000u | byte)), -8388736.0f));
}
// Two consecutive complex entries of one logical row: 4 BF16 per slice.  ROLE 0 (A): row r holds
// (re, im).  ROLE 1 (B): row 2 r holds (re, -im), row 2 r + 1 (im, re).
template <int ROLE>
__device__ __forceinline__ void store_digits(const cplx z[2], int E, __nv_bfloat16* out, long long row, int ldk,
                                             int k2, long long slice) {
  const unsigned long long r0 = biased_digits(z[0].x, E), i0 = biased_digits(z[0].y, E);
  const unsigned long long r1 = biased_digits(z[1].x, E), i1 = biased_digits(z[1].y, E);
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const unsigned a = digit_bits(r0, s), b = digit_bits(i0, s), c = digit_bits(r1, s), d = digit_bits(i1, s);
    if (ROLE == 0) {
      *reinterpret_cast<uint2*>(out + s * slice + row * ldk + k2) =
          make_uint2((a >> 16) | (b & 0xffff0000u), (c >> 16) | (d & 0xffff0000u));
    } else {
      const unsigned nb = b ^ 0x80000000u, nd = d ^ 0x80000000u;
      __nv_bfloat16* o = out + s * slice + 2 * row * ldk + k2;
      *reinterpret_cast<uint2*>(o) = make_uint2((a >> 16) | (nb & 0xffff0000u), (c >> 16) | (nd & 0xffff0000u));
      *reinterpret_cast<uint2*>(o + ldk) = make_uint2((b >> 16) | (a & 0xffff0000u), (d >> 16) | (c & 0xffff0000u));
    }
  }
}
template <int ROLE>
__device__ __forceinline__ void mark_chunk(unsigned* mask, int mw, long long row, int ch) {
  atomicOr(&mask[((ROLE == 0 ? row : 2 * row) >> 7) * mw + (ch >> 5)], 1u << (ch & 31));
}

// Entry (row, k) of a logical operand at p[row * ld + k], rows in the order given by wl: with
// wl > 0, row = w * ml + a is read from [a][w] (the channel-major rows of a left environment).
template <int ROLE>
__global__ void __launch_bounds__(128)
    k_digits_k(const cplx* __restrict__ p, long long ld, int rows, int K, int conj, int ml, int wl, int rows_pad,
               int ldk, __nv_bfloat16* __restrict__ out, int* __restrict__ eout, unsigned* __restrict__ mask, int mw) {
  __shared__ unsigned red[4];
  const long long row = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool live = row < rows;
  const long long src = wl > 0 ? (row % ml) * wl + row / ml : row;
  const cplx* x = p + (live ? src * ld : 0);
  unsigned h = 0;
  if (live)
    for (int k = tid; k < K; k += 128) h = max(h, high_word(x[k]));
  h = __reduce_max_sync(0xffffffffu, h);
  if (lane == 0) red[wid] = h;
  __syncthreads();
  const int E = row_exponent(max(max(red[0], red[1]), max(red[2], red[3])));
  const long long slice = (long long)rows_pad * ldk;
  for (int base = 64 * wid; 2 * base < ldk; base += 256) {  // a warp covers one chunk of 64 complex entries
    const int k = base + 2 * lane;
    cplx z[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      z[q] = live && k + q < K ? x[k + q] : mkc(0.0, 0.0);
      if (conj) z[q].y = -z[q].y;
    }
    if (2 * k < ldk) store_digits<ROLE>(z, E, out, row, ldk, 2 * k, slice);
    if (__any_sync(0xffffffffu, high_word(z[0]) | high_word(z[1])) && lane == 0) mark_chunk<ROLE>(mask, mw, row, base >> 6);
  }
  if (tid == 0) {
    if (ROLE == 0) {
      eout[row] = E;
    } else {
      eout[2 * row] = eout[2 * row + 1] = E;
    }
  }
}

// Entry (row, k) at p[k * ld + row]: blocks of 8 rows (128-byte reads), turned in shared memory.
template <int ROLE>
__global__ void __launch_bounds__(256)
    k_digits_r(const cplx* __restrict__ p, long long ld, int rows, int K, int conj, int rows_pad, int ldk,
               __nv_bfloat16* __restrict__ out, int* __restrict__ eout, unsigned* __restrict__ mask, int mw) {
  constexpr int TR = 8;
  __shared__ unsigned hmax[TR];
  __shared__ cplx t[TR][65];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const long long r0 = (long long)blockIdx.x * TR;
  const int rl = tid % TR, kk = tid / TR;  // 8 rows x 32 k
  if (tid < TR) hmax[tid] = 0;
  __syncthreads();
  unsigned h = 0;
  if (r0 + rl < rows)
    for (int k = kk; k < K; k += 32) h = max(h, high_word(p[(long long)k * ld + r0 + rl]));
  atomicMax(&hmax[rl], h);
  __syncthreads();
  const long long row = r0 + wid;  // warp w turns row w
  const int E = row_exponent(hmax[wid]);
  const long long slice = (long long)rows_pad * ldk;
  for (int base = 0; 2 * base < ldk; base += 64) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = base + kk + 32 * q;
      cplx z = r0 + rl < rows && k < K ? p[(long long)k * ld + r0 + rl] : mkc(0.0, 0.0);
      if (conj) z.y = -z.y;
      t[rl][kk + 32 * q] = z;
    }
    __syncthreads();
    const int k = base + 2 * lane;
    const cplx z[2] = {t[wid][2 * lane], t[wid][2 * lane + 1]};
    if (2 * k < ldk) store_digits<ROLE>(z, E, out, row, ldk, 2 * k, slice);
    if (__any_sync(0xffffffffu, high_word(z[0]) | high_word(z[1])) && lane == 0) mark_chunk<ROLE>(mask, mw, row, base >> 6);
    __syncthreads();
  }
  if (lane == 0) {
    if (ROLE == 0) {
      eout[row] = E;
    } else {
      eout[2 * row] = eout[2 * row + 1] = E;
    }
  }
}

// ---------------------------------------------------------------- host side
inline int pad_to(int x, int q) { return (x + q - 1) / q * q; }

// Digits [7][rows_pad][ldk] of an operand, row exponents [rows_pad] and the chunk mask.
struct Digits {
  RawBuf data, exps, mask;
  int rows_pad = 0, ldk = 0, mw = 0;
};

// role 0 (A): M rows; role 1 (B): 2 N rows.  kcontig: entry (row, k) at p[row * ld + k], else at
// p[k * ld + row].
void make_digits(cudaStream_t st, DevicePool* pool, int role, bool kcontig, const cplx* p, long long ld, int rows,
                 int K, bool conj, Digits& o, int ml = 0, int wl = 0) {
  const int real_rows = role == 0 ? rows : 2 * rows;
  o.rows_pad = pad_to(std::max(real_rows, 1), 128);
  o.ldk = pad_to(std::max(2 * K, 1), BK);
  o.mw = ((o.ldk + KC - 1) / KC + 31) / 32;
  const size_t mask_bytes = sizeof(unsigned) * (size_t)(o.rows_pad / 128) * o.mw;
  o.data.ensure(pool, sizeof(__nv_bfloat16) * (size_t)NS * o.rows_pad * o.ldk);
  o.exps.ensure(pool, sizeof(int) * (size_t)o.rows_pad);
  o.mask.ensure(pool, mask_bytes);
  TDVP_CUDA(cudaMemsetAsync(o.mask.as<void>(), 0, mask_bytes, st));
  const int log_rows = role == 0 ? o.rows_pad : o.rows_pad / 2;
  auto* d = o.data.as<__nv_bfloat16>();
  auto* e = o.exps.as<int>();
  auto* mk = o.mask.as<unsigned>();
  if (kcontig) {
    if (role == 0)
      k_digits_k<0><<<log_rows, 128, 0, st>>>(p, ld, rows, K, conj, ml, wl, o.rows_pad, o.ldk, d, e, mk, o.mw);
    else
      k_digits_k<1><<<log_rows, 128, 0, st>>>(p, ld, rows, K, conj, ml, wl, o.rows_pad, o.ldk, d, e, mk, o.mw);
  } else {
    if (role == 0)
      k_digits_r<0><<<log_rows / 8, 256, 0, st>>>(p, ld, rows, K, conj, o.rows_pad, o.ldk, d, e, mk, o.mw);
    else
      k_digits_r<1><<<log_rows / 8, 256, 0, st>>>(p, ld, rows, K, conj, o.rows_pad, o.ldk, d, e, mk, o.mw);
  }
  TDVP_CHECK_LAUNCH();
}

CUtensorMap digits_map(const Digits& o, int nslices) {
  const void* base = o.data.as<void>();
  tdvp_require((reinterpret_cast<uintptr_t>(base) & 15) == 0, TDVP_ERR_INVALID_ARG, "TMA base not 16B aligned");
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  cuuint64_t dims[3] = {(cuuint64_t)o.ldk, (cuuint64_t)o.rows_pad, (cuuint64_t)NS};
  cuuint64_t strides[2] = {(cuuint64_t)o.ldk * 2, (cuuint64_t)o.rows_pad * o.ldk * 2};
  cuuint32_t box[3] = {(cuuint32_t)BK, 128, (cuuint32_t)nslices};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  tdvp_require(r == CUDA_SUCCESS, TDVP_ERR_CUDA, "cuTensorMapEncodeTiled (f64 digits) failed: " + std::to_string((int)r));
  return m;
}

// C[M x N] (complex) = alpha A B + beta C over the digits of A (role 0) and B (role 1)
void gemm_digits(cudaStream_t st, DevicePool* pool, const Digits& A, const Digits& B, int M, int N, cplx alpha,
                 cplx beta, cplx* C, long long ldc, int* err) {
  tdvp_require(A.ldk == B.ldk && A.mw == B.mw && M <= A.rows_pad && 2 * N <= B.rows_pad, TDVP_ERR_INVALID_ARG,
               "gemm_digits: operands differ");
  const int sms = per_device([] {
    cudaFuncAttributes fa;
    TDVP_CUDA(cudaFuncGetAttributes(&fa, k_gemm_f64s));
    tdvp_require(fa.numRegs == REGS_LAUNCH, TDVP_ERR_CUDA,
                 "gemm_f64s: kernel built with " + std::to_string(fa.numRegs) + " registers, expected " +
                     std::to_string(REGS_LAUNCH));
    TDVP_CUDA(cudaFuncSetAttribute(k_gemm_f64s, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    int dev = 0, n = 0;
    TDVP_CUDA(cudaGetDevice(&dev));
    TDVP_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    return n > 0 ? n : 148;
  });
  const int nkb = A.ldk / BK, nchunks = (nkb + KC_KB - 1) / KC_KB;
  const long long tiles = (long long)ceil_div(M, BM) * ceil_div(2 * N, BN);
  // Splits of the two passes along K.  One product of one chunk takes about 0.5 us of an SM and a
  // CTA about 4 us beside its products; one CTA per SM runs at a time.  The pair of splits with the
  // smallest estimate: the longest CTA, or the whole work over the SMs and half a CTA for the tail.
  const int need = (nchunks + kMaxChunks - 1) / kMaxChunks;
  int s_hi = need, s_lo = need, c_hi = nchunks, c_lo = nchunks;
  double best = 1e300;
  for (int a = need; a <= std::min(nchunks, need + 31); ++a)
    for (int b = a; b <= std::min(nchunks, need + 31); ++b) {
      const int ca = (nchunks + a - 1) / a, cb = (nchunks + b - 1) / b;
      const int sa = (nchunks + ca - 1) / ca, sb = (nchunks + cb - 1) / cb;
      const double ta = 4.0 + 0.5 * 10 * ca, tb = 4.0 + 0.5 * 24 * cb, top = std::max(ta, tb);
      const double all = tiles * (sa * ta + sb * tb) / sms;
      const double t = (tiles * (sa + sb) <= sms ? top : std::max(top, all) + 0.5 * top) + 0.02 * (sa + sb);
      if (t < best) {
        best = t;
        s_hi = sa;
        s_lo = sb;
        c_hi = ca;
        c_lo = cb;
      }
    }
  const dim3 grid(ceil_div(2 * N, BN), ceil_div(M, BM), s_hi + s_lo);
  tdvp_require(grid.y <= 65535 && grid.z <= 65535, TDVP_ERR_INVALID_ARG, "gemm_f64s: grid too large");
  RawBuf ws;
  ws.ensure(pool, sizeof(cplx) * (size_t)(s_hi + s_lo) * M * N);
  const CUtensorMap a4 = digits_map(A, 4), b4 = digits_map(B, 4), a7 = digits_map(A, 7), b7 = digits_map(B, 7);
  k_gemm_f64s<<<grid, THREADS, SMEM_BYTES, st>>>(a4, b4, a7, b7, M, 2 * N, nkb, s_hi, c_hi * KC_KB, c_lo * KC_KB,
                                                  A.exps.as<int>(), B.exps.as<int>(), ws.as<double>(), err,
                                                  A.mask.as<unsigned>(), B.mask.as<unsigned>(), A.mw);
  TDVP_CHECK_LAUNCH();
  const long long n = (long long)M * N;
  k_f64_reduce<<<(int)std::min<long long>(ceil_div(n, 256), 16LL * sms), 256, 0, st>>>(ws.as<cplx>(), s_hi + s_lo, M, N,
                                                                                    alpha, beta, C, ldc);
  TDVP_CHECK_LAUNCH();
}
}  // namespace tcf

using namespace tcf;

struct F64EnvDigits {
  long long key = -1;
  Digits L, R;
};

// Below: the digit kernels, the GEMM and the reduction are four launches of 3-5 us each, so the
// plain FP64 GEMM (6.6 ns per 1000 complex multiply-adds on the whole device) is faster under
// about 4 M of them, and thin operands fill too little of a 128-wide tile.
bool f64_on_tensor_cores(long long M, long long N, long long K) {
  return M >= 64 && N >= 32 && K >= 32 && M * N * K >= (1LL << 22) && M < (1LL << 30) && N < (1LL << 29) &&
         K < (1LL << 29);
}

// Device memory that the digits and partial results of one product may take, and with H_eff's kept digits
// those of an apply.  Digits take 1.75 and 3.5 times their operands and the partials twice the output:
// 3 GB for H_eff at 1024 x 1024, w = 14, where T1 and T2 are 0.9 GB.  Beyond the limit a product runs in
// panels of A's rows and B's columns and H_eff keeps no digits, so that a size that fits the device
// without them still does, and a pool holding more than the limit in unused blocks gives them back.
// (A product that large runs for 50 ms and more, its digits and the allocations for a few.)
constexpr size_t kWorkBytes = size_t(8) << 30;
size_t digits_bytes(long long rows, long long K) {  // of `rows` real rows
  return sizeof(__nv_bfloat16) * NS * (size_t)((rows + 127) / 128 * 128) * (size_t)((2 * K + BK - 1) / BK * BK);
}
size_t partial_bytes(long long M, long long N) { return 2 * sizeof(cplx) * (size_t)M * (size_t)N; }
void give_back(DevicePool* pool) {
  if (pool->cached_bytes() > kWorkBytes) pool->trim();
}

void zgemm_f64s(cudaStream_t st, Scratch& s, int opA, int opB, int M, int N, int K, cplx alpha, const cplx* A,
                long long lda, const cplx* B, long long ldb, cplx beta, cplx* C, long long ldc) {
  int* err = tc_error_word(st, s);
  int mp = M, np = N;  // a panel: mp x np of the output, in steps of a tile (128 real rows each)
  while (digits_bytes(mp, K) + digits_bytes(2LL * np, K) + partial_bytes(mp, np) > kWorkBytes && (mp > 128 || np > 64)) {
    if (mp > 128 && (np <= 64 || mp >= 2LL * np))
      mp = pad_to((mp + 1) / 2, 128);
    else
      np = pad_to((np + 1) / 2, 64);
  }
  const bool ka = opA == OP_N || opA == OP_R, kb = opB == OP_T || opB == OP_C;
  Digits a, b;
  for (int n0 = 0; n0 < N; n0 += np) {
    const int nn = std::min(np, N - n0);
    make_digits(st, s.pool, 1, kb, kb ? B + n0 * ldb : B + n0, ldb, nn, K, opB == OP_C || opB == OP_R, b);
    for (int m0 = 0; m0 < M; m0 += mp) {
      const int mm = std::min(mp, M - m0);
      if (n0 == 0 || mp < M)
        make_digits(st, s.pool, 0, ka, ka ? A + m0 * lda : A + m0, lda, mm, K, opA == OP_C || opA == OP_R, a);
      gemm_digits(st, s.pool, a, b, mm, nn, alpha, beta, C + m0 * ldc + n0, ldc, err);
    }
  }
  if (mp < M || np < N) {
    a = Digits();
    b = Digits();
    give_back(s.pool);
  }
}

// H_eff with the digits of L and R kept for the applies that share op.env_key.  T1 has its rows
// in (w, a) order, so that a 128-row tile of L holds one MPO channel and under a conserved charge
// meets one sector of its columns.
void heff_f64s(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y) {
  const int ml = op.ml, mr = op.mr, wl = op.wl, wr = op.wr, d = op.d;
  const cplx one = mkc(1.0, 0.0), zero = mkc(0.0, 0.0);
  int* err = tc_error_word(st, s);
  const size_t kept = digits_bytes((long long)ml * wl, ml) + digits_bytes(2LL * mr, (long long)wr * mr);
  const size_t first = digits_bytes(2LL * d * mr, ml) + partial_bytes((long long)ml * wl, (long long)d * mr);
  const size_t second = digits_bytes((long long)ml * d, (long long)wr * mr) + partial_bytes((long long)ml * d, mr);
  if (kept + std::max(first, second) > kWorkBytes) {
    s.f64.reset();
    s.t1.ensure(s.pool, (size_t)ml * wl * d * mr);
    s.t2.ensure(s.pool, (size_t)ml * d * wr * mr);
    zgemm_f64s(st, s, OP_N, OP_N, ml * wl, d * mr, ml, one, op.L, ml, x, (long long)d * mr, zero, s.t1.data(),
               (long long)d * mr);
    wstage_left(st, *op.W, s.t1.data(), s.t2.data(), ml, mr);
    zgemm_f64s(st, s, OP_N, OP_T, ml * d, mr, wr * mr, one, s.t2.data(), (long long)wr * mr, op.R, (long long)wr * mr,
               zero, y, mr);
    give_back(s.pool);
    return;
  }
  if (!s.f64) s.f64 = std::make_shared<F64EnvDigits>();
  F64EnvDigits& c = *s.f64;
  if (op.env_key < 0 || c.key != op.env_key) {
    c.key = -1;
    make_digits(st, s.pool, 0, true, op.L, ml, ml * wl, ml, false, c.L, ml, wl);
    make_digits(st, s.pool, 1, true, op.R, (long long)wr * mr, mr, wr * mr, false, c.R);
    c.key = op.env_key;
  }
  s.t1.ensure(s.pool, (size_t)ml * wl * d * mr);
  s.t2.ensure(s.pool, (size_t)ml * d * wr * mr);
  {
    Digits xd;
    make_digits(st, s.pool, 1, false, x, (long long)d * mr, d * mr, ml, false, xd);
    gemm_digits(st, s.pool, c.L, xd, ml * wl, d * mr, one, zero, s.t1.data(), (long long)d * mr, err);
  }
  wstage_left(st, *op.W, s.t1.data(), s.t2.data(), ml, mr, true);
  Digits td;
  make_digits(st, s.pool, 0, true, s.t2.data(), (long long)wr * mr, ml * d, wr * mr, false, td);
  gemm_digits(st, s.pool, td, c.R, ml * d, mr, one, zero, y, mr, err);
}
