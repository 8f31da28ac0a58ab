// Tensor-core complex GEMMs with BF16 "exact slices" (sm_103a, tcgen05 kind::f16).
//
// Each real operand (the 4M embedding of the complex one, as in the TF32 path)
// is cut into fixed-point slices.  For one scaling group, with 2^e the smallest
// power of two above its largest magnitude, every entry is written as
//   x = 2^e (a1 2^-8 + a2 2^-16 + a3 2^-24 + a4 2^-32) + r,   |r| <= 2^(e-33),
// with integers |a1| <= 256 and |a_s| <= 128 (s > 1), exact in BF16.  Slice s is
// stored as a_s 2^(-8(s-1)) (exact) and the group scale as the float 2^(e-8).
// A-operand groups are one row and one chunk of 128 along K; B-operand groups
// are whole rows, so the B scale is one factor per output column, applied once.
//
// The products of slices s, t (0-based) with s + t <= S - 1 are summed: the
// leading product a1 b1 in accumulator P, all others in accumulator Q.  Within a
// chunk P is a sum of at most 128 integers of magnitude <= 2^16, so every partial
// sum is an integer below 2^24 and the tensor core's FP32 accumulation of P is
// exact whatever its rounding.  Q is about 2^-7 of P; its 72 (S = 4) MMA
// accumulations per chunk, each rounding near 2^-23 of Q, leave about 2^-24 of P.  The epilogue scales each chunk by its A chunk scale
// (a power of two: exact) and adds it into a double-float (hi, lo) pair per output
// with Knuth's two-sum, so no error accrues across chunks.  GB300 runs FP64 at a
// small fraction of its FP32 rate, which is why the promotion uses FP32 pairs.
// S = 4 (10 products) represents the operands to 2^-33 of their group maxima and
// the products to about 2^-24 (the rounding of Q); S = 3 (6 products) to 2^-25.
//
// Kernel layout (one CTA per 128 x 128 output tile, three warpgroups):
//   warp 0       TMA producer: one 3-D box per operand and stage (all S slices)
//   warp 1       TMEM allocator and single-thread tcgen05.mma issuer
//   warps 2, 3   idle
//   warps 4..11  epilogue: warp w reads TMEM lanes 32*(w%4)..+31, columns 64*((w-4)/4)..+63
// The first warpgroup gives registers back (setmaxnreg 40) so that the epilogue
// warpgroups can hold 64 (hi, lo) pairs per thread (setmaxnreg 232):
// 128 * 40 + 256 * 232 = 384 * 168, the launch's own allocation.
// Tensor memory: two chunk buffers (ping-pong) x (P, Q) x 128 columns = 512 columns.
// Every mbarrier wait is bounded; on expiry the CTA records an error word, drains
// its copies and MMAs (bounded) and frees its tensor memory.
#include <cuda_bf16.h>

#include <cstring>

#include "contract.cuh"
#include "tc_ptx.cuh"

namespace tcb {
using namespace tc;

constexpr int BM = 128, BN = 128, BK = 32, STAGES = 3;
constexpr int KC = 128;                 // K elements per chunk (exactness bound of P: 128 * 2^16 < 2^24)
constexpr int kMaxChunks = 1024;        // chunks one CTA can walk (K up to 131072 real entries per split)
constexpr int KC_KB = KC / BK;          // k-blocks per chunk
constexpr int EPI_WARPS = 8;
constexpr int EPI_WARP0 = 4;            // first epilogue warp (second warpgroup)
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr int REGS_LAUNCH = 168, REGS_LOW = 40, REGS_HIGH = 232;
static_assert(128 * REGS_LOW + 32 * EPI_WARPS * REGS_HIGH <= THREADS * REGS_LAUNCH, "register split");
constexpr int TILE = BM * BK * 2;       // one slice of one operand tile (bytes); BM == BN
constexpr int TMEM_COLS = 512;
constexpr int EC = 64;                  // output columns per epilogue thread
constexpr int EPI_ROW = EC * 8 + 16;    // bytes of a row of a warp's turned output (odd in 16-byte units)

template <int S>
struct SCfg {
  static constexpr int STAGE_BYTES = 2 * S * TILE;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static_assert(EPI_WARPS * 32 * EPI_ROW <= STAGES * STAGE_BYTES, "output tile in the stages");
};

// Two floats in one 64-bit register: sm_103a adds and multiplies both with one instruction (each
// rounded to nearest as alone).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(uint32_t a, uint32_t b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a - b (b times -1 plus a: one rounding)
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xbf800000bf800000ull), "l"(a));
  return r;
}
// hi + lo += v without loss (Knuth's two-sum into hi, its error into lo), two entries at once
__device__ __forceinline__ void two_sum_acc(f32x2& hi, f32x2& lo, f32x2 v) {
  const f32x2 s = add2(hi, v);
  const f32x2 bb = sub2(s, hi);
  const f32x2 e = add2(sub2(hi, sub2(s, bb)), sub2(v, bb));
  hi = s;
  lo = add2(lo, e);
}

// a float as a double by its bits (exact; an FP64 conversion would run on the FP64 pipe)
__device__ __forceinline__ double float_bits_to_double(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
  if (e == 0 || e == 255) return (double)x;  // zero, subnormal, not finite
  return __hiloint2double((int)((u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu)), (int)(u << 29));
}

// (double)h + (double)l, the same bits, by integer operations on the sum's mantissa when l is the
// smaller part: an FP64 addition holds the FP64 pipe for 16 cycles per warp, these 25 integer
// operations for 7 issue slots of each scheduler.
__device__ __forceinline__ double df_to_double(float h, float l) {
  const unsigned hb = __float_as_uint(h), lb = __float_as_uint(l);
  const int eh = (int)((hb >> 23) & 0xffu), el = (int)((lb >> 23) & 0xffu), sh = eh - el;
  const double d = float_bits_to_double(h);
  if (lb << 1 == 0u) return d;
  if (eh == 0 || el == 0 || eh == 255 || sh < 1) return d + float_bits_to_double(l);
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned m = (lb & 0x7fffffu) | 0x800000u;  // l = m 2^(29 - sh) units in the last place of d
  const bool minus = (hb ^ lb) >> 31;
  unsigned long long t;
  if (sh <= 29) {
    t = (unsigned long long)m << (29 - sh);
  } else {
    const int k = min(sh - 29, 25);  // from 25 on l is below half a unit
    const unsigned q = m >> k, rem = m & ((1u << k) - 1u), half = 1u << (k - 1);
    const unsigned odd = (unsigned)(minus ? u - q : u + q) & 1u;
    t = q + ((rem > half || (rem == half && odd)) ? 1u : 0u);  // to nearest even
  }
  const unsigned long long r = minus ? u - t : u + t;
  // the exponent changes, or a power of two loses a part that only the finer half below it resolves
  if ((r ^ u) >> 52 || (minus && !(u & 0xfffffffffffffull))) return d + float_bits_to_double(l);
  return __longlong_as_double((long long)r);
}

// x as a float pair: hi = (float)x, lo = (float)(x - hi), the same bits by integer operations where
// both parts are normal (four operations of the FP64 pipe otherwise)
__device__ __forceinline__ float2 double_to_df(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((u >> 52) & 0x7ff) - 1023;
  if (e < -74 || e > 126) {
    if (u << 1 == 0ull) return make_float2((float)x, 0.f);
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
  }
  const unsigned sign = (unsigned)(u >> 63) << 31;
  const unsigned top = (unsigned)((u & 0xfffffffffffffull) >> 29);  // 23 bits after the leading one
  const unsigned rest = (unsigned)u & 0x1fffffffu;                  // 29 bits below
  const unsigned up = rest > 0x10000000u || (rest == 0x10000000u && (top & 1u));  // to nearest even
  const float hi = __uint_as_float((sign | ((unsigned)(e + 127) << 23) | top) + up);
  const int rem = (int)rest - (up ? 0x20000000 : 0);  // x - hi in units 2^(e-52), of x's sign
  const float lo = __int2float_rn(sign ? -rem : rem) * __uint_as_float((unsigned)(e - 52 + 127) << 23);
  return make_float2(hi, rem == 0 ? 0.f : lo);
}

// x 2^e for a power of two s = 2^e given as a float, by the exponent bits when both sides are normal
__device__ __forceinline__ double scale_pow2(double x, float s) {
  const int e = (int)((__float_as_uint(s) >> 23) & 0xffu) - 127;
  const int h = __double2hiint(x), ex = (h >> 20) & 0x7ff;
  if (ex == 0 || ex == 0x7ff || ex + e <= 0 || ex + e >= 0x7ff || e == 128 || e == -127) return x * (double)s;
  return __hiloint2double(h + (e << 20), __double2loint(x));
}

// (output tile, K chunk) pairs visited by k_gemm_bf16s since load: [0] all, [1] multiplied
__device__ unsigned long long g_chunk_pairs[2];

template <int S>
__global__ void __launch_bounds__(THREADS, 1)
    k_gemm_bf16s(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M, int N,
                 int nkb_total, int kb_split, const float* __restrict__ sA, long long lsA,
                 const float* __restrict__ sB, void* __restrict__ out, long long ldo, long long split_stride,
                 int out_df, int skip_empty, int* __restrict__ err, const unsigned* __restrict__ maskA,
                 const unsigned* __restrict__ maskB, int mwords) {
  constexpr int STAGE_BYTES = SCfg<S>::STAGE_BYTES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + STAGES;
  uint64_t* tfull = bars + 2 * STAGES;
  uint64_t* tempty = bars + 2 * STAGES + 2;
  uint64_t* done = bars + 2 * STAGES + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  // split K: this CTA takes k-blocks [kb0, kb0 + nkb) (kb0 a multiple of a chunk)
  const int kb0 = blockIdx.z * kb_split;
  const int nkb = min(nkb_total, kb0 + kb_split) - kb0;
  const int c0 = kb0 / KC_KB;
  const int nchunks = (nkb + KC_KB - 1) / KC_KB;
  // Chunks whose A tile (these BM rows) or B tile (these BN rows) holds only zeros add exact
  // zeros to this output tile: the list of the others, built once (the slicing kernels set a
  // bit per 128-row tile and chunk that holds a nonzero entry) by one warp.  All three roles walk it.
  __shared__ int act[kMaxChunks];
  __shared__ int n_act;
  if (warp == 0) {
    const int n = active_chunks(maskA + (long long)blockIdx.y * mwords, maskB + (long long)blockIdx.x * mwords, c0,
                                nchunks, kMaxChunks, act);
    if (lane == 0) {
      n_act = n;
      atomicAdd(&g_chunk_pairs[0], (unsigned long long)nchunks);
      atomicAdd(&g_chunk_pairs[1], (unsigned long long)n);
    }
  }

  if (threadIdx.x == 32) {
    prefetch_map(&tmA);
    prefetch_map(&tmB);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
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
  if (warp < EPI_WARP0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LOW));
  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer: all S slices of the A and B tiles of one k-block
    int issued = 0;  // running count of k-blocks loaded (stage = issued % STAGES)
    for (int ai = 0; ai < n_act && !*abort_flag; ++ai) {
      const int c = act[ai];
      const int kb_end = min(nkb, (c + 1) * KC_KB);
      for (int kb = c * KC_KB; kb < kb_end; ++kb) {
        const int s = issued % STAGES, it = issued / STAGES;
        if (it > 0 && !mbar_wait(smem_u32(&empty[s]), (it - 1) & 1)) {
          *abort_flag = 1;
          break;
        }
        if (*abort_flag) break;
        uint8_t* st = smem + s * STAGE_BYTES;
        const uint32_t fb = smem_u32(&full[s]);
        mbar_expect_tx(fb, STAGE_BYTES);
        tma_load_3d(smem_u32(st), &tmA, fb, (kb0 + kb) * BK, m0, 0);
        tma_load_3d(smem_u32(st + S * TILE), &tmB, fb, (kb0 + kb) * BK, n0, 0);
        ++issued;
      }
    }
    if (*abort_flag) {
      for (int q = (issued > STAGES ? issued - STAGES : 0); q < issued; ++q)
        (void)mbar_wait(smem_u32(&full[q % STAGES]), (q / STAGES) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    const uint32_t idesc = idesc_bf16(BM, BN);
    const uint64_t desc = sdesc<64>(smem_u32(smem));
    const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
    int used = 0;  // running count of k-blocks consumed, in the producer's order
    for (int ai = 0; ai < n_act && !*abort_flag; ++ai) {
      const int c = act[ai];
      const int b = ai & 1, u = ai >> 1;
      if (u > 0 && !mbar_wait(smem_u32(&tempty[b]), (u - 1) & 1)) {
        *abort_flag = 1;
        break;
      }
      fence_after();
      const uint32_t accP = tmem + (uint32_t)(b * 2 * BN);
      const uint32_t accQ = accP + BN;
      const int kb_end = min(nkb, (c + 1) * KC_KB);
      for (int kb = c * KC_KB; kb < kb_end; ++kb) {
        const int s = used % STAGES, it = used / STAGES;
        ++used;
        if (!mbar_wait(smem_u32(&full[s]), it & 1)) {
          *abort_flag = 1;
          break;
        }
        fence_after();
        const uint32_t a0 = desc_lo + s * (STAGE_BYTES >> 4);
        const uint32_t b0 = a0 + (S * TILE >> 4);
        const uint32_t cont = kb == c * KC_KB ? 0u : 1u;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) {
          constexpr int KS = 2;  // 16 bf16 = 32 bytes along K inside the 64-byte swizzle atom
          if (k == 0)
            mma_bf16_first(accP, a0, b0, desc_hi, idesc, cont);
          else
            mma_bf16_acc(accP, a0 + k * KS, b0 + k * KS, desc_hi, idesc);
#pragma unroll
          for (int sa = 0; sa < S; ++sa)
#pragma unroll
            for (int sb = 0; sb + sa < S; ++sb) {
              if (sa == 0 && sb == 0) continue;
              const uint32_t da = a0 + (sa * TILE >> 4) + k * KS, db = b0 + (sb * TILE >> 4) + k * KS;
              if (k == 0 && sa == 0 && sb == 1)
                mma_bf16_first(accQ, da, db, desc_hi, idesc, cont);
              else
                mma_bf16_acc(accQ, da, db, desc_hi, idesc);
            }
        }
        mma_commit(smem_u32(&empty[s]));
      }
      if (*abort_flag) break;
      mma_commit(smem_u32(&tfull[b]));
    }
    mma_commit(smem_u32(done));
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_HIGH));
    // ---------------- epilogue: scale each chunk and add it into (hi, lo) pairs
    const int q = warp & 3;
    const int half = (warp - EPI_WARP0) >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const int gm = m0 + q * 32 + lane;  // this thread's row in the accumulators
    const int nb = n0 + half * EC;
    f32x2 hi[EC / 2], lo[EC / 2];
#pragma unroll
    for (int j = 0; j < EC / 2; ++j) hi[j] = lo[j] = 0ull;
    bool ok = true;
    for (int ai = 0; ai < n_act; ++ai) {
      const int c = act[ai];
      const int b = ai & 1, u = ai >> 1;
      bool got = mbar_wait(smem_u32(&tfull[b]), u & 1);
      if (!got) *abort_flag = 1;
      ok = __all_sync(0xffffffffu, got && !*abort_flag);
      if (!ok) break;
      fence_after();
      const uint32_t sab = __float_as_uint(sA[(long long)(c0 + c) * lsA + gm]);
      const f32x2 sa = pack2(sab, sab);
#pragma unroll
      for (int e0 = 0; e0 < EC; e0 += 16) {
        uint32_t vp[16], vq[16];
        const uint32_t col = tmem + lane_base + (uint32_t)(b * 2 * BN + half * EC + e0);
        tmem_ld16(vp, col);
        tmem_ld16(vq, col + BN);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          two_sum_acc(hi[e0 / 2 + j], lo[e0 / 2 + j], mul2(pack2(vp[2 * j], vp[2 * j + 1]), sa));
          two_sum_acc(hi[e0 / 2 + j], lo[e0 / 2 + j], mul2(pack2(vq[2 * j], vq[2 * j + 1]), sa));
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&tempty[b]));
    }
    if (ok) {  // warp-uniform
      // A thread holds 64 columns of one row; written straight out, every store of a warp would touch
      // 32 rows (8 us per tile).  The warp turns its 32 x 64 entries through its own part of the
      // stages (all MMAs have read them) and stores whole 512-byte rows.
      uint8_t* reg = smem + (warp - EPI_WARP0) * 32 * EPI_ROW;
#pragma unroll
      for (int j = 0; j < EC / 2; ++j)
        *reinterpret_cast<uint4*>(reg + lane * EPI_ROW + j * 16) =
            make_uint4((uint32_t)hi[j], (uint32_t)lo[j], (uint32_t)(hi[j] >> 32), (uint32_t)(lo[j] >> 32));
      __syncwarp();
      // column scales: lane i holds those of columns nb + 2i, nb + 2i + 1 (inside the padded rows)
      const float2 sbv = __ldg(reinterpret_cast<const float2*>(sB + nb) + lane);
      const int col = nb + 2 * lane;
      const bool vec = col + 1 < N && (ldo & 1) == 0;
      // partials without a chunk are zeros that the reduction, which knows the masks, does not read
      const int rows = skip_empty && n_act == 0 ? 0 : min(32, M - (m0 + q * 32));
      for (int r = 0; r < rows; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(reg + r * EPI_ROW + lane * 16);
        const long long at = (long long)(m0 + q * 32 + r) * ldo + col;
        if (out_df) {
          // double-float output: (hi, lo) FP32 pairs, scaled exactly by the power-of-two column scale
          float2* o = static_cast<float2*>(out) + blockIdx.z * split_stride + at;
          const float4 t = make_float4(__fmul_rn(v.x, sbv.x), __fmul_rn(v.y, sbv.x), __fmul_rn(v.z, sbv.y),
                                       __fmul_rn(v.w, sbv.y));
          if (vec) {
            *reinterpret_cast<float4*>(o) = t;
          } else {
            if (col < N) o[0] = make_float2(t.x, t.y);
            if (col + 1 < N) o[1] = make_float2(t.z, t.w);
          }
        } else {
          double* o = static_cast<double*>(out) + at;
          const double d0 = scale_pow2(df_to_double(v.x, v.y), sbv.x);
          const double d1 = scale_pow2(df_to_double(v.z, v.w), sbv.y);
          if (vec) {
            *reinterpret_cast<double2*>(o) = make_double2(d0, d1);
          } else {
            if (col < N) o[0] = d0;
            if (col + 1 < N) o[1] = d1;
          }
        }
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

// ---------------------------------------------------------------- operand slicing
// GB300 executes FP64 at a small fraction of its FP32 and integer rates, so the
// slicing runs without FP64 arithmetic: FP64 sources are cut into digits with
// integer operations on their bit patterns, double-float sources (FP32 hi, lo
// pairs) with exact FP32 operations.
//
// Sources give the real operand entries (k2, k2+1, k2+2, k2+3) of one row (k2 a
// multiple of 4), zero outside the logical matrix.  FP64 sources (kDF = false)
// fill double v[4]; double-float sources (kDF = true) fill float hi[4], lo[4].

// Rows m of opA(A) with K interleaved (re, im): the A operand of the 4M form.
struct SrcA {
  static constexpr bool kDF = false;
  const cplx* p;
  long long ld;
  int rows, K, op;
  __device__ void load4(long long m, int k2, double v[4]) const {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = (k2 >> 1) + h;
      double re = 0.0, im = 0.0;
      if (m < rows && k < K) {
        const cplx z = (op == OP_N || op == OP_R) ? p[m * ld + k] : p[(long long)k * ld + m];
        re = z.x;
        im = (op == OP_C || op == OP_R) ? -z.y : z.y;
      }
      v[2 * h] = re;
      v[2 * h + 1] = im;
    }
  }
};
// Rows (w, a) of the stage-1 A operand of H_eff, read from L[a][w][a'] channel by channel:
// a 128-row tile then holds one MPO channel w over a run of sector-ordered a, and under a
// conserved charge its nonzero columns a' lie in the one sector q_a - c_w.  In (a, w) order a
// tile mixes every channel and reaches the sectors of all channel charges at once.
struct SrcLwa {
  static constexpr bool kDF = false;
  const cplx* p;
  int ML, WL;
  __device__ void load4(long long m, int k2, double v[4]) const {
    const long long w = m / ML, a = m % ML;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = (k2 >> 1) + h;
      double re = 0.0, im = 0.0;
      if (w < WL && k < ML) {
        const cplx z = p[(a * WL + w) * ML + k];
        re = z.x;
        im = z.y;
      }
      v[2 * h] = re;
      v[2 * h + 1] = im;
    }
  }
};
// s_hi + s_lo += (a_hi + a_lo)(b_hi + b_lo) in double-float arithmetic (about 2^-48)
__device__ __forceinline__ void df_mac(float& sh, float& sl, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  const float pe = __fmaf_rn(ah, bh, -p);  // exact rounding error of ah * bh
  const float cross = __fmaf_rn(ah, bl, __fmul_rn(al, bh));
  const float s = __fadd_rn(sh, p);
  const float bb = __fadd_rn(s, -sh);
  const float err = __fadd_rn(__fadd_rn(sh, -__fadd_rn(s, -bb)), __fadd_rn(p, -bb));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, __fadd_rn(pe, cross)));
}

// Rows (a, s) of the stage-3 A operand of H_eff: K index (v, b', re/im),
//   T2[(a,s)][(v,b')] = sum_{(w,t)} W[w,s,t,v] T1[w][a][t][b']   (T1 rows in (w, a) order)
// with T1 and W as double-float complex (re hi, re lo, im hi, im lo).
struct SrcStage2 {
  static constexpr bool kDF = true;
  const float4* T1;
  const int* off;
  const int* idx;
  const float4* val;
  int ML, WL, WR, D, MR;
  __device__ void load4(long long row, int k2, float hi[4], float lo[4]) const {
    const long long a = row / D;
    const int s = (int)(row % D);
    const int j = k2 >> 1;
    const int vv = j / MR, b = j % MR;
    float r[2][2], i[2][2];  // (hi, lo) of the real and imaginary parts of the entries j, j + 1
#pragma unroll
    for (int h = 0; h < 2; ++h) r[h][0] = r[h][1] = i[h][0] = i[h][1] = 0.f;
    auto add = [&](int h, const float4 c, const float4 x) {
      df_mac(r[h][0], r[h][1], c.x, c.y, x.x, x.y);     // + Re c Re x
      df_mac(r[h][0], r[h][1], -c.z, -c.w, x.z, x.w);   // - Im c Im x
      df_mac(i[h][0], i[h][1], c.x, c.y, x.z, x.w);     // + Re c Im x
      df_mac(i[h][0], i[h][1], c.z, c.w, x.x, x.y);     // + Im c Re x
    };
    if (a < ML && vv < WR && b + 1 < MR) {  // one MPO column: both loads of an entry in flight together
      const int sv = s * WR + vv;
      for (int e = off[sv]; e < off[sv + 1]; ++e) {
        const float4* x = T1 + ((idx[2 * e] * ML + a) * D + idx[2 * e + 1]) * (long long)MR + b;
        const float4 x0 = x[0], x1 = x[1], c = val[e];
        add(0, c, x0);
        add(1, c, x1);
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v1 = (j + h) / MR, b1 = (j + h) % MR;
        if (a < ML && v1 < WR) {
          const int sv = s * WR + v1;
          for (int e = off[sv]; e < off[sv + 1]; ++e)
            add(h, val[e], T1[((idx[2 * e] * ML + a) * D + idx[2 * e + 1]) * (long long)MR + b1]);
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // renormalise so that |lo| <= ulp(hi) / 2
      float t = __fadd_rn(r[h][0], r[h][1]);
      r[h][1] = __fadd_rn(r[h][1], -__fadd_rn(t, -r[h][0]));
      r[h][0] = t;
      t = __fadd_rn(i[h][0], i[h][1]);
      i[h][1] = __fadd_rn(i[h][1], -__fadd_rn(t, -i[h][0]));
      i[h][0] = t;
      hi[2 * h] = r[h][0];
      lo[2 * h] = r[h][1];
      hi[2 * h + 1] = i[h][0];
      lo[2 * h + 1] = i[h][1];
    }
  }
};

// Group exponent: the smallest e with (largest magnitude) < 2^e.  Groups whose largest
// magnitude is below 2^-100 (or zero) are taken as zero (live = false); a non-finite
// entry makes the scale NaN, so that it shows in the output.
struct GroupScale {
  int e = 0;
  bool live = false;
  float sc = 0.f;  // 2^(e-8)
};
__device__ __forceinline__ GroupScale scale_from_exponent(int unbiased, bool bad) {
  GroupScale g;
  if (bad) {
    g.sc = __int_as_float(0x7fc00000);
  } else if (unbiased >= -100) {
    g.live = true;
    g.e = unbiased + 1;
    g.sc = ldexpf(1.f, g.e - 8);
  }
  return g;
}
// |x| as an ordered integer key (larger magnitude, larger key; NaN/Inf above all finite)
__device__ __forceinline__ unsigned long long abs_key(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ GroupScale scale_from_key(unsigned long long key) {
  const int ex = (int)(key >> 52);
  if (ex == 0x7ff) return scale_from_exponent(0, true);
  if (ex == 0) return scale_from_exponent(-2000, false);  // zero or subnormal
  return scale_from_exponent(ex - 1023, false);
}
__device__ __forceinline__ GroupScale scale_from_float(float m, bool bad) {
  const int ex = (int)((__float_as_uint(m) >> 23) & 0xff);
  if (bad || ex == 0xff) return scale_from_exponent(0, true);
  if (ex == 0) return scale_from_exponent(-2000, false);
  return scale_from_exponent(ex - 127, false);
}

// integer value a (|a| < 2^22) as an exact float
__device__ __forceinline__ float int_to_float_exact(int a) {
  return __fadd_rn(__int_as_float(0x4B400000 + a), -12582912.0f);
}

// Digits of an FP64 entry: X = round(|x| 2^(32-e)) (|X| <= 2^32) from the bit pattern,
// then X = a1 2^24 + a2 2^16 + a3 2^8 + a4 with rounded signed digits; out[s] = a_{s+1} 2^(-8s).
template <int S>
__device__ __forceinline__ void digits_fp64(double x, const GroupScale& g, float out[S]) {
  long long X = 0;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (g.live && ex != 0) {
    const int shift = 20 + g.e - (ex - 1023);  // >= 21
    if (shift < 64) {
      const unsigned long long m53 = (b & 0xfffffffffffffull) | (1ull << 52);
      X = (long long)((m53 + (1ull << (shift - 1))) >> shift);
      if (b >> 63) X = -X;
    }
  }
  const int a1 = (int)((X + (1ll << 23)) >> 24);
  int r = (int)(X - ((long long)a1 << 24));  // [-2^23, 2^23)
  const int a2 = (r + (1 << 15)) >> 16;
  r -= a2 << 16;
  int a3, a4;
  if (S == 4) {
    a3 = (r + (1 << 7)) >> 8;
    a4 = r - (a3 << 8);
  } else {
    a3 = (r + (1 << 7)) >> 8;
    a4 = 0;
  }
  const int dg[4] = {a1, a2, a3, a4};
#pragma unroll
  for (int s = 0; s < S; ++s) out[s] = __fmul_rn(int_to_float_exact(dg[s]), __int_as_float((127 - 8 * s) << 23));
}

// Digits of a double-float entry hi + lo with exact FP32 steps: peel the rounded
// top digit off the head, fold the tail back in with a two-sum, repeat.
template <int S>
__device__ __forceinline__ void digits_df(float hi, float lo, const GroupScale& g, float out[S]) {
  if (!g.live) {
#pragma unroll
    for (int s = 0; s < S; ++s) out[s] = 0.f;
    return;
  }
  const float up = ldexpf(1.f, 32 - g.e);
  float H = __fmul_rn(hi, up), L = __fmul_rn(lo, up);  // |H + L| < 2^32
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int sh = 24 - 8 * s;                          // digit weight 2^sh
    const float w = __int_as_float((127 + sh) << 23), iw = __int_as_float((127 - sh) << 23);
    const float a = rintf(__fmul_rn(H, iw));
    out[s] = __fmul_rn(a, __int_as_float((127 - 8 * s) << 23));
    const float r = __fmaf_rn(-a, w, H);  // exact
    const float t = __fadd_rn(r, L);
    const float bb = __fadd_rn(t, -r);
    L = __fadd_rn(__fadd_rn(r, -__fadd_rn(t, -bb)), __fadd_rn(L, -bb));
    H = t;
  }
}

template <int S>
__device__ __forceinline__ void store_slices(const float d[4][S], __nv_bfloat16* out, long long slice_stride) {
#pragma unroll
  for (int s = 0; s < S; ++s) {
    // every digit has at most 8 significant bits: the top half of its FP32 pattern is its BF16
    uint2 pk;
    pk.x = (__float_as_uint(d[0][s]) >> 16) | (__float_as_uint(d[1][s]) & 0xffff0000u);
    pk.y = (__float_as_uint(d[2][s]) >> 16) | (__float_as_uint(d[3][s]) & 0xffff0000u);
    *reinterpret_cast<uint2*>(out + s * slice_stride) = pk;
  }
}

// The entries of one row segment: group-max contribution and the source values.
template <class Src>
struct Seg {
  double v[4];
  float hi[4], lo[4];
  __device__ void load(const Src& src, long long row, int k2) {
    if constexpr (Src::kDF) {
      src.load4(row, k2, hi, lo);
    } else {
      src.load4(row, k2, v);
    }
  }
  __device__ void zero() {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = 0.0;
      hi[i] = lo[i] = 0.f;
    }
  }
  // max key (FP64) or max |hi| (double-float); bad = non-finite seen
  __device__ unsigned long long key() const {
    unsigned long long k = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) k = max(k, abs_key(v[i]));
    return k;
  }
  __device__ float fmaxabs(bool& bad) const {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float a = fabsf(hi[i]);
      bad = bad || !(a <= 3.0e38f) || !(fabsf(lo[i]) <= 3.0e38f);
      m = fmaxf(m, a);
    }
    return m;
  }
  template <int S>
  __device__ void write(const GroupScale& g, __nv_bfloat16* out, long long slice_stride) const {
    float d[4][S];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (Src::kDF)
        digits_df<S>(hi[i], lo[i], g, d[i]);
      else
        digits_fp64<S>(v[i], g, d[i]);
    }
    store_slices<S>(d, out, slice_stride);
  }
};

// warp-wide group scale of the segments held by the 32 lanes
template <class Src>
__device__ __forceinline__ GroupScale warp_scale(const Seg<Src>& sg) {
  if constexpr (Src::kDF) {
    bool bad = false;
    float m = sg.fmaxabs(bad);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    bad = __any_sync(0xffffffffu, bad);
    return scale_from_float(m, bad);
  } else {
    unsigned long long k = sg.key();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
    return scale_from_key(k);
  }
}

// Marks (row tile, chunk) as nonzero.  (Reading the word first to spare the atomic doubles the
// slicing time: the atomic needs no answer, the read does.)
__device__ __forceinline__ void mark_chunk(unsigned* mask, int mw, long long row, int ch) {
  atomicOr(&mask[(row >> 7) * mw + (ch >> 5)], 1u << (ch & 31));
}

// A operands: one warp per (row, chunk of 128 K entries).
// out: [S][rows_pad][ldk] bf16; scale: [nch][rows_pad] float.
// mask: bit ch of word (row / 128) * mw + ch / 32 is set when the group is not
// zero (its scale is nonzero or NaN), i.e. when the chunk holds a nonzero entry of the row tile.
template <int S, class Src>
__global__ void k_slice_chunks(Src src, int rows_pad, int ldk, int nch, __nv_bfloat16* __restrict__ out,
                               float* __restrict__ scale, unsigned* __restrict__ mask, int mw) {
  const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= (long long)rows_pad * nch) return;  // warp-uniform
  const long long row = gw / nch;
  const int ch = (int)(gw % nch);
  const int k2 = ch * KC + 4 * lane;
  Seg<Src> sg;
  sg.zero();
  if (k2 < ldk) sg.load(src, row, k2);
  const GroupScale g = warp_scale(sg);
  if (k2 < ldk) sg.template write<S>(g, out + row * ldk + k2, (long long)rows_pad * ldk);
  if (lane == 0) {
    scale[(long long)ch * rows_pad + row] = g.sc;
    if (g.sc != 0.f) mark_chunk(mask, mw, row, ch);
  }
}

__device__ __forceinline__ unsigned long long cplx_key(cplx z) { return max(abs_key(z.x), abs_key(z.y)); }
__device__ __forceinline__ bool cplx_nonzero(cplx z) {
  return z.x != 0.0 || z.y != 0.0 || !(z.x == z.x) || !(z.y == z.y);
}

// B operands, expanded to the real rows (n, re): (Re, -Im) and (n, im): (Im, Re) over the K index
// (k, re/im), one scale for both rows of a complex row n < N of opB(B)[k][n] (two passes over the
// source: the largest magnitude, then the slices).  Bound: HBM, 16 B read and 2 x 4 S B written per
// entry (the first pass over a row leaves it in L1 or L2).
// Two consecutive entries z of one complex row: 4 BF16 per slice and real row.
template <int S>
__device__ __forceinline__ void store_b(const cplx z[2], const GroupScale& g, __nv_bfloat16* out, long long n, int ldk,
                                        int k2, long long slice) {
  float re[2][S], im[2][S], ni[2][S];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    digits_fp64<S>(z[q].x, g, re[q]);
    digits_fp64<S>(z[q].y, g, im[q]);
    digits_fp64<S>(-z[q].y, g, ni[q]);
  }
  float d[4][S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    d[0][s] = re[0][s];
    d[1][s] = ni[0][s];
    d[2][s] = re[1][s];
    d[3][s] = ni[1][s];
  }
  store_slices<S>(d, out + 2 * n * ldk + k2, slice);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    d[0][s] = im[0][s];
    d[1][s] = re[0][s];
    d[2][s] = im[1][s];
    d[3][s] = re[1][s];
  }
  store_slices<S>(d, out + (2 * n + 1) * ldk + k2, slice);
}

// entry (n, k) at p[n * ld + k]: one block per complex row.  chi = 1024, w = 14 (235 MB): 436 -> 197 us
// against one block per real row (each complex row read four times).
template <int S>
__global__ void __launch_bounds__(128)
    k_slice_b_k(const cplx* __restrict__ p, long long ld, int N, int K, int conj, int rows_pad, int ldk,
                __nv_bfloat16* __restrict__ out, float* __restrict__ scale, unsigned* __restrict__ mask, int mw) {
  __shared__ unsigned long long red[4];
  const long long n = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool live = n < N;
  const cplx* x = p + (live ? n * ld : 0);
  unsigned long long h = 0;
  if (live)
    for (int k = tid; k < K; k += 128) h = max(h, cplx_key(x[k]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
  if (lane == 0) red[wid] = h;
  __syncthreads();
  const GroupScale g = scale_from_key(max(max(red[0], red[1]), max(red[2], red[3])));
  const long long slice = (long long)rows_pad * ldk;
  for (int base = 64 * wid; 2 * base < ldk; base += 256) {  // a warp covers one chunk: 64 complex entries
    const int k = base + 2 * lane;
    cplx z[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      z[q] = live && k + q < K ? x[k + q] : mkc(0.0, 0.0);
      if (conj) z[q].y = -z[q].y;
    }
    if (2 * k < ldk) store_b<S>(z, g, out, n, ldk, 2 * k, slice);
    if (__any_sync(0xffffffffu, cplx_nonzero(z[0]) || cplx_nonzero(z[1])) && lane == 0)
      mark_chunk(mask, mw, 2 * n, base >> 6);
  }
  if (tid == 0) scale[2 * n] = scale[2 * n + 1] = g.sc;
}

// entry (n, k) at p[k * ld + n]: blocks of 8 complex rows (128-byte reads), turned in shared memory
template <int S>
__global__ void __launch_bounds__(256)
    k_slice_b_r(const cplx* __restrict__ p, long long ld, int N, int K, int conj, int rows_pad, int ldk,
                __nv_bfloat16* __restrict__ out, float* __restrict__ scale, unsigned* __restrict__ mask, int mw) {
  constexpr int TR = 8;
  __shared__ unsigned long long hmax[TR];
  __shared__ cplx t[TR][65];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const long long n0 = (long long)blockIdx.x * TR;
  const int rl = tid % TR, kk = tid / TR;  // 8 rows x 32 k
  if (tid < TR) hmax[tid] = 0;
  __syncthreads();
  unsigned long long h = 0;
  if (n0 + rl < N)
    for (int k = kk; k < K; k += 32) h = max(h, cplx_key(p[(long long)k * ld + n0 + rl]));
  atomicMax(&hmax[rl], h);
  __syncthreads();
  const long long n = n0 + wid;  // warp w turns row w
  const GroupScale g = scale_from_key(hmax[wid]);
  const long long slice = (long long)rows_pad * ldk;
  for (int base = 0; 2 * base < ldk; base += 64) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = base + kk + 32 * q;
      cplx z = n0 + rl < N && k < K ? p[(long long)k * ld + n0 + rl] : mkc(0.0, 0.0);
      if (conj) z.y = -z.y;
      t[rl][kk + 32 * q] = z;
    }
    __syncthreads();
    const int k = base + 2 * lane;
    const cplx z[2] = {t[wid][2 * lane], t[wid][2 * lane + 1]};
    if (2 * k < ldk) store_b<S>(z, g, out, n, ldk, 2 * k, slice);
    if (__any_sync(0xffffffffu, cplx_nonzero(z[0]) || cplx_nonzero(z[1])) && lane == 0)
      mark_chunk(mask, mw, 2 * n, base >> 6);
    __syncthreads();
  }
  if (lane == 0) scale[2 * n] = scale[2 * n + 1] = g.sc;
}

// ---------------------------------------------------------------- host side
inline int pad32(int k) { return (k + 31) / 32 * 32; }
inline int pad128(int k) { return (k + 127) / 128 * 128; }

// A sliced operand: bf16 slices [S][rows_pad][ldk] and scales, per (chunk, row)
// ([nch][rows_pad], A operands) or per row ([rows_pad], B operands).
struct Sliced {
  RawBuf data, scale, mask;
  unsigned* mk = nullptr;  // the mask in use: mask, or a part of a shared buffer
  int rows_pad = 0, ldk = 0, nch = 0, S = 0, mw = 0;
  bool row_scale = false;
  void shape(DevicePool* pool, int S_, int rows, int K2, bool per_row) {
    S = S_;
    row_scale = per_row;
    rows_pad = pad128(std::max(rows, 1));
    ldk = pad32(std::max(K2, 1));
    nch = (ldk + KC - 1) / KC;
    mw = (nch + 31) / 32;
    data.ensure(pool, sizeof(__nv_bfloat16) * (size_t)S * rows_pad * ldk);
    scale.ensure(pool, sizeof(float) * (size_t)(per_row ? 1 : nch) * rows_pad);
    // one bit per (128-row tile, chunk) holding a nonzero entry (exact zeros of conserved charges)
    mask.ensure(pool, mask_words() * sizeof(unsigned));
    mk = mask.as<unsigned>();
  }
  size_t mask_words() const { return (size_t)(rows_pad / 128) * mw; }
};

void clear_mask(cudaStream_t st, Sliced& o) {
  TDVP_CUDA(cudaMemsetAsync(o.mk, 0, sizeof(unsigned) * o.mask_words(), st));
}
// gives two shaped operands masks side by side and clears both at once (a memset is a launch)
void clear_masks(cudaStream_t st, DevicePool* pool, Sliced& a, Sliced& b) {
  const size_t na = a.mask_words(), nb = b.mask_words();
  a.mask.ensure(pool, (na + nb) * sizeof(unsigned));
  a.mk = a.mask.as<unsigned>();
  b.mk = a.mk + na;
  TDVP_CUDA(cudaMemsetAsync(a.mk, 0, (na + nb) * sizeof(unsigned), st));
}

// A operand (its mask cleared before)
template <class Src>
void slice(cudaStream_t st, const Src& src, Sliced& o) {
  tdvp_require(!o.row_scale, TDVP_ERR_INVALID_ARG, "slice: A operands carry chunk scales");
  auto* d = o.data.as<__nv_bfloat16>();
  const int blocks = ceil_div((long long)o.rows_pad * o.nch * 32, 256);
  if (o.S == 4)
    k_slice_chunks<4, Src><<<blocks, 256, 0, st>>>(src, o.rows_pad, o.ldk, o.nch, d, o.scale.as<float>(),
                                                   o.mk, o.mw);
  else
    k_slice_chunks<3, Src><<<blocks, 256, 0, st>>>(src, o.rows_pad, o.ldk, o.nch, d, o.scale.as<float>(),
                                                   o.mk, o.mw);
  TDVP_CHECK_LAUNCH();
}

// B operand from opB(B)[k][n] (B row-major with leading dimension ld; its mask cleared before)
void slice_b(cudaStream_t st, const cplx* B, long long ld, int K, int N, int op, Sliced& o) {
  tdvp_require(o.row_scale, TDVP_ERR_INVALID_ARG, "slice_b: B operands carry row scales");
  auto* d = o.data.as<__nv_bfloat16>();
  float* sc = o.scale.as<float>();
  unsigned* mk = o.mk;
  const bool kcontig = op == OP_T || op == OP_C;
  const int conj = op == OP_C || op == OP_R, rows = o.rows_pad / 2;
  if (kcontig) {
    if (o.S == 4)
      k_slice_b_k<4><<<rows, 128, 0, st>>>(B, ld, N, K, conj, o.rows_pad, o.ldk, d, sc, mk, o.mw);
    else
      k_slice_b_k<3><<<rows, 128, 0, st>>>(B, ld, N, K, conj, o.rows_pad, o.ldk, d, sc, mk, o.mw);
  } else {
    if (o.S == 4)
      k_slice_b_r<4><<<rows / 8, 256, 0, st>>>(B, ld, N, K, conj, o.rows_pad, o.ldk, d, sc, mk, o.mw);
    else
      k_slice_b_r<3><<<rows / 8, 256, 0, st>>>(B, ld, N, K, conj, o.rows_pad, o.ldk, d, sc, mk, o.mw);
  }
  TDVP_CHECK_LAUNCH();
}

CUtensorMap make_map3(const Sliced& o, int box_rows) {
  const void* base = o.data.as<void>();
  tdvp_require((reinterpret_cast<uintptr_t>(base) & 15) == 0, TDVP_ERR_INVALID_ARG, "TMA base not 16B aligned");
  tdvp_require(o.ldk % 32 == 0 && o.rows_pad % box_rows == 0, TDVP_ERR_INVALID_ARG, "sliced operand not padded");
  CUtensorMap m;
  std::memset(&m, 0, sizeof(m));
  cuuint64_t dims[3] = {(cuuint64_t)o.ldk, (cuuint64_t)o.rows_pad, (cuuint64_t)o.S};
  cuuint64_t strides[2] = {(cuuint64_t)o.ldk * 2, (cuuint64_t)o.rows_pad * o.ldk * 2};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)o.S};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  tdvp_require(r == CUDA_SUCCESS, TDVP_ERR_CUDA, "cuTensorMapEncodeTiled (bf16) failed: " + std::to_string((int)r));
  return m;
}

template <int S>
void launch_bf16s(cudaStream_t st, const CUtensorMap& ma, const CUtensorMap& mb, int M, int N, int nkb,
                  int kb_split, int splits, const float* sA, long long lsA, const float* sB, void* out,
                  long long ldo, long long split_stride, int out_df, int* d_err, const unsigned* maskA,
                  const unsigned* maskB, int mw) {
  per_device([] {
    // the register hand-over inside the kernel is sized for exactly this launch allocation
    cudaFuncAttributes fa;
    TDVP_CUDA(cudaFuncGetAttributes(&fa, k_gemm_bf16s<S>));
    tdvp_require(fa.numRegs == REGS_LAUNCH, TDVP_ERR_CUDA,
                 "gemm_bf16s: kernel built with " + std::to_string(fa.numRegs) + " registers, expected " +
                     std::to_string(REGS_LAUNCH));
    TDVP_CUDA(cudaFuncSetAttribute(k_gemm_bf16s<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   SCfg<S>::SMEM_BYTES));
    return true;
  });
  dim3 grid(ceil_div(N, BN), ceil_div(M, BM), splits);
  tdvp_require(grid.y <= 65535 && splits <= 65535, TDVP_ERR_INVALID_ARG, "gemm_bf16s: grid too large");
  k_gemm_bf16s<S><<<grid, THREADS, SCfg<S>::SMEM_BYTES, st>>>(ma, mb, M, N, nkb, kb_split, sA, lsA, sB, out, ldo,
                                                              split_stride, out_df, splits > 1 ? 1 : 0, d_err, maskA, maskB,
                                                              mw);
  TDVP_CHECK_LAUNCH();
}

// Sum of the split-K partials (double-float pairs, one [M][N] slab per split of `cps` chunks) into
// the output: FP64, or double-float pairs when out_df.  One block per row and 256 columns (N even).
// Bound: FP64 (2 operations per cycle and SM against 8 bytes per partial) and, for the short sums,
// latency.  So a warp first reads off the masks which splits of its tile hold a chunk (the GEMM has
// not written the others: zeros of other charge sectors), loads those all at once, skips partials
// that are zero in the whole warp, and joins hi and lo by integer operations: one FP64 addition per
// nonzero partial after the first where there were 4 operations for every one.  The order of the
// splits is kept.
// Average over a sweep at bond dimension 256: 37 -> 13 us (the partials themselves are 58 MB there).
__global__ void __launch_bounds__(128) k_splitk_df(const float2* __restrict__ ws, int splits, int cps, int nchunks,
                                                   int M, int N, void* __restrict__ out, long long ldo, int out_df,
                                                   const unsigned* __restrict__ maskA,
                                                   const unsigned* __restrict__ maskB, int mwords) {
  constexpr int U = 4;  // splits in flight per thread, two columns each
  const int m = blockIdx.y, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * 256 + 2 * (threadIdx.x & ~31), n = n0 + 2 * lane;
  if (n0 >= N) return;  // warp-uniform; N is even
  const long long per = (long long)M * N, e = (long long)m * N + n;
  const bool in = n < N;
  unsigned todo;  // splits with a chunk (at most 32); a warp's 64 columns lie in one 128-column tile
  {
    const unsigned* a = maskA + (long long)(m >> 7) * mwords;
    const unsigned* b = maskB + (long long)(n0 >> 7) * mwords;
    unsigned on = 0;
    if (lane < splits) {
      const int lo = lane * cps, hi = min(nchunks, lo + cps) - 1;  // first and last chunk
      for (int w = lo >> 5; w <= hi >> 5; ++w) {
        unsigned x = a[w] & b[w];
        if (w == lo >> 5) x &= ~0u << (lo & 31);
        if (w == hi >> 5) x &= ~0u >> (31 - (hi & 31));
        on |= x;
      }
    }
    todo = __ballot_sync(0xffffffffu, on != 0u);
  }
  double s0 = 0.0, s1 = 0.0;
  bool first = true;  // no partial added yet (warp-uniform)
  while (todo) {
    float4 v[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const int z = __ffs(todo) - 1;  // -1: none left
      todo &= todo - 1;
      v[q] = in && z >= 0 ? *reinterpret_cast<const float4*>(ws + z * per + e) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const unsigned bits = __float_as_uint(v[q].x) | __float_as_uint(v[q].y) | __float_as_uint(v[q].z) |
                            __float_as_uint(v[q].w);
      if (!__any_sync(0xffffffffu, (bits << 1) != 0u)) continue;
      const double t0 = df_to_double(v[q].x, v[q].y), t1 = df_to_double(v[q].z, v[q].w);
      s0 = first ? t0 : s0 + t0;
      s1 = first ? t1 : s1 + t1;
      first = false;
    }
  }
  if (!in) return;
  if (out_df) {
    float2* o = static_cast<float2*>(out) + m * ldo + n;
    o[0] = double_to_df(s0);
    o[1] = double_to_df(s1);
  } else {
    double* o = static_cast<double*>(out) + m * ldo + n;
    o[0] = s0;
    o[1] = s1;
  }
}

// Splits of K (whole 128-deep chunks) that minimise waves of CTAs x work per CTA:
// few output tiles (a narrow product or a long K) would otherwise leave most SMs idle.
int choose_splits(long long tiles, int nchunks) {
  const int sms = per_device([] {
    int dev = 0, n = 0;
    TDVP_CUDA(cudaGetDevice(&dev));
    TDVP_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    return n > 0 ? n : 148;
  });
  int best = 1;
  double best_t = (double)((tiles + sms - 1) / sms);
  for (int sp = 2; sp <= std::min(32, nchunks); ++sp) {
    const int cps = (nchunks + sp - 1) / sp;
    const int real = (nchunks + cps - 1) / cps;
    const double t = (double)((tiles * real + sms - 1) / sms) * cps / nchunks + 0.02;  // + reduction pass
    if (t < 0.9 * best_t) {
      best_t = t;
      best = real;
    }
  }
  return best;
}

// out[M x N] (row-major, ldo) = A B^T over the sliced real operands; FP64 entries, or
// double-float (hi, lo) FP32 pairs when out_df.  Products with few output tiles split
// K over more CTAs (partials in a pool workspace, summed by k_splitk_df).
void gemm_bf16s(cudaStream_t st, DevicePool* pool, const Sliced& A, const Sliced& B, int M, int N, void* out,
                long long ldo, bool out_df, int* d_err) {
  if (M <= 0 || N <= 0) return;
  tdvp_require(A.ldk == B.ldk && A.S == B.S, TDVP_ERR_INVALID_ARG, "gemm_bf16s: operand K or slices differ");
  tdvp_require(M <= A.rows_pad && N <= B.rows_pad, TDVP_ERR_INVALID_ARG, "gemm_bf16s: operand rows");
  tdvp_require(!A.row_scale && B.row_scale, TDVP_ERR_INVALID_ARG, "gemm_bf16s: operand scaling groups");
  const CUtensorMap ma = make_map3(A, BM), mb = make_map3(B, BN);
  const int nkb = A.ldk / BK;
  const int nchunks = (nkb + KC_KB - 1) / KC_KB;
  const long long tiles = (long long)ceil_div(N, BN) * ceil_div(M, BM);
  const int splits = pool && M <= 65535 ? choose_splits(tiles, nchunks) : 1;  // at most 32
  const int kb_split = splits > 1 ? ((nchunks + splits - 1) / splits) * KC_KB : nkb;
  RawBuf ws;
  void* dst = out;
  long long ld = ldo, stride = 0;
  int df = out_df ? 1 : 0;
  if (splits > 1) {
    ws.ensure(pool, sizeof(float2) * (size_t)splits * M * N);
    dst = ws.as<void>();
    ld = N;
    stride = (long long)M * N;
    df = 1;
  }
  tdvp_require(A.mw == B.mw && (kb_split + KC_KB - 1) / KC_KB <= kMaxChunks, TDVP_ERR_INVALID_ARG,
               "gemm_bf16s: chunk masks or chunks per split out of range");
  const unsigned* mA = A.mk;
  const unsigned* mB = B.mk;
  if (A.S == 4)
    launch_bf16s<4>(st, ma, mb, M, N, nkb, kb_split, splits, A.scale.as<float>(), A.rows_pad, B.scale.as<float>(),
                    dst, ld, stride, df, d_err, mA, mB, A.mw);
  else
    launch_bf16s<3>(st, ma, mb, M, N, nkb, kb_split, splits, A.scale.as<float>(), A.rows_pad, B.scale.as<float>(),
                    dst, ld, stride, df, d_err, mA, mB, A.mw);
  if (splits > 1) {
    k_splitk_df<<<dim3(ceil_div(N, 256), M), 128, 0, st>>>(ws.as<float2>(), splits, kb_split / KC_KB, nchunks, M, N, out,
                                                          ldo, out_df ? 1 : 0, mA, mB, A.mw);
    TDVP_CHECK_LAUNCH();
  }
}
}  // namespace tcb

using namespace tcb;

struct TcSliceCache {
  long long key = -1;
  int S = 0;
  Sliced L, R, X, T2;
  RawBuf T1;
};

namespace {
TcSliceCache& slice_cache(Scratch& s) {
  if (!s.tcs) s.tcs = std::make_shared<TcSliceCache>();
  return *s.tcs;
}
}  // namespace

int* tc_error_word(cudaStream_t st, Scratch& s) {
  TcEnvCache& c = s.tc;
  if (c.err.bytes() == 0) {
    c.err.ensure(s.pool, sizeof(int));
    TDVP_CUDA(cudaMemsetAsync(c.err.as<int>(), 0, sizeof(int), st));
  }
  c.pending = true;
  return c.err.as<int>();
}

int bf16_slices(int precision) { return precision == TDVP_PREC_BF16X6 ? 3 : 4; }

void gemm_chunk_pairs(long long out[2]) {
  unsigned long long h[2] = {0, 0};
  TDVP_CUDA(cudaMemcpyFromSymbol(h, tcb::g_chunk_pairs, sizeof(h)));
  out[0] = (long long)h[0];
  out[1] = (long long)h[1];
}

void heff_bf16s(cudaStream_t st, Scratch& s, const SiteOp& op, const cplx* x, cplx* y, int S) {
  const int ml = op.ml, mr = op.mr, wl = op.wl, wr = op.wr, d = op.d;
  TcSliceCache& c = slice_cache(s);
  DevicePool* pool = s.pool;
  int* err = tc_error_word(st, s);
  if (op.env_key < 0 || c.key != op.env_key || c.S != S) {
    // L as the A operand: rows (w, a), K = (a', re/im)
    c.L.shape(pool, S, ml * wl, 2 * ml, false);
    c.R.shape(pool, S, 2 * mr, 2 * wr * mr, true);
    clear_mask(st, c.L);
    clear_mask(st, c.R);
    slice(st, SrcLwa{op.L, ml, wl}, c.L);
    // R[b][(v,b')] is B[k=(v,b')][n=b] stored n-major (op T)
    slice_b(st, op.R, (long long)wr * mr, wr * mr, mr, OP_T, c.R);
    c.key = op.env_key;
    c.S = S;
  }
  // stage 1: T1[(w,a)][(s',b',c)] = L x     (x[a'][(s',b')] is B[k=a'][n=(s',b')])
  c.X.shape(pool, S, 2 * d * mr, 2 * ml, true);
  c.T2.shape(pool, S, ml * d, 2 * wr * mr, false);
  clear_masks(st, pool, c.X, c.T2);
  slice_b(st, x, (long long)d * mr, ml, d * mr, OP_N, c.X);
  const int M1 = ml * wl, N1 = 2 * d * mr;
  c.T1.ensure(pool, sizeof(float2) * (size_t)M1 * N1);  // double-float
  gemm_bf16s(st, pool, c.L, c.X, M1, N1, c.T1.as<void>(), N1, true, err);
  // stage 2: MPO tensor, sliced straight into the stage-3 A operand
  const WSparse& ws = *op.W;
  tdvp_require(ws.d_l_val_df != nullptr, TDVP_ERR_INVALID_ARG, "heff_bf16s: MPO site without double-float values");
  slice(st, SrcStage2{c.T1.as<float4>(), ws.d_l_off, ws.d_l_idx, ws.d_l_val_df, ml, wl, wr, d, mr}, c.T2);
  // stage 3: y[(a,s)][(b,c)] = T2 R^T
  gemm_bf16s(st, pool, c.T2, c.R, ml * d, 2 * mr, y, 2 * mr, false, err);
}

void zgemm_bf16s(cudaStream_t st, Scratch& s, int S, int opA, int opB, int M, int N, int K, const cplx* A,
                 long long lda, const cplx* B, long long ldb, cplx* C, long long ldc) {
  if (M <= 0 || N <= 0) return;
  DevicePool* pool = s.pool;
  int* err = tc_error_word(st, s);
  Sliced a, b;
  a.shape(pool, S, M, 2 * std::max(K, 1), false);
  b.shape(pool, S, 2 * N, 2 * std::max(K, 1), true);
  clear_masks(st, pool, a, b);
  slice(st, SrcA{A, lda, M, K, opA}, a);
  slice_b(st, B, ldb, K, N, opB, b);
  gemm_bf16s(st, pool, a, b, M, 2 * N, C, 2 * ldc, false, err);
}
