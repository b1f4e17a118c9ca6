// FP64 matrix products on the tensor cores by error-free splitting (Ozaki, Ogita, Oishi, Rump,
// Numer. Algorithms 59, 95 (2012); on fp16 tensor cores: Mukunoki, Ozaki, Ogita, Imamura, ISC 2020).
//
// GB300's FP64 pipes run at ~1 TFLOP/s, its fp16 tensor cores at ~1900. Every operand row is scaled
// by a power of two to |x| < 1 and written as a 56-bit fixed-point number of seven balanced 8-bit
// digits, x = 2^e sum_i d_i 2^(-7 - 8 i), |d_i| <= 128, each digit an exact fp16 value. A product of
// two rows is then sum_s 2^(-14 - 8 s) L_s with L_s = sum_k sum_(i + j = s) a_i b_j, an integer. The
// levels s = 0 .. 6 (28 digit products) are formed on the tensor cores, one FP32 accumulator in
// tensor memory per level, over blocks of 192 k: |L_s| <= (s + 1) 192 2^14 < 2^24 for s <= 4, so the
// FP32 sums are exact there (at s = 5, 6 an extreme coherent row could round, by 2^-54 of the sum of
// |a b|). The blocks' levels are added up in 64-bit integers and become one double per element at
// the end. What is lost is the rounding of each operand to 2^-56 of its row's scale 2^e (2^(e-1) <= max|x| < 2^e)
// and the levels above 6: per term at most (2 + 6.03) 2^-56 2^(ea + eb), below 2^-50 max|a| max|b|; about 2^-56
// 2^(ea + eb) in the root mean square. That is below the rounding errors of an FP64 accumulation for rows
// whose entries are of one scale (measured errors of P and Sigma^c against exact sums on such data are below the
// CUDA-core kernels'), but it is relative to the rows' largest entries: a = [1, 2^-60], b = [2^-60, 1] gives 0, where
// FP64 gives 2^-59. GW_TUNE_FP64_FORM 1 takes the CUDA-core kernels, whose error is relative to each term.
// Rows that hold an infinity or a nan give nan.
//
// Short sums leave FP64 fewer roundings to make: of the digits' loss most is the first level left out (six products,
// 2^-56 of the rows' largest values, in the root mean square), so such a GEMM keeps eight levels (34
// products) and every bit of its integer sums.
//
// Tile 128 x 64: the seven levels of 64 columns take 448 of the 512 TMEM columns. A 128 x 64 x 16 MMA
// takes 48 clocks (its operands' 6 KB at 128 bytes per clock of shared memory; 32 of arithmetic), so
// the bound is 28 x 48 clocks per chunk of 16 k and SM; the levels' readout overlaps the next block's
// MMAs level by level (67 clocks per MMA with it, in the polarization of Nk 27, Nb 32, NI 128).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "gw_internal.h"
#include "tc_common.cuh"

namespace gwi {
namespace {

using namespace tc;

constexpr int XS_N = 7;                       // digits per operand
constexpr int XK = 16;                        // K values per chunk: one MMA step
constexpr int XL_MAX = 8;                     // levels a GEMM may keep (OP::LV: 7 or 8)
constexpr int X_BLK = 12;                     // chunks per accumulation block (192 k)
constexpr int XN = 64;                        // output columns per tile: 8 levels x 64 = 512 TMEM columns at most
constexpr int XA_SL = 128 * 32, XB_SL = XN * 32;  // bytes of one digit of an operand chunk
constexpr int XA_BYTES = XS_N * XA_SL, XB_BYTES = XS_N * XB_SL;
constexpr int XST_BYTES = XA_BYTES + XB_BYTES;    // 42 KB per stage
constexpr int X_ST = 5;                       // stages: a chunk's copy has four chunks' MMAs to land in
constexpr int X_EPI = 16;                     // epilogue warps: 4 per TMEM lane quadrant, 16 columns each
constexpr int X_THREADS = (X_EPI + 2) * 32;
constexpr int kBadExp = 1 << 20;              // row exponent of a row that is not finite

// ------------------------------------------------------------------ fixed point and digits
// |x| in units of 2^e, as a float that is not smaller (x finite, |x| < 2^(e + 126)); 0 for x = 0.
__device__ __forceinline__ float norm_up(double x, int e) {
  const uint32_t hi = (uint32_t)(__double_as_longlong(x) >> 32) & 0x7FFFFFFFu;
  if ((hi | (uint32_t)__double_as_longlong(x)) == 0) return 0.f;
  const int ef = (int)(hi >> 20);
  if (ef == 0) return __uint_as_float(1u << 23);
  const int k = ef - 1023 - e;
  if (k < -125) return __uint_as_float(1u << 23);
  return __uint_as_float((((uint32_t)(k + 127) << 23) | ((hi & 0xFFFFFu) << 3)) + 8u);
}
// smallest e with |x| < 2^e for every x whose |high word| is at most h
__device__ __forceinline__ int exp_of(uint32_t h) { return h >= 0x7FF00000u ? kBadExp : (int)(h >> 20) - 1022; }

// rint(x 2^(55 - e)), |x| < 2^e: a 56-bit integer (0 for a row that is not finite)
__device__ __forceinline__ long long to_fix(double x, int e) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int ef = (int)(b >> 52) & 2047;
  const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull);
  const int sh = (ef ? ef : 1) - 1020 - e;
  uint64_t t;
  if (sh >= 0)
    t = sh < 3 ? m << sh : 0;
  else
    t = sh > -55 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0;
  return (long long)b < 0 ? -(long long)t : (long long)t;
}

// sign, exponent field and left-justified 64-bit mantissa (0 for zero) of a double
struct Fl64 {
  uint64_t m;
  int e;  // |x| = m 2^(e - 1086)
};
__device__ __forceinline__ Fl64 fl64(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int ef = (int)(b >> 52) & 2047;
  Fl64 r;
  r.m = ((b & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull)) << 11;
  r.e = ef ? ef : 1;
  return r;
}
// rint(|x| |w| 2^(55 - e)), |x w| < 2^e (0 where the shift leaves the word: a row that is not finite)
__device__ __forceinline__ uint64_t mul_fix(const Fl64& x, const Fl64& w, int e) {
  const uint64_t h = __umul64hi(x.m, w.m);  // |x w| = h 2^(xe + we - 2108)
  const int sr = 2053 - x.e - w.e + e;
  return sr >= 1 && sr < 64 ? (h >> sr) + ((h >> (sr - 1)) & 1) : 0;
}

// the digits of 8 values as 16 bytes of fp16 per slice: the six lower digits are the bytes of the
// biased integer minus 128 (0x6400 | byte is the half 1024 + byte)
__device__ __forceinline__ void digits8(const long long (&t)[8], uint4 (&out)[XS_N]) {
  uint32_t w[XS_N][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint64_t u0 = (uint64_t)(t[2 * q] + 0x0000808080808080ll), u1 = (uint64_t)(t[2 * q + 1] + 0x0000808080808080ll);
    const uint32_t l0 = (uint32_t)u0, l1 = (uint32_t)u1, h0 = (uint32_t)(u0 >> 32), h1 = (uint32_t)(u1 >> 32);
    const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
    auto put = [&](int s, uint32_t r) {
      const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&r), bias);
      w[s][q] = *reinterpret_cast<const uint32_t*>(&d);
    };
#pragma unroll
    for (int j = 0; j < 4; ++j)
      put(6 - j, (__byte_perm(l0, l1, j | ((4 + j) << 8)) & 0x00FF00FFu) | 0x64006400u);
#pragma unroll
    for (int j = 0; j < 2; ++j)
      put(2 - j, (__byte_perm(h0, h1, j | ((4 + j) << 8)) & 0x00FF00FFu) | 0x64006400u);
    const uint32_t t0 = (uint32_t)(((int)h0 >> 16) + 128), t1 = (uint32_t)(((int)h1 >> 16) + 128);
    put(0, (t0 | (t1 << 16)) + 0x64006400u);
  }
#pragma unroll
  for (int s = 0; s < XS_N; ++s) out[s] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// 8 consecutive K values (k8 = 0, 1 of the chunk) of one row of an operand chunk [digit][k8][rows][16 B]
template <int ROWS>
__device__ __forceinline__ void put8(unsigned char* chunk, int row, int k8, const long long (&t)[8]) {
  uint4 d[XS_N];
  digits8(t, d);
  unsigned char* o = chunk + (k8 * ROWS + row) * 16;
#pragma unroll
  for (int s = 0; s < XS_N; ++s) *reinterpret_cast<uint4*>(o + s * ROWS * 32) = d[s];
}

__device__ __forceinline__ uint32_t abs_hi(double x) {
  return (uint32_t)(__double_as_longlong(x) >> 32) & 0x7FFFFFFFu;
}
__device__ __forceinline__ uint32_t warp_max(uint32_t v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// y 2^e rounded to nearest even, on the integer pipes (a conversion from 64-bit integers and a
// product would take two slots of the FP64 pipe, which two such slots per element already fill);
// nan when a row of the element is not finite
__device__ __forceinline__ double fix_to_double(long long y, int e) {
  if (e > kBadExp / 2) return __longlong_as_double(0x7FF8000000000000ll);
  if (y == 0) return 0.0;
  const uint64_t a = y < 0 ? 0ull - (uint64_t)y : (uint64_t)y;
  const int lz = __clzll((long long)a), ex = 1023 + 63 - lz + e;
  if (ex < 1 || ex > 2045) return scalbn((double)y, e);
  const uint64_t m = a << lz, r = m >> 11, rest = m & 2047;
  const uint64_t up = rest > 1024 || (rest == 1024 && (r & 1)) ? 1 : 0;
  const uint64_t b = ((uint64_t)(ex - 1) << 52) + r + up;  // r carries the implicit bit
  return __longlong_as_double((long long)(b | ((uint64_t)y & 0x8000000000000000ull)));
}

// (hi 2^32 + lo) 2^e with all of the sum's leading bits (|lo| < 2^61), where a fixed number of dropped bits, which
// has to cover the largest sum that K allows, would cost a short or cancelling one its last bits
__device__ __forceinline__ double fix_to_double(long long hi, long long lo, int e) {
  const int s = max(0, 34 - __clzll(hi ^ (hi >> 63)));
  return fix_to_double((hi << (32 - s)) + (lo >> s), e + s);
}

// ------------------------------------------------------------------ the digit GEMM
struct XSmem {
  uint64_t full[X_ST], empty[X_ST], done, lvl[XL_MAX], fin, never;
  uint32_t tslot;
  int abort_flag, no_dealloc;
  double red[3][128];
};

// The GEMM C = A B^T of digit images, one persistent kernel; what a unit is and what becomes of its tiles
// is an OP class:
//   OP::Job  kernel parameters (with sh, the bits of the 96-bit sums dropped at the end: drop_bits)
//   OP::LV   levels kept: 7, or 8 with tile(J, U, n, hi, lo), the elements being (hi 2^32 + lo) 2^(ea + eb - 62)
//   OP::Unit (J, u): n0, n1 (the tiles n of the unit, one after another), A(J, n), B(J, n) (operand images,
//            chunks XA_BYTES / XB_BYTES apart), range(J, n, c0, c1) (the chunks of tile n)
//   OP(J, U, r, part): the epilogue thread of row r (0 .. 127) and columns 16 part .. + 15 of the unit's tiles;
//   tile(J, U, n, y): y[16] = the thread's elements, in units of 2^(ea + eb - 62 + sh);
//   finish(J, U, red, ok): after the unit's last tile (all 512 threads; red: 3 x 128 doubles; ok false: no
//            tile may be used, a wait ran out).
template <class OP>
__global__ void __launch_bounds__(X_THREADS, 1)
    k_digit_gemm(const __grid_constant__ typename OP::Job J, int nunits, int* __restrict__ err, long long wait_cycles, int stall) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  XSmem& S = *reinterpret_cast<XSmem*>(base + X_ST * XST_BYTES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < X_ST; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], 1);
    }
    mbar_init(&S.done, 1);
    for (int s = 0; s < OP::LV; ++s) mbar_init(&S.lvl[s], X_EPI);
    mbar_init(&S.fin, 1);
    mbar_init(&S.never, 1);
    S.abort_flag = 0;
    S.no_dealloc = 0;
    fence_mbar_init();
  }
  if (warp == X_EPI + 1) tmem_alloc(&S.tslot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = S.tslot;

  if (warp == X_EPI) {
    // ------------------------------------------------------------ producer: one bulk copy per operand and chunk
    if (lane == 0) {
      int i = 0;  // running chunk: stage i % X_ST, its phase i / X_ST
      bool live = true;
      for (int u = blockIdx.x; u < nunits && live; u += gridDim.x) {
        const typename OP::Unit U(J, u);
        for (int n = U.n0; n < U.n1 && live; ++n) {
          int c0, c1;
          U.range(J, n, c0, c1);
          const unsigned char *a = U.A(J, n), *b = U.B(J, n);
          for (int c = c0; c < c1; ++c, ++i) {
            const int s = i % X_ST;
            if (S.abort_flag ||
                (i >= X_ST && !wait_bar(&S.empty[s], (i / X_ST + 1) & 1, &S.abort_flag, err, wait_cycles))) {
              live = false;
              break;
            }
            unsigned char* st = base + s * XST_BYTES;
            mbar_arrive_expect_tx(&S.full[s], XST_BYTES);
            bulk_g2s(st, a + (size_t)c * XA_BYTES, XA_BYTES, &S.full[s]);
            bulk_g2s(st + XA_BYTES, b + (size_t)c * XB_BYTES, XB_BYTES, &S.full[s]);
          }
        }
      }
      // the copies of every issued chunk land before the block exits
      for (int j = i > X_ST ? i - X_ST : 0; j < i; ++j)
        if (!drain_bar(&S.full[j % X_ST], (j / X_ST) & 1)) S.no_dealloc = 1;
    }
    __syncwarp();  // the warp meets the block barrier converged
  } else if (warp == X_EPI + 1) {
    // ------------------------------------------------------------ MMA issuer: the warp stays converged
    const uint32_t id = idesc_f16(128, XN, false, false), lead = elect_one();
    const uint32_t dh = (uint32_t)(sdesc_none(0, 0) >> 32);
    const uint32_t a0 = (uint32_t)sdesc_none(smem_u32(base), 128 * 16);
    const uint32_t b0 = (uint32_t)sdesc_none(smem_u32(base) + XA_BYTES, XN * 16);
    int s = 0, ph = 0, blk = 0;  // stage and its phase of the running chunk
    bool live = true;
    if (stall && lead) wait_bar(&S.never, 0, &S.abort_flag, err, wait_cycles);  // injected stall: runs out
    __syncwarp();
    for (int u = blockIdx.x; u < nunits && live; u += gridDim.x) {
      const typename OP::Unit U(J, u);
      for (int n = U.n0; n < U.n1 && live; ++n) {
        int c0, c1;
        U.range(J, n, c0, c1);
        for (int cb = c0; cb < c1 && live; cb += X_BLK, ++blk) {
          const int ce = min(cb + X_BLK, c1);
          for (int c = cb; c < ce; ++c) {
            live = __all_sync(0xffffffffu, wait_bar(&S.full[s], ph, &S.abort_flag, err, wait_cycles));
            if (!live) break;
            tc_fence_after();
            const uint32_t a = a0 + s * (XST_BYTES >> 4), b = b0 + s * (XST_BYTES >> 4);
            if (c == cb) {
#pragma unroll
              for (int l = 0; l < OP::LV; ++l) {
                // the previous block's level l has been read (its first MMA overwrites it)
                if (blk > 0) {
                  live = live && __all_sync(0xffffffffu, wait_bar(&S.lvl[l], (blk - 1) & 1, &S.abort_flag, err, wait_cycles));
                  tc_fence_after();
                }
                if (lead) {
#pragma unroll
                  for (int x = l < XS_N ? 0 : l - XS_N + 1; x <= l && x < XS_N; ++x)
                    mma_f16_lo(tbase + XN * l, a + x * (XA_SL >> 4), b + (l - x) * (XB_SL >> 4), dh, id,
                               x > (l < XS_N ? 0 : l - XS_N + 1));
                }
                __syncwarp();
              }
            } else {
              if (lead) {
#pragma unroll
                for (int l = 0; l < OP::LV; ++l)
#pragma unroll
                  for (int x = l < XS_N ? 0 : l - XS_N + 1; x <= l && x < XS_N; ++x)
                    mma_f16_lo(tbase + XN * l, a + x * (XA_SL >> 4), b + (l - x) * (XB_SL >> 4), dh, id, 1);
              }
            }
            if (lead) mma_commit(&S.empty[s]);
            __syncwarp();
            if (++s == X_ST) {
              s = 0;
              ph ^= 1;
            }
            if (!live) break;
          }
          if (live && lead) mma_commit(&S.done);
          __syncwarp();
        }
      }
    }
    if (lead) mma_commit(&S.fin);
    __syncwarp();
    if (!drain_bar(&S.fin, 0)) S.no_dealloc = 1;  // every MMA issued here has completed
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue: 16 warps, 16 columns each
    const int quad = warp & 3, part = warp >> 2;
    const int r = 32 * quad + lane;
    const uint32_t tw = tbase + ((uint32_t)(32 * quad) << 16) + 16 * part;
    int blk = 0;
    bool ok = true;  // uniform over the warp; a warp that gave up still takes part in the block barriers below
    for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
      const typename OP::Unit U(J, u);
      OP op(J, U, r, part);
      for (int n = U.n0; n < U.n1 && ok; ++n) {
        int c0, c1;
        U.range(J, n, c0, c1);
        long long hi[16], lo[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) hi[e] = lo[e] = 0;
        for (int cb = c0; cb < c1 && ok; cb += X_BLK, ++blk) {
          ok = __all_sync(0xffffffffu, wait_bar(&S.done, blk & 1, &S.abort_flag, err, wait_cycles));
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int l = 0; l < OP::LV; ++l) {
            constexpr int kShift[XL_MAX] = {16, 8, 0, 24, 16, 8, 0, 0};
            float v[16];
            tmem_ld16(tw + XN * l, v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.lvl[l]);  // the next block may overwrite this level
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const long long t = (long long)__float2int_rn(l < XS_N ? v[e] : v[e] * 0.00390625f) * (1 << kShift[l]);
              if (l < 3) hi[e] += t; else lo[e] += t;
            }
          }
        }
        if (!ok) break;
        // element = (hi 2^32 + lo) 2^(ea + eb - 62) = y 2^(ea + eb - 62 + sh), |y| < 2^63
        if constexpr (OP::LV == XL_MAX) {
          op.tile(J, U, n, hi, lo);
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) hi[e] = (hi[e] << (32 - J.sh)) + (lo[e] >> J.sh);
          op.tile(J, U, n, hi);
        }
      }
      op.finish(J, U, S.red, ok);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == X_EPI + 1 && !S.no_dealloc) tmem_dealloc(tbase, 512);
}


// Host side: the context's digit workspaces, one for each use, grown on use (grow_ws: a captured call keeps
// the one it was captured with). False (nothing launched, no error set) when it cannot be had: no memory, or a
// capture in progress, where nothing may be allocated; the callers then run kernels that need none.
inline bool x_workspace(gw_ctx* c, int use, size_t need) {
  if (need > c->x_ws_bytes[use] && capturing(c)) return false;
  return grow_ws(c, &c->x_ws[use], &c->x_ws_bytes[use], need);
}
enum { XW_POL = 0, XW_SIGMA = 1, XW_BOSE = 2, XW_SCREEN = 3, XW_OFFDIAG = 4 };

// the sum of K products is below K 2^14 2^48 (1 + 2^-7): bits to drop so that it fits 63 bits
inline int drop_bits(int64_t k) {
  int b = 1;
  while ((1ll << (b - 1)) < k) ++b;
  return b;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// persistent over the SMs: unit u runs in block u mod grid
template <class OP>
gw_status run_gemm(gw_ctx* c, const typename OP::Job& J, int nunits, const char* what) {
  const size_t smem = 1024 + X_ST * XST_BYTES + sizeof(XSmem);
  cudaFuncSetAttribute(k_digit_gemm<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int sms = num_sms(c);
  k_digit_gemm<OP><<<nunits < sms ? nunits : sms, X_THREADS, smem, c->stream>>>(J, nunits, c->d_err, c->wait_cycles,
                                                                                c->fault_stall);
  return check_launch(c, what);
}

}  // namespace
}  // namespace gwi
