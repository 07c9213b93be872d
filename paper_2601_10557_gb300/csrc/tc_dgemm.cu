// FP64-accurate sliced GEMM on tcgen05 tensor cores (see tc_dgemm.cuh).
//
// Kernel (persistent CTAs of 384 threads, each working through 128 x 32 output tiles, or K
// splits of them; the ring and the two accumulator buffers run on from one tile to the next):
//   warp 0    TMA producer: per 32-long K block, all 7 digit planes of the A tile
//             (one 3-D box of 32 x 128 x 7) and of the B tile (32 x 32 x 7), 64-byte
//             swizzle, into a 3-stage ring (70 KB per stage)
//   warp 1    allocates 512 TMEM columns; one lane issues, per 16-long K step and
//             A digit t, one MMA against the B digits u = 0 .. 6 - t stacked along N
//             (N = (7 - t) * 32), accumulating into the TMEM columns of the weight
//             groups w = t + u = t .. 6; two buffers of 7 x 32 columns alternate
//             every 128 K
//   warps 4-11 drain each finished buffer (warps 4-7 columns 0-15, warps 8-11
//             columns 16-31 of every group): the exact integer group sums of
//             weights 2^0 .. 2^-24 into one 64-bit integer per output, those of
//             2^-32 .. 2^-48 into a second one; at the end they round their exact sum
//             to FP64, apply the row and column exponents and write the result with
//             arbitrary strides, while the next tile's MMAs run (with a K split: both
//             integers to a partial tile, and a second kernel sums the splits)
// Bound: shared memory.  A K step of 16 reads 56 KB of operand digits in 448 MMA cycles
// (128 bytes a cycle) while the ring takes in 78 bytes a cycle.  Measured on one GB300,
// before (one CTA per tile, int64 partial tiles of every product) and after: the two
// products of the gradient at n = 8192 (16384 x 8192, K = 400) 11.7 -> 6.35 ms, 3.67 ms
// with only the lower triangle computed; the FP64_TC
// filter of 130 vectors at n = 2048 (24 products 4096 x 260, K = 4096, their slices and the
// recurrence) 8.1 -> 5.1 ms.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "tc_common.cuh"
#include "solver.cuh"
#include "tc_dgemm.cuh"

namespace cb {
namespace tcd {

using namespace cb::tc;

constexpr int S = SLICES;
constexpr int BM = 128, BNS = 32, BK = 32;
constexpr int A_SLICE = BM * BK * 2;                    // 8 KB
constexpr int B_SLICE = BNS * BK * 2;                   // 2 KB
constexpr int STAGE_BYTES = S * (A_SLICE + B_SLICE);    // 70 KB
constexpr int ST = 3;
constexpr int CHUNK = 4;                                // K blocks per exact partial sum (128 K)
constexpr int GCOLS = S * BNS;                          // TMEM columns per buffer
constexpr uint32_t TMEM_COLS = 512;
constexpr int THREADS = 384;
constexpr int DRAIN_WARPS = 8;
constexpr int NBAR = 2 * ST + 5;
constexpr int SMEM_BYTES = ST * STAGE_BYTES + 1024 + 256;
static_assert(2 * GCOLS <= (int)TMEM_COLS, "two accumulator buffers must fit in TMEM");
// a weight group holds at most S digit products of |d| <= 128 over CHUNK * BK terms
static_assert((double)S * 16384.0 * CHUNK * BK < 16777216.0, "group sums must stay exact in FP32");

__device__ __forceinline__ uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
// K-major tile with 64-byte rows and 64-byte swizzle: 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;  // 64-byte swizzle
  return d;
}

// Exponent of an operand row with an infinity or a NaN: its products are NaN.
constexpr int EXP_NONFINITE = 1 << 20;

struct Args {
  int num_m, num_n, kb_total, kb_per_split;
  int items;           // tiles x splits
  int n_fast;          // raster: the CTAs of one A tile (1) or of one B tile (0) run together
  int64_t mp;          // rows of a partial tile column (A rows_pad)
  int64_t np;          // columns per split (B rows_pad)
  long long* hi;       // [split][col][row]; NULL: one split, the tiles go to out
  long long* lo;
  const int* ea;       // row and column exponents
  const int* eb;
  int64_t M, N;
  double alpha;
  double* out;
  int64_t rs, cs;
  int neg_odd;
  int sym;             // 1 hermitian, 2 symmetric: only the lower triangle is computed (see sliced_gemm)
  int* err;
};

// (h 2^24 + l) 2^(e - 62) rounded once to FP64 (to nearest, ties to even): the sum and the
// rounding in integers, whose pipe is 32 times as wide as the FP64 one
__device__ __forceinline__ double fold(long long h, long long l, int e) {
  const __int128 sum = ((__int128)h << 24) + l;
  if (sum == 0) return 0.0;
  unsigned __int128 a = sum < 0 ? (unsigned __int128)(-sum) : (unsigned __int128)sum;
  const unsigned long long up = (unsigned long long)(a >> 64);
  const int lz = up ? __clzll((long long)up) : 64 + __clzll((long long)(unsigned long long)a);
  a <<= lz;
  const unsigned long long top = (unsigned long long)(a >> 64), low = (unsigned long long)a;
  unsigned long long m = top >> 11;  // 53 bits, the leading one among them
  const unsigned long long rem = top & 0x7ff;
  m += (rem > 0x400 || (rem == 0x400 && (low != 0 || (m & 1)))) ? 1 : 0;
  // the leading bit weighs 2^(127 - lz); a carry out of m raises the exponent by itself
  const int x = 127 - lz - 48, x1 = x + e - 14;
  const unsigned long long sign = sum < 0 ? 1ull << 63 : 0ull;
  if (x1 > -1022 && x1 < 1023) return __longlong_as_double((long long)(sign | (((unsigned long long)(x1 + 1022) << 52) + m)));
  return ldexp(__longlong_as_double((long long)(sign | (((unsigned long long)(x + 1022) << 52) + m))), e - 14);
}
__device__ __forceinline__ double result(const Args& g, int64_t r, int64_t c, long long h, long long l) {
  const int ea = g.ea[r], eb = g.eb[c];
  double y = max(ea, eb) >= EXP_NONFINITE ? nan("") : fold(h, l, ea + eb);
  if (g.alpha != 1.0) y *= g.alpha;
  return g.neg_odd && (r & 1) ? -y : y;
}
__device__ __forceinline__ void put_out(const Args& g, int64_t r, int64_t c, long long h, long long l) {
  g.out[r * g.rs + c * g.cs] = result(g, r, c, h, l);
}
// The 16 columns from col on of row `row` (lanes: consecutive rows from an even one) of a
// hermitian or symmetric complex result: entries (i, j), i = row / 2 >= j, and their mirrors.  Of
// a lane pair, which holds Re and Im of the same entries, one lane writes the mirrors of the
// first eight columns and one those of the other eight, 128 contiguous bytes each.
template <int NC>
__device__ __forceinline__ void put_sym(const Args& g, int64_t row, int64_t col, const long long* hi,
                                        const long long* lo) {
  const bool rv = row < g.M, odd = row & 1;
  const int64_t i = row >> 1;
  double y[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    y[c] = 0.0;
    if (rv && col + c < g.N && i >= col + c) {
      y[c] = result(g, row, col + c, hi[c], lo[c]);
      g.out[row + (col + c) * g.cs] = y[c];
    }
  }
#pragma unroll
  for (int c = 0; c < NC / 2; ++c) {
    const double got = __shfl_xor_sync(0xffffffffu, odd ? y[c] : y[c + NC / 2], 1);
    const double re = odd ? got : y[c], im = odd ? y[c + NC / 2] : got;
    const int64_t j = col + c + (odd ? NC / 2 : 0);
    if (rv && j < g.N && i > j)
      *reinterpret_cast<double2*>(g.out + i * g.cs + 2 * j) = make_double2(re, g.sym == 1 ? -im : im);
  }
}

__global__ void __launch_bounds__(THREADS, 1)
    sliced_gemm_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
                       const __grid_constant__ Args g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + ST * STAGE_BYTES);
  uint32_t full[ST], empty[ST];
#pragma unroll
  for (int s = 0; s < ST; ++s) {
    full[s] = smem_u32(bars + s);
    empty[s] = smem_u32(bars + ST + s);
  }
  const uint32_t accf[2] = {smem_u32(bars + 2 * ST), smem_u32(bars + 2 * ST + 1)};
  const uint32_t acce[2] = {smem_u32(bars + 2 * ST + 2), smem_u32(bars + 2 * ST + 3)};
  const uint32_t done = smem_u32(bars + 2 * ST + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NBAR);
  volatile int* abort_sh = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* issued_sh = reinterpret_cast<int*>(tmem_slot + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // the CTAs sharing a tile of the larger operand run together, so that it is read
  // from DRAM once and the other operand's tiles come from L2
  auto item = [&](int id, int& mt, int& nt, int& sp, int& kb0, int& nkb) {
    if (g.sym) {  // the 2 mt + 2 column tiles of row tile mt that reach the lower triangle
      mt = (int)((sqrtf(4.0f * (float)id + 1.0f) - 1.0f) * 0.5f);
      while (mt * (mt + 1) > id) --mt;
      while ((mt + 1) * (mt + 2) <= id) ++mt;
      nt = id - mt * (mt + 1);
      sp = kb0 = 0;
      nkb = g.kb_total;
      return;
    }
    mt = g.n_fast ? (id / g.num_n) % g.num_m : id % g.num_m;
    nt = g.n_fast ? id % g.num_n : (id / g.num_m) % g.num_n;
    sp = id / (g.num_m * g.num_n);
    kb0 = sp * g.kb_per_split;
    nkb = min(g.kb_per_split, g.kb_total - kb0);
  };
  int mt, nt, sp, kb0, nkb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full[s], 1);
      mbar_init(empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf[b], 1);
      mbar_init(acce[b], DRAIN_WARPS);
    }
    mbar_init(done, 1);
    *abort_sh = 0;
    *issued_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sbase = smem_u32(smem);

  if (warp == 0 && lane == 0) {
    int issued = 0, s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int id = blockIdx.x; ok && id < g.items; id += gridDim.x) {
      item(id, mt, nt, sp, kb0, nkb);
      for (int kb = 0; kb < nkb; ++kb) {
        if (issued >= ST && !mbar_wait(empty[0] + 8 * s, ph ^ 1u, abort_sh, g.err, true)) {
          ok = false;
          break;
        }
        const uint32_t st = sbase + s * STAGE_BYTES;
        mbar_expect_tx(full[0] + 8 * s, STAGE_BYTES);
        tma_load_3d(st, &ma, (kb0 + kb) * BK, mt * BM, 0, full[0] + 8 * s);
        tma_load_3d(st + S * A_SLICE, &mb, (kb0 + kb) * BK, nt * BNS, 0, full[0] + 8 * s);
        ++issued;
        if (++s == ST) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    *issued_sh = issued;
  } else if (warp == 1 && lane == 0) {
    const uint64_t dbase = sdesc64(sbase);
    int s = 0, grp = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int id = blockIdx.x; ok && id < g.items; id += gridDim.x) {
      item(id, mt, nt, sp, kb0, nkb);
      for (int kb = 0; kb < nkb; ++kb) {
        const int b = grp & 1;
        const bool first = (kb % CHUNK) == 0;
        const bool last = (kb % CHUNK) == CHUNK - 1 || kb == nkb - 1;
        if ((first && grp >= 2 && !mbar_wait(acce[b], (uint32_t)((grp >> 1) - 1) & 1u, abort_sh, g.err, true)) ||
            !mbar_wait(full[0] + 8 * s, ph, abort_sh, g.err, true)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t st = sbase + s * STAGE_BYTES;
        const uint32_t buf = tmem + (uint32_t)(b * GCOLS);
  #pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          // sdesc64 is linear in the address here (its 14-bit start field holds address / 16
          // of a ring below 256 KB and cannot carry): a hoisted base plus constants
          const uint64_t sd = dbase + (uint64_t)((uint32_t)(st - sbase) >> 4);
          const uint64_t bd = sd + (uint64_t)((S * A_SLICE + kk * 32) >> 4);
  #pragma unroll
          for (int t = 0; t < S; ++t) {
            const uint64_t ad = sd + (uint64_t)((t * A_SLICE + kk * 32) >> 4);
            const uint32_t acc = (first && kk == 0 && t == 0) ? 0u : 1u;
            mma_bf16(buf + (uint32_t)(t * BNS), ad, bd, idesc_n((S - t) * BNS), acc);
          }
        }
        mma_commit(empty[0] + 8 * s);
        if (last) {
          mma_commit(accf[b]);
          ++grp;
        }
        if (++s == ST) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    mma_commit(done);
  } else if (warp >= 4) {
    // TMEM lanes 32 (warp % 4) .. +31 are the rows; half selects columns 0-15 or 16-31
    const int q = warp & 3, half = (warp - 4) >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    constexpr int NC = BNS / 2;
    bool ok = true;
    int grp0 = 0;
    for (int id = blockIdx.x; ok && id < g.items; id += gridDim.x) {
      item(id, mt, nt, sp, kb0, nkb);
      long long hi[NC], lo[NC];
  #pragma unroll
      for (int i = 0; i < NC; ++i) {
        hi[i] = 0;
        lo[i] = 0;
      }
      const int ngrp = (nkb + CHUNK - 1) / CHUNK;
      for (int grp = grp0; grp < grp0 + ngrp; ++grp) {
        const int b = grp & 1;
        const bool w = mbar_wait(accf[b], (uint32_t)(grp >> 1) & 1u, abort_sh, g.err, true);
        if (!__all_sync(0xffffffffu, w)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t col = tmem + lane_base + (uint32_t)(b * GCOLS + half * NC);
        uint32_t r0[NC], r1[NC], r2[NC];
        // group sums g_w are integers below 2^24 (exact in FP32)
        // hi += (g0 2^8 + g1) 2^16 + g2 2^8 + g3       (each bracket below 2^31)
        tmem_ld16_nowait(col, r0);
        tmem_ld16_nowait(col + 32, r1);
        tmem_wait_ld();
  #pragma unroll
        for (int i = 0; i < NC; ++i) {
          const int v = __float2int_rn(__uint_as_float(r0[i])) * 256 + __float2int_rn(__uint_as_float(r1[i]));
          hi[i] += (long long)v * 65536;
        }
        tmem_ld16_nowait(col + 64, r0);
        tmem_ld16_nowait(col + 96, r1);
        tmem_wait_ld();
  #pragma unroll
        for (int i = 0; i < NC; ++i) {
          const int v = __float2int_rn(__uint_as_float(r0[i])) * 256 + __float2int_rn(__uint_as_float(r1[i]));
          hi[i] += (long long)v;
        }
        // lo += g4 2^16 + g5 2^8 + g6
        tmem_ld16_nowait(col + 128, r0);
        tmem_ld16_nowait(col + 160, r1);
        tmem_ld16_nowait(col + 192, r2);
        tmem_wait_ld();
  #pragma unroll
        for (int i = 0; i < NC; ++i) {
          lo[i] += (long long)__float2int_rn(__uint_as_float(r0[i])) * 65536 +
                   (long long)__float2int_rn(__uint_as_float(r1[i])) * 256 +
                   (long long)__float2int_rn(__uint_as_float(r2[i]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce[b]);
      }
      grp0 += ngrp;
      // warp-uniform: another role may abort at this moment, and put_sym shuffles over the whole warp
      if (ok && __all_sync(0xffffffffu, *abort_sh == 0)) {
        const int64_t row = (int64_t)mt * BM + q * 32 + lane;  // < mp: rows are padded to whole tiles
        const int64_t col = (int64_t)nt * BNS + half * NC;
        if (g.hi) {
          const int64_t base = ((int64_t)sp * g.np + col) * g.mp + row;
  #pragma unroll
          for (int i = 0; i < NC; ++i) {
            g.hi[base + (int64_t)i * g.mp] = hi[i];
            g.lo[base + (int64_t)i * g.mp] = lo[i];
          }
        } else if (g.sym) {
          put_sym<NC>(g, row, col, hi, lo);
        } else if (row < g.M) {
  #pragma unroll
          for (int i = 0; i < NC; ++i)
            if (col + i < g.N) put_out(g, row, col + i, hi[i], lo[i]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_sh) {
    const int issued = *issued_sh;
    for (int kb = max(0, issued - ST); kb < issued; ++kb)
      mbar_wait(full[kb % ST], (uint32_t)(kb / ST) & 1u, abort_sh, g.err, false);
  }
  if (warp == 1) {
    if (lane == 0) mbar_wait(done, 0, abort_sh, g.err, false);
    __syncwarp();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// The sum of the splits' integers
__global__ void sliced_finalize_kernel(const __grid_constant__ Args g, int splits) {
  const int64_t total = g.M * g.N;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = idx % g.M, c = idx / g.M;
    long long h = 0, l = 0;
    for (int sp = 0; sp < splits; ++sp) {
      const int64_t o = ((int64_t)sp * g.np + c) * g.mp + r;
      h += g.hi[o];
      l += g.lo[o];
    }
    put_out(g, r, c, h, l);
  }
}

// ---------------------------------------------------------------- slicing
// One warp per row: exponent e with |x| < 2^e on the row, then the digits
// d_t = rint(r_t), r_0 = x 2^(7-e), r_{t+1} = (r_t - d_t) 2^8.
// Balanced base-256 digits of s = x 2^(7 - e) (|x| <= 2^e), in integer arithmetic:
// N = round(x 2^(55 - e)) from the exponent and mantissa bits (|N| < 2^55, rounded half
// away from zero), then d_6 .. d_1 the balanced low bytes of N (in [-128, 127]) and d_0
// what is left (|d_0| <= 128): s = sum_t d_t 2^(-8t) up to 2^-49.
__device__ __forceinline__ void int_digits(double x, int e, int* d) {
  const long long b = __double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7ff);
  long long mant = b & 0xfffffffffffffLL;
  int ex = ef;
  if (ef == 0) ex = 1;
  else mant |= 1LL << 52;
  const int sh = ex - 1020 - e;  // N = mant 2^sh; sh <= 2 for every |x| <= 2^e
  long long N = 0;
  if (sh >= 0) N = mant << sh;
  else if (sh > -63) N = (mant + (1LL << (-sh - 1))) >> (-sh);
  if (b < 0) N = -N;
#pragma unroll
  for (int t = S - 1; t >= 1; --t) {
    const int dt = (int)((N + 128) & 255) - 128;
    d[t] = dt;
    N = (N - dt) >> 8;
  }
  d[0] = (int)N;
}
// frexp exponent of the largest |x| of a row from the magnitudes' bit patterns
// (non-negative doubles order like their bits): 0 for a zero row.
__device__ __forceinline__ int row_exponent(unsigned long long mbits) {
  if (mbits == 0) return 0;
  const int ef = (int)(mbits >> 52);
  if (ef == 0x7ff) return EXP_NONFINITE;
  if (ef) return ef - 1022;
  return (64 - __clzll((long long)mbits)) - 1074;  // subnormal
}
__device__ __forceinline__ unsigned long long abs_bits(double2 v) {
  const unsigned long long a0 = (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull;
  const unsigned long long a1 = (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull;
  return max(a0, a1);
}
__device__ __forceinline__ void put_digits(double2 v, int e, __nv_bfloat16* p, int64_t plane) {
  int d0[S], d1[S];
  int_digits(v.x, e, d0);
  int_digits(v.y, e, d1);
#pragma unroll
  for (int t = 0; t < S; ++t)
    *reinterpret_cast<__nv_bfloat162*>(p + t * plane) =
        __halves2bfloat162(__int2bfloat16_rn(d0[t]), __int2bfloat16_rn(d1[t]));
}
// max over the CTA of one value per thread (blockDim.x a multiple of 32)
__device__ __forceinline__ unsigned long long cta_max(unsigned long long m) {
  __shared__ unsigned long long w[32];
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = max(m, w[i]);
  __syncthreads();
  return m;
}
// One CTA per row (32 to 256 threads by its length: a block of vectors has too few rows to
// occupy the GPU with one warp each).
template <class Src>
__global__ void slice_kernel(Src src, int64_t K, int64_t kpad, int64_t plane, __nv_bfloat16* planes, int* exps) {
  const int64_t r = blockIdx.x;
  unsigned long long m = 0;
  for (int64_t p = threadIdx.x; 2 * p < K; p += blockDim.x) m = max(m, abs_bits(src.pair(r, p)));
  const int e = row_exponent(cta_max(m));
  __nv_bfloat16* row = planes + r * kpad;
  for (int64_t p = threadIdx.x; 2 * p < kpad; p += blockDim.x)
    put_digits(2 * p < K ? src.pair(r, p) : make_double2(0.0, 0.0), e, row + 2 * p, plane);
  if (threadIdx.x == 0) exps[r] = e;
}
// The real form P' of H, one CTA per row i, which gives rows 2i and 2i + 1 from
// one read of A and B each pass: y = A x + B conj(x) in (re, im) interleaved form,
// Re y: (Ar + Br, Bi - Ai), Im y: (Ai + Bi, Ar - Br).  The FP64 additions (4 per entry and pass)
// take as long as the memory traffic.
__global__ void slice_ham_kernel(const cplx* A, const cplx* B, int64_t n, int64_t kpad, int64_t plane,
                                 __nv_bfloat16* planes, int* exps) {
  const int64_t i = blockIdx.x;
  const cplx *Ai = A + i * n, *Bi = B + i * n;
  unsigned long long m0 = 0, m1 = 0;
#pragma unroll 2
  for (int64_t l = threadIdx.x; l < n; l += blockDim.x) {
    const cplx a = Ai[l], b = Bi[l];
    m0 = max(m0, abs_bits(make_double2(a.x + b.x, b.y - a.y)));
    m1 = max(m1, abs_bits(make_double2(a.y + b.y, a.x - b.x)));
  }
  const int e0 = row_exponent(cta_max(m0)), e1 = row_exponent(cta_max(m1));
  __nv_bfloat16* row = planes + 2 * i * kpad;
  for (int64_t l = threadIdx.x; 2 * l < kpad; l += blockDim.x) {
    double2 v0 = make_double2(0.0, 0.0), v1 = v0;
    if (l < n) {
      const cplx a = Ai[l], b = Bi[l];
      v0 = make_double2(a.x + b.x, b.y - a.y);
      v1 = make_double2(a.y + b.y, a.x - b.x);
    }
    put_digits(v0, e0, row + 2 * l, plane);
    put_digits(v1, e1, row + kpad + 2 * l, plane);
  }
  if (threadIdx.x == 0) {
    exps[2 * i] = e0;
    exps[2 * i + 1] = e1;
  }
}

struct RowsSrc {  // row r at p + r * ld, pairs transformed by mode
  const double* p;
  int64_t ld;
  int mode;
  __device__ double2 pair(int64_t r, int64_t q) const {
    const double2 v = *reinterpret_cast<const double2*>(p + r * ld + 2 * q);
    if (mode == 1) return make_double2(v.y, -v.x);
    if (mode == 2) return make_double2(v.x, -v.y);
    return v;
  }
};
struct RowsSrcUnaligned {  // same, for an odd ld or offset
  const double* p;
  int64_t ld;
  int mode;
  __device__ double2 pair(int64_t r, int64_t q) const {
    const double a = p[r * ld + 2 * q], b = p[r * ld + 2 * q + 1];
    if (mode == 1) return make_double2(b, -a);
    if (mode == 2) return make_double2(a, -b);
    return make_double2(a, b);
  }
};
// The blocks of H^2 as C = [A | -B] R, R = [[A, B], [conj B, conj A]], computed as
// C^T = R^T [A | -B]^T so that the result lands row-major: the A operand holds the
// real-form rows of the columns j0 + r/2 of R's left (part 0: P2) or right (part 1: Q2)
// block column, the B operand the rows of [A | -B] as (re, im) pairs.
struct H2ColsSrc {
  const cplx* A;
  const cplx* B;
  int64_t n, j0;
  int part;
  __device__ double2 pair(int64_t r, int64_t l) const {
    const int64_t j = j0 + (r >> 1);
    cplx v;
    if (l < n) v = part == 0 ? A[l * n + j] : B[l * n + j];
    else v = cconj(part == 0 ? B[(l - n) * n + j] : A[(l - n) * n + j]);
    // row 2j: (Re, -Im); row 2j + 1: (Im, Re) -> (Re, Im) of sum_l R_lj w_l for w pairs (Re, Im)
    return (r & 1) == 0 ? make_double2(v.x, -v.y) : make_double2(v.y, v.x);
  }
};
struct H2RowsSrc {  // row i of [A | -B] as (re, im) pairs
  const cplx* A;
  const cplx* B;
  int64_t n;
  __device__ double2 pair(int64_t i, int64_t l) const {
    if (l < n) {
      const cplx v = A[i * n + l];
      return make_double2(v.x, v.y);
    }
    const cplx v = B[i * n + (l - n)];
    return make_double2(-v.x, -v.y);
  }
};

struct ComplexRowsSrc {  // row r of the complex column-major M, optionally conjugated
  const cplx* M;
  int64_t ld;
  double sign;  // -1: conjugate
  __device__ double2 pair(int64_t r, int64_t l) const {
    const cplx v = M[r + l * ld];
    return make_double2(v.x, sign * v.y);
  }
};

// out (2n x 2m, row-major): rows 2i, 2i+1 of the real form of row i of X.
__global__ void complex_rows_kernel(const cplx* X, int64_t ldx, int64_t n, int64_t m, double* out) {
  __shared__ cplx t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32, l0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int j = ty; j < 32; j += 8) {
    const int64_t i = i0 + tx, l = l0 + j;
    t[j][tx] = (i < n && l < m) ? X[i + l * ldx] : mk(0, 0);
  }
  __syncthreads();
  for (int j = ty; j < 32; j += 8) {
    const int64_t i = i0 + j, l = l0 + tx;
    if (i < n && l < m) {
      const cplx x = t[tx][j];
      double* r0 = out + (2 * i) * (2 * m) + 2 * l;
      double* r1 = r0 + 2 * m;
      r0[0] = x.x;
      r0[1] = -x.y;
      r1[0] = x.y;
      r1[1] = x.x;
    }
  }
}

// Z (n x 2k, column-major) from W (2n x k): the J-fixed halves of w_j = [x; y],
// a_j = (x + conj(y))/2 and c_j = i (x - conj(y))/2, so that w = [a; conj(a)] - i [c; conj(c)].
__global__ void jsplit_kernel(const cplx* W, int64_t n, int64_t k, cplx* Z) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, j = idx / n;
    const cplx x = W[j * 2 * n + i], y = W[j * 2 * n + n + i];
    const cplx a = mk(0.5 * (x.x + y.x), 0.5 * (x.y - y.y));
    const cplx d = mk(0.5 * (x.x - y.x), 0.5 * (x.y + y.y));  // (x - conj(y)) / 2
    Z[(2 * j) * n + i] = a;
    Z[(2 * j + 1) * n + i] = mk(-d.y, d.x);                  // i d
  }
}
// H w_j from T = [P'a_j, P'c_j] (y = A z + B conj(z) of the J-fixed halves):
// top = P'a - i P'c, bottom = -conj(P'a) + i conj(P'c).
__global__ void jcombine_kernel(const cplx* T, int64_t n, int64_t k, cplx* out) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, j = idx / n;
    const cplx ta = T[(2 * j) * n + i], tc = T[(2 * j + 1) * n + i];
    out[j * 2 * n + i] = mk(ta.x + tc.y, ta.y - tc.x);       // ta - i tc
    out[j * 2 * n + n + i] = mk(-ta.x + tc.y, ta.y + tc.x);  // -conj(ta) + i conj(tc)
  }
}

// W (2n x k) from the halves in the columns 2v, 2v + 1 of the block Zsel[v]
__global__ void jmerge_kernel(cplx* W, const cplx* Z0, const cplx* Z1, const cplx* Z2, const int* sel, int64_t n,
                              int64_t k) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, j = idx / n;
    const cplx* Z = sel[j] == 0 ? Z0 : (sel[j] == 1 ? Z1 : Z2);
    const cplx a = Z[2 * j * n + i], c = Z[(2 * j + 1) * n + i];
    W[j * 2 * n + i] = mk(a.x + c.y, a.y - c.x);       // a - i c
    W[j * 2 * n + n + i] = mk(a.x - c.y, -a.y - c.x);  // conj(a) - i conj(c)
  }
}

static unsigned gsz(int64_t total) {
  const int64_t b = (total + 255) / 256;
  return (unsigned)std::min<int64_t>(std::max<int64_t>(b, 1), 16384);
}

static int make_map3(CUtensorMap* m, const void* base, int64_t kpad, int64_t rows_pad, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return CHASE_BSE_UNSUPPORTED;
  const cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)rows_pad, (cuuint64_t)S};
  const cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)(rows_pad * kpad * 2)};
  const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)S};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? CHASE_BSE_OK : CHASE_BSE_CUDA_ERROR;
}

template <class Src>
static int run_slice(const Src& src, SlicedOp& op, cudaStream_t s) {
  const int threads = op.K >= 4096 ? 256 : (op.K >= 512 ? 128 : 32);
  slice_kernel<Src><<<(unsigned)op.rows, threads, 0, s>>>(src, op.K, op.kpad, op.rows_pad * op.kpad, op.planes,
                                                          op.exps);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}

}  // namespace tcd

int sliced_alloc(Workspace& ws, SlicedOp& op, int64_t rows, int64_t K, cudaStream_t s) {
  using namespace tcd;
  if (rows <= 0 || K <= 0 || (K % 2) != 0) return CHASE_BSE_BAD_ARG;
  op.rows = rows;
  op.K = K;
  op.rows_pad = ((rows + BM - 1) / BM) * BM;
  op.kpad = ((K + BK - 1) / BK) * BK;
  const int64_t elems = (int64_t)S * op.rows_pad * op.kpad;
  CB_TRY(ws.alloc(&op.planes, elems));
  CB_TRY(ws.alloc(&op.exps, op.rows_pad));
  // rows beyond `rows` stay zero (and their exponent 0)
  if (op.rows_pad > rows) {
    for (int t = 0; t < S; ++t)
      CB_CUDA(cudaMemsetAsync(op.planes + (int64_t)t * op.rows_pad * op.kpad + rows * op.kpad, 0,
                              sizeof(__nv_bfloat16) * (op.rows_pad - rows) * op.kpad, s));
    CB_CUDA(cudaMemsetAsync(op.exps + rows, 0, sizeof(int) * (op.rows_pad - rows), s));
  }
  CB_TRY(make_map3(&op.map_a, op.planes, op.kpad, op.rows_pad, BM));
  CB_TRY(make_map3(&op.map_b, op.planes, op.kpad, op.rows_pad, BNS));
  return CHASE_BSE_OK;
}

int slice_rows(const double* src, int64_t ld, int mode, SlicedOp& op, cudaStream_t s) {
  if ((reinterpret_cast<uintptr_t>(src) % 16) == 0 && (ld % 2) == 0)
    return tcd::run_slice(tcd::RowsSrc{src, ld, mode}, op, s);
  return tcd::run_slice(tcd::RowsSrcUnaligned{src, ld, mode}, op, s);
}

int slice_complex_rows(const cplx* X, int64_t ldx, int64_t n, int64_t m, double* tmp, SlicedOp& op,
                       cudaStream_t s) {
  if (op.rows != 2 * n || op.K != 2 * m) return CHASE_BSE_BAD_ARG;
  dim3 grid((unsigned)((n + 31) / 32), (unsigned)((m + 31) / 32));
  tcd::complex_rows_kernel<<<grid, dim3(32, 8), 0, s>>>(X, ldx, n, m, tmp);
  count_launch();
  CB_LAUNCH();
  return slice_rows(tmp, 2 * m, 0, op, s);
}

int slice_conj_rows(const cplx* M, int64_t ld, SlicedOp& op, cudaStream_t s) {
  return tcd::run_slice(tcd::ComplexRowsSrc{M, ld, -1.0}, op, s);
}

int slice_plain_rows(const cplx* M, int64_t ld, SlicedOp& op, cudaStream_t s) {
  return tcd::run_slice(tcd::ComplexRowsSrc{M, ld, 1.0}, op, s);
}

int hop_sliced(const SlicedOp& ph, const cplx* W, int64_t n, int64_t k, cplx* out, cudaStream_t s) {
  if (k == 0) return CHASE_BSE_OK;
  if (ph.rows != 2 * n || ph.K != 2 * n) return CHASE_BSE_BAD_ARG;
  Workspace ws(s);
  cplx *Z, *T;
  CB_TRY(ws.alloc(&Z, n * 2 * k));
  CB_TRY(ws.alloc(&T, n * 2 * k));
  SlicedOp sz;
  CB_TRY(sliced_alloc(ws, sz, 2 * k, 2 * n, s));
  const int64_t tid = timer_begin(2, 32.0 * (double)n * (double)n * (double)k, s);
  tcd::jsplit_kernel<<<tcd::gsz(n * k), 256, 0, s>>>(W, n, k, Z);
  count_launch();
  CB_LAUNCH();
  CB_TRY(slice_rows(reinterpret_cast<const double*>(Z), 2 * n, 0, sz, s));
  CB_TRY(sliced_gemm(ph, sz, 1.0, reinterpret_cast<double*>(T), 1, 2 * n, false, s));
  tcd::jcombine_kernel<<<tcd::gsz(n * k), 256, 0, s>>>(T, n, k, out);
  timer_end(tid, s);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}

int form_h2(const cplx* A, const cplx* B, int64_t n, cplx* P2, cplx* Q2, cudaStream_t s) {
  Workspace ws(s);
  SlicedOp rows;  // [A | -B]: n rows of 2n complex entries
  CB_TRY(sliced_alloc(ws, rows, n, 4 * n, s));
  CB_TRY(tcd::run_slice(tcd::H2RowsSrc{A, B, n}, rows, s));
  // columns of R in chunks: the A operand of a chunk of cj columns holds 7 digit planes of
  // 2 cj x 4n BF16 values (about 8 GB at most)
  int64_t cj = std::max<int64_t>(64, (int64_t)(8.0e9 / (112.0 * (double)n)) / 64 * 64);
  cj = std::min(cj, n);
  for (int part = 0; part < 2; ++part) {
    cplx* out = part == 0 ? P2 : Q2;
    for (int64_t j0 = 0; j0 < n; j0 += cj) {
      const int64_t m = std::min(cj, n - j0);
      Workspace cws(s);
      SlicedOp cols;
      CB_TRY(sliced_alloc(cws, cols, 2 * m, 4 * n, s));
      CB_TRY(tcd::run_slice(tcd::H2ColsSrc{A, B, n, j0, part}, cols, s));
      // C^T[2(j - j0) + t][i] -> (Re, Im) of C_ij at double 2 (i n + j) + t
      CB_TRY(sliced_gemm(cols, rows, 1.0, reinterpret_cast<double*>(out + j0), 1, 2 * n, false, s));
    }
  }
  return CHASE_BSE_OK;
}

int slice_hamiltonian(const cplx* A, const cplx* B, int64_t n, SlicedOp& op, cudaStream_t s) {
  if (op.rows != 2 * n || op.K != 2 * n) return CHASE_BSE_BAD_ARG;
  tcd::slice_ham_kernel<<<(unsigned)n, 256, 0, s>>>(A, B, n, op.kpad, op.rows_pad * op.kpad, op.planes, op.exps);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}

int jsplit(const cplx* W, int64_t n, int64_t k, cplx* Z, cudaStream_t s) {
  tcd::jsplit_kernel<<<tcd::gsz(n * k), 256, 0, s>>>(W, n, k, Z);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}
int jmerge(cplx* W, const cplx* Z0, const cplx* Z1, const cplx* Z2, const int* sel, int64_t n, int64_t k,
           cudaStream_t s) {
  tcd::jmerge_kernel<<<tcd::gsz(n * k), 256, 0, s>>>(W, Z0, Z1, Z2, sel, n, k);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}

int sliced_gemm(const SlicedOp& a, const SlicedOp& b, double alpha, double* out, int64_t rs, int64_t cs,
                bool neg_odd, cudaStream_t s, int* err, int sym) {
  using namespace tcd;
  if (a.K != b.K || a.kpad != b.kpad) return CHASE_BSE_BAD_ARG;
  static bool attr = false;
  if (!attr) {
    CB_CUDA(cudaFuncSetAttribute(sliced_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    attr = true;
  }
  const int num_m = (int)(a.rows_pad / BM);
  const int num_n = (int)((b.rows + BNS - 1) / BNS);
  const int kb_total = (int)(a.kpad / BK);
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // K splits (whole 128-long chunks): the number of least estimated time, in K blocks (about
  // 0.75 us each): waves of CTAs x (blocks of a split + 2 for the tile's end), and with a split
  // the partial tiles' traffic (32 bytes an output and split, about 5 TB/s) and a second launch
  const int64_t tiles = (int64_t)num_m * num_n;
  const int64_t np = (int64_t)num_n * BNS, mp = a.rows_pad;
  int splits = 1, kb_per = ((kb_total + CHUNK - 1) / CHUNK) * CHUNK;
  double best = 0.0;
  for (int want = 1; want <= std::max(1, kb_total / CHUNK) && want <= 64; ++want) {
    const int per = ((kb_total + want - 1) / want + CHUNK - 1) / CHUNK * CHUNK;
    const int sp = (kb_total + per - 1) / per;
    const double waves = (double)((tiles * sp + sms - 1) / sms);
    double t = waves * (std::min(per, kb_total) + 2.0);
    if (sp > 1) t += 8.0 + (double)sp * (double)np * (double)mp * 32.0 / 3.75e6;
    if (best == 0.0 || t < best * 0.98) {
      best = t;
      splits = sp;
      kb_per = per;
    }
    if (tiles * sp > 4 * (int64_t)sms) break;
  }
  // a triangle's tiles, where they alone keep the SMs busy and need no K split
  const int64_t tri = (int64_t)num_m * (num_m + 1);
  const bool half = sym != 0 && rs == 1 && a.rows == 2 * b.rows && cs == a.rows && tri >= 2 * (int64_t)sms;
  if (half) splits = 1, kb_per = kb_total;
  Workspace ws(s);
  Args g{};
  g.sym = half ? sym : 0;
  g.num_m = num_m;
  g.num_n = num_n;
  g.n_fast = a.rows_pad >= b.rows_pad ? 1 : 0;
  g.kb_total = kb_total;
  g.kb_per_split = kb_per;
  g.items = (int)(half ? tri : tiles * splits);
  g.mp = mp;
  g.np = np;
  g.ea = a.exps;
  g.eb = b.exps;
  g.M = a.rows;
  g.N = b.rows;
  g.alpha = alpha;
  g.out = out;
  g.rs = rs;
  g.cs = cs;
  g.neg_odd = neg_odd ? 1 : 0;
  g.err = err;
  if (splits > 1) {
    CB_TRY(ws.alloc(&g.hi, (size_t)splits * np * mp));
    CB_TRY(ws.alloc(&g.lo, (size_t)splits * np * mp));
  }
  if (!err) {
    CB_TRY(ws.alloc(&g.err, 1));
    CB_CUDA(cudaMemsetAsync(g.err, 0, sizeof(int), s));
  }
  sliced_gemm_kernel<<<(unsigned)std::min<int64_t>(g.items, sms), THREADS, SMEM_BYTES, s>>>(a.map_a, b.map_b, g);
  count_launch();
  CB_LAUNCH();
  if (splits > 1) {
    sliced_finalize_kernel<<<gsz(a.rows * b.rows), 256, 0, s>>>(g, splits);
    count_launch();
    CB_LAUNCH();
  }
  if (err) return CHASE_BSE_OK;
  int herr = 0;
  CB_CUDA(cudaMemcpyAsync(&herr, g.err, sizeof(int), cudaMemcpyDeviceToHost, s));
  CB_CUDA(cudaStreamSynchronize(s));
  return herr ? CHASE_BSE_DEVICE_TIMEOUT : CHASE_BSE_OK;
}

}  // namespace cb
