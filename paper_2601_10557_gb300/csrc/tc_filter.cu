// Mixed-precision Chebyshev filter on H^2 with tcgen05 tensor cores (sm_103a).
//
// One application of H to a block of k vectors is one real GEMM on 5th-generation tensor
// cores, FP32 in TMEM, in one of two forms:
//
// Blocks: C (n x 4k) = P (n x 4n) * W (4n x 4k), P the rows of [A | B] as (re, im) pairs.  A vector
// w = [x; y] gives four columns: w and i w for the top half of H w, u = [conj y; conj x] and
// i u for -conj of the bottom half.  32 n^2 k operations.  Each half is a sum of its own
// products, so both keep the scheme's accuracy relative to their own size (the lower half of an
// eigenvector is smaller than the upper one by the coupling |B| / |A|).  The filter entry points.
//
// J form: w is the sum [a; conj a] - i [c; conj c] of two vectors fixed by J = K conj,
// a = (x + conj y) / 2 and c = i (x - conj y) / 2, and H maps [z; conj z] to i [z'; conj z']
// with z' = -i (A z + B conj z), a real-linear map of the real 2n-vector (Re z, Im z):
//   M = [[Ai + Bi, Ar - Br], [-(Ar + Br), Ai - Bi]]   (2n x 2n),   H^2: z -> -M M z.
// So the whole recurrence runs on two real columns per vector and one application is
//   C (2n x 2k) = M (2n x 2n) * Z (2n x 2k),
// 16 n^2 k operations and a quarter of the operand bytes to write per step; rows of M and
// entries of a column are interleaved, 2i is Re, 2i + 1 is Im.  The smaller half of a vector
// comes out as a difference of two numbers of the size of the larger one and is accurate relative
// to that (lower half of a degree-20 filter at n = 512, FP16x3: coupling 0.3 1.4e-5 instead of
// 2.0e-6, coupling 1e-3 6e-4 instead of 3e-6).  The solves: their QR and Rayleigh-Ritz steps hold
// the basis as J-fixed vectors, the correction form below lets a filter's error shrink with
// the residual, and the lower half y of a locked pair is off by (conj A + lambda)^{-1} times its
// residual whatever the form (measured equal at couplings 0.3 to 1e-6 and tolerances to 1e-12).
//
// Split products on 16-bit tensor cores: an operand x is written as a sum of
// pieces x = x0 + x1 (+ x2), x0 = rn(x), x1 = rn(x - x0), ..., and the product
// keeps the cross terms down to the target accuracy, all accumulated in FP32:
//   FP16x3: 2 FP16 pieces each (11 + 11 bits), x0 y0 + x0 y1 + x1 y0   (~2^-22)
//   BF16x3: 2 BF16 pieces each (8 + 8 bits), same products             (~2^-16)
//   BF16x6: 3 BF16 pieces each, adds x0 y2 + x1 y1 + x2 y0             (~2^-24)
// (FP16 pieces of this kind: Ootomo and Yokota, Int. J. HPC Appl. 2022.)  FP16 has
// a 5-bit exponent, so every operand row is scaled by a power of two: row r of M
// or P by 2^prow[r] (its largest entry in [2^12, 2^13)), column (blocks: vector) v by 2^vexp[v], chosen
// from an upper bound of its entries below 2^13: the bound of an output of H is
// L * max|input| with L the largest absolute row sum of P, and that of the
// recurrence combines the maxima of its terms; every epilogue records the true
// maximum of each output column or vector (one atomic max per warp and column) for the
// next bound.  The epilogue divides the accumulator by 2^(prow + vexp).  Entries
// far below the bound only lose precision relative to the bound, which keeps the
// product's error below that of an FP32 GEMM (|dy| <~ 2^-22 L max|w|).  The
// BF16 schemes use the same scaling (harmless: BF16 has FP32's exponent range).
//
// Kernel structure: persistent CTA pairs (cta_group::2, one pair per two SMs, 512 threads
// a CTA), each working through 256 x BN output tiles (BN <= 256, chosen per launch); CTA r
// of a pair holds rows 128 r .. 128 r + 127 of the tile, its A rows and half of the B rows.
//   warp 0   TMA producer: the A pieces and the B half's pieces of 64 K-elements (128B
//            swizzle) into the shared-memory ring; both CTAs' bytes count on CTA 0's barrier
//   warp 1   allocates all 512 TMEM columns (x0*y0 and the cross products); one lane
//            of CTA 0 issues the tcgen05.mma of a K block, x0*y0 first
//   warps 4-11 drain x0*y0 after every FLUSH K blocks (tcgen05.ld) into FP32 registers,
//            because the tensor core's FP32 accumulation truncates, while the block's
//            cross products (2/3 of its MMA time) run (and, in tiles of up to 160 columns,
//            the next blocks' x0*y0 in a second buffer); at the end of a tile they add the
//            cross products, write the FP32 tile to a workspace that stays in L2 and go on
//            to the next tile
//   warps 12-15 finish a tile behind the next one's MMAs (the drain warps help with a pair's
//            last tile, and where several pairs hold K ranges of a tile the last writer sums
//            them): either
//            (mode 0) store the next GEMM's B-operand pieces, or
//            (mode 1) the fused three-term recurrence in FP32 plus the pieces, or
//            (mode 2) Z = H X + gamma * X (no pieces).
// Every mbarrier wait is bounded (2 s of %globaltimer); on expiry the kernel
// sets an error flag, waits (bounded) for its copies in flight into its shared
// memory, frees its TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "dense_kernels.cuh"
#include "fp64_kernels.cuh"
#include "solver.cuh"
#include "tc_common.cuh"

namespace cb {
namespace tc {

constexpr int BM = 128;
constexpr int KPAD = 64;              // K (2n) is padded to a multiple of this
constexpr int BNMAX = 256;            // widest output tile
constexpr uint32_t TMEM_COLS = 512;   // one or two x0*y0 buffers and the cross products
constexpr int VEXP_MAX = 100;         // |operand exponents| are clamped to this
// instruction descriptor, kind::f16: D = F32, A = B = BF16 (bf16) or FP16, both K-major, 256 x n
__device__ __forceinline__ uint32_t make_idesc(int n, bool bf16) {
  return (1u << 4) | (bf16 ? ((1u << 7) | (1u << 10)) : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(2 * BM >> 4) << 24);
}

// 16-bit piece types
template <class T>
struct Piece;
template <>
struct Piece<__nv_bfloat16> {
  using T2 = __nv_bfloat162;
  static constexpr bool BF16 = true;
  __device__ static __nv_bfloat16 rn(float x) { return __float2bfloat16_rn(x); }
  __device__ static float back(__nv_bfloat16 x) { return __bfloat162float(x); }
  __device__ static T2 pair(__nv_bfloat16 a, __nv_bfloat16 b) { return __halves2bfloat162(a, b); }
  __device__ static unsigned bits(T2 p) { return *reinterpret_cast<unsigned*>(&p); }
};
template <>
struct Piece<__half> {
  using T2 = __half2;
  static constexpr bool BF16 = false;
  __device__ static __half rn(float x) { return __float2half_rn(x); }
  __device__ static float back(__half x) { return __half2float(x); }
  __device__ static T2 pair(__half a, __half b) { return __halves2half2(a, b); }
  __device__ static unsigned bits(T2 p) { return *reinterpret_cast<unsigned*>(&p); }
};

// Scheme: piece type, pieces of A (NPA) and B (NPW), product list (product 0 is x0 * y0), K blocks
// per drained partial sum of x0 * y0 in the J form (FLUSH) and in the blocks form, whose sums are
// twice as long (FLUSH_BLOCKS; against FLUSH there: FP16x3 3-5 % longer for 0.5 to 0.8 of the
// error, BF16x6 3-5 % for 0.6 to 0.8 below n = 3500).
enum : int { SCH_BF16X3 = 1, SCH_BF16X6 = 2, SCH_FP16X3 = 3 };
template <int SCH>
struct Scheme;
template <>
struct Scheme<SCH_BF16X3> {
  using T = __nv_bfloat16;
  static constexpr int NPA = 2, NPW = 2, NPROD = 3, FLUSH = 4, FLUSH_BLOCKS = 4;
  __device__ static constexpr int pa(int i) { return i == 2 ? 1 : 0; }
  __device__ static constexpr int pb(int i) { return i == 1 ? 1 : 0; }
};
template <>
struct Scheme<SCH_FP16X3> {
  using T = __half;
  static constexpr int NPA = 2, NPW = 2, NPROD = 3, FLUSH = 4, FLUSH_BLOCKS = 2;
  __device__ static constexpr int pa(int i) { return i == 2 ? 1 : 0; }
  __device__ static constexpr int pb(int i) { return i == 1 ? 1 : 0; }
};
template <>
struct Scheme<SCH_BF16X6> {
  using T = __nv_bfloat16;
  static constexpr int NPA = 3, NPW = 3, NPROD = 6, FLUSH = 2, FLUSH_BLOCKS = 1;
  // (0,0) (0,1) (1,0) (0,2) (1,1) (2,0)
  __device__ static constexpr int pa(int i) { return i == 2 ? 1 : (i == 4 ? 1 : (i == 5 ? 2 : 0)); }
  __device__ static constexpr int pb(int i) { return i == 1 ? 1 : (i == 3 ? 2 : (i == 4 ? 1 : 0)); }
};
// Form of an application: operand rows per row of A, operand columns per vector and, of
// those, how many differ in scale (a master, an exponent and a maximum each); K elements per
// row of A.
enum : int { FORM_J = 0, FORM_BLOCKS = 1 };
template <int FORM>
struct Form;
template <>
struct Form<FORM_J> {
  static constexpr int ROWS = 2, COLS = 2, SCALES = 2, KEL = 2;
};
template <>
struct Form<FORM_BLOCKS> {
  static constexpr int ROWS = 1, COLS = 4, SCALES = 1, KEL = 4;
};
// Geometry.  A K block is 64 K-elements (128-byte swizzle); a stage of the ring holds the
// pieces of 128 A rows and of BN / 2 B rows, so a pair takes in 64 KB per CTA and 1536 MMA
// cycles at BN = 256 where one CTA per 128 x 128 tile takes 64 KB per 768: shared-memory
// traffic (operand reads of the MMAs plus the fill) bounds the smaller tile.  Of x0 * y0
// 16 truncating MMA additions go into a drained sum with two pieces (8 cost 2-8 %), 8 with
// three, whose 24 bits the truncation of 16 would show (1.9 times the error).  K blocks of 32 in
// twice the stages lost 10-25 % (64-byte rows).
//
// Measured on one GB300, FP16x3, time of one launch of a degree's two, before (one CTA per
// 128 x 128 tile, blocks form) and after, blocks and J form: n = 16384, k = 1300 26.8 -> 24.0 and
// 11.5 ms (J form: three products of 16 n^2 k at 1446 TFLOP/s; cuBLAS bf16 1702 sustained); n = 8192,
// k = 300 1707 -> 1218 and 715 us; n = 4096, k = 260 370 -> 315 and 185 us; n = 3001, k = 83 89 -> 85
// and 60 us; n = 512, k = 30 30 -> 21 and 20 us.  Whole filters in blocks form: degree 20 at n = 4096
// 15.2 -> 12.5 ms, degree 8 at n = 16384 436 -> 390 ms; of 28 sizes only those below n = 80 are not
// faster (n = 40, k = 4, degree 28 0.75 -> 0.83 ms, n = 64, k = 6 0.79 -> 0.82).  Errors against 64 bits, of the
// earlier kernel's: each half in blocks form 0.5 to 1.03 (n = 128 to 16384), the whole vector in J form 0.46
// to 1.03.
constexpr int BK = 64;
constexpr int A_BYTES = BM * BK * 2;
constexpr int MAX_ST = 8;                // most ring stages
constexpr int RING_BYTES = 196608;       // (all 227 KB, 4 stages at BN = 192, ran 2-5 % slower)
constexpr int NBAR = 2 * MAX_ST + 10;    // full, empty, acc_full[2], acc_empty[2], cross_full, cross_empty, out_full[2], out_empty[2]
constexpr int SMEM_BYTES = RING_BYTES + 1024 + 256;
constexpr int DC = 128;                  // most columns per drain warp
constexpr int DRAIN_WARPS = 4 * (BNMAX / DC);
constexpr int EPI_WARPS = 4;
constexpr int THREADS = 128 + 32 * (DRAIN_WARPS + EPI_WARPS);
// Registers a thread: 128 at launch (65536 over 16 warps); the warpgroup of the producer and
// the MMA issuer and that of the finishing warps give theirs to the drain warps, whose sums
// take 128.  40, 184 and 96 spilled the finishing warps' addresses: blocks form 5-8 % slower (n = 1301,
// k = 67 42 -> 39 us a launch, n = 3001, k = 83 91 -> 84), the n = 4096 solve 1 %.
constexpr int REGS_LAUNCH = 128, REGS_ROLES = 48, REGS_DRAIN = 176, REGS_EPI = 104;
// The warpgroups draw on what the block was launched with: a kernel compiled to fewer registers a
// thread than the shares add up to would wait for the rest forever (see mixed_filter_available).
constexpr bool register_split_fits(int regs) {
  return 128 * REGS_ROLES + 32 * DRAIN_WARPS * REGS_DRAIN + 32 * EPI_WARPS * REGS_EPI <= THREADS * regs;
}
static_assert(register_split_fits(REGS_LAUNCH) && register_split_fits(126) && !register_split_fits(125),
              "126 registers a thread hold the shares");
static_assert(SMEM_BYTES <= 232448, "shared memory");

struct Epi {
  int mode;           // 0: operand pieces, 1: recurrence, 2: H X + gamma X
  int h2;             // the operand holds the blocks of H^2
  int64_t n;          // rows of A
  int64_t rows, cols; // rows of the operand, active columns
  int64_t kpad;       // elements per piece row
  void* out[3];       // output operand pieces (NPW used)
  float* Znext;       // masters: 2n reals per column (J form), 2n complex per vector (blocks)
  const float* Zcur;
  const float* Zprev;
  const float* src;
  const float* gamma;  // per column
  float alpha, beta, c;
  // operand scaling: M' = diag(2^prow) M, scaled column v times 2^vexp_in[v]; the pieces this
  // launch writes get 2^vexp_out[v] chosen from the bound
  //   ca * L * amax_a[v] + cb * amax_b[v] + cc * amax_c[v] + |gamma[v]| * amax_d[v]
  // (L: largest absolute row sum of M; amax_*: largest |entry| of each input column);
  // amax_out receives the largest |entry| of each output column
  const float* L;
  const int* prow;
  const int* vexp_in;
  int* vexp_out;
  float* amax_out;
  const float* amax_a;
  const float* amax_b;
  const float* amax_c;
  const float* amax_d;
  float ca, cb, cc;
  int* err;
  float* part;  // FP32 (partial) tiles, two per CTA in turn, column-major 128 x BN
  int* cnt;     // per half tile, partial tiles written so far (zero between launches)
  int sms;      // SMs of the device
};

// 2^e as a float, |e| <= 126
__device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }
// Operand exponent for entries bounded by b: b 2^e < 2^13 (b = m 2^x, m in [1/2, 1) -> e = 13 - x);
// 0 for a zero, infinite or NaN bound.
__device__ __forceinline__ int out_exp(float b) {
  if (!(b > 0.0f) || !(b <= 3.0e38f)) return 0;
  const int bits = __float_as_int(b);
  const int x = ((bits >> 23) & 0xff) - 126;  // subnormal b: a smaller x, still a valid scale
  return min(max(13 - x, -VEXP_MAX), VEXP_MAX);
}
__device__ __forceinline__ float vec_bound(const Epi& ep, int64_t v) {
  float b = ep.ca * *ep.L * ep.amax_a[v];
  if (ep.cb != 0.0f) b += ep.cb * ep.amax_b[v];
  if (ep.cc != 0.0f) b += ep.cc * ep.amax_c[v];
  if (ep.amax_d) b += fabsf(ep.gamma[v]) * ep.amax_d[v];
  return b;
}

// Work of one launch: 256 x BN output tiles in a grouped raster (group_m row tiles x all
// column tiles), so that the pairs running at the same time stream the same K blocks of A
// and B from L2.  Pair c takes the whole tiles w * pairs + c of the full waves; the K blocks of the
// `rest` tiles that are left, one tile's after the other's, are shared out to `tail` pairs (rest <=
// tail <= pairs), so a pair holds one K range of a tile or the end of one and the start of the next.
// Where a tile is cut, the CTA that writes a half tile's last partial tile (a counter per half
// tile) sums them in K order and finishes the tile, so no CTA waits for another and the result does
// not depend on timing.
struct Sched {
  int nkb, num_m, num_n, bn, n_last;  // K blocks; tiles; columns of a tile and of the last one
  int stages, stage_bytes, bufs, dcols, flush;
  int pairs, waves, rest, tail;
  int group_m;
  __device__ void tile_of(int t, int& mt, int& nt) const {
    const int per_group = group_m * num_n;
    const int g = t / per_group, first = g * group_m;
    const int gm = min(group_m, num_m - first);
    const int rem = t - g * per_group;
    nt = rem / gm;
    mt = first + rem % gm;
  }
  // First of the tail's K blocks that pair c holds, and the pair that holds block x (32-bit
  // products: rest * nkb * tail < 2^31 up to n = 10^6).
  __device__ int tail_start(int c) const { return (int)((unsigned)(rest * nkb * c) / (unsigned)tail); }
  __device__ int tail_owner(int x) const { return (int)((unsigned)((x + 1) * tail - 1) / (unsigned)(rest * nkb)); }
};
// The segments (tile, K range) of pair c in order; all roles of both CTAs walk the same list.
struct Walk {
  const Sched& sc;
  int c, w;
  int mt, nt, cols;  // the current segment's tile and its columns
  int kb0, kb1;
  int pos, end;      // the pair's K blocks of the tail not yet walked
  __device__ Walk(const Sched& s, int pair) : sc(s), c(pair), w(-1), pos(0), end(0) {
    if (c < sc.tail) {
      pos = sc.tail_start(c);
      end = sc.tail_start(c + 1);
    }
  }
  __device__ bool next() {
    ++w;
    int t;
    if (w < sc.waves) {
      t = w * sc.pairs + c;
      kb0 = 0;
      kb1 = sc.nkb;
    } else if (pos < end) {
      const int r = (unsigned)pos / (unsigned)sc.nkb, x = r * sc.nkb;
      t = sc.waves * sc.pairs + r;
      kb0 = pos - x;
      pos = min(x + sc.nkb, end);
      kb1 = pos - x;
    } else {
      return false;
    }
    sc.tile_of(t, mt, nt);
    cols = nt == sc.num_n - 1 ? sc.n_last : sc.bn;
    return true;
  }
  __device__ int tail_tile() const { return (unsigned)(pos - 1) / (unsigned)sc.nkb; }
  __device__ bool split() const { return w >= sc.waves && sc.tail > sc.rest; }
  __device__ bool final() const { return pos >= end && w >= sc.waves - 1; }
};

// Shared-memory matrix descriptor: K-major tile written by TMA with 128-byte rows and
// 128-byte swizzle; 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused for these layouts)
  d |= (uint64_t)((8 * 2 * BK) >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)2 << 61;                    // 128-byte swizzle
  return d;
}
// sum[0..cols) += the warp's TMEM lanes at columns [col, col + cols), cols a multiple of 16
__device__ __forceinline__ void drain_add(uint32_t col, int cols, float* sum) {
#pragma unroll
  for (int c = 0; c < DC; c += 32) {
    if (c + 16 < cols) {  // uniform over the warp
      uint32_t r[32];
      tmem_ld32_nowait(col + (uint32_t)c, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) sum[c + i] += __uint_as_float(r[i]);
    } else if (c < cols) {
      uint32_t r[16];
      tmem_ld16_nowait(col + (uint32_t)c, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i) sum[c + i] += __uint_as_float(r[i]);
    }
  }
}

// NPC pieces of the pair (a, b) at element offset off of every piece plane
template <class T, int NPC>
__device__ __forceinline__ void put(void* const* pc, int64_t off, float a, float b) {
  using PT = Piece<T>;
#pragma unroll
  for (int q = 0; q < NPC; ++q) {
    const T ha = PT::rn(a), hb = PT::rn(b);
    *reinterpret_cast<typename PT::T2*>(static_cast<T*>(pc[q]) + off) = PT::pair(ha, hb);
    a -= PT::back(ha);
    b -= PT::back(hb);
  }
}
// and of one value
template <class T, int NPC>
__device__ __forceinline__ void put1(void* const* pc, int64_t off, float a) {
  using PT = Piece<T>;
#pragma unroll
  for (int q = 0; q < NPC; ++q) {
    const T ha = PT::rn(a);
    static_cast<T*>(pc[q])[off] = ha;
    a -= PT::back(ha);
  }
}

// The four operand rows of vector v in the blocks form at K positions 2i (top entry t) and
// 2(n + i) (bottom entry b): w, i w, u, i u as (re, -im), (im, re) pairs, u = [conj(b); conj(t)],
// times sc.
template <class T, int NPC>
__device__ __forceinline__ void store_operand(void* const* pc, int64_t kpad, int64_t n, int64_t v, int64_t i, float2 t,
                                              float2 b, float sc) {
  using PT = Piece<T>;
  t.x *= sc; t.y *= sc; b.x *= sc; b.y *= sc;
#pragma unroll
  for (int q = 0; q < NPC; ++q) {
    // each value is rounded once; the eight pairs are its pieces swapped and negated
    const T tx = PT::rn(t.x), ty = PT::rn(t.y), bx = PT::rn(b.x), by = PT::rn(b.y);
    const unsigned tt = PT::bits(PT::pair(tx, ty)), bb = PT::bits(PT::pair(bx, by));
    const unsigned ts = __byte_perm(tt, tt, 0x1032), bs = __byte_perm(bb, bb, 0x1032);
    unsigned* r = reinterpret_cast<unsigned*>(static_cast<T*>(pc[q]) + 4 * v * kpad) + i;  // kpad even
    const int64_t row = kpad / 2;
    r[0] = tt ^ 0x80000000u;
    r[n] = bb ^ 0x80000000u;
    r += row;
    r[0] = ts;
    r[n] = bs;
    r += row;
    r[0] = bb;
    r[n] = tt;
    r += row;
    r[0] = bs ^ 0x00008000u;
    r[n] = ts ^ 0x00008000u;
    t.x -= PT::back(tx);
    t.y -= PT::back(ty);
    b.x -= PT::back(bx);
    b.y -= PT::back(by);
  }
}

struct Maps {
  CUtensorMap a[3];
  CUtensorMap b[3];
};

// The end of one half tile: sums its partial tiles, undoes the scaling and runs the mode's epilogue for the 32 rows of TMEM lane quarter q and
// the groups of EB columns first, first + step, ...  It is a chain of L2 latencies, so the scales of
// four groups are prepared at a time and all loads of a group are in flight together.
constexpr int EB = 8;
// The n partial tiles of a half tile in K order: the first, and tile j of the others at
// rest + j * PART_STRIDE (one pair's two slots in both CTAs further).
constexpr size_t PART_STRIDE = (size_t)4 * BM * BNMAX;
struct Partials {
  const float* first;
  const float* rest;
  int n;
};
template <int SCH>
__device__ __forceinline__ void finish_jform(const Epi& ep, const Sched& sc, const Walk& wk, uint32_t rank, int q,
                                            int lane, int first, int step, const Partials& pt) {
  using T = typename Scheme<SCH>::T;
  const int row_t = q * 32 + lane;
  const int64_t row = (int64_t)(2 * wk.mt + (int)rank) * BM + row_t;
  const bool rvalid = row < ep.rows;
  const float rs = rvalid ? exp2i(-ep.prow[row]) : 0.0f;  // undo the row scaling of M
  const float hsign = ep.h2 ? 1.0f : -1.0f;               // H^2 = -M M
  const int64_t v0 = (int64_t)wk.nt * sc.bn;
  const int cols = (int)min((int64_t)wk.cols, ep.cols - v0);  // even
#pragma unroll 1
  for (int g0 = first; g0 * EB < cols; g0 += 4 * step) {
    // lane l prepares column l % 8 of group l / 8: the input column's scale (undone), the
    // output's, gamma
    const int pc = (g0 + (lane >> 3) * step) * EB + (lane & 7);
    float s_in = 0.0f, s_out = 0.0f, gmm = 0.0f;
    if (pc < cols) {
      const int64_t v = v0 + pc;
      const int ein = ep.vexp_in[v];
      if (ep.gamma) gmm = ep.gamma[v];
      if (ep.mode != 2) {
        const int e = out_exp(vec_bound(ep, v));
        s_out = exp2i(e);
        if (q == 0) ep.vexp_out[v] = e;  // the same value from every tile
      }
      s_in = exp2i(-ein);
    }
    unsigned amax = 0;
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {
      const int g = (g0 + t * step) * EB;
      if (g >= cols) break;
      const int left = cols - g;
      const int64_t vb = v0 + g;
      // loads at clamped rows and columns instead of under a predicate each
      const int64_t oz = vb * ep.rows + min(row, ep.rows - 1);
      const size_t off = (size_t)g * BM + row_t;
      float x[EB], zc[EB], zp[EB];
#pragma unroll
      for (int i = 0; i < EB; ++i) x[i] = __ldcg(pt.first + off + i * BM);
      if (ep.mode != 0) {
#pragma unroll
        for (int i = 0; i < EB; ++i) zc[i] = ep.Zcur[oz + (i < left ? i : 0) * ep.rows];
      }
      if (ep.mode == 1 && ep.beta != 0.0f) {
#pragma unroll
        for (int i = 0; i < EB; ++i) zp[i] = ep.Zprev[oz + (i < left ? i : 0) * ep.rows];
      }
#pragma unroll 1
      for (int j = 1; j < pt.n; j += 3) {
        float y[3][EB];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
          for (int i = 0; i < EB; ++i) y[p][i] = __ldcg(pt.rest + off + min(j + p, pt.n - 1) * PART_STRIDE + i * BM);
#pragma unroll
        for (int p = 0; p < 3; ++p)
          if (j + p < pt.n) {
#pragma unroll
            for (int i = 0; i < EB; ++i) x[i] += y[p][i];
          }
      }
#pragma unroll
      for (int i = 0; i < EB; ++i) x[i] *= rs * __shfl_sync(0xffffffffu, s_in, t * EB + i);
      if (ep.mode == 1) {
#pragma unroll
        for (int i = 0; i < EB; ++i) x[i] = ep.alpha * (hsign * x[i] - ep.c * zc[i]);
        if (ep.beta != 0.0f) {
#pragma unroll
          for (int i = 0; i < EB; ++i) x[i] += ep.beta * zp[i];
        }
        if (ep.src) {
#pragma unroll
          for (int i = 0; i < EB; ++i) zc[i] = ep.src[oz + (i < left ? i : 0) * ep.rows];
#pragma unroll
          for (int i = 0; i < EB; ++i) x[i] += __shfl_sync(0xffffffffu, gmm, t * EB + i) * zc[i];
        }
      } else if (ep.mode == 2) {
        // H w + gamma w: the two columns of a vector trade places, a' = M c, c' = -M a
#pragma unroll
        for (int i = 0; i < EB; i += 2) {
          const float a = x[i];
          x[i] = x[i + 1] + __shfl_sync(0xffffffffu, gmm, t * EB + i) * zc[i];
          x[i + 1] = -a + __shfl_sync(0xffffffffu, gmm, t * EB + i + 1) * zc[i + 1];
        }
      }
#pragma unroll
      for (int i = 0; i < EB; ++i) {
        const bool lv = rvalid && i < left;
        const float so = __shfl_sync(0xffffffffu, s_out, t * EB + i);
        if (lv) {
          if (ep.mode != 2) put1<T, Scheme<SCH>::NPW>(ep.out, (vb + i) * ep.kpad + row, x[i] * so);
          if (ep.mode != 0) ep.Znext[oz + i * ep.rows] = x[i];
        }
        const unsigned mm = __reduce_max_sync(0xffffffffu, lv ? __float_as_uint(fabsf(x[i])) : 0u);
        if (lane == t * EB + i) amax = mm;
      }
    }
    if (pc < cols) atomicMax(reinterpret_cast<unsigned*>(ep.amax_out) + v0 + pc, amax);
  }
}

// The same for the blocks form: row i of the operand holds, per vector, top = P w (columns
// 4v, 4v + 1) and P u (4v + 2, 4v + 3), whose -conj (with the blocks of H^2, conj) is the bottom.
// A group of EB columns is two vectors.
template <int SCH>
__device__ __forceinline__ void finish_blocks(const Epi& ep, const Sched& sc, const Walk& wk, uint32_t rank, int q,
                                              int lane, int first, int step, const Partials& pt) {
  using T = typename Scheme<SCH>::T;
  const int row_t = q * 32 + lane;
  const int64_t row = (int64_t)(2 * wk.mt + (int)rank) * BM + row_t;
  const bool rvalid = row < ep.n;
  const float rs = rvalid ? exp2i(-ep.prow[row]) : 0.0f;  // undo the row scaling of the operand
  const int64_t v0 = (int64_t)wk.nt * (sc.bn / 4), n2 = 2 * ep.n, rc = min(row, ep.n - 1);
  const int vecs = (int)min((int64_t)(wk.cols / 4), ep.cols / 4 - v0);
#pragma unroll 1
  for (int g0 = first; 2 * g0 < vecs; g0 += 4 * step) {
    // lane l < 8 prepares vector l % 2 of group l / 2
    const int pv = 2 * (g0 + (lane >> 1) * step) + (lane & 1);
    const bool mine = lane < EB && pv < vecs;
    float s_in = 0.0f, s_out = 0.0f, gmm = 0.0f;
    if (mine) {
      const int64_t v = v0 + pv;
      const int ein = ep.vexp_in[v];
      if (ep.gamma) gmm = ep.gamma[v];
      if (ep.mode != 2) {
        const int e = out_exp(vec_bound(ep, v));
        s_out = exp2i(e);
        if (q == 0) ep.vexp_out[v] = e;  // the same value from every tile
      }
      s_in = exp2i(-ein);
    }
    unsigned amax = 0;
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {
      const int vb = 2 * (g0 + t * step);
      if (vb >= vecs) break;
      const size_t off = (size_t)(4 * vb) * BM + row_t;
      // masters of the group's two vectors (a missing second one reads the first)
      const int64_t o[2] = {(v0 + vb) * n2 + rc, (v0 + (vb + 1 < vecs ? vb + 1 : vb)) * n2 + rc};
      float x[EB];
      float2 zc[4], zp[4];
#pragma unroll
      for (int i = 0; i < EB; ++i) x[i] = __ldcg(pt.first + off + i * BM);
      if (ep.mode != 0) {
        const float2* Z = reinterpret_cast<const float2*>(ep.Zcur);
#pragma unroll
        for (int h = 0; h < 4; ++h) zc[h] = Z[o[h >> 1] + (h & 1) * ep.n];
      }
      if (ep.mode == 1 && ep.beta != 0.0f) {
        const float2* Z = reinterpret_cast<const float2*>(ep.Zprev);
#pragma unroll
        for (int h = 0; h < 4; ++h) zp[h] = Z[o[h >> 1] + (h & 1) * ep.n];
      }
#pragma unroll 1
      for (int j = 1; j < pt.n; j += 3) {
        float y[3][EB];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
          for (int i = 0; i < EB; ++i) y[p][i] = __ldcg(pt.rest + off + min(j + p, pt.n - 1) * PART_STRIDE + i * BM);
#pragma unroll
        for (int p = 0; p < 3; ++p)
          if (j + p < pt.n) {
#pragma unroll
            for (int i = 0; i < EB; ++i) x[i] += y[p][i];
          }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float vs = rs * __shfl_sync(0xffffffffu, s_in, 2 * t + u);
        const float so = __shfl_sync(0xffffffffu, s_out, 2 * t + u);
        const float gm = __shfl_sync(0xffffffffu, gmm, 2 * t + u);
        float2 z[2] = {make_float2(x[4 * u] * vs, x[4 * u + 1] * vs),
                       ep.h2 ? make_float2(x[4 * u + 2] * vs, -x[4 * u + 3] * vs)
                             : make_float2(-x[4 * u + 2] * vs, x[4 * u + 3] * vs)};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float2 c = zc[2 * u + h];
          if (ep.mode == 1) {
            z[h].x = ep.alpha * (z[h].x - ep.c * c.x);
            z[h].y = ep.alpha * (z[h].y - ep.c * c.y);
            if (ep.beta != 0.0f) {
              z[h].x += ep.beta * zp[2 * u + h].x;
              z[h].y += ep.beta * zp[2 * u + h].y;
            }
            if (ep.src) {
              const float2 r = reinterpret_cast<const float2*>(ep.src)[o[u] + h * ep.n];
              z[h].x += gm * r.x;
              z[h].y += gm * r.y;
            }
          } else if (ep.mode == 2) {
            z[h].x += gm * c.x;
            z[h].y += gm * c.y;
          }
        }
        const bool lv = rvalid && vb + u < vecs;
        if (lv) {
          if (ep.mode != 2) store_operand<T, Scheme<SCH>::NPW>(ep.out, ep.kpad, ep.n, v0 + vb + u, row, z[0], z[1], so);
          if (ep.mode != 0) {
            float2* Z = reinterpret_cast<float2*>(ep.Znext);
            Z[o[u]] = z[0];
            Z[o[u] + ep.n] = z[1];
          }
        }
        const float m = fmaxf(fmaxf(fabsf(z[0].x), fabsf(z[0].y)), fmaxf(fabsf(z[1].x), fabsf(z[1].y)));
        const unsigned mm = __reduce_max_sync(0xffffffffu, lv ? __float_as_uint(m) : 0u);
        if (lane == 2 * t + u) amax = mm;
      }
    }
    if (mine) atomicMax(reinterpret_cast<unsigned*>(ep.amax_out) + v0 + pv, amax);
  }
}
template <int SCH, int FORM>
__device__ __forceinline__ void finish_tile(const Epi& ep, const Sched& sc, const Walk& wk, uint32_t rank, int q,
                                            int lane, int first, int step, const Partials& pt) {
  if (FORM == FORM_J) finish_jform<SCH>(ep, sc, wk, rank, q, lane, first, step, pt);
  else finish_blocks<SCH>(ep, sc, wk, rank, q, lane, first, step, pt);
}

template <int SCH, int FORM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    tc_hop_kernel(const __grid_constant__ Maps maps, const __grid_constant__ Epi ep, const __grid_constant__ Sched sc) {
  using SC = Scheme<SCH>;
  using T = typename SC::T;
  const int FLUSH = FORM == FORM_J ? SC::FLUSH : sc.flush;  // a power of two
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RING_BYTES);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + MAX_ST);
  const uint32_t accf = smem_u32(bars + 2 * MAX_ST), acce = smem_u32(bars + 2 * MAX_ST + 2);  // two of each
  const uint32_t crossf = smem_u32(bars + 2 * MAX_ST + 4), crosse = smem_u32(bars + 2 * MAX_ST + 5);
  const uint32_t outf = smem_u32(bars + 2 * MAX_ST + 6), oute = smem_u32(bars + 2 * MAX_ST + 8);  // two of each
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NBAR);
  volatile int* abort_sh = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* issued_sh = reinterpret_cast<int*>(tmem_slot + 2);
  volatile int* last_sh = reinterpret_cast<volatile int*>(tmem_slot + 3);
  volatile int* last_epi_sh = reinterpret_cast<volatile int*>(tmem_slot + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1;
  const int ST = sc.stages;
  const int nb = sc.bufs;                             // x0 * y0 buffers, bn columns each
  const uint32_t cross = (uint32_t)(nb * sc.bn);      // the cross products' columns

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full0 + 8 * s, 1);   // CTA 0: its producer's expect_tx of both CTAs' bytes
      mbar_init(empty0 + 8 * s, 1);  // a commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf + 8 * b, 1);
      mbar_init(acce + 8 * b, 2 * DRAIN_WARPS);  // CTA 0: one arrival per drain warp of the pair
      mbar_init(outf + 8 * b, DRAIN_WARPS);
      mbar_init(oute + 8 * b, EPI_WARPS);
    }
    mbar_init(crossf, 1);
    mbar_init(crosse, 2 * DRAIN_WARPS);
    *abort_sh = 0;
    *issued_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t b_bytes = (uint32_t)(sc.bn / 2) * BK * 2;  // one piece of a stage's B half

  float* my_tiles = ep.part + (size_t)blockIdx.x * (2 * BM * BNMAX);
  // The partial tiles of the tail tile that wk is in: pairs c0 .. c1 hold its K ranges, c0 as its second
  // segment of the tail where it starts in the tile before, the others as their first.
  auto partials = [&](const Walk& wk) -> Partials {
    const int x = wk.tail_tile() * sc.nkb, c0 = sc.tail_owner(x), c1 = sc.tail_owner(x + sc.nkb - 1);
    const int slot = sc.waves & 1, slot0 = sc.rest * sc.nkb * c0 < x * sc.tail ? slot ^ 1 : slot;  // c0 starts before x
    const float* at = ep.part + (size_t)(4 * c0 + 2 * (int)rank) * (BM * BNMAX);
    return Partials{at + (size_t)slot0 * (BM * BNMAX), at + (size_t)slot * (BM * BNMAX), c1 - c0 + 1};
  };
  // Whether this CTA has written the last partial tile of its half of wk's tile (its drain warps
  // have fenced their writes); for N threads, all of which pass the barriers `bar`, `lead` among them.
  auto count_partial = [&](const Walk& wk, int bar, int N, int lead, volatile int* sh) -> bool {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(N) : "memory");
    if (threadIdx.x == lead) {
      int* cnt = ep.cnt + 2 * wk.tail_tile() + rank;
      const bool l = atomicAdd(cnt, 1) == partials(wk).n - 1;
      if (l) *cnt = 0;  // ready for the next launch
      *sh = l ? 1 : 0;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(N) : "memory");
    const bool last = *sh != 0;
    if (last) __threadfence();
    return last;
  };
  // A pair's last tile, for the drain and the finishing warps together: all of them pass the
  // barriers, also after a failed wait.  True where this CTA has the tile's last partial.
  auto final_tile = [&](bool ok, const Walk& wk) -> bool {
    constexpr int N = 32 * (DRAIN_WARPS + EPI_WARPS);
    bool last = true;
    if (wk.split()) {
      __threadfence();
      last = count_partial(wk, 1, N, 128, last_sh);
    } else {
      asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
    }
    return last && ok && __all_sync(0xffffffffu, *abort_sh == 0);  // warp-uniform
  };
  auto finish_final = [&](const Walk& wk, int slot, int third) {
    const float* mine = my_tiles + (size_t)slot * (BM * BNMAX);
    const Partials pt = wk.split() ? partials(wk) : Partials{mine, mine, 1};
    finish_tile<SCH, FORM>(ep, sc, wk, rank, warp & 3, lane, third, 3, pt);
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_ROLES));
    if (warp == 0 && lane == 0) {
      int issued = 0, s = 0;
      uint32_t ph = 0;
      const uint32_t lead = map_rank(full0, 0);
      bool ok = true;
      for (Walk wk(sc, pair); ok && wk.next();) {
        const int m0 = (2 * wk.mt + (int)rank) * BM, n0 = wk.nt * sc.bn + (int)rank * (wk.cols / 2);
        for (int kb = wk.kb0; kb < wk.kb1; ++kb) {
          if (issued >= ST && !mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_sh, ep.err, true)) {
            ok = false;
            break;
          }
          const uint32_t st = sbase + s * sc.stage_bytes;
          if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2 * sc.stage_bytes);
  #pragma unroll
          for (int q = 0; q < SC::NPA; ++q) tma_load_2d_pair(st + q * A_BYTES, &maps.a[q], kb * BK, m0, lead + 8 * s);
  #pragma unroll
          for (int q = 0; q < SC::NPW; ++q)
            tma_load_2d_pair(st + SC::NPA * A_BYTES + q * b_bytes, &maps.b[q], kb * BK, n0, lead + 8 * s);
          ++issued;
          if (++s == ST) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      *issued_sh = issued;
    } else if (warp == 1 && lane == 0 && rank == 0) {
      const uint64_t dbase = sdesc(sbase);
      int s = 0, b = 0, seg = 0;
      uint32_t ph = 0, accph = 1;  // the first pass over the buffers does not wait
      bool ok = true, used = false;
      for (Walk wk(sc, pair); ok && wk.next(); ++seg) {
        const uint32_t idesc = make_idesc(wk.cols, Piece<T>::BF16);
        for (int kb = wk.kb0; kb < wk.kb1; ++kb) {
          const int i = kb - wk.kb0;
          const bool first = (i & (FLUSH - 1)) == 0;
          const bool last = (i & (FLUSH - 1)) == FLUSH - 1 || kb == wk.kb1 - 1;
          if (!mbar_wait(full0 + 8 * s, ph, abort_sh, ep.err, true)) {
            ok = false;
            break;
          }
          // sdesc is linear in the address here (its 14-bit start field holds address / 16 of
          // a 1024-aligned ring below 256 KB and cannot carry): a hoisted base plus constants;
          // 16 K elements further along a swizzled row is 32 bytes further
          const uint64_t ad0 = dbase + (uint64_t)((uint32_t)(s * sc.stage_bytes) >> 4);
          const uint64_t bd0 = ad0 + (uint64_t)((SC::NPA * A_BYTES) >> 4);
          // x0 * y0 first, so that a finished buffer drains behind the cross products; but a new
          // buffer's x0 * y0 last, so that the drain has a second block's cross products to hide
          // behind (except at a tile's start, whose cross products wait for the previous drain)
          const bool big_last = first && i > 0;
          auto cross_products = [&]() {
  #pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
  #pragma unroll
              for (int pr = 1; pr < SC::NPROD; ++pr)
                mma_f16_pair(tmem + cross, ad0 + (uint64_t)((SC::pa(pr) * A_BYTES + kk * 32) >> 4),
                             bd0 + (uint64_t)((SC::pb(pr) * b_bytes + (uint32_t)(kk * 32)) >> 4), idesc,
                             (i > 0 || kk > 0 || pr > 1) ? 1u : 0u);
          };
          tc_fence_after();
          if (big_last) cross_products();
          if (first && used) {
            if (!mbar_wait(acce + 8 * b, accph, abort_sh, ep.err, true)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
  #pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_f16_pair(tmem + (uint32_t)(b * sc.bn), ad0 + (uint64_t)((kk * 32) >> 4),
                         bd0 + (uint64_t)((kk * 32) >> 4), idesc, (!first || kk > 0) ? 1u : 0u);
          if (last) {
            mma_commit_pair(accf + 8 * b);
            if (++b == nb) {
              b = 0;
              accph ^= 1u;
              used = true;
            }
          }
          if (i == 0 && seg > 0) {
            if (!mbar_wait(crosse, (uint32_t)(seg - 1) & 1u, abort_sh, ep.err, true)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
          if (!big_last) cross_products();
          mma_commit_pair(empty0 + 8 * s);
          if (++s == ST) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok) mma_commit_pair(crossf);
      }
    }
  } else if (warp < 4 + DRAIN_WARPS) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_DRAIN));
    const int dw = warp - 4;
    const int q = warp & 3;                  // TMEM lanes 32 q .. 32 q + 31 (rows of the half tile)
    const int col0 = (dw >> 2) * sc.dcols;   // this warp's columns [col0, col0 + dcols)
    const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
    const uint32_t acce0 = map_rank(acce, 0), crosse0 = map_rank(crosse, 0);
    int b = 0, seg = 0;
    uint32_t accph = 0;
    bool ok = true;
    // after a failed wait a warp walks on without waiting, for the named barriers' sake
    for (Walk wk(sc, pair); wk.next(); ++seg) {
      const int cols = min(sc.dcols, wk.cols - col0);  // may be <= 0
      float sum[DC];
#pragma unroll
      for (int i = 0; i < DC; ++i) sum[i] = 0.0f;
      const int ngrp = (wk.kb1 - wk.kb0 + FLUSH - 1) / FLUSH;
      for (int g = 0; ok && g < ngrp; ++g) {
        const bool w = mbar_wait(accf + 8 * b, accph, abort_sh, ep.err, true);
        if (!__all_sync(0xffffffffu, w)) {  // warp-uniform (tcgen05.ld is .sync.aligned)
          ok = false;
          break;
        }
        tc_fence_after();
        drain_add(tcol + (uint32_t)(b * sc.bn), cols, sum);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acce0 + 8 * b);
        if (++b == nb) {
          b = 0;
          accph ^= 1u;
        }
      }
      if (ok) {
        const bool w = mbar_wait(crossf, (uint32_t)seg & 1u, abort_sh, ep.err, true);
        ok = __all_sync(0xffffffffu, w);
      }
      if (ok) {
        tc_fence_after();
        drain_add(tcol + cross, cols, sum);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(crosse0);
      }
      // the tile into its workspace slot, once the tile before the last is finished
      const int slot = seg & 1;
      if (ok && seg >= 2) {
        const bool w = mbar_wait(oute + 8 * slot, (uint32_t)((seg >> 1) - 1) & 1u, abort_sh, ep.err, true);
        ok = __all_sync(0xffffffffu, w);
      }
      if (ok) {
        float* mine = my_tiles + (size_t)slot * (BM * BNMAX) + (size_t)col0 * BM + q * 32 + lane;
#pragma unroll
        for (int c = 0; c < DC; ++c)
          if ((c & ~15) < cols) __stcg(mine + c * BM, sum[c]);
      }
      if (wk.final()) {
        if (final_tile(ok, wk)) finish_final(wk, slot, 1 + (dw >> 2));
      } else {
        if (wk.split()) __threadfence();
        __syncwarp();
        if (lane == 0) mbar_arrive(outf + 8 * slot);
      }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_EPI));
    bool ok = true;
    int seg = 0;
    for (Walk wk(sc, pair); wk.next(); ++seg) {
      const int slot = seg & 1;
      if (wk.final()) {
        if (final_tile(ok, wk)) finish_final(wk, slot, 0);
        continue;
      }
      if (ok) {
        const bool w = mbar_wait(outf + 8 * slot, (uint32_t)(seg >> 1) & 1u, abort_sh, ep.err, true);
        ok = __all_sync(0xffffffffu, w);
      }
      const float* mine = my_tiles + (size_t)slot * (BM * BNMAX);
      Partials pt{mine, mine, 1};
      bool last = true;
      if (wk.split()) {  // the first of a pair's two K ranges of the tail
        last = count_partial(wk, 2, 32 * EPI_WARPS, 32 * (4 + DRAIN_WARPS), last_epi_sh);
        pt = partials(wk);
      }
      if (ok && last) finish_tile<SCH, FORM>(ep, sc, wk, rank, warp & 3, lane, 0, 1, pt);
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(oute + 8 * slot);
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // every MMA of the pair has been drained, or a wait has run out
  if (threadIdx.x == 0 && *abort_sh) {
    // copies and MMAs still in flight on the pair's shared memory and TMEM (bounded): CTA 0's
    // barriers count both CTAs' bytes
    if (rank == 0) {
      const int issued = *issued_sh;
      for (int i = max(0, issued - ST); i < issued; ++i)
        mbar_wait(full0 + 8 * (i % ST), (uint32_t)(i / ST) & 1u, abort_sh, ep.err, false);
    }
    const uint64_t t0 = gtimer();
    while (gtimer() - t0 < COPY_LIMIT_NS) __nanosleep(1000);
  }
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------- helpers
struct Pieces {
  void* p[3];
};

// block-wide max and sum of one value per thread (blockDim.x a multiple of 32, <= 1024)
__device__ __forceinline__ void block_max_sum(float& m, float& s) {
  __shared__ float wm[32], ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if (lane == 0) {
    wm[w] = m;
    ws[w] = s;
  }
  __syncthreads();
  if (w == 0) {
    m = lane < nw ? wm[lane] : 0.0f;
    s = lane < nw ? ws[lane] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    if (lane == 0) {
      wm[0] = m;
      ws[0] = s;
    }
  }
  __syncthreads();
  m = wm[0];
  s = ws[0];
}

// The real form of [A | B] (row-major complex128) -> NPC pieces, one CTA per row i of A and B,
// which gives rows 2i and 2i + 1; TWIST 1: M above (z -> -i (A z + B conj z)), 0: the plain
// z -> A z + B conj z.  Row r is scaled by 2^prow[r] (its largest entry in [2^12, 2^13)); L
// receives the largest row sum of absolute values (unscaled), the bound factor of an
// application.  Columns 2n .. kpad are zero.  The FP64 additions (4 an entry of A and B) bound it, so
// with CACHE their rounded results wait in shared memory (16 n bytes) for the row's exponent
// instead of being formed again: n = 4096 a
// degree-20 filter 8.2 -> 7.96 ms.
template <int TWIST>
__device__ __forceinline__ void real_form(cplx a, cplx b, float2& r0, float2& r1) {
  const float2 re = make_float2((float)(a.x + b.x), (float)(b.y - a.y));  // Re: (Re z, Im z) coefficients
  const float2 im = make_float2((float)(a.y + b.y), (float)(a.x - b.x));  // Im
  r0 = TWIST ? im : re;
  r1 = TWIST ? make_float2(-re.x, -re.y) : im;
}
template <class T, int NPC, int TWIST, bool CACHE>
__global__ void split_p_kernel(const cplx* A, const cplx* B, int64_t n, int64_t kpad, Pieces out, int* prow,
                               float* L) {
  extern __shared__ float4 row_cache[];
  const int64_t i = blockIdx.x;
  float m0 = 0.0f, m1 = 0.0f, s0 = 0.0f, s1 = 0.0f;
  float2 r0, r1;
#pragma unroll 4
  for (int64_t l = threadIdx.x; l < n; l += blockDim.x) {
    real_form<TWIST>(A[i * n + l], B[i * n + l], r0, r1);
    if (CACHE) row_cache[l] = make_float4(r0.x, r0.y, r1.x, r1.y);  // read back by this thread
    m0 = fmaxf(m0, fmaxf(fabsf(r0.x), fabsf(r0.y)));
    m1 = fmaxf(m1, fmaxf(fabsf(r1.x), fabsf(r1.y)));
    s0 += fabsf(r0.x) + fabsf(r0.y);
    s1 += fabsf(r1.x) + fabsf(r1.y);
  }
  block_max_sum(m0, s0);
  __syncthreads();
  block_max_sum(m1, s1);
  const int e0 = out_exp(m0), e1 = out_exp(m1);
  if (threadIdx.x == 0) {
    prow[2 * i] = e0;
    prow[2 * i + 1] = e1;
    atomicMax(reinterpret_cast<unsigned*>(L), __float_as_uint(fmaxf(s0, s1)));
  }
  const float c0 = exp2i(e0), c1 = exp2i(e1);
  for (int64_t l = threadIdx.x; 2 * l < kpad; l += blockDim.x) {
    r0 = r1 = make_float2(0.0f, 0.0f);
    if (CACHE && l < n) {
      const float4 v = row_cache[l];
      r0 = make_float2(v.x, v.y);
      r1 = make_float2(v.z, v.w);
    } else if (l < n) {
      real_form<TWIST>(A[i * n + l], B[i * n + l], r0, r1);
    }
    put<T, NPC>(out.p, (2 * i) * kpad + 2 * l, r0.x * c0, r0.y * c0);
    put<T, NPC>(out.p, (2 * i + 1) * kpad + 2 * l, r1.x * c1, r1.y * c1);
  }
}
// The rows of [A | B] (row-major complex128) as (re, im) pairs -> NPC pieces, one CTA per row,
// scaled by 2^prow[i] (largest entry in [2^12, 2^13)); L as above; columns 4n .. kpad are zero.
// CACHE: the FP32 entries (16 n bytes) wait in shared memory for the row's exponent.
template <class T, int NPC, bool CACHE>
__global__ void split_blocks_kernel(const cplx* A, const cplx* B, int64_t n, int64_t kpad, Pieces out, int* prow,
                                    float* L) {
  extern __shared__ float4 row_cache[];
  const int64_t i = blockIdx.x;
  float m = 0.0f, sum = 0.0f;
  auto load = [&](int64_t l) {
    const cplx a = A[i * n + l], b = B[i * n + l];
    return make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
  };
#pragma unroll 4
  for (int64_t l = threadIdx.x; l < n; l += blockDim.x) {
    const float4 v = load(l);
    if (CACHE) row_cache[l] = v;  // read back by this thread
    m = fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
    sum += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
  }
  block_max_sum(m, sum);
  const int e = out_exp(m);
  if (threadIdx.x == 0) {
    prow[i] = e;
    atomicMax(reinterpret_cast<unsigned*>(L), __float_as_uint(sum));
  }
  const float c = exp2i(e);
  for (int64_t l = threadIdx.x; l < n; l += blockDim.x) {
    const float4 v = CACHE ? row_cache[l] : load(l);
    put<T, NPC>(out.p, i * kpad + 2 * l, v.x * c, v.y * c);
    put<T, NPC>(out.p, i * kpad + 2 * (n + l), v.z * c, v.w * c);
  }
  for (int64_t l = 4 * n + 2 * threadIdx.x; l < kpad; l += 2 * blockDim.x) put<T, NPC>(out.p, i * kpad + l, 0.0f, 0.0f);
}
// amax[v] = largest |Re|, |Im| of column v of W, rounded to FP32, and its operand exponent
__global__ void col_amax_blocks_kernel(const cplx* W, int64_t n, float* amax, int* vexp) {
  const int64_t v = blockIdx.x;
  float m = 0.0f, unused = 0.0f;
  for (int64_t i = threadIdx.x; i < 2 * n; i += blockDim.x) {
    const cplx w = W[v * 2 * n + i];
    m = fmaxf(m, fmaxf(fabsf((float)w.x), fabsf((float)w.y)));
  }
  block_max_sum(m, unused);
  if (threadIdx.x == 0) {
    amax[v] = m;
    vexp[v] = out_exp(m);
  }
}
// complex128 block (2n x k) -> FP32 masters and operand pieces (exponents vexp)
template <class T, int NPC>
__global__ void pack_blocks_kernel(const cplx* W, int64_t n, int64_t k, float2* Z, Pieces out, int64_t kpad,
                                   const int* vexp) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, v = idx / n, o = v * 2 * n + i;
    const cplx x = W[o], y = W[o + n];
    const float2 t = make_float2((float)x.x, (float)x.y), b = make_float2((float)y.x, (float)y.y);
    Z[o] = t;
    Z[o + n] = b;
    store_operand<T, NPC>(out.p, kpad, n, v, i, t, b, exp2i(vexp[v]));
  }
}
// Z = scale * X (masters) and its operand pieces, as scale_pack_kernel
template <class T, int NPC>
__global__ void scale_pack_blocks_kernel(const float2* X, int64_t n, int64_t k, float scale, float2* Z, Pieces out,
                                         int64_t kpad, const float* amax_x, float* amax_z, int* vexp_z) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, v = idx / n, o = v * 2 * n + i;
    const float am = fabsf(scale) * amax_x[v];
    const int e = out_exp(am);
    if (i == 0) {
      amax_z[v] = am;
      vexp_z[v] = e;
    }
    const float2 x = X[o], y = X[o + n];
    const float2 t = make_float2(scale * x.x, scale * x.y), b = make_float2(scale * y.x, scale * y.y);
    Z[o] = t;
    Z[o + n] = b;
    store_operand<T, NPC>(out.p, kpad, n, v, i, t, b, exp2i(e));
  }
}
// out[:, v] = the master of vector v in Zsel, in FP64, + coef[v] * base[:, v] (coef/base optional)
__global__ void combine_blocks_kernel(cplx* out, const float2* Z0, const float2* Z1, const float2* Z2, const int* sel,
                                      const double* coef, const cplx* base, int64_t n2, int64_t k) {
  const int64_t total = n2 * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = idx / n2;
    const int q = sel[v];
    const float2 z = (q == 0 ? Z0 : (q == 1 ? Z1 : Z2))[idx];
    cplx r = mk((double)z.x, (double)z.y);
    if (coef) r = cadd(r, cscale(base[idx], coef[v]));
    out[idx] = r;
  }
}
// The halves a and c of w = [x; y]; and w from them
__device__ __forceinline__ void j_split(cplx x, cplx y, float2& a, float2& c) {
  a = make_float2((float)(0.5 * (x.x + y.x)), (float)(0.5 * (x.y - y.y)));
  c = make_float2((float)(-0.5 * (x.y + y.y)), (float)(0.5 * (x.x - y.x)));
}
// amax[2v], amax[2v + 1] = largest |entry| of the halves of column v of the complex128 block
// W (2n x k), rounded to FP32, and vexp their operand exponents; one CTA per column
__global__ void col_amax_kernel(const cplx* W, int64_t n, float* amax, int* vexp) {
  const int64_t v = blockIdx.x;
  float m0 = 0.0f, m1 = 0.0f, unused = 0.0f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    float2 a, c;
    j_split(W[v * 2 * n + i], W[v * 2 * n + n + i], a, c);
    m0 = fmaxf(m0, fmaxf(fabsf(a.x), fabsf(a.y)));
    m1 = fmaxf(m1, fmaxf(fabsf(c.x), fabsf(c.y)));
  }
  block_max_sum(m0, unused);
  __syncthreads();
  block_max_sum(m1, unused);
  if (threadIdx.x == 0) {
    amax[2 * v] = m0;
    amax[2 * v + 1] = m1;
    vexp[2 * v] = out_exp(m0);
    vexp[2 * v + 1] = out_exp(m1);
  }
}
// complex128 block (2n x k) -> FP32 columns (2n x 2k) and their operand pieces (exponents
// vexp), zero in the entries 2n .. kpad
template <class T, int NPC>
__global__ void pack_kernel(const cplx* W, int64_t n, int64_t k, float2* Z, Pieces out, int64_t kpad,
                            const int* vexp) {
  const int64_t half = kpad / 2, total = half * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % half, v = idx / half;
    float2 a = make_float2(0.0f, 0.0f), c = a;
    if (i < n) {
      j_split(W[v * 2 * n + i], W[v * 2 * n + n + i], a, c);
      Z[2 * v * n + i] = a;
      Z[(2 * v + 1) * n + i] = c;
    }
    const float sa = exp2i(vexp[2 * v]), sc = exp2i(vexp[2 * v + 1]);
    put<T, NPC>(out.p, 2 * v * kpad + 2 * i, a.x * sa, a.y * sa);
    put<T, NPC>(out.p, (2 * v + 1) * kpad + 2 * i, c.x * sc, c.y * sc);
  }
}
// Z = scale * X (FP32 columns) and its operand pieces; the largest entry of column v
// is |scale| amax_x[v] (up to rounding), which sets its exponent
template <class T, int NPC>
__global__ void scale_pack_kernel(const float2* X, int64_t n, int64_t k2, float scale, float2* Z, Pieces out,
                                  int64_t kpad, const float* amax_x, float* amax_z, int* vexp_z) {
  const int64_t total = n * k2;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, v = idx / n;
    const float am = fabsf(scale) * amax_x[v];
    const int e = out_exp(am);
    if (i == 0) {
      amax_z[v] = am;
      vexp_z[v] = e;
    }
    const float2 x = X[idx], z = make_float2(scale * x.x, scale * x.y);
    const float sz = exp2i(e);
    Z[idx] = z;
    put<T, NPC>(out.p, v * kpad + 2 * i, z.x * sz, z.y * sz);
  }
}
// out[:, v] = the vector of the halves in columns 2v, 2v + 1 of Zsel, in FP64,
// + coef[v] * base[:, v]   (coef/base optional)
__global__ void combine_kernel(cplx* out, const float2* Z0, const float2* Z1, const float2* Z2, const int* sel,
                               const double* coef, const cplx* base, int64_t n, int64_t k) {
  const int64_t total = n * k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, v = idx / n;
    const int q = sel[v];
    const float2* Z = q == 0 ? Z0 : (q == 1 ? Z1 : Z2);
    const float2 a = Z[2 * v * n + i], c = Z[(2 * v + 1) * n + i];
    cplx x = mk((double)a.x + (double)c.y, (double)a.y - (double)c.x);   // a - i c
    cplx y = mk((double)a.x - (double)c.y, -(double)a.y - (double)c.x);  // conj(a) - i conj(c)
    const int64_t o = v * 2 * n + i;
    if (coef) {
      x = cadd(x, cscale(base[o], coef[v]));
      y = cadd(y, cscale(base[o + n], coef[v]));
    }
    out[o] = x;
    out[o + n] = y;
  }
}

// Tensor map of a piece plane (rows x kpad, K contiguous) with boxes of BK x box_rows and
// 128-byte swizzle; rows of a box beyond the plane read as zero.
static int make_map(CUtensorMap* m, const void* base, int64_t kpad, int64_t rows, int box_rows, bool bf16) {
  auto fn = encode_fn();
  if (!fn) return CHASE_BSE_UNSUPPORTED;
  const cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)kpad * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                  const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? CHASE_BSE_OK : CHASE_BSE_CUDA_ERROR;
}

static inline unsigned gsz(int64_t total) {
  const int64_t b = (total + 255) / 256;
  return (unsigned)std::min<int64_t>(std::max<int64_t>(b, 1), 16384);
}

// The operand of A and B in NPA pieces, with its tensor maps, row exponents and the
// bound factor L (device scalar).
constexpr size_t CACHE_MAX = 220 * 1024;  // shared memory for a row's FP32 entries
struct POperand {
  int64_t n = 0, rows = 0, kpad = 0;
  Pieces pc{};
  CUtensorMap map[3];
  int* prow = nullptr;
  float* L = nullptr;
};

template <int SCH, int FORM, int TWIST>
static int prepare_p(const cplx* A, const cplx* B, int64_t n, Workspace& ws, POperand& P, cudaStream_t s) {
  using T = typename Scheme<SCH>::T;
  constexpr int NPA = Scheme<SCH>::NPA;
  P.n = n;
  P.rows = Form<FORM>::ROWS * n;
  P.kpad = ((Form<FORM>::KEL * n + KPAD - 1) / KPAD) * KPAD;
  for (int q = 0; q < NPA; ++q) {
    T* pq;
    CB_TRY(ws.alloc(&pq, P.rows * P.kpad));
    P.pc.p[q] = pq;
  }
  CB_TRY(ws.alloc(&P.prow, P.rows));
  CB_TRY(ws.alloc(&P.L, 1));
  CB_CUDA(cudaMemsetAsync(P.L, 0, sizeof(float), s));
  const size_t cache = sizeof(float4) * (size_t)n;
  void (*kern)(const cplx*, const cplx*, int64_t, int64_t, Pieces, int*, float*);
  // as many threads an SM where only one or two rows fit it
  const int threads = cache > 72 * 1024 && cache <= CACHE_MAX ? 512 : 256;
  if (cache <= CACHE_MAX) {
    if (FORM == FORM_J) kern = split_p_kernel<T, NPA, TWIST, true>;
    else kern = split_blocks_kernel<T, NPA, true>;
    static bool attr = false;
    if (!attr) {
      CB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CACHE_MAX));
      attr = true;
    }
    kern<<<(unsigned)n, threads, cache, s>>>(A, B, n, P.kpad, P.pc, P.prow, P.L);
  } else {
    if (FORM == FORM_J) kern = split_p_kernel<T, NPA, TWIST, false>;
    else kern = split_blocks_kernel<T, NPA, false>;
    kern<<<(unsigned)n, threads, 0, s>>>(A, B, n, P.kpad, P.pc, P.prow, P.L);
  }
  count_launch();
  CB_LAUNCH();
  for (int q = 0; q < NPA; ++q) CB_TRY(make_map(&P.map[q], P.pc.p[q], P.kpad, P.rows, BM, Piece<T>::BF16));
  return CHASE_BSE_OK;
}

// Cycles of one K block of a 256 x w tile in a launch of bn-wide tiles with a share `active` of the
// pairs at work: the MMAs (w / 2 each), the shared-memory traffic at 128 bytes a cycle (operand
// reads and the ring's fill), or 0.027 cycles a byte of a stage, a fit to what a K block was
// measured to take with all pairs busy (0.8-0.85 us for tiles of 160 and of 192 columns at n = 4096,
// whose MMAs take 0.5 and 0.6 at the top clock; the tensor pipe is active in 56-59 % of the cycles
// and L2 at 29 % of its rate, and replacing half of B's loads by multicasts between two pairs or
// alternating the accumulators changed nothing, so what the rest is has not been shown).  It
// favours wide tiles: n = 6000, k = 100 225 -> 182 us a launch in J form, n = 8192, k = 300 786 -> 704 us
// against a choice by the other two terms.
// Blocks form: a K block takes no less than 1400 cycles however narrow the tile (n = 1301, tiles of
// 32 to 160 columns in one K range: 78 to 88 us a launch, 82 blocks).
template <int SCH, int FORM>
static double block_cycles(int w, int bn, double active) {
  using SC = Scheme<SCH>;
  constexpr int MMAS = SC::NPROD * (BK / 16);
  const double mma = MMAS * (w / 2.0), stage = SC::NPA * A_BYTES + SC::NPW * 64.0 * bn;
  const double smem = (MMAS * (4096.0 + 16.0 * w) + stage) / 128.0;
  const double t = std::max(std::max(mma, smem), 0.027 * stage * std::max(active, 0.5));
  return FORM == FORM_J ? t : std::max(t, 1400.0);
}
// Cycles to finish a pair's last tile behind its MMAs, summing `parts` partial tiles: three sets of
// warps take its groups of 8 columns in turn, each a chain of L2 latencies (2 us, and 0.7 us for
// every three partial tiles more; n = 700 to 1301), and a cut tile is counted (n = 74, k = 8 in one
// K range 0.94, in two 0.98 ms a degree-28 filter).  The J form's choices rest on a constant fitted
// with the rest of its terms.
template <int FORM>
static double finish_cycles(int bn, int parts) {
  if (FORM == FORM_J) return parts > 1 ? 9000.0 + (parts + 1) * 8.0 * bn : 6000.0;
  return 10000.0 + (double)cdiv(bn, 3 * EB) * (3900.0 + 1350.0 * (double)cdiv(parts - 1, 3)) +
         (parts > 1 ? 1500.0 : 0.0);
}
// The schedule of a launch with m rows, k2 columns and nkb K blocks: of the column widths
// (multiples of 32) that ceil(k2 / 256) to 3 more column tiles need, and of the ways to cut the
// tiles left after the full waves into K ranges, the choice of least estimated time.
template <int SCH, int FORM>
static Sched plan(int64_t m, int64_t k2, int nkb, int pairs) {
  using SC = Scheme<SCH>;
  Sched best{};
  double best_t = 0.0;
  const int n0 = (int)cdiv(k2, BNMAX);
  for (int nn = n0; nn <= n0 + 3; ++nn) {
    Sched sc{};
    sc.nkb = nkb;
    sc.num_m = (int)cdiv(m, 2 * BM);
    sc.bn = (int)cdiv(cdiv(k2, nn), 32) * 32;
    sc.num_n = (int)cdiv(k2, sc.bn);
    if (sc.num_n != nn) continue;
    sc.n_last = (int)cdiv(k2 - (int64_t)(nn - 1) * sc.bn, 32) * 32;
    sc.stage_bytes = SC::NPA * A_BYTES + SC::NPW * (sc.bn / 2) * BK * 2;
    sc.stages = std::min(MAX_ST, RING_BYTES / sc.stage_bytes);
    sc.dcols = (int)cdiv(sc.bn, BNMAX / DC * 16) * 16;  // half of the tile, whole TMEM loads
    sc.bufs = 3 * sc.bn <= (int)TMEM_COLS ? 2 : 1;
    sc.group_m = 8;
    // narrow tiles of an operand that streams from HBM wait for their drains (n = 16384, k = 20
    // 833 us a launch drained every four K blocks, 901 every two)
    const bool streamed = sc.bn <= 128 && (double)m * nkb * BK * 4.0 > 126e6;
    // and with three pieces the FP32 additions of a long sum outweigh the truncation again (lower
    // halves at n = 4096, k = 260 3.9e-6, drained every K block 4.8e-6)
    sc.flush = streamed || (SC::NPA == 3 && nkb > 224) ? SC::FLUSH : SC::FLUSH_BLOCKS;
    const int64_t tiles = (int64_t)sc.num_m * nn;
    sc.pairs = pairs;
    sc.waves = (int)(tiles / pairs);
    sc.rest = (int)(tiles % pairs);
    const double full = block_cycles<SCH, FORM>(sc.bn, sc.bn, 1.0);
    const double avg = (full * (nn - 1) + block_cycles<SCH, FORM>(sc.n_last, sc.bn, 1.0)) / nn;
    const double fixed = 6000.0;  // prologue and epilogue of a tile in the full waves
    const double base = sc.waves * ((sc.waves > 1 ? avg : full) * nkb + fixed);
    auto consider = [&](int tail, double t) {
      if (best_t == 0.0 || base + t < best_t) {
        best = sc;
        best.tail = tail;
        best_t = base + t;
      }
    };
    if (sc.rest == 0) consider(0, 0.0);
    for (int f = 1; sc.rest > 0 && (f == 1 || (f * sc.rest <= pairs && nkb / f >= 2)); ++f)
      consider(f * sc.rest, std::ceil((double)nkb / f) *
                                    block_cycles<SCH, FORM>(sc.bn, sc.bn, (double)(f * sc.rest) / pairs) +
                                finish_cycles<FORM>(sc.bn, f));
    // blocks form: the tail's K blocks over all pairs, where a pair's range may cross from one tile
    // into the next (about 2000 cycles more for its second segment).  Equal parts of each tile leave
    // pairs idle where twice or thrice the tiles just miss their number: n = 4956, k = 79 (40 tiles of 76 pairs)
    // 278 -> 189 us a launch, n = 8100, k = 30 237 -> 210, n = 16384, k = 20 854 -> 731.
    const int64_t tail_blocks = (int64_t)sc.rest * nkb;
    if (FORM == FORM_BLOCKS && tail_blocks >= 4 * (int64_t)pairs)
      consider(pairs, std::ceil((double)tail_blocks / pairs) * block_cycles<SCH, FORM>(sc.bn, sc.bn, 1.0) +
                          finish_cycles<FORM>(sc.bn, pairs / sc.rest + 2) + 2000.0);
  }
  return best;
}

// One tensor-core application of M to the columns held in the operand pieces bp (rows
// columns allocated), with epilogue `ep`.
template <int SCH, int FORM>
static int apply(const POperand& P, const Pieces& bp, int64_t rows, Epi ep, cudaStream_t s) {
  using T = typename Scheme<SCH>::T;
  if (ep.cols <= 0) return CHASE_BSE_OK;
  static bool attr = false;
  if (!attr) {
    CB_CUDA(cudaFuncSetAttribute(tc_hop_kernel<SCH, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
    attr = true;
  }
  ep.prow = P.prow;
  ep.L = P.L;
  const Sched sc = plan<SCH, FORM>(ep.rows, ep.cols, (int)(P.kpad / BK), ep.sms / 2);
  Maps maps;
  for (int q = 0; q < Scheme<SCH>::NPA; ++q) maps.a[q] = P.map[q];
  for (int q = 0; q < Scheme<SCH>::NPW; ++q)
    CB_TRY(make_map(&maps.b[q], bp.p[q], P.kpad, rows, sc.bn / 2, Piece<T>::BF16));
  const unsigned grid = 2u * (unsigned)(sc.waves > 0 ? sc.pairs : sc.tail);
  const int64_t tid = timer_begin(0, 32.0 * (double)P.n * (double)P.n * (double)(ep.cols / Form<FORM>::COLS), s);
  tc_hop_kernel<SCH, FORM><<<grid, THREADS, SMEM_BYTES, s>>>(maps, ep, sc);
  timer_end(tid, s);
  count_launch();
  CB_LAUNCH();
  return CHASE_BSE_OK;
}

// Mixed-precision filter on columns sorted by descending degree.  If `ritz` and
// `R` are given, the filter runs in correction form: with m_i = ritz_i^2 and
// r2_i = (H^2 - m_i) v_i = (H + ritz_i)(H v_i - ritz_i v_i),
//   p(H^2) v_i = p(m_i) v_i + q(H^2) r2_i,  q(x) = (p(x) - p(m_i)) / (x - m_i),
// and only q(H^2) r2 runs on the tensor cores; its recurrence is the filter's
// with the source term alpha_j p_j(m_i) r2_i (divided differences of the
// three-term recurrence).  The low-precision error then scales with the
// residual of v_i instead of with v_i.
//
// With P2, Q2 (the blocks of H^2 = [[P2, Q2], [conj Q2, conj P2]], row-major n x n) the
// filter applies H^2 from its blocks, one launch per step (the explicit-H^2 variant, not
// the paper's method); H itself (A, B) is then used only for the correction source.
template <int SCH, int FORM>
static int filter_impl(const cplx* A, const cplx* B, int64_t n, const cplx* Y0, int64_t k, const int* degs,
                       double mu1, double mu_nevex, double muN, cplx* out, const double* ritz, const cplx* R,
                       cudaStream_t s, FilterStats* fs, const cplx* P2, const cplx* Q2) {
  using T = typename Scheme<SCH>::T;
  using F = Form<FORM>;
  constexpr int NPW = Scheme<SCH>::NPW;
  constexpr bool J = FORM == FORM_J;
  if (k == 0) return CHASE_BSE_OK;
  const int64_t n2 = 2 * n;
  const bool expl = P2 != nullptr && Q2 != nullptr;
  const bool corr = (ritz != nullptr && R != nullptr);
  Workspace ws(s);
  POperand P, PH2;  // [A | B] (H), [P2 | Q2] (H^2)
  if (!expl || corr) CB_TRY((prepare_p<SCH, FORM, 1>(A, B, n, ws, P, s)));
  if (expl) CB_TRY((prepare_p<SCH, FORM, 0>(P2, Q2, n, ws, PH2, s)));
  const POperand& PK = expl ? PH2 : P;  // the operand of the recurrence (its kpad and pieces layout)
  const int64_t kpad = PK.kpad, rows = PK.rows;  // the same for both operands
  const int64_t nc = F::COLS * k, ns = F::SCALES * k;  // columns, scales
  Pieces Zp{}, Tp{};
  for (int q = 0; q < NPW; ++q) {
    T *zq, *tq;
    CB_TRY(ws.alloc(&zq, nc * kpad));
    CB_TRY(ws.alloc(&tq, nc * kpad));
    Zp.p[q] = zq;
    Tp.p[q] = tq;
    const int64_t ke = F::KEL * n;
    if (kpad > ke) {  // zero past the entries of a column, as past those of an operand row
      CB_CUDA(cudaMemset2DAsync(zq + ke, sizeof(T) * kpad, 0, sizeof(T) * (kpad - ke), nc, s));
      CB_CUDA(cudaMemset2DAsync(tq + ke, sizeof(T) * kpad, 0, sizeof(T) * (kpad - ke), nc, s));
    }
  }
  // explicit H^2: the pieces of Z_j alternate between the two sets (j even: Zp)
  Pieces* zbuf[2] = {&Zp, &Tp};
  float *Zb[3], *src = nullptr;
  float* gam;
  int* err;
  for (int q = 0; q < 3; ++q) CB_TRY(ws.alloc(&Zb[q], 2 * n2 * k));
  CB_TRY(ws.alloc(&gam, ns));
  auto c2 = [](float* z) { return reinterpret_cast<float2*>(z); };
  CB_TRY(ws.alloc(&err, 1));
  CB_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
  // (partial) tiles, two per CTA, and a counter per half of a split tile
  int dev = 0, sms = 0;
  CB_CUDA(cudaGetDevice(&dev));
  CB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  float* part;
  int* cnt;
  CB_TRY(ws.alloc(&part, (int64_t)sms * 2 * BM * BNMAX));
  CB_TRY(ws.alloc(&cnt, sms));
  CB_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * sms, s));
  auto sk = [&](Epi& e) {
    e.part = part;
    e.cnt = cnt;
    e.sms = sms;
  };

  const double a = mu_nevex * mu_nevex, b = muN * muN;
  const double c = 0.5 * (a + b), e = 0.5 * (b - a);
  const double sigma1 = e / (mu1 * mu1 - c);
  const double tau = 2.0 / sigma1;
  const int maxdeg = degs[0];
  // per-column maxima and operand exponents, one slot of ns entries per block:
  // Z_j (j = 0 .. maxdeg), T_j = H Z_j (j < maxdeg), the residual block R and the
  // correction source r2
  const int64_t nslot = 2 * (int64_t)maxdeg + 3;
  float* amax;
  int* vexp;
  CB_TRY(ws.alloc(&amax, nslot * ns));
  CB_TRY(ws.alloc(&vexp, nslot * ns));
  CB_CUDA(cudaMemsetAsync(amax, 0, sizeof(float) * nslot * ns, s));
  CB_CUDA(cudaMemsetAsync(vexp, 0, sizeof(int) * nslot * ns, s));
  auto slotZ = [&](int j) { return (int64_t)j * ns; };
  auto slotT = [&](int j) { return (int64_t)(maxdeg + 1 + j) * ns; };
  const int64_t slotR = (int64_t)(2 * maxdeg + 1) * ns, slotS = (int64_t)(2 * maxdeg + 2) * ns;

  std::vector<double> al(maxdeg), be(maxdeg);  // alpha_j, beta_j of the scaled recurrence
  {
    double sigma = sigma1;
    al[0] = sigma1 / e;
    be[0] = 0.0;
    for (int j = 1; j < maxdeg; ++j) {
      const double sn = 1.0 / (tau - sigma);
      al[j] = 2.0 * sn / e;
      be[j] = -sigma * sn;
      sigma = sn;
    }
  }
  std::vector<double> pj;  // p_j(m_i), j = 0 .. maxdeg
  if (corr) {
    pj.assign((size_t)(maxdeg + 1) * k, 0.0);
    for (int64_t i = 0; i < k; ++i) {
      const double m = ritz[i] * ritz[i];
      double p0 = 1.0, p1 = al[0] * (m - c);
      pj[i] = p0;
      pj[(size_t)k + i] = p1;
      for (int j = 1; j < maxdeg; ++j) {
        const double p2 = al[j] * (m - c) * p1 + be[j] * p0;
        pj[(size_t)(j + 1) * k + i] = p2;
        p0 = p1;
        p1 = p2;
      }
    }
  }
  std::vector<float> gh(ns);
  // gamma of the first m vectors to the device, one entry per scaled column
  auto put_gamma = [&](int64_t m, auto value) -> int {
    for (int64_t i = 0; i < m; ++i)
      for (int q = 0; q < F::SCALES; ++q) gh[F::SCALES * i + q] = (float)value(i);
    CB_CUDA(cudaMemcpyAsync(gam, gh.data(), sizeof(float) * F::SCALES * m, cudaMemcpyHostToDevice, s));
    return CHASE_BSE_OK;
  };
  // a block of vectors -> masters and operand pieces, with their maxima and exponents in `slot`
  auto pack = [&](const cplx* W, float* Z, int64_t slot) -> int {
    if (J) {
      col_amax_kernel<<<(unsigned)k, 256, 0, s>>>(W, n, amax + slot, vexp + slot);
      pack_kernel<T, NPW><<<gsz(kpad / 2 * k), 256, 0, s>>>(W, n, k, c2(Z), Zp, kpad, vexp + slot);
    } else {
      col_amax_blocks_kernel<<<(unsigned)k, 256, 0, s>>>(W, n, amax + slot, vexp + slot);
      pack_blocks_kernel<T, NPW><<<gsz(n * k), 256, 0, s>>>(W, n, k, c2(Z), Zp, kpad, vexp + slot);
    }
    count_launch();
    count_launch();
    CB_LAUNCH();
    return CHASE_BSE_OK;
  };
  int j0 = 0;
  cudaEvent_t e0, e1;
  CB_CUDA(cudaEventCreate(&e0));
  CB_CUDA(cudaEventCreate(&e1));
  CB_CUDA(cudaEventRecord(e0, s));
  if (!corr) {
    CB_TRY(pack(Y0, Zb[0], slotZ(0)));  // Z_0 = W
  } else {
    // r2 = H R + ritz R on the tensor cores; Z_0 = 0; Z_1 = alpha_0 r2
    CB_TRY(ws.alloc(&src, 2 * n2 * k));
    CB_TRY(pack(R, Zb[2], slotR));
    CB_TRY(put_gamma(k, [&](int64_t i) { return ritz[i]; }));
    Epi ep{};
    ep.mode = 2; ep.n = n; ep.rows = rows; ep.cols = nc; ep.kpad = kpad; ep.err = err;
    ep.Znext = src; ep.Zcur = Zb[2]; ep.gamma = gam;
    ep.vexp_in = vexp + slotR;
    ep.amax_out = amax + slotS;
    sk(ep);
    CB_TRY((apply<SCH, FORM>(P, Zp, nc, ep, s)));
    CB_CUDA(cudaMemsetAsync(Zb[0], 0, sizeof(float) * 2 * n2 * k, s));
    if (J)
      scale_pack_kernel<T, NPW><<<gsz(n2 * k), 256, 0, s>>>(c2(src), n, 2 * k, (float)al[0], c2(Zb[1]), expl ? Tp : Zp,
                                                             kpad, amax + slotS, amax + slotZ(1), vexp + slotZ(1));
    else
      scale_pack_blocks_kernel<T, NPW><<<gsz(n * k), 256, 0, s>>>(c2(src), n, k, (float)al[0], c2(Zb[1]),
                                                                  expl ? Tp : Zp, kpad, amax + slotS, amax + slotZ(1),
                                                                  vexp + slotZ(1));
    count_launch();
    CB_LAUNCH();
    j0 = 1;
    if (fs) {
      fs->flops += 32.0 * (double)n * (double)n * (double)k;
      fs->launches += 1;
    }
  }
  for (int j = j0; j < maxdeg && expl; ++j) {
    // Z_{j+1} = alpha (H^2 Z_j - c Z_j) + beta Z_{j-1} (+ source): one launch on [P2 | Q2]
    int64_t kj = 0;
    while (kj < k && degs[kj] >= j + 1) ++kj;
    Epi ep{};
    ep.mode = 1; ep.h2 = 1; ep.n = n; ep.rows = rows; ep.cols = F::COLS * kj; ep.kpad = kpad; ep.err = err;
    sk(ep);
    for (int q = 0; q < NPW; ++q) ep.out[q] = zbuf[(j + 1) % 2]->p[q];
    ep.Znext = Zb[(j + 1) % 3]; ep.Zcur = Zb[j % 3]; ep.Zprev = Zb[(j + 2) % 3];
    ep.alpha = (float)al[j]; ep.beta = (float)be[j]; ep.c = (float)c;
    ep.vexp_in = vexp + slotZ(j);
    ep.vexp_out = vexp + slotZ(j + 1);
    ep.amax_out = amax + slotZ(j + 1);
    ep.amax_a = amax + slotZ(j);
    ep.amax_b = amax + slotZ(j);
    ep.amax_c = amax + slotZ(j > 0 ? j - 1 : 0);
    ep.ca = (float)std::fabs(al[j]);
    ep.cb = (float)std::fabs(al[j] * c);
    ep.cc = (float)std::fabs(be[j]);
    if (corr) {
      CB_TRY(put_gamma(kj, [&](int64_t i) { return al[j] * pj[(size_t)j * k + i]; }));
      ep.src = src;
      ep.gamma = gam;
      ep.amax_d = amax + slotS;
    }
    CB_TRY((apply<SCH, FORM>(PH2, *zbuf[j % 2], nc, ep, s)));
    if (fs) {
      fs->flops += 32.0 * (double)n * (double)n * (double)kj;  // the product with the blocks of H^2
      fs->launches += 1;
    }
  }
  for (int j = j0; j < maxdeg && !expl; ++j) {
    int64_t kj = 0;
    while (kj < k && degs[kj] >= j + 1) ++kj;
    Epi e1p{};
    e1p.mode = 0; e1p.n = n; e1p.rows = rows; e1p.cols = F::COLS * kj; e1p.kpad = kpad; e1p.err = err;
    sk(e1p);
    for (int q = 0; q < NPW; ++q) e1p.out[q] = Tp.p[q];
    e1p.vexp_in = vexp + slotZ(j);
    e1p.vexp_out = vexp + slotT(j);
    e1p.amax_out = amax + slotT(j);
    e1p.amax_a = amax + slotZ(j);
    e1p.ca = 1.0f;
    CB_TRY((apply<SCH, FORM>(P, Zp, nc, e1p, s)));  // T = H Z_j (J form: M Z_j)
    Epi e2p{};
    e2p.mode = 1; e2p.n = n; e2p.rows = rows; e2p.cols = F::COLS * kj; e2p.kpad = kpad; e2p.err = err;
    sk(e2p);
    for (int q = 0; q < NPW; ++q) e2p.out[q] = Zp.p[q];
    e2p.Znext = Zb[(j + 1) % 3]; e2p.Zcur = Zb[j % 3]; e2p.Zprev = Zb[(j + 2) % 3];
    e2p.alpha = (float)al[j]; e2p.beta = (float)be[j]; e2p.c = (float)c;
    e2p.vexp_in = vexp + slotT(j);
    e2p.vexp_out = vexp + slotZ(j + 1);
    e2p.amax_out = amax + slotZ(j + 1);
    e2p.amax_a = amax + slotT(j);
    e2p.amax_b = amax + slotZ(j);
    e2p.amax_c = amax + slotZ(j > 0 ? j - 1 : 0);
    e2p.ca = (float)std::fabs(al[j]);
    e2p.cb = (float)std::fabs(al[j] * c);
    e2p.cc = (float)std::fabs(be[j]);
    if (corr) {
      CB_TRY(put_gamma(kj, [&](int64_t i) { return al[j] * pj[(size_t)j * k + i]; }));
      e2p.src = src;
      e2p.gamma = gam;
      e2p.amax_d = amax + slotS;
    }
    CB_TRY((apply<SCH, FORM>(P, Tp, nc, e2p, s)));  // Z_{j+1} = alpha (H T - c Z_j) + beta Z_{j-1} (+ source)
    if (fs) {
      fs->flops += 64.0 * (double)n * (double)n * (double)kj;
      fs->launches += 2;
    }
  }
  CB_CUDA(cudaEventRecord(e1, s));
  std::vector<int> sel(k);
  std::vector<double> coef(k, 0.0);
  for (int64_t i = 0; i < k; ++i) {
    sel[i] = degs[i] % 3;
    if (corr) coef[i] = pj[(size_t)degs[i] * k + i];
  }
  int* dsel;
  double* dcoef;
  CB_TRY(ws.alloc(&dsel, k));
  CB_TRY(ws.alloc(&dcoef, k));
  CB_CUDA(cudaMemcpyAsync(dsel, sel.data(), sizeof(int) * k, cudaMemcpyHostToDevice, s));
  CB_CUDA(cudaMemcpyAsync(dcoef, coef.data(), sizeof(double) * k, cudaMemcpyHostToDevice, s));
  const double* dc = corr ? dcoef : nullptr;
  if (J) combine_kernel<<<gsz(n * k), 256, 0, s>>>(out, c2(Zb[0]), c2(Zb[1]), c2(Zb[2]), dsel, dc, Y0, n, k);
  else combine_blocks_kernel<<<gsz(n2 * k), 256, 0, s>>>(out, c2(Zb[0]), c2(Zb[1]), c2(Zb[2]), dsel, dc, Y0, n2, k);
  count_launch();
  CB_LAUNCH();
  int herr = 0;
  CB_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  CB_CUDA(cudaStreamSynchronize(s));
  if (fs) {
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    fs->ms_mixed += ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return herr ? CHASE_BSE_DEVICE_TIMEOUT : CHASE_BSE_OK;
}

}  // namespace tc

bool mixed_available() {
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  return major == 10 && minor == 3 && tc::encode_fn() != nullptr;
}

template <int SCH, int FORM>
static bool kernel_fits() {
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, tc::tc_hop_kernel<SCH, FORM>) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return tc::register_split_fits(fa.numRegs);
}
template <int SCH>
static bool scheme_fits() {
  return kernel_fits<SCH, tc::FORM_J>() && kernel_fits<SCH, tc::FORM_BLOCKS>();
}
bool mixed_filter_available() {
  if (!mixed_available()) return false;
  // a property of the build
  static const bool fits = scheme_fits<tc::SCH_BF16X3>() && scheme_fits<tc::SCH_BF16X6>() && scheme_fits<tc::SCH_FP16X3>();
  return fits;
}

// Where both forms are open the J form takes half the operations but, to form the entries of
// M, four FP64 additions per entry of A and B (1.6e-5 us n^2), and its launches are no shorter
// where M streams from HBM for few columns.  Measured, J form and blocks: n = 6000, k = 8,
// degree 4 2.00 and 1.35 ms; 8100, 30, 8 4.91 and 4.22; 16384, 20, 4 14.6 and 9.5; 3001, 10, 10 1.12
// and 1.14; against 4096, 60, 10 1.96 and 2.20; 16384, 100, 4 15.8 and 17.9; 1301, 6, 12 0.61 and 0.64.
static bool j_form_faster(int64_t n, int64_t k, const int* degs) {
  int64_t work = 0;
  for (int64_t i = 0; i < k; ++i) work += degs[i];
  return n < 3000 || work >= 300;
}
template <int SCH>
static int filter_form(bool jfixed, const cplx* A, const cplx* B, int64_t n, const cplx* V, int64_t k, const int* degs,
                       double mu1, double mu_nevex, double muN, cplx* out, const double* ritz, const cplx* R,
                       cudaStream_t s, FilterStats* fs, const cplx* P2, const cplx* Q2) {
  if (jfixed && j_form_faster(n, k, degs))
    return tc::filter_impl<SCH, tc::FORM_J>(A, B, n, V, k, degs, mu1, mu_nevex, muN, out, ritz, R, s, fs, P2, Q2);
  return tc::filter_impl<SCH, tc::FORM_BLOCKS>(A, B, n, V, k, degs, mu1, mu_nevex, muN, out, ritz, R, s, fs, P2, Q2);
}

int filter_mixed_sorted(const cplx* A, const cplx* B, int64_t n, const cplx* Y0, int64_t k, const int* degs_sorted,
                        double mu1, double mu_nevex, double muN, cplx* out, int scheme, bool jfixed, const double* ritz,
                        const cplx* R, cudaStream_t s, FilterStats* fs, const cplx* P2, const cplx* Q2) {
  switch (scheme) {
    case SCHEME_BF16X3:
      return filter_form<tc::SCH_BF16X3>(jfixed, A, B, n, Y0, k, degs_sorted, mu1, mu_nevex, muN, out, ritz, R, s, fs,
                                         P2, Q2);
    case SCHEME_BF16X6:
      return filter_form<tc::SCH_BF16X6>(jfixed, A, B, n, Y0, k, degs_sorted, mu1, mu_nevex, muN, out, ritz, R, s, fs,
                                         P2, Q2);
    case SCHEME_FP16X3:
      return filter_form<tc::SCH_FP16X3>(jfixed, A, B, n, Y0, k, degs_sorted, mu1, mu_nevex, muN, out, ritz, R, s, fs,
                                         P2, Q2);
    default:
      return CHASE_BSE_BAD_ARG;
  }
}

}  // namespace cb
