// FP64 kernels of the ChASE-BSE library.
//
// On GB300 the FP64 pipe issues 2 DFMA lanes per clock and SM (measured: 1.20 TFLOP/s
// with DFMA, 1.05 TFLOP/s with DMMA mma.sync.m8n8k4), 1/64 of the FP32 rate: a warp's
// DFMA occupies its SM for 16 clocks, so shared-memory and L2 traffic hide behind the
// arithmetic at any tile shape, and an FP64 product is bound by (1) the number of FP64
// instructions, padding included, and (2) how evenly they spread over the 152 pipes.
// Both kernels below therefore use a warp tile of 32 rows (one per lane) by a few columns,
// cut the rows and columns close to the matrix, and split K until the CTAs fill whole
// waves of SMs (plan_fp64); the K partials are summed in order by a second kernel.
#include <algorithm>

#include "fp64_kernels.cuh"

namespace cb {

namespace {
constexpr int ROWS = 32;   // rows of a tile: one per lane
constexpr int WARPS = 8;   // column groups of a tile: one per warp
constexpr int BK = 16;     // K elements staged at a time
constexpr int THREADS = 32 * WARPS;
constexpr double PART_LIMIT = 512e6;  // bytes of K partials

int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                 cudaSuccess || sms <= 0)
      sms = 152;
  }
  return sms;
}

// Tile width and K split of an FP64 product with M rows, N columns and K steps of
// `fma_step` DFMA per row and column, `tile_step` further FP64 instructions per row and K
// step of a tile (forming its left operand), and `sums` complex sums per row and column.  The
// estimated clocks of a split: waves of CTAs x (FP64 instructions of a CTA / 2 + 1500 for its
// loads' latency), plus the sum of the partials (two additions per sum and split over all SMs)
// and its launch.
struct Plan {
  int tn;       // columns per warp
  int split;
  int64_t chunk;
};
Plan plan_fp64(int64_t M, int64_t N, int64_t K, double fma_step, double tile_step, int sums, const int* widths,
               int nwidths, bool may_split) {
  const int sms = num_sms();
  Plan best{widths[0], 1, K};
  double best_t = 0.0;
  for (int w = 0; w < nwidths; ++w) {
    const int tn = widths[w];
    const int64_t tiles = (int64_t)cdiv(M, ROWS) * cdiv(N, WARPS * tn);
    const double step = 0.5 * ROWS * (fma_step * WARPS * tn + tile_step);
    for (int64_t sp = 1; sp <= 64; ++sp) {
      if (sp > 1 && (!may_split || K / sp < 2 || 16.0 * sums * (double)sp * (double)M * (double)N > PART_LIMIT)) break;
      const int64_t chunk = (K + sp - 1) / sp;
      const double waves = (double)((tiles * sp + sms - 1) / sms);
      double t = waves * ((double)chunk * step + 1500.0);
      if (sp > 1) t += 3000.0 + sums * (double)sp * (double)M * (double)N / sms;
      if (best_t == 0.0 || t < best_t * 0.999) {
        best_t = t;
        best = {tn, (int)((K + chunk - 1) / chunk), chunk};
      }
      if (tiles * sp > 8 * (int64_t)sms) break;
    }
  }
  return best;
}
}  // namespace

// ---------------------------------------------------------------------------
// H application, J-fixed form (HOP_JFIXED).  H is real on vectors [z; conj(z)]: H [z; conj(z)] = [t; -conj(t)] with
// t = A z + B conj(z), a real 2n x 2n matrix on (Re z, Im z):
//   Re t = (Ar + Br) Re z + (Bi - Ai) Im z,  Im t = (Ai + Bi) Re z + (Ar - Br) Im z.
// Every w = [x; y] is the sum of [a; conj(a)] and -i [c; conj(c)], a = (x + conj(y))/2 and
// c = i (x - conj(y))/2, so H w takes 2 x 4 n^2 DFMA instead of the 16 n^2 of the complex
// product with [A | B].  Both halves of H w are then sums and differences of two numbers of
// the size of A x, so the smaller half is exact only relative to the larger one: the form is
// for results of which that is all that is used (norms and inner products of whole vectors,
// and the filter of a solve, whose QR and Rayleigh-Ritz steps hold the basis as J-fixed vectors
// themselves).  The kernel stages the four sums of A and B (4 additions per
// element and tile) and 2a, 2c (4 per vector entry and tile), each a few per cent of the
// tile's DFMAs, and computes t for `cols` columns (2j: 2a_j, 2j + 1: 2c_j of vector j).
//
// Measured on one GB300, before (64 x 32 tiles, the complex product, K chunks >= 256) and
// after: residuals of 200 vectors at n = 4096 99.3 -> 47.7 ms (1.12 of 1.20 TFLOP/s), of 6
// vectors at n = 64 533 -> 42 us.

// Epilogue for output row i (< n) of vector j: top and bottom entry of H w.
__device__ __forceinline__ void hop_epilogue(const HopArgs& a, int64_t i, int64_t j, cplx top, cplx bot) {
  const int64_t n = a.n, n2 = 2 * a.n;
  const int64_t ot = j * n2 + i, ob = j * n2 + n + i;
  if (a.mode == HOP_STORE) {
    a.out[ot] = top;
    a.out[ob] = a.sflip ? mk(-bot.x, -bot.y) : bot;
  } else if (a.mode == HOP_CHEB) {
    cplx t = csub(top, cscale(a.Wc[ot], a.c));
    cplx b = csub(bot, cscale(a.Wc[ob], a.c));
    t = cscale(t, a.alpha);
    b = cscale(b, a.alpha);
    if (a.beta != 0.0) {
      t = cadd(t, cscale(a.Wp[ot], a.beta));
      b = cadd(b, cscale(a.Wp[ob], a.beta));
    }
    a.out[ot] = t;
    a.out[ob] = b;
  } else if (a.mode == HOP_RESID) {
    const double lam = a.lambda[j];
    a.out[ot] = csub(top, cscale(a.W[ot], lam));
    a.out[ob] = csub(bot, cscale(a.W[ob], lam));
  }
}
// ta, tc: the t of 2a_j and 2c_j.  H w: top = (ta - i tc)/2, bottom = (-conj(ta) + i conj(tc))/2.
__device__ __forceinline__ void hop_finish(const HopArgs& a, int64_t i, int64_t j, cplx ta, cplx tc) {
  hop_epilogue(a, i, j, mk(0.5 * (ta.x + tc.y), 0.5 * (ta.y - tc.x)), mk(0.5 * (tc.y - ta.x), 0.5 * (ta.y + tc.x)));
}

// GEN: general vectors W (2n x k, two columns each); else the columns of X = a.W are the z
// themselves (n x k, ld n) and a.out = t (ld n).  part != NULL: the t of K chunk blockIdx.z
// go to part + blockIdx.z * n * cols instead.
template <int TN, bool GEN>
__global__ void __launch_bounds__(THREADS)
hop_kernel(HopArgs a, cplx* part, int64_t chunk) {
  __shared__ double Ps[4][BK][ROWS + 1];
  __shared__ cplx Zs[BK][WARPS * TN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n = a.n, n2 = 2 * a.n, cols = GEN ? 2 * a.k : a.k;
  const int64_t row0 = (int64_t)blockIdx.x * ROWS;
  const int64_t col0 = (int64_t)blockIdx.y * (WARPS * TN);
  const int64_t kbeg = (int64_t)blockIdx.z * chunk;
  const int64_t kend = kbeg + chunk < n ? kbeg + chunk : n;
  const int64_t mycol = col0 + warp * TN;
  const bool active = mycol < cols;  // warp-uniform
  cplx acc[TN];
#pragma unroll
  for (int c = 0; c < TN; ++c) acc[c] = mk(0, 0);

  for (int64_t kb = kbeg; kb < kend; kb += BK) {
    const int kn = (int)(kend - kb < BK ? kend - kb : BK);
    for (int idx = tid; idx < ROWS * BK; idx += THREADS) {
      const int kk = idx % BK, r = idx / BK;
      const int64_t gi = row0 + r, gl = kb + kk;
      cplx p = mk(0, 0), q = mk(0, 0);
      if (gi < n && kk < kn) {
        p = a.A[gi * n + gl];
        q = a.B[gi * n + gl];
      }
      Ps[0][kk][r] = p.x + q.x;
      Ps[1][kk][r] = q.y - p.y;
      Ps[2][kk][r] = p.y + q.y;
      Ps[3][kk][r] = p.x - q.x;
    }
    if (GEN) {
      for (int idx = tid; idx < BK * (WARPS * TN / 2); idx += THREADS) {
        const int kk = idx % BK, j = idx / BK;
        const int64_t gj = col0 / 2 + j, gl = kb + kk;
        cplx za = mk(0, 0), zc = mk(0, 0);
        if (gj < a.k && kk < kn) {
          const cplx x = a.W[gj * n2 + gl], y = a.W[gj * n2 + n + gl];
          za = mk(x.x + y.x, x.y - y.y);
          zc = mk(-(x.y + y.y), x.x - y.x);
        }
        Zs[kk][2 * j] = za;
        Zs[kk][2 * j + 1] = zc;
      }
    } else {
      for (int idx = tid; idx < BK * (WARPS * TN); idx += THREADS) {
        const int kk = idx % BK, j = idx / BK;
        const int64_t gj = col0 + j;
        Zs[kk][j] = (gj < cols && kk < kn) ? a.W[gj * n + kb + kk] : mk(0, 0);
      }
    }
    __syncthreads();
    if (active) {
#pragma unroll 4
      for (int kk = 0; kk < kn; ++kk) {
        const double p0 = Ps[0][kk][lane], p1 = Ps[1][kk][lane], p2 = Ps[2][kk][lane], p3 = Ps[3][kk][lane];
#pragma unroll
        for (int c = 0; c < TN; ++c) {
          const cplx z = Zs[kk][warp * TN + c];
          acc[c].x = fma(p0, z.x, acc[c].x);
          acc[c].y = fma(p2, z.x, acc[c].y);
          acc[c].x = fma(p1, z.y, acc[c].x);
          acc[c].y = fma(p3, z.y, acc[c].y);
        }
      }
    }
    __syncthreads();
  }

  const int64_t i = row0 + lane;
  if (!active || i >= n) return;
  if (part) {
#pragma unroll
    for (int c = 0; c < TN; ++c)
      if (mycol + c < cols) part[((int64_t)blockIdx.z * cols + mycol + c) * n + i] = acc[c];
  } else if (GEN) {
#pragma unroll
    for (int c = 0; c + 1 < TN; c += 2)
      if (mycol + c < cols) hop_finish(a, i, (mycol + c) / 2, acc[c], acc[c + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < TN; ++c)
      if (mycol + c < cols) a.out[(mycol + c) * n + i] = acc[c];
  }
}

// Sum of the K partials in order, and the epilogue; one thread per row and vector.
template <bool GEN>
__global__ void hop_reduce_kernel(HopArgs a, const cplx* part, int nsplit) {
  const int64_t n = a.n, total = n * a.k, cols = GEN ? 2 * a.k : a.k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, j = idx / n;
    const cplx* p = part + (GEN ? 2 * j : j) * n + i;
    cplx ta = mk(0, 0), tc = mk(0, 0);
#pragma unroll 4
    for (int z = 0; z < nsplit; ++z) {
      ta = cadd(ta, p[(int64_t)z * cols * n]);
      if (GEN) tc = cadd(tc, p[(int64_t)z * cols * n + n]);
    }
    if (GEN) hop_finish(a, i, j, ta, tc);
    else a.out[idx] = ta;
  }
}

template <bool GEN>
static int hop_jfixed(const HopArgs& a, cudaStream_t s) {
  static const int widths_gen[4] = {2, 4, 6, 8}, widths_top[4] = {1, 2, 4, 8};
  const int64_t cols = GEN ? 2 * a.k : a.k;
  const Plan p = plan_fp64(a.n, cols, a.n, 4.0, 4.0, 1, GEN ? widths_gen : widths_top, 4, !a.no_split);
  cplx* part = nullptr;
  if (p.split > 1) CB_CUDA(dalloc(&part, sizeof(cplx) * p.split * a.n * cols, s));
  const dim3 grid(cdiv(a.n, ROWS), cdiv(cols, WARPS * p.tn), (unsigned)p.split);
  const int64_t tid = GEN ? timer_begin(1, 32.0 * (double)a.n * (double)a.n * (double)a.k, s) : -1;
  switch (p.tn) {
    case 1: hop_kernel<GEN ? 2 : 1, GEN><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
    case 2: hop_kernel<2, GEN><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
    case 4: hop_kernel<4, GEN><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
    case 6: hop_kernel<GEN ? 6 : 4, GEN><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
    default: hop_kernel<8, GEN><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
  }
  count_launch();
  if (part) {
    const int64_t blocks = (a.n * a.k + 127) / 128;
    hop_reduce_kernel<GEN><<<(unsigned)(blocks < 8192 ? blocks : 8192), 128, 0, s>>>(a, part, p.split);
    count_launch();
  }
  if (GEN) timer_end(tid, s);
  const cudaError_t e = cudaGetLastError();
  if (part) cudaFreeAsync(part, s);
  return e == cudaSuccess ? CHASE_BSE_OK : CHASE_BSE_CUDA_ERROR;
}

int hop_top_fp64(const cplx* A, const cplx* B, int64_t n, const cplx* X, int64_t k, cplx* Y, cudaStream_t s) {
  if (k <= 0 || n <= 0) return CHASE_BSE_OK;
  HopArgs a{};
  a.A = A; a.B = B; a.n = n; a.W = X; a.k = k; a.out = Y;
  return hop_jfixed<false>(a, s);
}

// The complex product [A | B] [x, conj(y); y, conj(x)] on the same tiles, two sums per row
// and vector over the 2n columns of [A | B]: the top half of H w and -conj of the bottom, each
// a sum of its own products, accurate relative to its own size (an eigenvector's lower half
// is smaller than the upper one by the coupling).  Twice the DFMAs of hop_kernel.  HOP_BLOCKS
// splits K by plan_fp64 and (FOLD) sums every 64 products by themselves first, so that the length
// of a K range does not show in the error (n = 1301, k = 67, degree 4 to 20: 1.1e-14 with one
// chain per range, 5.9e-15 so; 1 % more additions).  HOP_ORDERED keeps one chain and a fixed chunk rule: the phases of the Ritz vectors
// of a caller's basis come out of the last Jacobi rotations, whose pivots are rounding residue
// (a change of the last bit of H Q turns them by up to 1e-5).
// Measured on one GB300, before (64 x 32 tiles, K chunks >= 256) and after: a degree-20 filter
// of 30 vectors at n = 512 42.4 -> 9.6 ms, of 67 ragged ones at n = 1301 147 -> 80 ms (16 n^2 k
// DFMA at 1.17 of 1.20 TFLOP/s; the J-fixed form takes 5.25 and 41 ms, but leaves the lower half
// 1.3e-13 of its size off instead of 8.6e-15, and 1e-12 and more at a coupling of 1e-3).
template <int TN, bool FOLD>
__global__ void __launch_bounds__(THREADS)
hop_blocks_kernel(HopArgs a, cplx* part, int64_t kchunk) {
  __shared__ cplx Ps[BK][ROWS + 1];
  __shared__ cplx W1s[BK][WARPS * TN];
  __shared__ cplx W2s[BK][WARPS * TN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n = a.n, n2 = 2 * a.n;
  const int64_t row0 = (int64_t)blockIdx.x * ROWS, col0 = (int64_t)blockIdx.y * (WARPS * TN);
  const int64_t kbeg = (int64_t)blockIdx.z * kchunk;
  const int64_t kend = kbeg + kchunk < n2 ? kbeg + kchunk : n2;
  const int64_t mycol = col0 + warp * TN;
  const bool active = mycol < a.k;  // warp-uniform
  cplx acc1[TN], acc2[TN], sum1[TN], sum2[TN];
#pragma unroll
  for (int c = 0; c < TN; ++c) acc1[c] = acc2[c] = sum1[c] = sum2[c] = mk(0, 0);
  for (int64_t kb = kbeg; kb < kend; kb += BK) {
    if (FOLD && ((kb - kbeg) & 63) == 0) {
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        sum1[c] = cadd(sum1[c], acc1[c]);
        sum2[c] = cadd(sum2[c], acc2[c]);
        acc1[c] = acc2[c] = mk(0, 0);
      }
    }
    const int kn = (int)(kend - kb < BK ? kend - kb : BK);
    for (int idx = tid; idx < ROWS * BK; idx += THREADS) {
      const int kk = idx % BK, r = idx / BK;
      const int64_t gi = row0 + r, gl = kb + kk;
      cplx v = mk(0, 0);
      if (gi < n && kk < kn) v = (gl < n) ? a.A[gi * n + gl] : a.B[gi * n + (gl - n)];
      Ps[kk][r] = v;
    }
    for (int idx = tid; idx < BK * WARPS * TN; idx += THREADS) {
      const int kk = idx % BK, j = idx / BK;
      const int64_t gj = col0 + j, gl = kb + kk;
      cplx v1 = mk(0, 0), v2 = mk(0, 0);
      if (gj < a.k && kk < kn) {
        const cplx* w = a.W + gj * n2;
        v1 = w[gl];
        v2 = cconj(w[gl < n ? gl + n : gl - n]);
      }
      W1s[kk][j] = v1;
      W2s[kk][j] = v2;
    }
    __syncthreads();
    if (active) {
#pragma unroll 4
      for (int kk = 0; kk < kn; ++kk) {
        const cplx p = Ps[kk][lane];
#pragma unroll
        for (int c = 0; c < TN; ++c) {
          cfma(acc1[c], p, W1s[kk][warp * TN + c]);
          cfma(acc2[c], p, W2s[kk][warp * TN + c]);
        }
      }
    }
    __syncthreads();
  }
  const int64_t i = row0 + lane;
  if (!active || i >= n) return;
#pragma unroll
  for (int c = 0; c < TN; ++c) {
    const int64_t j = mycol + c;
    if (j >= a.k) continue;
    if (FOLD) {
      acc1[c] = cadd(sum1[c], acc1[c]);
      acc2[c] = cadd(sum2[c], acc2[c]);
    }
    if (part) {
      cplx* p = part + ((int64_t)blockIdx.z * a.k + j) * n2;
      p[i] = acc1[c];
      p[n + i] = acc2[c];
    } else {
      hop_epilogue(a, i, j, acc1[c], mk(-acc2[c].x, acc2[c].y));
    }
  }
}
__global__ void hop_blocks_reduce_kernel(HopArgs a, const cplx* part, int nsplit) {
  const int64_t n = a.n, n2 = 2 * n, total = n * a.k;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % n, j = idx / n;
    cplx c1 = mk(0, 0), c2 = mk(0, 0);
    for (int z = 0; z < nsplit; ++z) {
      const cplx* p = part + ((int64_t)z * a.k + j) * n2;
      c1 = cadd(c1, p[i]);
      c2 = cadd(c2, p[n + i]);
    }
    hop_epilogue(a, i, j, c1, mk(-c2.x, c2.y));
  }
}

// K chunks that fill the GPU twice with tiles of `tiles`, at least min_chunk long and a
// multiple of `round` (the fixed rule of the ordered products).
static void ordered_chunks(int64_t tiles, int64_t K, int64_t min_chunk, int64_t round, int64_t* chunk, int* splits) {
  const int64_t want = 2 * (int64_t)num_sms();
  int64_t s = 1;
  if (tiles < want && K >= 2 * min_chunk) s = std::max<int64_t>(1, std::min((want + tiles - 1) / tiles, K / min_chunk));
  *chunk = s == 1 ? std::max<int64_t>(K, 1) : ((K + s - 1) / s + round - 1) / round * round;
  *splits = (int)std::max<int64_t>(1, (K + *chunk - 1) / *chunk);
}

static int hop_blocks(const HopArgs& a, cudaStream_t s) {
  static const int widths[4] = {1, 2, 3, 4};
  const int64_t n2 = 2 * a.n;
  Plan p;
  if (a.form == HOP_ORDERED) {
    p.tn = a.k >= 32 ? 4 : (a.k >= 16 ? 2 : 1);
    ordered_chunks((int64_t)cdiv(a.n, 64) * cdiv(a.k, a.k <= 4 ? 4 : 32), n2, 256, 16, &p.chunk, &p.split);
  } else {
    p = plan_fp64(a.n, a.k, n2, 8.0, 0.0, 2, widths, 4, !a.no_split);
  }
  cplx* part = nullptr;
  if (p.split > 1) CB_CUDA(dalloc(&part, sizeof(cplx) * p.split * n2 * a.k, s));
  const dim3 grid(cdiv(a.n, ROWS), cdiv(a.k, WARPS * p.tn), (unsigned)p.split);
  const int64_t tid = timer_begin(1, 32.0 * (double)a.n * (double)a.n * (double)a.k, s);
  if (a.form == HOP_ORDERED) {
    if (p.tn == 4) hop_blocks_kernel<4, false><<<grid, THREADS, 0, s>>>(a, part, p.chunk);
    else if (p.tn == 2) hop_blocks_kernel<2, false><<<grid, THREADS, 0, s>>>(a, part, p.chunk);
    else hop_blocks_kernel<1, false><<<grid, THREADS, 0, s>>>(a, part, p.chunk);
  } else {
    switch (p.tn) {
      case 1: hop_blocks_kernel<1, true><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
      case 2: hop_blocks_kernel<2, true><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
      case 3: hop_blocks_kernel<3, true><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
      default: hop_blocks_kernel<4, true><<<grid, THREADS, 0, s>>>(a, part, p.chunk); break;
    }
  }
  count_launch();
  if (part) {
    const int64_t blocks = (a.n * a.k + 127) / 128;
    hop_blocks_reduce_kernel<<<(unsigned)(blocks < 8192 ? blocks : 8192), 128, 0, s>>>(a, part, p.split);
    count_launch();
  }
  timer_end(tid, s);
  const cudaError_t e = cudaGetLastError();
  if (part) cudaFreeAsync(part, s);
  return e == cudaSuccess ? CHASE_BSE_OK : CHASE_BSE_CUDA_ERROR;
}

int hop_fp64(const HopArgs& a, cudaStream_t s) {
  if (a.k <= 0 || a.n <= 0) return CHASE_BSE_OK;
  return a.form == HOP_JFIXED ? hop_jfixed<true>(a, s) : hop_blocks(a, s);
}

// ---------------------------------------------------------------------------
// Generic complex GEMM, column-major.
__device__ __forceinline__ cplx load_op(const cplx* X, int64_t ld, char op, int64_t r, int64_t c) {
  // element (r, c) of op(X)
  if (op == 'N') return X[r + c * ld];
  const cplx v = X[c + r * ld];
  return op == 'C' ? cconj(v) : v;
}

// Tiles of 32 rows (one per lane) by WN * TN columns (TN per warp), sized so that the FP64
// work spreads over all SMs: a product of the Rayleigh-Ritz steps has few outputs (80 x 80 with
// K = 512 at n = 512), and each is 4 K DFMA at 2 a clock and SM.  Every output is one chain of
// DFMAs in K order whatever the tile, so the tile does not change a bit of the result.
// kchunk > 0: K split over blockIdx.z; block z writes alpha * its partial product to
// C + z * ldc * N (beta ignored).
// Measured on one GB300, before (64 x 64 tiles of 256 threads) and after: a Gram matrix of
// 80 vectors at n = 512 2.1 ms -> 0.10 ms; a Rayleigh-Ritz step of 256 vectors at n = 2048
// 68.6 -> 64.3 ms; a solve and its gradient at n = 512 219 -> 143 ms.
template <int WN, int TN>
__global__ void __launch_bounds__(32 * WN)
zgemm_kernel(char opA, char opB, int64_t M, int64_t N, int64_t K, cplx alpha, const cplx* __restrict__ A,
             int64_t lda, const cplx* __restrict__ B, int64_t ldb, cplx beta, cplx* C, int64_t ldc, int64_t kchunk) {
  constexpr int BN = WN * TN;
  constexpr int NT = 32 * WN;
  __shared__ cplx As[BK][ROWS + 1];
  __shared__ cplx Bs[BK][BN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t row0 = (int64_t)blockIdx.x * ROWS;
  const int64_t col0 = (int64_t)blockIdx.y * BN;
  cplx acc[TN];
#pragma unroll
  for (int c = 0; c < TN; ++c) acc[c] = mk(0, 0);

  const int64_t kbeg = kchunk ? (int64_t)blockIdx.z * kchunk : 0;
  const int64_t kend = kchunk ? (kbeg + kchunk < K ? kbeg + kchunk : K) : K;
  if (kchunk) {
    C += (int64_t)blockIdx.z * ldc * N;
    beta = mk(0, 0);
  }
  for (int64_t kb = kbeg; kb < kend; kb += BK) {
    const int kn = (int)(kend - kb < BK ? kend - kb : BK);
    for (int idx = tid; idx < ROWS * BK; idx += NT) {
      int r, l;
      if (opA == 'N') { r = idx % ROWS; l = idx / ROWS; } else { l = idx % BK; r = idx / BK; }
      const int64_t gr = row0 + r;
      As[l][r] = (gr < M && l < kn) ? load_op(A, lda, opA, gr, kb + l) : mk(0, 0);
    }
    for (int idx = tid; idx < BN * BK; idx += NT) {
      int c, l;
      if (opB == 'N') { l = idx % BK; c = idx / BK; } else { c = idx % BN; l = idx / BN; }
      const int64_t gc = col0 + c;
      Bs[l][c] = (gc < N && l < kn) ? load_op(B, ldb, opB, kb + l, gc) : mk(0, 0);
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      const cplx av = As[kk][lane];
#pragma unroll
      for (int c = 0; c < TN; ++c) cfma(acc[c], av, Bs[kk][warp * TN + c]);
    }
    __syncthreads();
  }
  const bool use_beta = (beta.x != 0.0 || beta.y != 0.0);
  const int64_t i = row0 + lane;
  if (i >= M) return;
#pragma unroll
  for (int c = 0; c < TN; ++c) {
    const int64_t j = col0 + warp * TN + c;
    if (j >= N) continue;
    cplx v = cmul(alpha, acc[c]);
    if (use_beta) v = cadd(v, cmul(beta, C[i + j * ldc]));
    C[i + j * ldc] = v;
  }
}

// C = alpha * sum_z part[z] + beta * C
__global__ void zgemm_reduce_kernel(const cplx* part, int nsplit, int64_t M, int64_t N, cplx beta, cplx* C,
                                    int64_t ldc) {
  const int64_t total = M * N;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx % M, j = idx / M;
    cplx v = mk(0, 0);
    for (int z = 0; z < nsplit; ++z) v = cadd(v, part[(int64_t)z * M * N + idx]);
    if (beta.x != 0.0 || beta.y != 0.0) v = cadd(v, cmul(beta, C[i + j * ldc]));
    C[i + j * ldc] = v;
  }
}

// Number of K chunks so that a small output grid still fills the GPU (two CTAs per
// SM); 1 when the grid is large enough or K too short to split.
static int64_t split_count(int64_t tiles, int64_t K, int64_t min_chunk) {
  const int64_t want = 2 * (int64_t)num_sms();
  if (tiles >= want || K < 2 * min_chunk) return 1;
  int64_t s = (want + tiles - 1) / tiles;
  if (s > K / min_chunk) s = K / min_chunk;
  return s < 1 ? 1 : s;
}

int zgemm(char opA, char opB, int64_t M, int64_t N, int64_t K, cplx alpha, const cplx* A, int64_t lda,
          const cplx* B, int64_t ldb, cplx beta, cplx* C, int64_t ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0) return CHASE_BSE_OK;
  if (K < 0) K = 0;  // K = 0: C = beta C (empty K loop)
  // the K chunks follow a fixed rule (as if on tiles of 64 x 64, or 32 x 32 for few rows or
  // columns): they set the order of the sums
  const int rule = (M <= 16 || N <= 16) ? 32 : 64;
  const int64_t nsplit = split_count((int64_t)cdiv(M, rule) * cdiv(N, rule), K, 512);
  const int64_t kchunk = nsplit <= 1 ? 0 : ((K + nsplit - 1) / nsplit + 7) / 8 * 8;
  const int64_t ns = kchunk ? (K + kchunk - 1) / kchunk : 1;
  cplx* part = nullptr;
  if (ns > 1) CB_CUDA(dalloc(&part, sizeof(cplx) * ns * M * N, s));
  // of the tile widths, the one of least estimated time: waves of SMs x the columns of a tile
  // (16 clocks a row group, K step and column for 4 DFMA of 32 lanes), or what a CTA's loads take
  static const int widths[6] = {32, 16, 8, 4, 2, 1};
  int best = 32;
  double best_t = 0.0;
  for (int w : widths) {
    const double ctas = (double)cdiv(M, ROWS) * cdiv(N, w) * (double)ns;
    const double t = std::ceil(ctas / num_sms()) * std::max(64.0 * w, 40.0 + 30.0 * w);
    if (best_t == 0.0 || t < best_t * 0.999) {
      best_t = t;
      best = w;
    }
  }
  const dim3 grid(cdiv(M, ROWS), cdiv(N, best), (unsigned)ns);
  cplx* out = ns > 1 ? part : C;
  const int64_t ldo = ns > 1 ? M : ldc, kc = ns > 1 ? kchunk : 0;
#define CB_ZGEMM(WN, TN) \
  zgemm_kernel<WN, TN><<<grid, 32 * WN, 0, s>>>(opA, opB, M, N, K, alpha, A, lda, B, ldb, beta, out, ldo, kc)
  switch (best) {
    case 1: CB_ZGEMM(1, 1); break;
    case 2: CB_ZGEMM(2, 1); break;
    case 4: CB_ZGEMM(4, 1); break;
    case 8: CB_ZGEMM(8, 1); break;
    case 16: CB_ZGEMM(8, 2); break;
    default: CB_ZGEMM(8, 4); break;
  }
#undef CB_ZGEMM
  count_launch();
  if (ns > 1) {
    const int64_t total = M * N;
    const unsigned rb = (unsigned)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192);
    zgemm_reduce_kernel<<<rb, 256, 0, s>>>(part, (int)ns, M, N, beta, C, ldc);
    count_launch();
  }
  const cudaError_t e = cudaGetLastError();
  if (part) cudaFreeAsync(part, s);
  return e == cudaSuccess ? CHASE_BSE_OK : CHASE_BSE_CUDA_ERROR;
}

}  // namespace cb
