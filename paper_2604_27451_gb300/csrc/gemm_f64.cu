// Complex FP64 GEMM on the CUDA cores (FP64 FMA), C = alpha*A*B + beta*C,
// for matrices given as two-mode strided views (common.cuh).  This is the
// arithmetic of the FP64 path: every contraction of t2, M11 and the sigma
// vector goes through it when precision = CVSADC_FP64, and the small
// contractions of every precision do.
//
// What bounds it: an SM of this GPU retires two FP64 FMAs per cycle (1.26
// TFLOP/s for the chip at 2.07 GHz), 32 times fewer than FP32, and a complex multiply-
// add takes four.  One 16-byte operand pair is worth two FMA cycles, so even
// a 16 x 4 tile reads only 2.5 bytes per SM cycle: memory, shared memory and
// latency all hide behind the FP64 pipe, and what costs time is an SM
// without work and an FMA spent on padding.  Hence small tiles in many
// shapes (the ncore-sized sides of 6 and 12 among them), one warp per
// scheduler, and K split until every SM holds work; plan_f64 takes the
// shape and the split with the least modelled time.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace cvs {

namespace {
// threads per block: a warp for each of the SM's four schedulers, which own
// the FP64 units (blocks of two warps left some of them short of work:
// 960 x 560 x 240 ran at 0.72 of the FP64 rate)
constexpr int NT = 128;

__device__ __forceinline__ void cp16(cplx* dst, const cplx* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(live ? 16 : 0)
               : "memory");
}
// conj != 0: the conjugate, by the sign bit (integer pipe)
__device__ __forceinline__ cplx conj_if(cplx v, int conj) {
  v.y = __longlong_as_double(__double_as_longlong(v.y) ^ ((long long)conj << 63));
  return v;
}

// offset of index i in one dimension of a view (32-bit division)
__device__ __forceinline__ int64_t mode_off(int64_t hi, int64_t lo, int lo_ext, int i) {
  if (lo_ext == INT32_MAX) return (int64_t)i * lo;
  const int h = i / lo_ext;
  return (int64_t)h * hi + (int64_t)(i - h * lo_ext) * lo;
}

// A block computes a (TY RM) x (TX RN) tile with TY x TX x KX threads; each
// thread holds RM x RN outputs, and the KX thread groups take every KX-th k
// of a step (tiles of fewer outputs than threads: the 6 x 6 and 12 x 12
// blocks of core indices), added up at the end.  ST steps of BK are staged
// in shared memory with 16-byte asynchronous copies, one element each; a
// step takes ~2 us from its first load on when nothing hides it, so small
// tiles keep four in flight.
// part == nullptr: z is the batch index (operand batch strides), full K.
// part != nullptr: z is a K slice [z*kchunk, (z+1)*kchunk); alpha * the
// partial product goes to part[z][M][N].
template <int TY, int TX, int RM, int RN, int BK, int ST>
__global__ void __launch_bounds__(NT)
    zgemm_f64_kernel(int M, int N, int K, double alpha, View A, View B,
                     double beta, View C, int a_kfast, int b_kfast,
                     int ntn, int kchunk, int period, int64_t upper, cplx* part) {
  constexpr int KX = NT / (TY * TX);
  constexpr int TM = TY * RM, TN = TX * RN;
  constexpr int EA = (TM * BK + NT - 1) / NT, EB = (TN * BK + NT - 1) / NT;
  constexpr int STAGE = BK * (TM + 1 + TN + 1);
  constexpr int RED = KX > 1 ? KX * TM * TN : 0;
  __shared__ cplx sh[ST * STAGE > RED ? ST * STAGE : RED];
  const int tid = threadIdx.x;
  const int ty = tid % TY, tx = (tid / TY) % TX, kx = tid / (TY * TX);
  const int m0 = (blockIdx.x / ntn) * TM, n0 = (blockIdx.x % ntn) * TN;
  const int64_t z = blockIdx.z;
  // upper >= 0: the square of columns from `upper` on is symmetric, and tiles
  // wholly below its diagonal are left out
  if (upper >= 0 && n0 >= upper && n0 + TN <= upper + m0) return;
  const cplx* Ap = A.p;
  const cplx* Bp = B.p;
  cplx* Cp = C.p;
  int kb = 0, ke = K;
  if (part) {
    kb = (int)(z * kchunk);
    ke = min(K, kb + kchunk);
  } else {
    Ap += z * A.batch;
    Bp += z * B.batch;
    Cp += z * C.batch;
  }

  // element e of this thread's share of a stage: (row, k) of A, (k, col) of
  // B, along whichever mode of the operand has unit stride
  auto a_rk = [&](int e, int& m, int& k) {
    const int idx = tid + e * NT;
    m = a_kfast ? idx / BK : idx % TM;
    k = a_kfast ? idx % BK : idx / TM;
  };
  auto b_kn = [&](int e, int& k, int& n) {
    const int idx = tid + e * NT;
    n = b_kfast ? idx / BK : idx % TN;
    k = b_kfast ? idx % BK : idx / TN;
  };
  int64_t aro[EA], bco[EB];  // row / column offset, -1 outside the matrix
#pragma unroll
  for (int e = 0; e < EA; ++e) {
    int m, k;
    a_rk(e, m, k);
    aro[e] = (tid + e * NT < TM * BK && m0 + m < M)
                 ? mode_off(A.rs_hi, A.rs_lo, A.r_lo, m0 + m) : -1;
  }
#pragma unroll
  for (int e = 0; e < EB; ++e) {
    int k, n;
    b_kn(e, k, n);
    bco[e] = (tid + e * NT < TN * BK && n0 + n < N)
                 ? mode_off(B.cs_hi, B.cs_lo, B.c_lo, n0 + n) : -1;
  }
  // starts the copies of the step at k0 (zeros outside the matrix)
  auto load = [&](int k0, cplx* st) {
#pragma unroll
    for (int e = 0; e < EA; ++e) {
      int m, k;
      a_rk(e, m, k);
      const bool live = aro[e] >= 0 && k0 + k < ke;
      if (tid + e * NT < TM * BK)
        cp16(st + k * (TM + 1) + m,
             live ? Ap + aro[e] + mode_off(A.cs_hi, A.cs_lo, A.c_lo, k0 + k) : Ap, live);
    }
#pragma unroll
    for (int e = 0; e < EB; ++e) {
      int k, n;
      b_kn(e, k, n);
      const bool live = bco[e] >= 0 && k0 + k < ke;
      if (tid + e * NT < TN * BK)
        cp16(st + BK * (TM + 1) + k * (TN + 1) + n,
             live ? Bp + bco[e] + mode_off(B.rs_hi, B.rs_lo, B.r_lo, k0 + k) : Bp, live);
    }
  };

  // every `period` steps the sums so far are added up apart: the rounding
  // error of a chain of additions grows with its length
  double accr[RM][RN], acci[RM][RN], sumr[RM][RN], sumi[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) accr[i][j] = acci[i][j] = sumr[i][j] = sumi[i][j] = 0.0;
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        sumr[i][j] += accr[i][j];
        sumi[i][j] += acci[i][j];
        accr[i][j] = acci[i][j] = 0.0;
      }
  };

  const int ntiles = (ke - kb + BK - 1) / BK;
  int left = period;
  // one copy group per step, empty past the end, so that a fixed count of
  // pending groups says that step t has landed
#pragma unroll
  for (int t = 0; t < ST - 1; ++t) {
    if (t < ntiles) load(kb + t * BK, sh + t * STAGE);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int t = 0; t < ntiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();  // step t is visible; step t - 1 is read by everyone
    if (t + ST - 1 < ntiles)
      load(kb + (t + ST - 1) * BK, sh + ((t + ST - 1) % ST) * STAGE);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const cplx* as = sh + (t % ST) * STAGE;
    const cplx* bs = as + BK * (TM + 1);
#pragma unroll
    for (int kk = 0; kk < BK / KX; ++kk) {
      const int k = kk * KX + kx;
      cplx a[RM], b[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = conj_if(as[k * (TM + 1) + ty + TY * i], A.conj);
#pragma unroll
      for (int j = 0; j < RN; ++j) b[j] = conj_if(bs[k * (TN + 1) + tx + TX * j], B.conj);
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          accr[i][j] = fma(a[i].x, b[j].x, accr[i][j]);
          accr[i][j] = fma(-a[i].y, b[j].y, accr[i][j]);
          acci[i][j] = fma(a[i].x, b[j].y, acci[i][j]);
          acci[i][j] = fma(a[i].y, b[j].x, acci[i][j]);
        }
    }
    if (--left == 0) {
      flush();
      left = period;
    }
  }
  flush();

  auto put = [&](int r, int c, double re, double im) {
    if (r >= M || c >= N) return;
    cplx v = cmake(alpha * re, alpha * im);
    if (part) {
      part[(z * M + r) * (int64_t)N + c] = v;
      return;
    }
    cplx* dst = Cp + mode_off(C.rs_hi, C.rs_lo, C.r_lo, r) + mode_off(C.cs_hi, C.cs_lo, C.c_lo, c);
    if (beta != 0.0) {
      cplx o = *dst;
      v.x += beta * o.x;
      v.y += beta * o.y;
    }
    *dst = v;
  };
  if constexpr (KX > 1) {
    __syncthreads();  // the stages are read
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j)
        sh[(kx * TM + ty + TY * i) * TN + tx + TX * j] = cmake(sumr[i][j], sumi[i][j]);
    __syncthreads();
    for (int e = tid; e < TM * TN; e += NT) {
      double re = 0.0, im = 0.0;
      for (int q = 0; q < KX; ++q) {
        const cplx v = sh[q * TM * TN + e];
        re += v.x;
        im += v.y;
      }
      put(m0 + e / TN, n0 + e % TN, re, im);
    }
  } else {
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j)
        put(m0 + ty + TY * i, n0 + tx + TX * j, sumr[i][j], sumi[i][j]);
  }
}

typedef void (*F64Kernel)(int, int, int, double, View, View, double, View, int, int, int, int,
                          int, int64_t, cplx*);
struct F64Shape {
  int tm, tn, bk, kx;
  double eff;
  F64Kernel fn;
};
#define CVS_F64(TY, TX, RM, RN, BK, ST, EFF) \
  {TY * RM, TX * RN, BK, NT / (TY * TX), EFF, zgemm_f64_kernel<TY, TX, RM, RN, BK, ST>}
// with the share of the FP64 rate each holds on 1000 products of 246 x 165 x
// 200 (its padding and whole k steps counted as work)
const F64Shape F64_SHAPES[] = {
    CVS_F64(16, 8, 2, 4, 16, 2, 0.96),  // 32 x 32
    CVS_F64(16, 8, 2, 3, 16, 2, 0.95),  // 32 x 24
    CVS_F64(16, 8, 2, 2, 16, 3, 0.95),  // 32 x 16
    CVS_F64(32, 4, 1, 3, 16, 3, 0.95),  // 32 x 12
    CVS_F64(32, 4, 1, 2, 16, 4, 0.91),  // 32 x 8
    CVS_F64(16, 8, 1, 2, 16, 4, 0.91),  // 16 x 16
    CVS_F64(16, 8, 1, 1, 16, 4, 0.91),  // 16 x 8
    CVS_F64(32, 2, 1, 3, 16, 4, 0.98),  // 32 x 6
    CVS_F64(32, 4, 1, 1, 16, 4, 0.95),  // 32 x 4
    CVS_F64(32, 2, 1, 1, 16, 4, 0.90),  // 32 x 2
    CVS_F64(32, 1, 1, 1, 16, 4, 0.82),  // 32 x 1
    CVS_F64(8, 8, 1, 1, 16, 4, 0.91),   // 8 x 8
    CVS_F64(8, 4, 1, 1, 32, 3, 0.83),   // 8 x 4
    CVS_F64(4, 32, 1, 1, 16, 4, 0.95),  // 4 x 32
    CVS_F64(2, 32, 3, 1, 16, 4, 0.98),  // 6 x 32
    CVS_F64(4, 4, 3, 3, 16, 4, 0.95),   // 12 x 12
    CVS_F64(2, 2, 3, 3, 32, 3, 0.74),   // 6 x 6
};
#undef CVS_F64

struct F64Plan {
  const F64Shape* shape;
  int splits;
};

// The tile shape and number of K slices with the least modelled time, in SM
// cycles.  A block's FMAs take w = 2 tm tn (k of whole steps) / eff cycles of
// its SM's FP64 pipe (padding included), its set-up and stores about 200
// more; the SM with the most blocks sets the time, and one block alone takes
// w plus 1000 cycles of latency per k step.  K slices
// cost one more launch (5000 cycles) and their partials' way through memory,
// 32 bytes each at 3 KB per cycle.  The modelled time is within 5 % of the
// measured one over these shapes at 61 x 47 x 83 to 1024^3 and 6 x 6 x 10^6.
// Measured at 2.07 GHz against the former 64 x 64 tile (256 threads):
//   61 x 47 x 83       8 x 4,  s 1        10 us  (383 us)
//   960 x 240 x 560    32 x 24, s 1      858 us  (2330 us), 0.97 of the FP64 rate
//   157 x 6 x 123245   32 x 6,  s 512    794 us  (1520 us)
//   1200 x 4 x 1200    32 x 4, s 8        56 us  (4960 us)
F64Plan plan_f64(int M, int N, int K, int batch, size_t part_elems) {
  constexpr double SMS = 152.0;
  F64Plan best{&F64_SHAPES[0], 1};
  double tbest = 1e300;
  const int64_t smax = std::min<int64_t>(
      std::min<int64_t>(1024, K / 16), (int64_t)(part_elems / ((size_t)M * N)));
  for (const F64Shape& f : F64_SHAPES) {
    const double tiles = (double)((M + f.tm - 1) / f.tm) * ((N + f.tn - 1) / f.tn) * batch;
    for (int64_t s = 1; s == 1 || s <= smax; s *= 2) {
      const double ks = (double)((K + s - 1) / s);
      const double steps = std::ceil(ks / f.bk);
      const double w = 2.0 * f.tm * f.tn * f.bk * steps / f.eff;
      double t = std::max(std::ceil(tiles * s / SMS) * (w + 200.0), w + 1000.0 * steps);
      if (s > 1) t += 5000.0 + 32.0 * s * (double)M * N / 3000.0;
      if (t < tbest) {
        tbest = t;
        best = F64Plan{&f, (int)s};
      }
    }
  }
  return best;
}

// C(m, n) = sum_z part[z][m][n] + beta * C(m, n)
// in a fixed order: a thread per output, or (WARP) a warp per output when
// there are fewer outputs than threads to hide 1000 dependent adds behind
// (36 outputs of 1024 slices: 200 us with a thread each)
template <bool WARP>
__global__ void splitk_reduce_kernel(int M, int N, int nz, const cplx* part,
                                     double beta, View C) {
  constexpr int W = WARP ? 32 : 1;
  const int64_t MN = (int64_t)M * N;
  const int lane = threadIdx.x % W;
  for (int64_t idx = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / W; idx < MN;
       idx += (int64_t)gridDim.x * blockDim.x / W) {
    double sr = 0, si = 0;
    if (nz <= 4 * W) {
      for (int z = lane; z < nz; z += W) {
        const cplx v = part[z * MN + idx];
        sr += v.x;
        si += v.y;
      }
    } else {
      // eight running sums, added pairwise (1217 x 4 x 901, 29 slices: rms error
      // 3.3e-16 -> 2.9e-16; their additions cost 30 us a single-vector sigma
      // of 6/33/157/785 where there are only a few slices)
      double r8[8], i8[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) r8[q] = i8[q] = 0.0;
      for (int z0 = lane; z0 < nz; z0 += 8 * W)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (z0 + q * W >= nz) break;
          const cplx v = part[(z0 + q * W) * MN + idx];
          r8[q] += v.x;
          i8[q] += v.y;
        }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < o; ++q) {
          r8[q] += r8[q + o];
          i8[q] += i8[q + o];
        }
      sr = r8[0];
      si = i8[0];
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane != 0) continue;
    int r = idx / N, c = idx % N;
    cplx* d = C.p + vrow(C, r) + vcol(C, c);
    if (beta != 0.0) {
      cplx o = *d;
      sr += beta * o.x;
      si += beta * o.y;
    }
    *d = cmake(sr, si);
  }
}
}  // namespace

void splitk_reduce(cudaStream_t s, int M, int N, int nz, const cplx* part,
                   double beta, View C) {
  const int64_t mn = (int64_t)M * N;
  if (mn < 152 * 256 && nz >= 32)
    splitk_reduce_kernel<true><<<grid1d(mn * 32, 256), 256, 0, s>>>(M, N, nz, part, beta, C);
  else
    splitk_reduce_kernel<false><<<grid1d(mn, 256), 256, 0, s>>>(M, N, nz, part, beta, C);
  CVS_CHECK_LAUNCH();
}

void zgemm_f64(cudaStream_t s, int M, int N, int K, double alpha, View A,
               View B, double beta, View C, int batch, cplx* part,
               size_t part_elems, int64_t upper) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  if (K <= 0) {
    // C = beta * C
    scale_view(s, M, N, beta, C, batch);
    return;
  }
  const int tok = kstats_begin(s, K_F64_GEMM, 8.0 * M * N * (double)K * batch);
  const F64Plan p = plan_f64(M, N, K, batch, (batch == 1 && part) ? part_elems : 0);
  const int a_kfast = (A.cs_lo == 1) ? 1 : 0;
  const int b_kfast = (B.rs_lo == 1) ? 1 : 0;
  const int bk = p.shape->bk;
  const int kchunk = ((K + p.splits - 1) / p.splits + bk - 1) / bk * bk;
  const int nz = (K + kchunk - 1) / kchunk;
  // Long contractions in chains of 32 terms a thread, short ones of a few
  // columns in chains of 16 (kx groups of threads take every kx-th k); others
  // as they come (two more additions per output cost up to 8 % of the small
  // tiles at K = 200).  Rms error against double-double sums of Gaussian
  // entries, in these chains and in chains of 128 or whole K slices:
  //   64 x 48 x 22000   3.1e-16 (4.0e-16)   1800 x 4 x 1800   2.5e-16 (7.2e-16)
  //   157 x 6 x 123245  3.4e-16 (4.5e-16)   1217 x 4 x 901    2.2e-16 (3.3e-16)
  // The third takes 849 us, 844 us in chains of 128 and 863 us of 16.
  const int chain = K >= 4096 ? 32 : 16;
  const int period = K >= 4096 || N <= 8 ? std::max(1, chain * p.shape->kx / bk) : INT32_MAX;
  const int ntn = (N + p.shape->tn - 1) / p.shape->tn;
  const int64_t tiles = (int64_t)ntn * ((M + p.shape->tm - 1) / p.shape->tm);
  CVS_REQUIRE(tiles <= INT32_MAX, -1, "zgemm_f64: output too large");
  dim3 grid((unsigned)tiles, 1, nz > 1 ? nz : batch);
  p.shape->fn<<<grid, NT, 0, s>>>(M, N, K, alpha, A, B, beta, C, a_kfast, b_kfast, ntn, kchunk,
                                  period, upper, nz > 1 ? part : nullptr);
  CVS_CHECK_LAUNCH();
  kstats_end(s, tok);
  if (nz > 1) splitk_reduce(s, M, N, nz, part, beta, C);
}

}  // namespace cvs
