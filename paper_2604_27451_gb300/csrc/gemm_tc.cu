// Complex GEMM on the 5th-generation tensor cores (tcgen05, sm_103a).
//
//   C = alpha * A * B + beta * C, A: M x K, B: K x N complex (two-mode
//   views), C complex128.
//
// Precision: every real value x is split into bfloat16 parts x = x_h + x_l
// (x_h = bf16(x), x_l = bf16(x - x_h)); a real product keeps x_h y_h +
// x_h y_l + x_l y_h (~2^-16 relative), accumulated in FP32 in tensor
// memory.  The tensor-memory accumulation rounds each MMA step, so its
// error grows linearly with K (measured: ~1e-5 relative at K' ~ 10^4); the
// exact-slice kernel further down removes that limit.
//
// Layout: one real GEMM computes the complex product.  For every product
// term p = (pa, pb) the K dimension carries two segments of length Kp:
//   A row m       : [ re_pa(a) , im_pa(a) ]
//   B' row 2n     : [ re_pb(b) , -im_pb(b) ]   -> column 2n   = Re(a b)
//   B' row 2n + 1 : [ im_pb(b) ,  re_pb(b) ]   -> column 2n+1 = Im(a b)
// so K' = 2 * (number of product terms) * Kp and N' = 2 N, with real and
// imaginary parts of one output
// element in adjacent accumulator columns.  Packing (split + transpose into
// K-major rows, zero padding to the tile grid) is a bandwidth kernel; the
// GEMM itself is TMA -> shared memory (128B swizzle) -> tcgen05.mma with
// the accumulator in tensor memory -> tcgen05.ld -> complex128 epilogue.
//
// CTA: 128 threads.  Thread 0 issues the TMA loads, thread 32 issues the
// MMAs, all four warps drain TMEM (warp w owns TMEM lanes 32w..32w+31).
// Every mbarrier wait is bounded by a globaltimer deadline; on expiry the
// kernel records an error code, releases its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace cvs {

namespace {

constexpr int BM = 128;   // UMMA M
constexpr int BN = 256;   // UMMA N (real columns = 128 complex columns)
constexpr int BK = 64;    // bf16 elements per 128-byte swizzle row
constexpr int STAGES = 4;
constexpr int A_TILE = BM * BK * 2;
constexpr int B_TILE = BN * BK * 2;
constexpr int STAGE_BYTES = A_TILE + B_TILE;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr uint64_t WAIT_NS = 4000000000ull;  // 4 s bound on any wait

// product tables: (part of A, part of B), part 0 = hi, 1 = mid/lo, 2 = lo
template <int NP>
struct Split;
template <>
struct Split<3> {
  static constexpr int parts = 2;
  __device__ static int pa(int p) { return p == 2 ? 1 : 0; }
  __device__ static int pb(int p) { return p == 1 ? 1 : 0; }
};
template <>
struct Split<6> {
  static constexpr int parts = 3;
  // (0,0) (0,1) (1,0) (0,2) (1,1) (2,0)
  __device__ static int pa(int p) {
    return p == 2 ? 1 : p == 4 ? 1 : p == 5 ? 2 : 0;
  }
  __device__ static int pb(int p) {
    return p == 1 ? 1 : p == 3 ? 2 : p == 4 ? 1 : 0;
  }
};

// CTA rasterisation: consecutive CTAs walk groups of RASTER M-tiles
// column by column, so the CTAs resident at one time share A and B panels
// in L2 instead of streaming the whole B operand once per M-tile row.
constexpr int RASTER = 8;
__device__ __forceinline__ void tile_coords(int& mt, int& nt) {
  const int num_n = gridDim.x, num_m = gridDim.y;
  const int pid = blockIdx.y * num_n + blockIdx.x;
  const int per_group = RASTER * num_n;
  const int first_m = (pid / per_group) * RASTER;
  const int gsz = min(num_m - first_m, RASTER);
  const int local = pid - (first_m / RASTER) * per_group;
  mt = first_m + local % gsz;
  nt = local / gsz;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait on the phase with the given parity: try_wait suspends the
// thread in hardware for a while before it reports "not yet", so the loop
// polls without sleeping and reads the clock only every 64 tries
// true once the phase completes; false after limit_ns of the global timer
__device__ bool mbar_wait_for(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = gtime();
  for (uint32_t n = 1;; ++n) {
    if (mbar_try(bar, parity)) return true;
    if ((n & 63) == 0 && gtime() - t0 > limit_ns) return false;
  }
}
__device__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_for(bar, parity, WAIT_NS);
}

// an expired wait's code into the context's error word (mapped host memory;
// whichever thread writes last stands)
__device__ __forceinline__ void report(int* err, int code) {
  *(volatile int*)err = code;
  __threadfence_system();
}

// The error path of the bounded waits, on demand: one thread waits, with
// limit_ns, on an mbarrier that nothing arrives on.  The wait gives up, the
// kernel records code 5 in *err (as a GEMM's expired wait records its
// code) and returns.
__global__ void wait_probe_kernel(uint64_t limit_ns, int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait_for(&bar, 0, limit_ns)) report(err, 5);
  }
}
__device__ __forceinline__ void tma_load(const CUtensorMap* map, uint64_t* bar,
                                         void* dst, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::"
      "bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// shared-memory matrix descriptor: K-major, 128B swizzle, 8-row atoms of
// 1024 bytes stacked along M/N (stride 1024 B)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;            // leading byte offset (unused here)
  d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;            // descriptor version
  d |= (uint64_t)2 << 61;            // 128-byte swizzle
  return d;
}
// instruction descriptor, kind::f16: D f32, A/B bf16, both K-major
__device__ __forceinline__ uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t dtm, uint64_t a, uint64_t b,
                                     uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtm),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 "
      "[%0];" ::"r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]),
        "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__global__ void __launch_bounds__(128, 1)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                   const __grid_constant__ CUtensorMap tmB, int nkt, int zkt,
                   int M, int N, double alpha, double beta, View C,
                   cplx* part, int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_TILE;
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tslot = (uint32_t*)(done + 1);
  __shared__ int fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mt, nt;
  tile_coords(mt, nt);
  const int m0 = mt * BM, n0 = nt * BN;
  const int z = blockIdx.z;
  const int ktb = z * zkt, kte = min(nkt, ktb + zkt);  // non-empty by launch

  if (threadIdx.x == 0) {
    fail = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile(
        "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tslot)),
        "r"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (threadIdx.x == 0) {
    // TMA producer
    for (int i = 0; i < kte - ktb; ++i) {
      const int kt = ktb + i;
      const int s = i % STAGES;
      const uint32_t ph = (i / STAGES) & 1;
      if (i >= STAGES && !mbar_wait(&empty[s], ph ^ 1)) {
        fail = 1;
        break;
      }
      if (fail) break;
      mbar_expect_tx(&full[s], STAGE_BYTES);
      tma_load(&tmA, &full[s], sA + s * A_TILE, kt * BK, m0);
      tma_load(&tmB, &full[s], sB + s * B_TILE, kt * BK, n0);
    }
  } else if (threadIdx.x == 32) {
    // MMA issuer
    const uint32_t id = idesc_bf16(BM, BN);
    for (int i = 0; i < kte - ktb; ++i) {
      const int s = i % STAGES;
      const uint32_t ph = (i / STAGES) & 1;
      if (!mbar_wait(&full[s], ph)) {
        fail = 2;
        break;
      }
      fence_after();
      const uint64_t ad = sdesc(smem_u32(sA + s * A_TILE));
      const uint64_t bd = sdesc(smem_u32(sB + s * B_TILE));
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
        umma(tmem, ad + 2 * kk, bd + 2 * kk, id, (i | kk) ? 1u : 0u);
      umma_commit(&empty[s]);
    }
    umma_commit(done);
  }
  __syncwarp();
  const bool ok = mbar_wait(done, 0);
  __syncwarp();
  fence_after();
  if (ok && !fail) {
    const int m = m0 + warp * 32 + lane;
    const int64_t ro = (m < M && !part) ? vrow(C, m) : 0;
#pragma unroll 1
    for (int c = 0; c < BN; c += 16) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c, v);
      if (m < M) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int n = (n0 + c) / 2 + q;
          if (n < N) {
            cplx o = cmake(alpha * (double)v[2 * q], alpha * (double)v[2 * q + 1]);
            if (part) {
              part[((int64_t)z * M + m) * N + n] = o;
              continue;
            }
            cplx* d = C.p + ro + vcol(C, n);
            if (beta != 0.0) {
              cplx old = *d;
              o.x += beta * old.x;
              o.y += beta * old.y;
            }
            *d = o;
          }
        }
      }
    }
  } else if (lane == 0) {
    report(err, fail ? fail : 3);
  }
  fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(
                     tmem),
                 "r"(BN));
}

// ------------------------------------------------------------ packing
template <int PARTS>
__device__ __forceinline__ void split(double x, __nv_bfloat16* p) {
  double r = x;
#pragma unroll
  for (int q = 0; q < PARTS; ++q) {
    __nv_bfloat16 h = __double2bfloat16(r);
    p[q] = h;
    r -= (double)__bfloat162float(h);
  }
}

// A' [Mp][2 NP Kp]: row m, segment 2p + {0: re, 1: im} of part pa(p)
template <int NP>
__global__ void pack_a_kernel(View A, int M, int K, int k0, int Mp, int Kp,
                              __nv_bfloat16* out) {
  constexpr int PARTS = Split<NP>::parts;
  const int64_t ld = (int64_t)2 * NP * Kp;
  const int64_t total = (int64_t)Mp * Kp;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
       idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
    const int m = idx / Kp, k = idx % Kp;
    cplx a = cmake(0, 0);
    if (m < M && k < K) {
      a = A.p[vrow(A, m) + vcol(A, k0 + k)];
      if (A.conj) a.y = -a.y;
    }
    __nv_bfloat16 re[PARTS], im[PARTS];
    split<PARTS>(a.x, re);
    split<PARTS>(a.y, im);
    __nv_bfloat16* o = out + (int64_t)m * ld + k;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      o[(2 * p) * (int64_t)Kp] = re[Split<NP>::pa(p)];
      o[(2 * p + 1) * (int64_t)Kp] = im[Split<NP>::pa(p)];
    }
  }
}

// B' [Np2][2 NP Kp]: rows 2n (real part column) and 2n+1 (imaginary)
template <int NP>
__global__ void pack_b_kernel(View B, int K, int k0, int N, int Np2, int Kp,
                              __nv_bfloat16* out) {
  constexpr int PARTS = Split<NP>::parts;
  const int64_t ld = (int64_t)2 * NP * Kp;
  const int64_t total = (int64_t)(Np2 / 2) * Kp;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
       idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
    const int n = idx / Kp, k = idx % Kp;
    cplx b = cmake(0, 0);
    if (n < N && k < K) {
      b = B.p[vrow(B, k0 + k) + vcol(B, n)];
      if (B.conj) b.y = -b.y;
    }
    __nv_bfloat16 re[PARTS], im[PARTS];
    split<PARTS>(b.x, re);
    split<PARTS>(b.y, im);
    __nv_bfloat16* o0 = out + (int64_t)(2 * n) * ld + k;
    __nv_bfloat16* o1 = o0 + ld;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int q = Split<NP>::pb(p);
      o0[(2 * p) * (int64_t)Kp] = re[q];
      o0[(2 * p + 1) * (int64_t)Kp] = __hneg(im[q]);
      o1[(2 * p) * (int64_t)Kp] = im[q];
      o1[(2 * p + 1) * (int64_t)Kp] = re[q];
    }
  }
}

// ------------------------------------------------------- host helpers
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t,
                                  void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                         cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
    else
      (void)cudaGetLastError();
  });
  return fn;
}

CUtensorMap make_map(const void* base, int64_t rows, int64_t cols_bf16,
                     int box_rows) {
  EncodeTiledFn fn = encode_fn();
  CVS_REQUIRE(fn, -4, "cuTensorMapEncodeTiled unavailable");
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)cols_bf16, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols_bf16 * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base),
                  dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CVS_REQUIRE(r == CUDA_SUCCESS, -4, "cuTensorMapEncodeTiled failed");
  return m;
}

struct Dims {
  int Mp, Np2, Kp, nseg;
  size_t a_bytes, b_bytes;
};
Dims dims_of(int M, int N, int K, int nprod) {
  Dims d;
  d.Mp = (M + BM - 1) / BM * BM;
  d.Np2 = (2 * N + BN - 1) / BN * BN;
  d.Kp = (K + BK - 1) / BK * BK;
  d.nseg = 2 * nprod;
  d.a_bytes = (size_t)d.Mp * d.nseg * d.Kp * 2;
  d.b_bytes = (size_t)d.Np2 * d.nseg * d.Kp * 2;
  return d;
}

}  // namespace

bool tc_available() {
  static int avail = -1;
  static std::once_flag once;
  std::call_once(once, [] {
    int dev = 0, major = 0, minor = 0;
    avail = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) ==
            cudaSuccess &&
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) ==
            cudaSuccess)
      avail = (major == 10 && minor == 3 && encode_fn() != nullptr) ? 1 : 0;
    (void)cudaGetLastError();
    if (avail)
      cudaFuncSetAttribute(tc_gemm_kernel,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           SMEM_BYTES);
  });
  return avail == 1;
}

// packed-operand budget per K chunk
constexpr size_t PACK_BUDGET = (size_t)3 << 30;

int chunk_k(int Mp, int Np2, int K, int nseg) {
  // complex K per chunk so that both packed operands fit the budget
  const size_t per_k = (size_t)(Mp + Np2) * nseg * 2;
  int64_t kc = (int64_t)(PACK_BUDGET / per_k) / BK * BK;
  kc = std::max<int64_t>(kc, BK);
  return (int)std::min<int64_t>(kc, ((int64_t)K + BK - 1) / BK * BK);
}

size_t tc_workspace_bytes(int M, int N, int K, int nprod) {
  Dims d = dims_of(M, N, K, nprod);
  const int kc = chunk_k(d.Mp, d.Np2, K, d.nseg);
  return (size_t)(d.Mp + d.Np2) * d.nseg * kc * 2 + 256;
}

// number of K splits for an output of `tiles` CTA tiles over `kt` k-tiles
int tc_splits(int64_t tiles, int kt, int min_kt) {
  if (tiles >= 152) return 1;
  int64_t s = (2 * 152 + tiles - 1) / tiles;
  s = std::min<int64_t>(s, std::max(1, kt / min_kt));
  return (int)std::max<int64_t>(1, s);
}

void zgemm_tc(cudaStream_t s, int nprod, int M, int N, int K, double alpha,
              View A, View B, double beta, View C, void* work,
              size_t work_bytes, cplx* part, size_t part_elems, int* err) {
  if (M <= 0 || N <= 0) return;
  CVS_REQUIRE(nprod == 3 || nprod == 6, -1, "zgemm_tc: nprod must be 3 or 6");
  Dims d = dims_of(M, N, K, nprod);
  const int kc = chunk_k(d.Mp, d.Np2, K, d.nseg);
  CVS_REQUIRE(work_bytes >= (size_t)(d.Mp + d.Np2) * d.nseg * kc * 2, -1,
              "zgemm_tc: workspace too small");
  __nv_bfloat16* ap = (__nv_bfloat16*)work;
  __nv_bfloat16* bp = ap + (size_t)d.Mp * d.nseg * kc;
  const int64_t tiles = (int64_t)(d.Np2 / BN) * (d.Mp / BM);
  for (int k0 = 0; k0 < K; k0 += kc) {
    const int Kc = std::min(kc, K - k0);
    const int Kp = (Kc + BK - 1) / BK * BK;
    const unsigned ga = grid1d((int64_t)d.Mp * Kp, 256);
    const unsigned gb = grid1d((int64_t)(d.Np2 / 2) * Kp, 256);
    if (nprod == 3) {
      pack_a_kernel<3><<<ga, 256, 0, s>>>(A, M, Kc, k0, d.Mp, Kp, ap);
      CVS_CHECK_LAUNCH();
      pack_b_kernel<3><<<gb, 256, 0, s>>>(B, Kc, k0, N, d.Np2, Kp, bp);
    } else {
      pack_a_kernel<6><<<ga, 256, 0, s>>>(A, M, Kc, k0, d.Mp, Kp, ap);
      CVS_CHECK_LAUNCH();
      pack_b_kernel<6><<<gb, 256, 0, s>>>(B, Kc, k0, N, d.Np2, Kp, bp);
    }
    CVS_CHECK_LAUNCH();
    CUtensorMap ma = make_map(ap, d.Mp, (int64_t)d.nseg * Kp, BM);
    CUtensorMap mb = make_map(bp, d.Np2, (int64_t)d.nseg * Kp, BN);
    const int nkt = d.nseg * Kp / BK;
    int sp = tc_splits(tiles, nkt, 8);
    if (part == nullptr || (size_t)sp * M * N > part_elems) sp = 1;
    const int zkt = (nkt + sp - 1) / sp;
    const int nz = (nkt + zkt - 1) / zkt;
    const double beta_c = (k0 == 0) ? beta : 1.0;
    dim3 grid(d.Np2 / BN, d.Mp / BM, nz);
    const int tok = kstats_begin(s, K_TC_BF16X3, 8.0 * M * N * (double)Kc);
    tc_gemm_kernel<<<grid, 128, SMEM_BYTES, s>>>(ma, mb, nkt, zkt, M, N, alpha,
                                                 beta_c, C, nz > 1 ? part : nullptr,
                                                 err);
    CVS_CHECK_LAUNCH();
    kstats_end(s, tok);
    if (nz > 1) splitk_reduce(s, M, N, nz, part, beta_c, C);
  }
}

// ===========================================================================
// Exact-accumulation slice GEMM (an error-free splitting in the manner of
// Ozaki et al., Numer. Algorithms 59 (2012), mapped onto tcgen05).
//
// Every row m of A' and every output column n of B' gets a power-of-two
// scale 2^e with max |entry| < 2^e.  A scaled value a in (-1, 1) is cut into
// integer slices q_i in [-128, 128] with a = sum_i q_i 2^{-7(i+1)} + r,
// |r| <= 2^{-7 s - 1}; each slice is exactly a bf16.  A product of slices is
// an integer with |q q'| <= 2^14, and short runs of them sum exactly in the
// FP32 tensor-memory accumulator (up to 2^24; each kernel below counts its
// own: 512 products on pairs of CTAs, 256 in the tile kernel).  Slice
// products (i, j) with i + j <= s - 1 are kept; those of one order i + j
// share an accumulator.  Each finished run is drained from tensor memory
// while the next one is computed and added, times 2^{-7(i+j+2)}, to
// accumulators in registers (float-float, about 48 bits; 8 slices: 64-bit
// integers).  The epilogue applies 2^{e_m + f_n}, alpha and beta in FP64.
//
// The digits lie below a line's largest component, so a product is off by
// about 2^(1 - 7 s) of row max x column max per term, whatever the size of
// the term: small entries beside a large one are cut, and a line that holds
// an infinity or a not-a-number gives infinities or not-a-numbers.
//
// ===========================================================================
namespace {

constexpr int SLICE_BITS = 7;

__device__ __forceinline__ void ff_add(float& hi, float& lo, float x) {
  // TwoSum without contraction
  float s = __fadd_rn(hi, x);
  float bp = __fsub_rn(s, hi);
  float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  hi = s;
  lo = __fadd_rn(lo, e);
}

// ---------------------------------------------------------------------------
// The exact-slice GEMM on pairs of CTAs (cta_group::2, NS slices).  Packed
// operands: A'' row m = 2 NS segments (slice i, re / im) of Kp values, B''
// rows 2n (the real output column) and 2n + 1 (the imaginary one) = 2 NS
// segments (slice j, re-part / im-part: [re b, -im b] for row 2n and
// [im b, re b] for row 2n + 1).  One unit is one K block of 64 in one part:
// the NS tiles of A (128 rows in each CTA) and of B, from which all the NS
// (NS + 1) / 2 slice pairs are issued.  Pairs of one order o = i + j share
// the scale 2^{-7(o+2)} and one tensor-memory accumulator of PN columns; the
// orders lie side by side and fill the tensor memory (4 x 128, 7 x 64 and 64
// that nothing reads, or 8 x 64), so there is one set of them.
//
// Exact runs: |q_0| <= 2^7, |q_i| <= 2^6 for i > 0, so a run of 512 products
// (8 units) of every pair of an order stays within 2^23 (o = 0, 1), 2.5 2^22
// (o = 2), 3 2^22 (o = 3), 3.5 2^22 (o = 4) and 2^24 (o = 5) and sums exactly
// in FP32; order 6 may pass 2^24 by an eighth, where one rounding is 2^-55 of
// the order-0 product it is added to; order 7 may by a quarter (2^-62).  At
// the end of a run the orders finish one after the other, the drain warps add
// each to accumulators in registers (float-float; 8 slices: two 64-bit
// integers, so that FP64 rounds the whole sum once), and the next run
// overwrites an order once it is in registers.
//
// What bounds it: an MMA takes 90 to 100 cycles to issue and run whatever its
// width up to 128 columns, and a unit's operands arrive at ~11 TB/s over all
// SMs (96 KB a unit and CTA: 1.35 us).
// - 4 slices: a B slice is split over the CTAs by columns, 40 MMAs of 256 x
//   128 a unit.  One thread issues an MMA in 45 ns or more, so two warps do,
//   each with its own orders: 2.1 -> 1.8 us a unit.
// - 7 slices: the 112 MMAs of 256 x 64 took 5.0 us a unit however many warps
//   issued them.  B slices are whole in one CTA instead, so that one MMA
//   covers up to four (256 columns: two slices from either CTA, into four
//   adjacent orders): 44 MMAs, 2.75 us a unit.
// - 8 slices: the same with 15 MMAs of one to four slices per K step, 3.75 us.
// A's tiles free up one by one, so the copies run more than a unit ahead.
// The pairs of CTAs are persistent: the epilogue of a tile runs while the
// next one's first run is computed.  Measured (with the operands packed):
// 4096^3 4 slices 4.57 -> 3.23 ms (170 TFLOP/s, 0.91 of the measured bf16
// rate over 10 products; the tile kernel below before), 7 slices 21.2 -> 9.5
// ms (58 TFLOP/s, 0.87 over 28 products); 8 slices 11.5 ms (48 TFLOP/s, 0.92
// over 36 products; the FP64 kernels: 1.2 TFLOP/s), and 246000 x 200 by 200 x
// 150, one run a tile, 1.8 ms (33 TFLOP/s).
//
// Warps: 0 (lane 0) TMA producer; 1 .. ISSUERS of rank 0 (lane 0) MMA
// issuers; then 16 drain warps (warp w reads TMEM lanes 32 (w % 4) .. +31
// and CG columns of every order).  CTA rank r owns rows 128 r .. of the tile.
// ---------------------------------------------------------------------------
template <int NS>
struct PairCfg;
template <>
struct PairCfg<4> {
  static constexpr int PN = 128, ASLOTS = 8, BSTAGES = 3, ISSUERS = 2;
  static constexpr int R0 = 0, R1 = 0, R2 = 0, R3 = 0;
  static constexpr int B_ROWS = 4 * PN / 2;  // half of every slice
};
template <>
struct PairCfg<7> {
  static constexpr int PN = 64, ASLOTS = 9, BSTAGES = 2, ISSUERS = 1;
  // rows of the B regions of a stage: B_0 .. B_3 (two slices in each CTA),
  // B_4 | B_5, B_0 | B_1 (one in each), B_6 (half in each)
  static constexpr int R0 = 0, R1 = 128, R2 = 192, R3 = 256, B_ROWS = 288;
};
template <>
struct PairCfg<8> {
  static constexpr int PN = 64, ASLOTS = 7, BSTAGES = 2, ISSUERS = 1;
  // B_0 .. B_3 (two slices in each CTA), B_4 | B_5, B_6 | B_7, B_0 | B_1 (one
  // in each), then B_6, B_4, B_2, B_0 (half in each)
  static constexpr int R0 = 0, R1 = 128, R4 = 192, R2 = 256, R3 = 320, B_ROWS = 448;
};
constexpr int P_BM = 256;
constexpr int P_RUN = 8;  // units per exact run
template <int NS>
constexpr int pair_threads() {
  return 32 * (1 + PairCfg<NS>::ISSUERS + 16);
}
template <int NS>
constexpr int pair_smem() {
  using P = PairCfg<NS>;
  return P::ASLOTS * A_TILE + P::BSTAGES * P::B_ROWS * BK * 2 + 1024 + 512;
}

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the shared::cluster address of `p`'s counterpart in CTA 0 of the pair
__device__ __forceinline__ uint32_t leader_addr(const void* p) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(p)));
  return a;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// copy into this CTA's shared memory, counted on the leader's barrier
__device__ __forceinline__ void tma_load2(const CUtensorMap* map, uint32_t leader_bar,
                                          void* dst, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::"
      "bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(leader_bar), "r"(x), "r"(y)
      : "memory");
}
// 2^e for the exponents of a line (-1022 .. 1025; infinite above 1023)
__device__ __forceinline__ double pow2(int e) {
  return __hiloint2double(min(2047, 1023 + e) << 20, 0);
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void umma2(uint32_t dtm, uint64_t a, uint64_t b, uint32_t idesc,
                                      uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtm),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// arrives on the barrier's counterparts in both CTAs once this thread's MMAs
// issued so far are done
__device__ __forceinline__ void umma2_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster"
      ".b64 [%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

template <int NS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(pair_threads<NS>(), 1)
    tc_slice_pair_kernel(const __grid_constant__ CUtensorMap tmA,
                         const __grid_constant__ CUtensorMap tmB,
                         const __grid_constant__ CUtensorMap tmB2, int kpa, int ka_off,
                         int kpb, int kb_off, int nkb, int zl, int ntm, int ntn, int nitems,
                         int64_t upper, int M, int N, const int* __restrict__ eA, const int* __restrict__ eB,
                         double alpha, double beta, View C, cplx* part, int* err) {
  using P = PairCfg<NS>;
  constexpr int PN = P::PN, AS = P::ASLOTS, BS = P::BSTAGES, NI = P::ISSUERS;
  constexpr int CG = PN / 4;                       // columns of an order per drain warp
  constexpr int B_SLICE = (PN / 2) * BK * 2;       // this CTA's half of a B slice tile
  constexpr int B_STAGE = P::B_ROWS * BK * 2;
  constexpr uint32_t TMEM_COLS = 512;
  static_assert(NS * PN <= (int)TMEM_COLS, "accumulators fit the tensor memory");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + AS * A_TILE;
  uint64_t* fullA = (uint64_t*)(sB + BS * B_STAGE);
  uint64_t* emptyA = fullA + AS;
  uint64_t* fullB = emptyA + AS;
  uint64_t* emptyB = fullB + BS;
  uint64_t* afull = emptyB + BS;   // [NS]
  uint64_t* aempty = afull + NS;   // [NS]
  uint32_t* tslot = (uint32_t*)(aempty + NS);
  __shared__ int fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    fail = 0;
    for (int s = 0; s < AS; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&emptyA[s], NI);
    }
    for (int s = 0; s < BS; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyB[s], NI);
    }
    for (int o = 0; o < NS; ++o) {
      mbar_init(&afull[o], 1);
      mbar_init(&aempty[o], 32);  // the drain warps of both CTAs
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile(
        "tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tslot)),
        "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  cluster_sync();
  fence_after();
  const uint32_t tmem = *tslot;

  // item -> first row and column of its tile, its K blocks [kb0, kb1)
  auto item_at = [&](int it, int& m0, int& n0, int& z, int& kb0, int& kb1) {
    const int tiles = ntm * ntn;
    z = it / tiles;
    const int t = it - z * tiles;
    // groups of 4 M tiles walked column by column (shared panels in L2)
    const int per_group = 4 * ntn;
    const int g = t / per_group, first = 4 * g;
    const int gsz = min(ntm - first, 4);
    const int local = t - g * per_group;
    m0 = (first + local % gsz) * P_BM;
    n0 = (local / gsz) * (PN / 2);  // complex columns
    kb0 = z * zl;
    kb1 = min(nkb, kb0 + zl);
    // tiles wholly below the diagonal of a symmetric square are left out
    return !(upper >= 0 && n0 >= upper && n0 + PN / 2 <= upper + m0);
  };

  if (threadIdx.x == 0) {
    // TMA producer of this CTA's rows of A and half of the columns of B
    int u = 0, ia = 0;  // units and A tiles so far
    for (int it = pair; it < nitems && !fail; it += npairs) {
      int m0, n0, z, kb0, kb1;
      if (!item_at(it, m0, n0, z, kb0, kb1)) continue;
      const int ya = m0 + (int)rank * BM, yb = 2 * n0 + (int)rank * (PN / 2);
      for (int v = 0; v < 2 * (kb1 - kb0) && !fail; ++v, ++u) {
        const int kb = kb0 + v / 2, c = v & 1;
        const int sb = u % BS;
        if (u >= BS && !mbar_wait(&emptyB[sb], ((u / BS) & 1) ^ 1)) {
          fail = 1;
          break;
        }
        if (rank == 0) mbar_expect_tx(&fullB[sb], 2 * B_STAGE);
        const uint32_t fb = leader_addr(&fullB[sb]);
        uint8_t* st = sB + sb * B_STAGE;
        const int xb = c * kpb + (kb_off + kb) * BK;  // slice j: + 2 j kpb
        if constexpr (NS == 4) {
#pragma unroll
          for (int j = 0; j < NS; ++j)
            tma_load2(&tmB, fb, st + j * B_SLICE, 2 * j * kpb + xb, yb);
        } else if constexpr (NS == 8) {
          auto slice = [&](int row, int j) {  // all 64 columns of slice j
            tma_load2(&tmB, fb, st + row * BK * 2, 2 * j * kpb + xb, 2 * n0);
          };
          slice(P::R0, rank ? 2 : 0);
          slice(P::R0 + PN, rank ? 3 : 1);
          slice(P::R1, rank ? 5 : 4);
          slice(P::R4, rank ? 7 : 6);
          slice(P::R2, rank ? 1 : 0);
#pragma unroll
          for (int h = 0; h < 4; ++h)
            tma_load2(&tmB2, fb, st + (P::R3 + h * PN / 2) * BK * 2, 2 * (6 - 2 * h) * kpb + xb,
                      yb);
        } else {
          auto slice = [&](int row, int j) {  // all 64 columns of slice j
            tma_load2(&tmB, fb, st + row * BK * 2, 2 * j * kpb + xb, 2 * n0);
          };
          slice(P::R0, rank ? 2 : 0);
          slice(P::R0 + PN, rank ? 3 : 1);
          slice(P::R1, rank ? 5 : 4);
          slice(P::R2, rank ? 1 : 0);
          tma_load2(&tmB2, fb, st + P::R3 * BK * 2, 2 * 6 * kpb + xb, yb);
        }
        for (int i = 0; i < NS; ++i, ++ia) {
          const int sa = ia % AS;
          if (ia >= AS && !mbar_wait(&emptyA[sa], ((ia / AS) & 1) ^ 1)) {
            fail = 1;
            break;
          }
          if (rank == 0) mbar_expect_tx(&fullA[sa], 2 * A_TILE);
          tma_load2(&tmA, leader_addr(&fullA[sa]), sA + sa * A_TILE,
                    (2 * i + c) * kpa + (ka_off + kb) * BK, ya);
        }
      }
    }
    // The issuers' commits arrive in both CTAs' shared memory on their own
    // time, the last ones on barriers that no later copy waits for.  Each
    // producer waits for the last use of every slot, so that its CTA is still
    // there when they arrive: cluster_sync() does not order them.
    for (int j = max(0, u - BS); j < u && !fail; ++j)
      if (!mbar_wait(&emptyB[j % BS], (j / BS) & 1)) fail = 6;
    for (int j = max(0, ia - AS); j < ia && !fail; ++j)
      if (!mbar_wait(&emptyA[j % AS], (j / AS) & 1)) fail = 6;
  } else if (warp >= 1 && warp <= NI) {
    if (rank == 0 && lane == 0) {
      const uint32_t dhi = (uint32_t)(sdesc(0) >> 32);
      auto desc = [&](uint32_t lo) { return ((uint64_t)dhi << 32) | lo; };
      // NS = 4: issuer w takes the orders 3 - w and w, five pairs a step
      [[maybe_unused]] auto issue4 = [&](auto W) {
        constexpr int w = decltype(W)::value;
        constexpr int O1 = NS - 1 - w, O2 = w;
        const uint32_t id = idesc_bf16(P_BM, PN);
        int u = 0, ia = 0, r = 0;
        for (int it = pair; it < nitems && !fail; it += npairs) {
          int m0, n0, z, kb0, kb1;
          if (!item_at(it, m0, n0, z, kb0, kb1)) continue;
          const int nu = 2 * (kb1 - kb0);
          for (int v = 0; v < nu && !fail; ++v, ++u) {
            const bool first = v % P_RUN == 0;
            const bool last = v % P_RUN == P_RUN - 1 || v == nu - 1;
            const int sb = u % BS;
            bool ok = mbar_wait(&fullB[sb], (u / BS) & 1);
            // low words of the descriptors (the high word is the same for all)
            const uint32_t bd = (uint32_t)sdesc(smem_u32(sB + sb * B_STAGE));
            // pair (i, o - i) into order o
            auto mma = [&](int i, int o, uint32_t ad, bool start) {
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                umma2(tmem + o * PN, desc(ad + 2 * kk),
                      desc(bd + (o - i) * (B_SLICE >> 4) + 2 * kk), id,
                      (start && kk == 0) ? 0u : 1u);
            };
            if (first || last) {
              // by order: it waits for its drain at the start of a run and is
              // handed to the drain warps at the end
              uint32_t ad[NS];
#pragma unroll
              for (int i = 0; i < NS; ++i) {
                const int sa = (ia + i) % AS;
                ok = ok && mbar_wait(&fullA[sa], ((ia + i) / AS) & 1);
                ad[i] = (uint32_t)sdesc(smem_u32(sA + sa * A_TILE));
              }
#pragma unroll
              for (int o = 0; o < NS; ++o) {
                if (o != O1 && o != O2) continue;
                if (first && r > 0) ok = ok && mbar_wait(&aempty[o], (r - 1) & 1);
                if (!ok) break;
                fence_after();
#pragma unroll
                for (int i = 0; i <= o; ++i) mma(i, o, ad[i], first && i == 0);
                if (last) umma2_commit(&afull[o]);
              }
              if (ok)
#pragma unroll
                for (int i = 0; i < NS; ++i) umma2_commit(&emptyA[(ia + i) % AS]);
            } else {
              // by slice of A, whose slot is freed early
#pragma unroll
              for (int i = 0; i < NS; ++i) {
                const int sa = (ia + i) % AS;
                // also where no pair needs A_i: its slot is not given back
                // before it has been filled
                ok = ok && mbar_wait(&fullA[sa], ((ia + i) / AS) & 1);
                if (!ok) break;
                fence_after();
                const uint32_t ad = (uint32_t)sdesc(smem_u32(sA + sa * A_TILE));
                if (O1 >= i) mma(i, O1, ad, false);
                if (O2 >= i) mma(i, O2, ad, false);
                umma2_commit(&emptyA[sa]);
              }
            }
            if (!ok) {
              fail = 2;
              break;
            }
            umma2_commit(&emptyB[sb]);
            ia += NS;
            if (last) ++r;
          }
        }
      };
      // NS = 7, 8: one issuer, up to four slices of B per MMA
      [[maybe_unused]] auto issue_wide = [&]() {
        int u = 0, ia = 0, r = 0;
        for (int it = pair; it < nitems && !fail; it += npairs) {
          int m0, n0, z, kb0, kb1;
          if (!item_at(it, m0, n0, z, kb0, kb1)) continue;
          const int nu = 2 * (kb1 - kb0);
          for (int v = 0; v < nu && !fail; ++v, ++u) {
            const bool first = v % P_RUN == 0;
            const bool last = v % P_RUN == P_RUN - 1 || v == nu - 1;
            const int sb = u % BS;
            bool ok = mbar_wait(&fullB[sb], (u / BS) & 1);
            const uint32_t bd = (uint32_t)sdesc(smem_u32(sB + sb * B_STAGE));
            // A_i with the slices of the region at `row` into orders o ..
            auto mma = [&](int o, uint32_t ad, int row, int n, bool start) {
              const uint32_t id = idesc_bf16(P_BM, n);
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                umma2(tmem + o * PN, desc(ad + 2 * kk),
                      desc(bd + row * (BK * 2 >> 4) + 2 * kk), id, (start && kk == 0) ? 0u : 1u);
            };
            // the drains of orders [o0, o1) at the start of a run
            auto drained = [&](int o0, int o1) {
              for (int o = o0; o < o1 && first && r > 0; ++o)
                ok = ok && mbar_wait(&aempty[o], (r - 1) & 1);
              if (ok) fence_after();
              return ok;
            };
#pragma unroll
            for (int i = 0; i < NS; ++i) {
              const int sa = (ia + i) % AS;
              ok = ok && mbar_wait(&fullA[sa], ((ia + i) / AS) & 1);
              if (!ok) break;
              fence_after();
              const uint32_t ad = (uint32_t)sdesc(smem_u32(sA + sa * A_TILE));
              const bool start = first && i == 0;
              if (i < 5) {
                if (i == 0 && !drained(0, 4)) break;
                mma(i, ad, P::R0, 4 * PN, start);
              }
              if (i < 3) {
                if (i == 0 && !drained(4, 6)) break;
                mma(i + 4, ad, P::R1, 2 * PN, start);
              }
              if (i == 0 && !drained(6, NS)) break;
              if constexpr (NS == 7) {
                if (i == 0) mma(6, ad, P::R3, PN, first);
                if (i >= 5) mma(i, ad, P::R2, 2 * PN, false);
              } else if constexpr (NS == 8) {
                if (i == 0) mma(6, ad, P::R4, 2 * PN, first);
                if (i == 5 || i == 6) mma(i, ad, P::R2, 2 * PN, false);
                // (1, 6), (3, 4), (5, 2) and (7, 0)
                if (i & 1) mma(7, ad, P::R3 + (i / 2) * (PN / 2), PN, false);
              }
              umma2_commit(&emptyA[sa]);
              // no later pair of this unit adds to order i
              if (last) umma2_commit(&afull[i]);
            }
            if (!ok) {
              fail = 2;
              break;
            }
            umma2_commit(&emptyB[sb]);
            ia += NS;
            if (last) ++r;
          }
        }
      };
      if constexpr (NS == 4) {
        if (warp == 1) issue4(std::integral_constant<int, 0>());
        if (warp == 2) issue4(std::integral_constant<int, 1>());
      } else {
        issue_wide();
      }
    }
  } else if (warp > NI) {
    // drain warps
    const int q = warp & 3;               // TMEM lane quarter
    const int cq = (warp - 1 - NI) >> 2;  // CG columns of every order
    const uint32_t ae = leader_addr(aempty);
    bool ok = true;
    int r = 0;
    for (int it = pair; it < nitems && ok; it += npairs) {
      int m0, n0, z, kb0, kb1;
      if (!item_at(it, m0, n0, z, kb0, kb1)) continue;
      const int nruns = (2 * (kb1 - kb0) + P_RUN - 1) / P_RUN;
      // NS < 8: float-float sums; 8: the orders 0 .. 3 and 4 .. 7 as exact
      // integers in units of 2^-35 and 2^-63 (a run adds at most 2^46)
      using Acc = std::conditional_t<NS == 8, long long, float>;
      Acc hi[CG], lo[CG];
#pragma unroll
      for (int i = 0; i < CG; ++i) hi[i] = lo[i] = 0;
      for (int rr = 0; rr < nruns && ok; ++rr, ++r) {
        // order o is handed over, then f(i, value) for this warp's columns
        auto drain = [&](int o, auto f) {
          if (!mbar_wait(&afull[o], r & 1)) return false;
          fence_after();
#pragma unroll
          for (int h = 0; h < CG / 8; ++h) {
            float v[8];
            tmem_ld8(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(o * PN + cq * CG + 8 * h), v);
            if (h == CG / 8 - 1) {
              // the order is in registers: the next run may overwrite it
              fence_before();
              __syncwarp();
              if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(
                                 ae + 8 * o)
                             : "memory");
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) f(8 * h + i, v[i]);
          }
          return true;
        };
        if constexpr (NS == 8) {
#pragma unroll 1
          for (int o = 0; o < 4 && ok; ++o) {
            const int mul = 1 << SLICE_BITS * (3 - o);
            ok = drain(o, [&](int i, float v) { hi[i] += (long long)__float2int_rn(v) * mul; });
          }
#pragma unroll 1
          for (int o = 4; o < 8 && ok; ++o) {
            const int mul = 1 << SLICE_BITS * (7 - o);
            ok = drain(o, [&](int i, float v) { lo[i] += (long long)__float2int_rn(v) * mul; });
          }
        } else {
#pragma unroll 1
          for (int o = 0; o < NS && ok; ++o) {
            // 2^{-7 (o + 2)}
            const float sc = __int_as_float((127 - SLICE_BITS * (o + 2)) << 23);
            ok = drain(o, [&](int i, float v) {
              ff_add(hi[i], lo[i], v * sc);
              // one group of 8 at a time: the accumulators take most registers
              asm volatile("" : "+f"(hi[i]), "+f"(lo[i]));
            });
          }
        }
      }
      if (!ok || fail) {
        ok = false;
        if (lane == 0) report(err, fail ? fail : 3);
        break;
      }
      const int m = m0 + (int)rank * BM + q * 32 + lane;
      if (m < M) {
        const int64_t ro = part ? 0 : vrow(C, m);
        const double em = alpha * pow2(eA[m]);
#pragma unroll
        for (int i = 0; i < CG / 2; ++i) {
          const int n = n0 + cq * (CG / 2) + i;
          if (n < N) {
            // one column at a time (nothing hoisted): the accumulators take
            // most registers
            if constexpr (NS != 8)
              asm volatile("" : "+f"(hi[2 * i]), "+f"(lo[2 * i]), "+f"(hi[2 * i + 1]),
                           "+f"(lo[2 * i + 1]) :: "memory");
            else
              asm volatile("" : "+l"(hi[2 * i]), "+l"(lo[2 * i]), "+l"(hi[2 * i + 1]),
                           "+l"(lo[2 * i + 1]) :: "memory");
            const double sc = em * pow2(eB[n]);
            auto sum = [&](int j) {
              if constexpr (NS == 8)
                return fma((double)hi[j], 0x1p-35, (double)lo[j] * 0x1p-63);
              else
                return (double)hi[j] + (double)lo[j];
            };
            cplx o = cmake(sc * sum(2 * i), sc * sum(2 * i + 1));
            if (part) {
              part[((int64_t)z * M + m) * N + n] = o;
              continue;
            }
            cplx* d = C.p + ro + vcol(C, n);
            if (beta != 0.0) {
              const cplx old = *d;
              o.x += beta * old.x;
              o.y += beta * old.y;
            }
            *d = o;
          }
        }
      }
    }
  }
  __syncwarp();
  // an expired wait: let the copies in flight land before the memory goes
  if (threadIdx.x == 0 && fail) {
    const uint64_t t0 = gtime();
    for (int n = 0; n < (1 << 20) && gtime() - t0 < 2000000; ++n) __nanosleep(1000);
  }
  if (threadIdx.x == 0 && fail) report(err, fail);
  fence_before();
  __syncthreads();
  __syncwarp();
  cluster_sync();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS));
}

// Exponents and slices work on the IEEE bits with integer arithmetic (this
// GPU runs FP64 at a small fraction of its integer and FP32 rates).  For a
// normal double the biased exponent field E gives |x| < 2^(E - 1022); zeros
// and subnormals count as 0.

__device__ __forceinline__ int exp_field(double x) {
  return (int)((__double_as_longlong(x) >> 52) & 0x7FF);
}

// column offset of a view for an int column index (32-bit index math)
__device__ __forceinline__ int64_t vcol32(const View& v, int c) {
  if (v.c_lo == INT32_MAX) return (int64_t)c * v.cs_lo;
  const int h = c / v.c_lo, r = c - h * v.c_lo;
  return (int64_t)h * v.cs_hi + (v.ctab ? (int64_t)v.ctab[r] : (int64_t)r * v.cs_lo);
}

// Operands are packed line by line: rows of A, columns of B (a transposed
// view), so that lines are the view's rows and k its columns.

// Exponents over [k0, k0 + K): e with max |re|, |im| < 2^e for every element
// of a line; an all-zero line gets -1022.  The caller presets e[] below
// -1022 (bytes 0x80); maxima are folded into it with atomicMax, so that an
// operand with few lines and a K in the millions still spreads over every
// SM.  KFAST: a warp takes a (line, segment of EXP_SEG) task, lanes along k.
// Otherwise (the lines are the contiguous mode: columns of a row-major B,
// (a, b) rows of B^P) lanes take adjacent lines and walk a segment, so that
// the warp reads 512 contiguous bytes a step instead of half a sector each.
// (942 lines of 5181: 56 us in segments of 4096, 16 us of 1024.)
constexpr int EXP_SEG = 1024, EXP_SEG_LINES = 64;
template <bool KFAST>
__global__ void __launch_bounds__(256) line_exp_kernel(View X, int L, int K, int k0, int* e) {
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  constexpr int SEG = KFAST ? EXP_SEG : EXP_SEG_LINES;
  const int nsg = (K + SEG - 1) / SEG;
  const int64_t nlg = KFAST ? L : (L + 31) / 32;  // lines, or groups of 32
  for (int64_t t = warp; t < nlg * nsg; t += nwarp) {
    const int64_t lg = t / nsg;
    const int k1 = (int)(t % nsg) * SEG, k2 = min(K, k1 + SEG);
    const int l = (int)(KFAST ? lg : lg * 32 + lane);
    int mx = 0;
    if (l < L) {
      const cplx* x = X.p + vrow(X, l);
      for (int k = KFAST ? k1 + lane : k1; k < k2; k += KFAST ? 32 : 1) {
        const cplx a = x[vcol32(X, k0 + k)];
        mx = max(mx, max(exp_field(a.x), exp_field(a.y)));
      }
    }
    if (KFAST) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) atomicMax(e + l, mx - 1022);
    } else if (l < L) {
      atomicMax(e + l, mx - 1022);
    }
  }
}

unsigned warp_tasks_grid(int64_t lines, int K, int seg) {
  const int64_t ntask = lines * ((K + seg - 1) / seg);
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((ntask + 7) / 8, 152 * 32));
}

// S balanced 7-bit slices of t = x 2^-e (|t| < 1): T = round(t 2^(7S)),
// then digits q_{S-1} .. q_1 in [-64, 63] from the bottom and q_0 = the
// rest, in [-128, 128], so that t = sum_i q_i 2^(-7(i+1)) + r with |r| <=
// 2^(-7S-1); each q_i is exact in bf16, the upper half of its float.
//
// In 32-bit integer arithmetic: with s = 1075 + e - 7S - E >= 53 - 7S
// the bits to drop, T = ((m >> (s - 1)) + 1) >> 1.  Adding 64 at every lower
// digit's place makes its balanced digit the plain one less 64, and a digit
// n becomes the float n - 64 by an OR into the mantissa of 1.5 2^23 and a
// subtraction.  (64-bit digits and int-to-float conversions held the packing
// kernels to 2 TB/s.)
__device__ __forceinline__ float digit(int n) {  // n in [0, 127]: n - 64
  return __int_as_float(0x4B400000 | n) - 12582976.0f;
}
template <int S>
__device__ __forceinline__ void slices(double x, int e, float* q) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int E = (hi >> 20) & 0x7FF;
  const uint32_t mh = (hi & 0xFFFFF) | 0x100000;
  const int s = 1075 + e - 7 * S - E;  // >= 53 - 7 S, since |x| < 2^e
  if constexpr (S == 4) {
    const int h = (int)__funnelshift_l(lo, mh, 8);  // m >> 24
    int T = ((h >> min(31, max(0, s - 25))) + 1) >> 1;
    T = E == 0 ? 0 : ((int)hi < 0 ? -T : T);
    T += 64 + (64 << 7) + (64 << 14);
    q[3] = digit(T & 127);
    q[2] = digit((T >> 7) & 127);
    q[1] = digit((T >> 14) & 127);
    q[0] = __int_as_float(0x4B400000 + (T >> 21)) - 12582912.0f;
  } else if constexpr (S == 8) {
    // (s >= -3: four more bits below the significand)
    const long long m = (((long long)mh << 32) | lo) << 4;
    long long T = ((m >> min(63, max(0, s + 3))) + 1) >> 1;
    T = E == 0 ? 0 : ((int)hi < 0 ? -T : T);
    T += 64ll * (1 + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35) +
                 (1ll << 42));
    const int tl = (int)(T & 0xFFFFFFF), th = (int)(T >> 28);
    q[7] = digit(tl & 127);
    q[6] = digit((tl >> 7) & 127);
    q[5] = digit((tl >> 14) & 127);
    q[4] = digit((tl >> 21) & 127);
    q[3] = digit(th & 127);
    q[2] = digit((th >> 7) & 127);
    q[1] = digit((th >> 14) & 127);
    q[0] = __int_as_float(0x4B400000 + (th >> 21)) - 12582912.0f;
  } else {
    static_assert(S == 7, "4, 7 or 8 slices");
    const long long m = ((long long)mh << 32) | lo;
    long long T = ((m >> min(63, max(0, s - 1))) + 1) >> 1;
    T = E == 0 ? 0 : ((int)hi < 0 ? -T : T);
    // 64 at the places of digits 6 .. 1
    T += 64ll * (1 + (1ll << 7) + (1ll << 14) + (1ll << 21) + (1ll << 28) + (1ll << 35));
    const int tl = (int)(T & 0xFFFFFFF), th = (int)(T >> 28);
    q[6] = digit(tl & 127);
    q[5] = digit((tl >> 7) & 127);
    q[4] = digit((tl >> 14) & 127);
    q[3] = digit((tl >> 21) & 127);
    q[2] = digit(th & 127);
    q[1] = digit((th >> 7) & 127);
    q[0] = __int_as_float(0x4B400000 + (th >> 14)) - 12582912.0f;
  }
}
// two exact bf16 values as one word
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// Packed lines: out line l (A: one, B: the two lines 2l and 2l + 1) = 2 S
// segments of Kp, segment 2 i + {0: re, 1: im} of slice i; for B line 2l
// holds [re, -im] and line 2l + 1 [im, re].  Two adjacent k per lane.
template <int S, bool ISB>
__device__ __forceinline__ void pack_two(cplx a0, cplx a1, int e, __nv_bfloat16* o, int64_t ld,
                                         int Kp) {
  float r0[S], i0[S], r1[S], i1[S];
  slices<S>(a0.x, e, r0);
  slices<S>(a0.y, e, i0);
  slices<S>(a1.x, e, r1);
  slices<S>(a1.y, e, i1);
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const uint32_t re = bf16_pair(r0[i], r1[i]), im = bf16_pair(i0[i], i1[i]);
    __nv_bfloat16* p = o + (2 * i) * (int64_t)Kp;
    *(uint32_t*)p = re;
    if (!ISB) {
      *(uint32_t*)(p + Kp) = im;
    } else {
      *(uint32_t*)(p + Kp) = bf16_pair(-i0[i], -i1[i]);
      *(uint32_t*)(p + ld) = im;
      *(uint32_t*)(p + ld + Kp) = re;
    }
  }
}

// Lp padded lines.  k contiguous: a warp takes a (line, segment of PACK_SEG)
// task.
constexpr int PACK_SEG = 2048;
template <int S, bool ISB>
__global__ void __launch_bounds__(256)
    slice_pack_kernel(View X, int L, int K, int k0, int Lp, int Kp,
                      const int* __restrict__ eX, __nv_bfloat16* out) {
  const int64_t ld = (int64_t)2 * S * Kp;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nsg = (Kp + PACK_SEG - 1) / PACK_SEG;
  for (int64_t t = warp; t < (int64_t)Lp * nsg; t += nwarp) {
    const int l = (int)(t / nsg), k1 = (int)(t % nsg) * PACK_SEG;
    const int k2 = min(Kp, k1 + PACK_SEG);
    const bool live = l < L;
    const cplx* x = X.p + (live ? vrow(X, l) : 0);
    const int e = live ? eX[l] : 0;
    __nv_bfloat16* o = out + (int64_t)l * (ISB ? 2 : 1) * ld;
    for (int k = k1 + 2 * lane; k < k2; k += 64) {
      cplx a0 = cmake(0, 0), a1 = cmake(0, 0);
      if (live && k < K) a0 = x[vcol32(X, k0 + k)];
      if (live && k + 1 < K) a1 = x[vcol32(X, k0 + k + 1)];
      if (X.conj) {
        a0.y = -a0.y;
        a1.y = -a1.y;
      }
      pack_two<S, ISB>(a0, a1, e, o + k, ld, Kp);
    }
  }
}

// Lines contiguous: a block takes tiles of 32 lines x 64 k, reads them along
// the lines (512 bytes a warp) and packs them along k from shared memory.
template <int S, bool ISB>
__global__ void __launch_bounds__(256)
    slice_pack_lines_kernel(View X, int L, int K, int k0, int Lp, int Kp,
                            const int* __restrict__ eX, __nv_bfloat16* out) {
  __shared__ cplx tile[64][33];
  const int64_t ld = (int64_t)2 * S * Kp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkt = Kp / 64;
  const int64_t ntask = (int64_t)((Lp + 31) / 32) * nkt;
  for (int64_t t = blockIdx.x; t < ntask; t += gridDim.x) {
    const int l0 = (int)(t / nkt) * 32, kt = (int)(t % nkt) * 64;
    const bool live = l0 + lane < L;
    const cplx* x = X.p + (live ? vrow(X, l0 + lane) : 0);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int k = kt + warp + 8 * r;
      cplx a = cmake(0, 0);
      if (live && k < K) a = x[vcol32(X, k0 + k)];
      if (X.conj) a.y = -a.y;
      tile[warp + 8 * r][lane] = a;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int l = l0 + warp * 4 + r;
      if (l >= Lp) break;
      const int e = l < L ? eX[l] : 0;
      pack_two<S, ISB>(tile[2 * lane][l - l0], tile[2 * lane + 1][l - l0], e,
                       out + (int64_t)l * (ISB ? 2 : 1) * ld + kt + 2 * lane, ld, Kp);
    }
  }
}

// exponents and packed slices of L lines (padded to Lp) of X over [k0, k0 + K)
template <int S, bool ISB>
void pack_lines(cudaStream_t s, View X, int L, int K, int k0, int Lp, int Kp, int* e,
                size_t e_count, __nv_bfloat16* out) {
  CVS_CUDA(cudaMemsetAsync(e, 0x80, e_count * sizeof(int), s));
  // lanes go along the contiguous mode (along k when neither or both are)
  const bool lines = X.cs_lo != 1 && X.rs_lo == 1 && (X.r_lo == INT32_MAX || X.r_lo >= 16);
  if (lines) {
    line_exp_kernel<false><<<warp_tasks_grid((L + 31) / 32, K, EXP_SEG_LINES), 256, 0, s>>>(
        X, L, K, k0, e);
    CVS_CHECK_LAUNCH();
    const int64_t tiles = (int64_t)((Lp + 31) / 32) * (Kp / 64);
    slice_pack_lines_kernel<S, ISB>
        <<<(unsigned)std::min<int64_t>(tiles, 152 * 16), 256, 0, s>>>(X, L, K, k0, Lp, Kp, e,
                                                                      out);
  } else {
    line_exp_kernel<true><<<warp_tasks_grid(L, K, EXP_SEG), 256, 0, s>>>(X, L, K, k0, e);
    CVS_CHECK_LAUNCH();
    slice_pack_kernel<S, ISB><<<warp_tasks_grid(Lp, Kp, PACK_SEG), 256, 0, s>>>(X, L, K, k0, Lp,
                                                                               Kp, e, out);
  }
  CVS_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// SLICE4 with slice reuse.  The packed operands hold each slice once: A''
// row m = 8 segments (slice i, re / im) of Kp values; B'' rows 2n (the real
// output column) and 2n+1 (the imaginary one) = 8 segments (slice j,
// re-part / im-part: [re b, -im b] for row 2n and [im b, re b] for row
// 2n+1).  One pipeline stage is one K block of 64 in one part c (re or im):
// the four A tiles A_{i,c} (128 x 64) and four B tiles B_{j,c} (64 x 64),
// 96 KB, from which all ten slice pairs are issued.  Pairs of one order
// o = i + j share the scale 2^{-7(o+2)} and one tensor-memory accumulator;
// a run is 2 K blocks x 2 parts: at most 4 pairs x 256 products of
// |q q'| <= 2^13 (2^14 for order 0, one pair) per element, so every run
// sums exactly in FP32.  TMEM: 2 buffers x 4 orders x 64 columns = 512.
// The B tiles of a stage lie back to back (one 256-row K-major operand) and
// the orders of a buffer side by side, so the pairs (i, 0..3-i) are one MMA
// of A_i with B_0..B_{3-i} (N = 64 (4 - i)) into orders i..3: four MMAs
// per K step instead of ten, and each A tile is read from shared memory
// once.  The drain adds each order, times its scale, to float-float
// accumulators.
//
// It serves the narrow and small products that the pairs of CTAs above would
// pad (plan_slices).
//
// CTA: 576 threads, tile 128 x 64 (N' = 64: 32 complex columns).  Warp 0
// lane 0: TMA producer; warp 1 lane 0: MMA issuer; warps 2..17: drain (warp
// w reads TMEM lanes 32 (w % 4) .. +31 and the 16 columns [16 c, 16 c + 16),
// c = (w - 2) / 4, of every order).
// ---------------------------------------------------------------------------
constexpr int RBN = 64;                  // N' per CTA
constexpr int R_A_TILE = BM * BK * 2;    // 16 KB
constexpr int R_B_TILE = RBN * BK * 2;   // 8 KB
constexpr int R_STAGE = 4 * R_A_TILE + 4 * R_B_TILE;  // 96 KB
constexpr int R_STAGES = 2;
constexpr int R_SMEM = R_STAGES * R_STAGE + 1024 + 512;
constexpr int R_RUN = 4;                 // units (K block, part) per exact run

__global__ void __launch_bounds__(576, 1)
    tc_slice4r_kernel(const __grid_constant__ CUtensorMap tmA,
                      const __grid_constant__ CUtensorMap tmB, int kpa, int ka_off,
                      int kpb, int kb_off, int nkb, int zl, int M, int N,
                      const int* __restrict__ eA,
                      const int* __restrict__ eB, double alpha, double beta,
                      View C, cplx* part, int64_t upper, int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + R_STAGES * R_STAGE);
  uint64_t* empty = full + R_STAGES;
  uint64_t* afull = empty + R_STAGES;  // [2]
  uint64_t* aempty = afull + 2;        // [2]
  uint32_t* tslot = (uint32_t*)(aempty + 2);
  __shared__ int fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mt, nt;
  tile_coords(mt, nt);
  const int m0 = mt * BM, n0 = nt * RBN;
  const int z = blockIdx.z;
  // a tile wholly below the diagonal of a symmetric square is left out
  if (upper >= 0 && n0 / 2 >= upper && (n0 + RBN) / 2 <= upper + m0) return;
  // this CTA's K blocks [kb0, kb1); units u = 2 (kb - kb0) + c
  const int kb0 = z * zl, kb1 = min(nkb, kb0 + zl);
  const int nunits = 2 * max(0, kb1 - kb0);
  const int nruns = (nunits + R_RUN - 1) / R_RUN;

  if (threadIdx.x == 0) {
    fail = 0;
    for (int s = 0; s < R_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&afull[b], 1);
      mbar_init(&aempty[b], 16);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile(
        "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            smem_u32(tslot)),
        "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (threadIdx.x == 0) {
    // TMA producer: unit u -> K block kb0 + u / 2, part c = u % 2
    for (int u = 0; u < nunits; ++u) {
      const int s = u % R_STAGES;
      const uint32_t ph = (u / R_STAGES) & 1;
      if (u >= R_STAGES && !mbar_wait(&empty[s], ph ^ 1)) {
        fail = 1;
        break;
      }
      if (fail) break;
      const int kb = kb0 + u / 2, c = u & 1;
      uint8_t* st = smem + s * R_STAGE;
      mbar_expect_tx(&full[s], R_STAGE);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        tma_load(&tmA, &full[s], st + i * R_A_TILE, (2 * i + c) * kpa + (ka_off + kb) * BK,
                 m0);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        tma_load(&tmB, &full[s], st + 4 * R_A_TILE + j * R_B_TILE,
                 (2 * j + c) * kpb + (kb_off + kb) * BK, n0);
    }
  } else if (threadIdx.x == 32) {
    // MMA issuer: for each unit, the ten pairs into their order's
    // accumulator of the run's buffer
    // N = 64 (4 - i) for the MMA of A_i
    uint32_t idn[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) idn[i] = idesc_bf16(BM, RBN * (4 - i));
    for (int r = 0; r < nruns && !fail; ++r) {
      const int b = r & 1;
      if (r >= 2 && !mbar_wait(&aempty[b], ((r >> 1) + 1) & 1)) {
        fail = 4;
        break;
      }
      fence_after();
      const int u0 = r * R_RUN, u1 = min(nunits, u0 + R_RUN);
      for (int u = u0; u < u1; ++u) {
        const int s = u % R_STAGES;
        const uint32_t ph = (u / R_STAGES) & 1;
        if (!mbar_wait(&full[s], ph)) {
          fail = 2;
          break;
        }
        fence_after();
        const uint32_t st = smem_u32(smem + s * R_STAGE);
        const uint64_t bd = sdesc(st + 4 * R_A_TILE);  // B_0 .. B_3
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // pairs (i, 0 .. 3 - i) into orders i .. 3; the first MMA of a
          // run (i = 0 covers every order) starts the accumulators
          const uint32_t dt = tmem + (uint32_t)((b * 4 + i) * RBN);
          const uint64_t ad = sdesc(st + i * R_A_TILE);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            umma(dt, ad + 2 * kk, bd + 2 * kk, idn[i],
                 (u != u0 || i != 0 || kk != 0) ? 1u : 0u);
        }
        umma_commit(&empty[s]);
      }
      umma_commit(&afull[b]);
    }
  } else if (warp >= 2) {
    // drain warps
    const int q = warp & 3;          // TMEM lane quarter
    const int cq = (warp - 2) >> 2;  // 16-column chunk of the 64
    float hi[16], lo[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) hi[i] = lo[i] = 0.f;
    bool ok = true;
    for (int r = 0; r < nruns; ++r) {
      const int b = r & 1;
      if (!mbar_wait(&afull[b], (r >> 1) & 1)) {
        ok = false;
        break;
      }
      fence_after();
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const float sc = exp2f(-(float)(SLICE_BITS * (o + 2)));
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((b * 4 + o) * RBN + cq * 16), v);
#pragma unroll
        for (int i = 0; i < 16; ++i) ff_add(hi[i], lo[i], v[i] * sc);
      }
      fence_before();
      __syncwarp();
      if (lane == 0) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&aempty[b]))
                     : "memory");
      }
    }
    if (!ok || fail) {
      if (lane == 0) report(err, fail ? fail : 3);
    } else {
      const int m = m0 + q * 32 + lane;
      if (m < M) {
        const int64_t ro = part ? 0 : vrow(C, m);
        const double em = ldexp(1.0, eA[m]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int n = (n0 + cq * 16) / 2 + i;
          if (n < N) {
            const double sc = alpha * em * ldexp(1.0, eB[n]);
            cplx o = cmake(sc * ((double)hi[2 * i] + (double)lo[2 * i]),
                           sc * ((double)hi[2 * i + 1] + (double)lo[2 * i + 1]));
            if (part) {
              part[((int64_t)z * M + m) * N + n] = o;
              continue;
            }
            cplx* d = C.p + ro + vcol(C, n);
            if (beta != 0.0) {
              const cplx old = *d;
              o.x += beta * old.x;
              o.y += beta * old.y;
            }
            *d = o;
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// packed geometry: every slice once (2 segments each), rows padded to the
// tiles.  K runs in chunks of kc, each with its own exponents; a B operand
// held in a cache is packed once over its whole K (KpF) and only A's pack
// counts against the budget.  kc is what PACK_BUDGET holds at 8 (SLICE4) or
// 56 (SLICE7) segments: a chunk's length is also the reach of its exponents,
// so the 7-slice chunks stay as short as when every slice pair had segments
// of its own.
struct SDims {
  int Mp, Np2, nseg, cseg, kc, KpF;
  size_t a_bytes, b_bytes, e_bytes;
};
SDims sdims_of(int M, int N, int K, int nslices, bool b_cached, bool a_cached = false) {
  SDims d;
  const int tn = nslices == 4 ? RBN : 128;
  d.Mp = (M + BM - 1) / BM * BM;
  d.Np2 = (2 * N + tn - 1) / tn * tn;
  d.nseg = 2 * nslices;
  d.cseg = nslices == 7 ? nslices * (nslices + 1) : d.nseg;
  d.KpF = (int)(((int64_t)K + BK - 1) / BK * BK);
  const size_t per_k = (size_t)((a_cached ? 0 : d.Mp) + (b_cached ? 0 : d.Np2)) * d.cseg * 2;
  int64_t kc = per_k ? (int64_t)(PACK_BUDGET / per_k) / BK * BK : (int64_t)d.KpF;
  kc = std::max<int64_t>(kc, BK);
  d.kc = (int)std::min<int64_t>(kc, d.KpF);
  d.a_bytes = a_cached ? 0 : (size_t)d.Mp * d.nseg * d.kc * 2;
  d.b_bytes = b_cached ? 0 : (size_t)d.Np2 * d.nseg * d.kc * 2;
  d.e_bytes = ((size_t)d.Mp + d.Np2 / 2 + 64) * sizeof(int);
  return d;
}

// How a product of nkb K blocks is laid out on the GPU, by modelled time in
// us.  Pairs of CTAs: 1.8 (4 slices), 2.75 (7) or 3.75 (8) us per unit of a tile, tiles
// (times K slices) dealt out to 76 pairs, about 7 units of start and end.
// SLICE4's 128 x 64 tiles: 1.3 us per unit, a CTA per tile, 8 units of start
// and end: they keep narrow (2 N <= 64) and small products.  K slices need
// an output that fits the scratch, and cost its way through memory (32 bytes
// per partial at 6 TB/s) and a launch.  Up to 64 of them: 300 x 24 outputs
// with K = 450000 are 3 tiles (1410 -> 910 us against at most 32).
struct SlicePlan {
  bool pair;
  int splits;
};
SlicePlan plan_slices(int nslices, int M, int N, int nkb, size_t part_elems) {
  SlicePlan best{true, 1};
  double tbest = 1e300;
  auto consider = [&](bool pair, double tiles, double workers, double unit, double fixed) {
    for (int sp = 1; sp <= 64; ++sp) {
      if (sp > 1 && (nkb / sp < 4 || (size_t)sp * M * N > part_elems)) break;
      const double units = 2.0 * ((nkb + sp - 1) / sp);
      double t = std::ceil(tiles * sp / workers) * (units + fixed) * unit;
      if (sp > 1) t += 3.0 + 32.0 * sp * (double)M * N / 6e6;
      if (t < tbest) {
        tbest = t;
        best = SlicePlan{pair, sp};
      }
    }
  };
  const int pn = nslices == 4 ? PairCfg<4>::PN : PairCfg<7>::PN;
  const double tm = (M + P_BM - 1) / P_BM, tn = (2 * N + pn - 1) / pn;
  consider(true, tm * tn, 76.0, nslices == 4 ? 1.8 : nslices == 7 ? 2.75 : 3.75, 7.0);
  if (nslices == 4)
    consider(false, (double)((M + BM - 1) / BM) * ((2 * N + RBN - 1) / RBN), 152.0, 1.3, 8.0);
  return best;
}

template <int NS>
void launch_pair(cudaStream_t s, const CUtensorMap& ma, const CUtensorMap& mb,
                 const CUtensorMap& mb2, int kpa,
                 int ka_off, int kpb, int kb_off, int nkb, int zl, int nz, int M, int N,
                 const int* eA, const int* eB, double alpha, double beta, View C, cplx* part,
                 int64_t upper, int* err) {
  const int ntm = (M + P_BM - 1) / P_BM, ntn = (2 * N + PairCfg<NS>::PN - 1) / PairCfg<NS>::PN;
  const int64_t items = (int64_t)ntm * ntn * nz;
  CVS_REQUIRE(items <= INT32_MAX, -1, "zgemm_slice: output too large");
  const unsigned grid = 2 * (unsigned)std::min<int64_t>(items, 76);
  tc_slice_pair_kernel<NS><<<grid, pair_threads<NS>(), pair_smem<NS>(), s>>>(
      ma, mb, mb2, kpa, ka_off, kpb, kb_off, nkb, zl, ntm, ntn, (int)items, upper, M, N, eA, eB, alpha,
      beta, C, part, err);
  CVS_CHECK_LAUNCH();
}

}  // namespace

void wait_probe(cudaStream_t s, int64_t limit_ns, int* err) {
  const uint64_t lim = (uint64_t)std::min<int64_t>(std::max<int64_t>(limit_ns, 1000000),
                                                   (int64_t)WAIT_NS);
  wait_probe_kernel<<<1, 32, 0, s>>>(lim, err);
  CVS_CHECK_LAUNCH();
}

size_t slice_workspace_bytes(int M, int N, int K, int nslices, bool b_cached, bool a_cached) {
  SDims d = sdims_of(M, N, K, nslices, b_cached, a_cached);
  return d.a_bytes + d.b_bytes + d.e_bytes + 256;
}

size_t slice_acache_bytes(int M, int K, int nslices) {
  SDims d = sdims_of(M, 1, K, nslices, true, true);
  return (size_t)d.Mp * d.nseg * d.KpF * 2 + (size_t)d.Mp * sizeof(int) + 256;
}

size_t slice_bcache_bytes(int N, int K, int nslices) {
  SDims d = sdims_of(1, N, K, nslices, true);
  return (size_t)d.Np2 * d.nseg * d.KpF * 2 + ((size_t)d.Np2 / 2 + 64) * sizeof(int) + 256;
}

int64_t slice_row_slab(int M, int N, int K, int nslices) {
  SDims d = sdims_of(M, N, K, nslices, false);
  if (d.kc >= d.KpF) return M;  // K is whole already
  const size_t per_row = (size_t)d.cseg * d.KpF * 2;
  const size_t bfull = (size_t)d.Np2 * d.cseg * d.KpF * 2;
  if (bfull >= PACK_BUDGET / 2) return M;
  const int64_t rows = (int64_t)((PACK_BUDGET - bfull) / per_row) / BM * BM;
  return rows >= 16 * BM ? rows : M;
}

void zgemm_slice(cudaStream_t s, int nslices, int M, int N, int K,
                 double alpha, View A, View B, double beta, View C, void* work,
                 size_t work_bytes, cplx* part, size_t part_elems, int* err,
                 SliceBCache* bc, SliceBCache* ac, int64_t upper) {
  if (M <= 0 || N <= 0) return;
  CVS_REQUIRE(nslices == 4 || nslices == 7 || nslices == 8, -1, "zgemm_slice: 4, 7 or 8 slices");
  CVS_REQUIRE(!ac || nslices == 4, -1, "zgemm_slice: cached A needs 4 slices");
  SDims d = sdims_of(M, N, K, nslices, bc != nullptr, ac != nullptr);
  CVS_REQUIRE(work_bytes >= d.a_bytes + d.b_bytes + d.e_bytes, -1,
              "zgemm_slice: workspace too small");
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(tc_slice_pair_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         pair_smem<4>());
    cudaFuncSetAttribute(tc_slice_pair_kernel<7>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         pair_smem<7>());
    cudaFuncSetAttribute(tc_slice_pair_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         pair_smem<8>());
    cudaFuncSetAttribute(tc_slice4r_kernel,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, R_SMEM);
  });
  auto pack_a = [&](int Kc, int k0, int Kp, int* e, __nv_bfloat16* out) {
    if (nslices == 4)
      pack_lines<4, false>(s, A, M, Kc, k0, d.Mp, Kp, e, d.Mp, out);
    else if (nslices == 8)
      pack_lines<8, false>(s, A, M, Kc, k0, d.Mp, Kp, e, d.Mp, out);
    else
      pack_lines<7, false>(s, A, M, Kc, k0, d.Mp, Kp, e, d.Mp, out);
  };
  const size_t eb_n = (size_t)d.Np2 / 2 + 64;
  auto pack_b = [&](int Kc, int k0, int Kp, int* e, __nv_bfloat16* out) {
    if (nslices == 4)
      pack_lines<4, true>(s, trans(B), N, Kc, k0, d.Np2 / 2, Kp, e, eb_n, out);
    else if (nslices == 8)
      pack_lines<8, true>(s, trans(B), N, Kc, k0, d.Np2 / 2, Kp, e, eb_n, out);
    else
      pack_lines<7, true>(s, trans(B), N, Kc, k0, d.Np2 / 2, Kp, e, eb_n, out);
  };
  __nv_bfloat16* ap = (__nv_bfloat16*)work;
  __nv_bfloat16* bp = (__nv_bfloat16*)((char*)work + d.a_bytes);
  int* eA = (int*)((char*)work + d.a_bytes + d.b_bytes);
  int* eB = eA + d.Mp;
  const size_t bfull = (size_t)d.Np2 * d.nseg * d.KpF * 2;
  if (bc) {
    // the cached B: packed once over the whole K, with whole-column exponents
    CVS_REQUIRE(bc->bytes >= bfull + eb_n * sizeof(int), -1, "zgemm_slice: B cache too small");
    if (!bc->filled) {
      pack_b(K, 0, d.KpF, (int*)((char*)bc->base + bfull), (__nv_bfloat16*)bc->base);
      bc->filled = true;
    }
  }
  // the cached A: packed once over the whole K, with whole-row exponents
  const size_t afull = (size_t)d.Mp * d.nseg * d.KpF * 2;
  if (ac) {
    CVS_REQUIRE(ac->bytes >= afull + (size_t)d.Mp * sizeof(int), -1,
                "zgemm_slice: A cache too small");
    if (!ac->filled) {
      pack_a(K, 0, d.KpF, (int*)((char*)ac->base + afull), (__nv_bfloat16*)ac->base);
      ac->filled = true;
    }
  }
  for (int k0 = 0; k0 < K; k0 += d.kc) {
    const int Kc = std::min(d.kc, K - k0);
    const int Kp = (Kc + BK - 1) / BK * BK;
    // B's packed slices and exponents: the cache (whole K; this chunk starts
    // at K block k0 / BK of each segment of KpF) or this chunk's packs in
    // the workspace
    const __nv_bfloat16* bpc = bc ? (const __nv_bfloat16*)bc->base : bp;
    const int* eBc = bc ? (const int*)((const char*)bc->base + bfull) : eB;
    const int kpb = bc ? d.KpF : Kp, kb_off = bc ? k0 / BK : 0;
    // A's packed slices and exponents: the cache (whole K) or this chunk's
    const __nv_bfloat16* apc = ac ? (const __nv_bfloat16*)ac->base : ap;
    const int* eAc = ac ? (const int*)((const char*)ac->base + afull) : eA;
    const int kpa = ac ? d.KpF : Kp, ka_off = ac ? k0 / BK : 0;
    if (!ac) pack_a(Kc, k0, Kp, eA, ap);
    if (!bc) pack_b(Kc, k0, Kp, eB, bp);
    const double beta_c = (k0 == 0) ? beta : 1.0;
    const int nkb = Kp / BK;  // K blocks
    const SlicePlan pl = plan_slices(nslices, M, N, nkb, part ? part_elems : 0);
    const int zl = (nkb + pl.splits - 1) / pl.splits;
    const int nz = (nkb + zl - 1) / zl;
    cplx* pp = nz > 1 ? part : nullptr;
    CUtensorMap ma = make_map(apc, d.Mp, (int64_t)d.nseg * kpa, BM);
    // boxes of 64 rows: half a 128-column slice (4 slices) or a whole
    // 64-column one; of 32 rows: half of that
    CUtensorMap mb = make_map(bpc, d.Np2, (int64_t)d.nseg * kpb, 64);
    CUtensorMap mb2 = make_map(bpc, d.Np2, (int64_t)d.nseg * kpb, 32);
    const int tok = kstats_begin(s, K_TC_SLICE, 8.0 * M * N * (double)Kc);
    if (pl.pair && nslices == 4) {
      launch_pair<4>(s, ma, mb, mb2, kpa, ka_off, kpb, kb_off, nkb, zl, nz, M, N, eAc, eBc, alpha,
                     beta_c, C, pp, upper, err);
    } else if (nslices == 8) {
      launch_pair<8>(s, ma, mb, mb2, kpa, ka_off, kpb, kb_off, nkb, zl, nz, M, N, eAc, eBc, alpha,
                     beta_c, C, pp, upper, err);
    } else if (pl.pair) {
      launch_pair<7>(s, ma, mb, mb2, kpa, ka_off, kpb, kb_off, nkb, zl, nz, M, N, eAc, eBc, alpha,
                     beta_c, C, pp, upper, err);
    } else {
      dim3 grid(d.Np2 / RBN, d.Mp / BM, nz);
      tc_slice4r_kernel<<<grid, 576, R_SMEM, s>>>(ma, mb, kpa, ka_off, kpb, kb_off, nkb, zl, M, N,
                                                  eAc, eBc, alpha, beta_c, C, pp, upper, err);
      CVS_CHECK_LAUNCH();
    }
    kstats_end(s, tok);
    if (nz > 1) splitk_reduce(s, M, N, nz, part, beta_c, C);
  }
}

}  // namespace cvs
