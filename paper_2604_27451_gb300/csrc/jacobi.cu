// FP64 complex Hermitian eigensolver: cyclic Jacobi with the round-robin
// (Brent-Luk) pair ordering, so that the n/2 rotations of one step act on
// disjoint index pairs.  Used for the Davidson subspace matrix, for the MP2
// vv density and the truncated Fock block of the frozen-natural-spinor step
// (Eqs. 17 and 19) and for the Schur-complement preconditioner.
//
// A rotation is the unitary J = [[c, s], [-conj(s), c]] on the pair (p, q):
// A <- J^H A J, V <- V J, with s = c t a_pq / |a_pq|, c = (1 + t^2)^-1/2,
// t = sgn(tau) / (|tau| + sqrt(1 + tau^2)), tau = (a_qq - a_pp) / (2 |a_pq|).
//
// Up to SMALL_N indices one CTA runs the whole solve; above, every step of a
// sweep is one grid-wide launch (jstep_kernel).
#include <cmath>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"

namespace cvs {

namespace {

__global__ void __launch_bounds__(1024)
    jacobi_kernel(cplx* A, int n, double* w, cplx* V, int max_sweeps) {
  extern __shared__ char smem[];
  const int np = (n + 1) & ~1;
  const int half = np / 2;
  cplx* se = (cplx*)smem;                 // [half] s * e per pair
  double* cc = (double*)(se + half);      // [half] c per pair
  int* arr = (int*)(cc + half);           // [np] tournament positions
  __shared__ double red[32];
  __shared__ int stop;
  const int tid = threadIdx.x, nt = blockDim.x;

  for (int64_t e = tid; e < (int64_t)n * n; e += nt) {
    int r = e / n, c = e % n;
    V[e] = cmake(r == c ? 1.0 : 0.0, 0.0);
  }
  for (int k = tid; k < np; k += nt) arr[k] = k;
  __syncthreads();

  int sweep = 0;
  double ratio = 0.0;
  for (; sweep <= max_sweeps; ++sweep) {
    // convergence: off-diagonal norm against the full norm
    double off = 0.0, tot = 0.0;
    for (int64_t e = tid; e < (int64_t)n * n; e += nt) {
      int r = e / n, c = e % n;
      cplx a = A[e];
      double m2 = a.x * a.x + a.y * a.y;
      tot += m2;
      if (r != c) off += m2;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_down_sync(0xffffffffu, off, o);
      tot += __shfl_down_sync(0xffffffffu, tot, o);
    }
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = off;
    __syncthreads();
    if (tid == 0) {
      double s = 0;
      for (int q = 0; q < (nt + 31) / 32; ++q) s += red[q];
      red[0] = s;
    }
    __syncthreads();
    double offs = red[0];
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = tot;
    __syncthreads();
    if (tid == 0) {
      double s = 0;
      for (int q = 0; q < (nt + 31) / 32; ++q) s += red[q];
      ratio = s > 0 ? sqrt(offs / s) : 0.0;
      stop = (ratio < 1e-15) || (sweep == max_sweeps);
      red[1] = ratio;
    }
    __syncthreads();
    ratio = red[1];
    if (stop) break;

    for (int step = 0; step < np - 1; ++step) {
      // rotation parameters from the current matrix
      for (int k = tid; k < half; k += nt) {
        int p = arr[k], q = arr[np - 1 - k];
        if (p > q) {
          int t = p;
          p = q;
          q = t;
        }
        double c = 1.0;
        cplx sv = cmake(0, 0);
        if (q < n) {
          cplx apq = A[(int64_t)p * n + q];
          double r = hypot(apq.x, apq.y);
          double app = A[(int64_t)p * n + p].x, aqq = A[(int64_t)q * n + q].x;
          if (r > 1e-300 && r > 1e-18 * sqrt(fabs(app * aqq))) {
            double tau = (aqq - app) / (2.0 * r);
            double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            c = 1.0 / sqrt(1.0 + t * t);
            double s = t * c;
            sv = cmake(s * apq.x / r, s * apq.y / r);  // s * e
          }
        }
        cc[k] = c;
        se[k] = sv;
      }
      __syncthreads();
      // rows: A <- J^H A
      for (int64_t e = tid; e < (int64_t)half * n; e += nt) {
        int k = e / n, col = e % n;
        int p = arr[k], q = arr[np - 1 - k];
        if (p > q) {
          int t = p;
          p = q;
          q = t;
        }
        if (q >= n) continue;
        double c = cc[k];
        cplx sv = se[k];
        if (sv.x == 0.0 && sv.y == 0.0) continue;
        cplx ap = A[(int64_t)p * n + col], aq = A[(int64_t)q * n + col];
        // row p: c a_p - (s e) a_q ; row q: conj(s e) a_p + c a_q
        A[(int64_t)p * n + col] = csub(cscale(ap, c), cmul(sv, aq));
        A[(int64_t)q * n + col] = cadd(cmul(cconj(sv), ap), cscale(aq, c));
      }
      __syncthreads();
      // columns: A <- A J, V <- V J
      for (int64_t e = tid; e < (int64_t)half * n; e += nt) {
        int k = e / n, row = e % n;
        int p = arr[k], q = arr[np - 1 - k];
        if (p > q) {
          int t = p;
          p = q;
          q = t;
        }
        if (q >= n) continue;
        double c = cc[k];
        cplx sv = se[k];
        if (sv.x == 0.0 && sv.y == 0.0) continue;
        // col p: c a_p - conj(s e) a_q ; col q: (s e) a_p + c a_q
        cplx ap = A[(int64_t)row * n + p], aq = A[(int64_t)row * n + q];
        A[(int64_t)row * n + p] = csub(cscale(ap, c), cmul(cconj(sv), aq));
        A[(int64_t)row * n + q] = cadd(cmul(sv, ap), cscale(aq, c));
        cplx vp = V[(int64_t)row * n + p], vq = V[(int64_t)row * n + q];
        V[(int64_t)row * n + p] = csub(cscale(vp, c), cmul(cconj(sv), vq));
        V[(int64_t)row * n + q] = cadd(cmul(sv, vp), cscale(vq, c));
      }
      __syncthreads();
      // advance the tournament: position 0 fixed, the rest rotate
      if (tid == 0) {
        int last = arr[np - 1];
        for (int k = np - 1; k > 1; --k) arr[k] = arr[k - 1];
        arr[1] = last;
      }
      __syncthreads();
    }
  }

  // ascending eigenvalues: rank sort, permuted copy of V through A
  for (int i = tid; i < n; i += nt) {
    double wi = A[(int64_t)i * n + i].x;
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      double wj = A[(int64_t)j * n + j].x;
      rank += (wj < wi) || (wj == wi && j < i);
    }
    arr[i] = rank;
  }
  __syncthreads();
  for (int i = tid; i < n; i += nt) w[arr[i]] = A[(int64_t)i * n + i].x;
  __syncthreads();
  for (int64_t e = tid; e < (int64_t)n * n; e += nt) {
    int r = e / n, c = e % n;
    A[(int64_t)r * n + arr[c]] = V[e];
  }
  __syncthreads();
  for (int64_t e = tid; e < (int64_t)n * n; e += nt) V[e] = A[e];
}

// ------------------------------------------------------- one step per launch
// Pairs of step s of the round-robin tournament over np (even) positions:
// position 0 stays, the others rotate by one per step.  q = n (odd n) is the
// bye: the pair's one index is left alone.
__device__ __forceinline__ void rr_pair(int k, int np, int s, int& p, int& q) {
  auto pos = [&](int kk) {
    int t = kk - 1 - s;  // > -2 np
    t += t < 0 ? np - 1 : 0;
    t += t < 0 ? np - 1 : 0;
    return kk == 0 ? 0 : 1 + t;
  };
  p = pos(k);
  q = pos(np - 1 - k);
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// A step's kernels are launched while their predecessor drains: their blocks
// come up, work out indices and wait here until it is complete and its
// writes are visible, which hides most of a launch.  Whole solves whose
// preconditioner has n = 240: 51.5 -> 46.5 ms, n = 600: 221 -> 199 ms.  No
// load of what the predecessor writes may stand above this, nor be a
// read-only (non-coherent) one.
__device__ __forceinline__ void after_predecessor() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... Q>
void launch_chained(cudaStream_t s, void (*kernel)(P...), int grid, int block, Q... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  CVS_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  CVS_CHECK_LAUNCH();
}

// the rotation of a_pq, skipped for |a_pq| <= 1e-18 sqrt(|a_pp a_qq|)
__device__ __forceinline__ void rotation(cplx apq, double app, double aqq, double& c, cplx& sv) {
  c = 1.0;
  sv = cmake(0.0, 0.0);
  const double r = hypot(apq.x, apq.y);
  // (the square root only where the squares do not tell)
  const double r2 = r * r, pq = fabs(app * aqq);
  if (!(r > 1e-300) || (!(r2 > 2e-36 * pq && r2 > 1e-290) && !(r > 1e-18 * sqrt(pq)))) return;
  const double tau = (aqq - app) / (2.0 * r);
  const double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
  c = 1.0 / sqrt(1.0 + t * t);
  const double sn = t * c;
  sv = cmake(sn * apq.x / r, sn * apq.y / r);
}

struct Rot {
  cplx s;
  double c, pad;
};
// the rotation of pair k of step s, and its indices (p = n: no such pair)
__device__ __forceinline__ Rot rotation_of(const cplx* A, int n, int np, int s, int k, int& p,
                                           int& q) {
  Rot r{cmake(0.0, 0.0), 1.0, 0.0};
  p = q = n;
  if (k < np / 2) rr_pair(k, np, s, p, q);
  if (q < n)
    rotation(A[(int64_t)p * n + q], A[(int64_t)p * n + p].x, A[(int64_t)q * n + q].x, r.c, r.s);
  return r;
}

// An = J^H A J on the 2 x 2 block of rows (pk, qk) and columns (pl, ql)
__device__ __forceinline__ void rotate_block(const cplx* A, cplx* An, int n, int pk, int qk,
                                             const Rot& rk, int pl, int ql, const Rot& rl) {
  auto get = [&](int r, int c) {
    return r < n && c < n ? A[(int64_t)r * n + c] : cmake(0.0, 0.0);
  };
  auto put = [&](int r, int c, cplx v) {
    if (r < n && c < n) An[(int64_t)r * n + c] = v;
  };
  const double ck = rk.c, cl = rl.c;
  const cplx sk = rk.s, sl = rl.s;
  cplx a = get(pk, pl), b = get(pk, ql), c = get(qk, pl), d = get(qk, ql);
  if (sk.x != 0.0 || sk.y != 0.0) {  // rows: p' = c p - s q, q' = conj(s) p + c q
    const cplx a0 = a, b0 = b;
    a = csub(cscale(a0, ck), cmul(sk, c));
    c = cadd(cmul(cconj(sk), a0), cscale(c, ck));
    b = csub(cscale(b0, ck), cmul(sk, d));
    d = cadd(cmul(cconj(sk), b0), cscale(d, ck));
  }
  if (sl.x != 0.0 || sl.y != 0.0) {  // columns: p' = c p - conj(s) q, q' = s p + c q
    const cplx a0 = a, c0 = c;
    a = csub(cscale(a0, cl), cmul(cconj(sl), b));
    b = cadd(cmul(sl, a0), cscale(b, cl));
    c = csub(cscale(c0, cl), cmul(cconj(sl), d));
    d = cadd(cmul(sl, c0), cscale(d, cl));
  }
  put(pk, pl, a);
  put(pk, ql, b);
  put(qk, pl, c);
  put(qk, ql, d);
}

// columns (p, q) of the rows r0, r0 + dr, .. < r1 of V: V <- V J
__device__ __forceinline__ void rotate_rows(cplx* V, int n, int p, int q, const Rot& r, int r0,
                                            int r1, int dr) {
  if (q >= n || (r.s.x == 0.0 && r.s.y == 0.0)) return;
  for (int i = r0; i < r1; i += dr) {
    cplx* v = V + (int64_t)i * n;
    const cplx vp = v[p], vq = v[q];
    v[p] = csub(cscale(vp, r.c), cmul(cconj(r.s), vq));
    v[q] = cadd(cmul(r.s, vp), cscale(vq, r.c));
  }
}

// One step as one launch: An = J^H A J and V = V J for all pairs of step s.
// A is only read, so a block takes a tile of 8 x 8 pairs, computes their
// rotations and both sides of its 16 x 16 elements in one pass; blocks from
// na on rotate 8 pairs of columns of 32 rows of V.  What bounds it is the
// chain of ~150 FP64 operations of a rotation (64 cycles each on a warp's
// scheduler: ~5 us) and the launch.  Against three launches and two passes:
// n = 240 11.6 us a step (20 us); n = 200 against one block: 11 us (~190 us);
// before launches overlapped.
constexpr int JT = 8, JV = 32;
__global__ void __launch_bounds__(JT * JT)
    jstep_kernel(const cplx* A, cplx* An, cplx* V, int n, int np, int s, int nt, int na) {
  __shared__ Rot rot[2 * JT];
  __shared__ int ip[2 * JT], iq[2 * JT];
  const int tid = threadIdx.x, ti = tid / JT, tj = tid % JT;
  const bool vblk = (int)blockIdx.x >= na;
  const int blk = vblk ? (int)blockIdx.x - na : (int)blockIdx.x;
  const int tk = blk / nt, tl = blk % nt;  // tk of a V block: its tile of rows
  after_predecessor();
  // pairs of the tile's columns at [0, JT), of its rows at [JT, 2 JT)
  if (tid < (vblk ? JT : 2 * JT))
    rot[tid] = rotation_of(A, n, np, s, (tid < JT ? tl : tk) * JT + tid % JT, ip[tid], iq[tid]);
  __syncthreads();
  if (vblk)
    rotate_rows(V, n, ip[tj], iq[tj], rot[tj], tk * JV + ti, min(n, (tk + 1) * JV), JT);
  else
    rotate_block(A, An, n, ip[JT + ti], iq[JT + ti], rot[JT + ti], ip[tj], iq[tj], rot[tj]);
}

// One step as two launches, for n where the FP64 pipes are the bound and
// rotations worked out in every block take a third of them: the tiles of A
// (8 x 8 pairs a block) from the step's rotations in rot; then, side by
// side, V of this step and the rotations of the next one, s1, a warp of
// pairs a block (blocks below nr).  n = 600: 20.7 us a step, 24 us as one
// launch, 33 us as three, before launches overlapped.
constexpr int LT = 8, LV = 32;
__global__ void __launch_bounds__(LT * LT)
    jtiles_kernel(const cplx* A, cplx* An, int n, int np, int s, int nt, const Rot* rot) {
  const int k = blockIdx.x / nt * LT + threadIdx.x / LT;
  const int l = blockIdx.x % nt * LT + threadIdx.x % LT;
  int pk, qk, pl, ql;
  rr_pair(k, np, s, pk, qk);
  rr_pair(l, np, s, pl, ql);
  after_predecessor();
  if (k >= np / 2 || l >= np / 2) return;
  rotate_block(A, An, n, pk, qk, rot[k], pl, ql, rot[l]);
}
__global__ void __launch_bounds__(LT * LT)
    jnext_kernel(const cplx* A, cplx* V, int n, int np, int s, int s1, int nt, int nr,
                 const Rot* rot, Rot* rot1) {
  after_predecessor();
  int p, q;
  if ((int)blockIdx.x < nr) {
    const int k = blockIdx.x * 32 + threadIdx.x;
    if (threadIdx.x < 32 && k < np / 2) rot1[k] = rotation_of(A, n, np, s1, k, p, q);
    return;
  }
  const int blk = (int)blockIdx.x - nr;
  const int l = blk % nt * LT + threadIdx.x % LT, r0 = blk / nt * LV;
  if (l >= np / 2) return;
  rr_pair(l, np, s, p, q);
  rotate_rows(V, n, p, q, rot[l], r0 + threadIdx.x / LT, min(n, r0 + LV), LT);
}

__global__ void jidentity_kernel(cplx* V, int n) {
  const int64_t total = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x)
    V[e] = cmake(e / n == e % n ? 1.0 : 0.0, 0.0);
}

// per-block partial sums of the off-diagonal and total squared modulus
constexpr int JPART = 304;
__global__ void __launch_bounds__(256)
    joffnorm_kernel(const cplx* __restrict__ A, int n, double* __restrict__ part) {
  __shared__ double so[8], st[8];
  double off = 0.0, tot = 0.0;
  const int64_t total = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const cplx a = A[e];
    const double m2 = a.x * a.x + a.y * a.y;
    tot += m2;
    if (e / n != e % n) off += m2;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    off += __shfl_xor_sync(0xffffffffu, off, o);
    tot += __shfl_xor_sync(0xffffffffu, tot, o);
  }
  if ((threadIdx.x & 31) == 0) {
    so[threadIdx.x >> 5] = off;
    st[threadIdx.x >> 5] = tot;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) {
      off += so[q];
      tot += st[q];
    }
    part[2 * blockIdx.x] = off;
    part[2 * blockIdx.x + 1] = tot;
  }
}

// rank[i] = place of eigenvalue i in ascending order, w sorted
__global__ void jrank_kernel(const cplx* __restrict__ A, int n, double* __restrict__ w,
                             int* __restrict__ rank) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double wi = A[(int64_t)i * n + i].x;
    int r = 0;
    for (int j = 0; j < n; ++j) {
      const double wj = A[(int64_t)j * n + j].x;
      r += (wj < wi) || (wj == wi && j < i);
    }
    w[r] = wi;
    rank[i] = r;
  }
}

__global__ void jcolumns_kernel(const cplx* __restrict__ V, int n, const int* __restrict__ rank,
                                cplx* __restrict__ U) {
  const int64_t total = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x)
    U[e / n * n + rank[e % n]] = V[e];
}

}  // namespace

// The one-CTA solve runs at an SM's two FP64 FMAs per cycle (18 n^3 a
// sweep); a step launch costs ~3 us.  They meet near n = 24 (one sweep: 60
// against 70 us).
constexpr int SMALL_N = 24;

// scratch of jacobi_eigh_grid: a second A, the rotations of two steps,
// partial sums, ranks
static size_t grid_work_bytes(int n) {
  return (size_t)n * n * sizeof(cplx) + (size_t)(n + 2) * sizeof(Rot) +
         2 * JPART * sizeof(double) + ((size_t)n * sizeof(int) + 15) / 16 * 16;
}
size_t jacobi_work_bytes(int n) {
  return (size_t)n * n * sizeof(cplx) + grid_work_bytes(n);
}

int jacobi_eigh_grid(cudaStream_t s, cplx* A, int n, double* w, cplx* U, cplx* V, void* work,
                     int max_sweeps, double tol, double floor) {
  CVS_REQUIRE(n >= 1 && n <= 16384, -1, "jacobi_eigh_grid: n out of range");
  const int np = (n + 1) & ~1, half = np / 2;
  cplx* bufs[2] = {A, (cplx*)work};
  Rot* rots[2] = {(Rot*)((cplx*)work + (size_t)n * n), nullptr};
  rots[1] = rots[0] + half;
  double* part = (double*)(rots[0] + (n + 2));
  int* rank = (int*)(part + 2 * JPART);
  // 8 x 8 pairs give 345 blocks at n = 240 (2.3 per SM); at n = 600 two
  // launches save a seventh of the step (jtiles_kernel)
  const bool two = n >= 400;
  const int nt = (half + (two ? LT : JT) - 1) / (two ? LT : JT);
  const int na = nt * nt, nr = (half + 31) / 32;
  const int nv = nt * ((n + (two ? LV : JV) - 1) / (two ? LV : JV));
  if (two) {  // the rotations of the first step
    jnext_kernel<<<nr, LT * LT, 0, s>>>(A, V, n, np, 0, 0, nt, nr, rots[1], rots[0]);
    CVS_CHECK_LAUNCH();
  }
  jidentity_kernel<<<grid1d((int64_t)n * n, 256), 256, 0, s>>>(V, n);
  CVS_CHECK_LAUNCH();
  int sweep = 0, cur = 0;
  double prev = 1e300;
  std::vector<double> hp(2 * JPART);
  for (; sweep < max_sweeps; ++sweep) {
    joffnorm_kernel<<<JPART, 256, 0, s>>>(bufs[cur], n, part);
    CVS_CHECK_LAUNCH();
    CVS_CUDA(cudaMemcpyAsync(hp.data(), part, hp.size() * sizeof(double),
                             cudaMemcpyDeviceToHost, s));
    CVS_CUDA(cudaStreamSynchronize(s));
    double off = 0.0, tot = 0.0;
    for (int b = 0; b < JPART; ++b) {
      off += hp[2 * b];
      tot += hp[2 * b + 1];
    }
    const double ratio = tot > 0.0 ? std::sqrt(off / tot) : 0.0;
    // converged, or stalled at the rounding level of the largest entries
    if (ratio < tol || (ratio < floor && ratio > 0.5 * prev)) break;
    prev = ratio;
    for (int st = 0; st < np - 1; ++st, cur ^= 1) {
      if (!two) {
        launch_chained(s, jstep_kernel, na + nv, JT * JT, bufs[cur], bufs[cur ^ 1], V, n, np, st,
                       nt, na);
        continue;
      }
      launch_chained(s, jtiles_kernel, na, LT * LT, bufs[cur], bufs[cur ^ 1], n, np, st, nt,
                     rots[cur]);
      launch_chained(s, jnext_kernel, nr + nv, LT * LT, bufs[cur ^ 1], V, n, np, st,
                     (st + 1) % (np - 1), nt, nr, rots[cur], rots[cur ^ 1]);
    }
  }
  jrank_kernel<<<(n + 127) / 128, 128, 0, s>>>(bufs[cur], n, w, rank);
  CVS_CHECK_LAUNCH();
  jcolumns_kernel<<<grid1d((int64_t)n * n, 256), 256, 0, s>>>(V, n, rank, U);
  CVS_CHECK_LAUNCH();
  return sweep;
}

void jacobi_eigh(cudaStream_t s, cplx* A, int n, double* w, cplx* Vec, int max_sweeps,
                 void* work) {
  CVS_REQUIRE(n >= 1 && n <= 4096, -1, "jacobi_eigh: n out of range");
  if (n > SMALL_N) {
    cplx* V = (cplx*)work;
    jacobi_eigh_grid(s, A, n, w, Vec, V, V + (size_t)n * n, max_sweeps, 1e-15, 1e-13);
    return;
  }
  const int np = (n + 1) & ~1, half = np / 2;
  size_t sh = (size_t)(np + 2) * sizeof(int) + (size_t)(half + 2) * sizeof(double) +
              (size_t)half * sizeof(cplx) + 64;
  jacobi_kernel<<<1, 1024, sh, s>>>(A, n, w, Vec, max_sweeps);
  CVS_CHECK_LAUNCH();
}

}  // namespace cvs
