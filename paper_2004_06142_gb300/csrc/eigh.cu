// Symmetric FP64 eigensolver of the orbital update (Sec. III.B: the new orbitals are the
// eigenvectors of the symmetric matrix F of Eq. Fockian, and its eigenvalues the next
// diagonal).  Laid out for this GPU's narrow FP64 pipe and large L2:
//   1. A = Q T Q^T by Householder reflections, one barrier per column: small matrices in one
//      cluster of CTAs, larger ones in a cooperative launch of one CTA per SM.  Each step forms
//      the next column of the rank-2-updated matrix in every CTA (from one row, by symmetry) and
//      its reflector; every row warp updates its own row of the trailing matrix, which it keeps
//      in registers (in L2 above n 1216), and takes its part of the next matrix-vector product
//      while a scalar warp forms the reflector's scalars.  A is first scaled by a power of two (exact) to a largest element in
//      [1/2, 1).
//   2. T is split where an off-diagonal element is at most 16 N eps ||T||_inf (a perturbation
//      of that size moves no eigenvalue by more) and scaled by a power of two to
//      ||T||_inf <= 1; eigenvalues of each block by multisection on Sturm counts, a half-warp
//      per eigenvalue: float rounds, then double rounds from the three-term recurrence of the
//      leading minors with exact power-of-two rescaling.
//   3. Eigenvectors of T from twisted factorisations T - lambda I = N_r D_r N_r^T, two threads
//      per eigenvalue, the twist r where |gamma_r| is smallest; eigenvalues of one block closer
//      than 1e-5 ||T||_inf form clusters: each member's own inverse iteration (all members at
//      once), then a block orthonormalisation inside the cluster (one warp for small
//      clusters, panels on the GEMM kernel for large ones).
//   4. V = Q Z by the compact WY form of blocks of 64 reflectors: the blocks' triangular
//      factors from their Gram matrices, and two products per block as exact digit products on
//      the tensor cores (digits.cu).
#include <float.h>

#include <atomic>
#include <map>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "tcptx.cuh"

namespace donof {
namespace {

constexpr int kRowWarps = 8;                  // warps of a tridiagonal-reduction CTA that own rows
constexpr int kTriWarps = kRowWarps + 1;      // ... and the scalar warp
constexpr int kTriThreads = 32 * kTriWarps;
static_assert(kTriWarps <= 16, "warps_sum_d adds at most 16 sums");
constexpr int kNb = 64;           // reflectors per WY block
constexpr int kFixCTAs = 32;      // CTAs (one warp each) of the small-cluster kernel
constexpr int kSmallCl = 32;      // clusters up to this size are orthonormalised by one warp
constexpr int kClDesc = 5;        // ints per cluster: first slot, members, block start, block
                                  // length, offset of its vectors in the scratch (large ones)
// tridiagonal reduction: vector elements per thread held in registers, and the largest n whose
// trailing rows (one per warp) stay in registers, kTriRowRegs elements per lane
constexpr int kTriVec = 5;  // (kTriRegMaxN + kTriThreads - 1) / kTriThreads
constexpr int kTriRegMaxN = 1216;
constexpr int kTriRowRegs = (kTriRegMaxN - 2 + 31) / 32;
// its cluster form: the most CTAs, rows per row warp, and the largest n
constexpr int kRowGroup = 4;  // 32-column pieces of a row handled together
constexpr int kClCtas = 16, kClRows = 1, kClCols = 128;
constexpr double kClusterTol = 1e-5;
constexpr unsigned long long kBarrierLimitNs = 2000000000ull;

struct EighHdr {
  unsigned int ctr;   // grid-barrier arrivals of the tridiagonal reduction
  int abort;          // set when a barrier wait ran out
  int ncl;            // clusters found
  int maxcl;          // members of the largest cluster
  int nonfinite;      // A holds a NaN or an infinity
  int abort_code;     // the status word of the digit products' bounded waits
  unsigned long long amax_bits;  // max |A_ij| (bit pattern of a non-negative double)
  double scale;       // the power of two applied to A
  double tscale;      // the power of two applied to T: ||T||_inf * tscale in [1/2, 1)
  double tnorm;       // ||T||_inf after that scaling
  double pivmin;      // pivot floor of the twisted factorisations (scaled units)
};

struct EighLayout {
  size_t hdr, Yr, A, Wd, Wp, d, e, ds, es, e2, df, e2f, tau, pbuf, lam, glo, ghi, col, bstart,
      bend, incl, cl, cj, T, G, W1, W2, part, total;
  int nref, nblk;
};

EighLayout eigh_layout(int N) {
  EighLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align_up(off + (bytes ? bytes : 1));
    return o;
  };
  const size_t n = (size_t)N, nn = n * n;
  L.nref = N > 2 ? N - 2 : 0;
  L.nblk = (L.nref + kNb - 1) / kNb;
  L.hdr = take(sizeof(EighHdr));
  L.Yr = take(nn * 8);
  // A, Wd and Wp in turn; afterwards the operands of the digit products of the
  // back-transformation, and of the caller's own (eigh_scratch)
  L.A = take(nn * 8);
  L.Wd = take(nn * 8);
  L.Wp = take(nn * 8);
  {
    const size_t r = digit_reflect_bytes(N), p = digit_product_bytes(N, N, N), m = r > p ? r : p;
    if (off < L.A + m) off = align_up(L.A + m);
  }
  L.d = take(n * 8);
  L.e = take(n * 8);
  L.ds = take(n * 8);
  L.es = take(n * 8);
  L.e2 = take(n * 8);
  L.df = take(n * 4);
  L.e2f = take(n * 4);
  L.tau = take(n * 8);
  L.pbuf = take(2 * n * 8);
  L.lam = take(n * 8);
  L.glo = take(n * 8);
  L.ghi = take(n * 8);
  L.col = take(n * 4);
  L.bstart = take(n * 4);
  L.bend = take(n * 4);
  L.incl = take(n * 4);
  L.cl = take((size_t)kClDesc * n * 4);
  L.cj = take(n * 4);
  L.T = take((size_t)L.nblk * kNb * kNb * 8);
  L.G = take((size_t)L.nblk * kNb * kNb * 8);
  L.W1 = take((size_t)32 * n * 8);  // the large clusters' panel products
  L.W2 = take((size_t)32 * 32 * 8);
  size_t part = 0;
  // the large clusters' panel products: (r0 x 32) and (32 x 32) with contraction length <= N
  for (int r0 = 32; r0 < N; r0 += 32) {
    const size_t k = (size_t)splitk_count(r0, 32, N);
    if (k > 1 && k * r0 * 32 > part) part = k * r0 * 32;
  }
  {
    const size_t k = (size_t)splitk_count(32, 32, N);
    if (k > 1 && k * 32 * 32 > part) part = k * 32 * 32;
  }
  L.part = take(part * 8);
  L.total = off;
  return L;
}

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The sum of the warps' sums in red[kTriWarps], in a fixed order; in lanes 0 .. 15 of the warp that
// calls it.
__device__ __forceinline__ double warps_sum_d(const double* red) {
  const int lane = threadIdx.x & 31;
  double t = lane < kTriWarps ? red[lane] : 0.0;
#pragma unroll
  for (int o = 8; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Grid barrier of the cooperative launch: arrivals counted in hdr->ctr (zeroed before the
// launch); the wait gives up after kBarrierLimitNs and raises hdr->abort, which ends every
// other CTA's wait at once.  grid_wait returns false when the CTA must leave.  Release and acquire
// at device scope, cumulative over what the CTA's own barrier ordered before.
__device__ __forceinline__ void grid_arrive(EighHdr* h) {
  __syncthreads();
  if (threadIdx.x == 0)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&h->ctr) : "memory");
}
__device__ __forceinline__ bool grid_wait(EighHdr* h, unsigned target, int* s_flag) {
  if (threadIdx.x == 0) {
    const unsigned long long t0 = gtimer();
    int ok = 1;
    for (unsigned it = 1;; ++it) {
      unsigned c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&h->ctr) : "memory");
      if (c >= target) break;
      if (it & 15) continue;
      if (*(volatile int*)&h->abort) { ok = 0; break; }
      if (gtimer() - t0 > kBarrierLimitNs) {
        atomicExch(&h->abort, 1);
        ok = 0;
        break;
      }
    }
    *s_flag = ok;
  }
  __syncthreads();
  return *s_flag != 0;
}

// ---------------------------------------------------------------------------
// 0. max |A| (and a non-finite check), then the scaled copy
// ---------------------------------------------------------------------------
__global__ void k_eigh_amax(const double* __restrict__ A, long long nn, EighHdr* h) {
  __shared__ unsigned long long red[8];
  unsigned long long m = 0;
  int bad = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nn;
       i += (long long)gridDim.x * blockDim.x) {
    const double a = fabs(A[i]);
    if (!isfinite(a)) bad = 1;
    else m = max(m, (unsigned long long)__double_as_longlong(a));
  }
  for (int o = 16; o; o >>= 1) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  if ((threadIdx.x & 31) == 0 && bad) h->nonfinite = 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = max(m, red[i]);
    atomicMax(&h->amax_bits, m);
  }
}

__device__ __forceinline__ double eigh_scale(const EighHdr* h) {
  const double amax = __longlong_as_double((long long)h->amax_bits);
  if (amax == 0.0 || h->nonfinite) return 1.0;
  int ex = 0;
  frexp(amax, &ex);  // amax = f 2^ex, f in [1/2, 1)
  return ldexp(1.0, -ex);
}

__global__ void k_eigh_scale_copy(const double* __restrict__ A, long long nn, EighHdr* h,
                                  double* __restrict__ out) {
  const double s = eigh_scale(h);
  if (blockIdx.x == 0 && threadIdx.x == 0) h->scale = s;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nn;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = A[i] * s;
}

// ---------------------------------------------------------------------------
// 1. Householder tridiagonalisation: a cooperative launch of CTAs that exchange through L2 and a
//    grid barrier, or (CL) one cluster of up to 16 CTAs that exchange through each other's shared
//    memory and the cluster's hardware barrier.  Both form the same sums in the same order.
// ---------------------------------------------------------------------------
struct TriArgs {
  int N;
  double* A;     // N x N, row-major, symmetric; the updated rows that others need (rows in memory: all)
  double* Yr;    // reflector k in row k, columns k+1 .. N-1 (zero elsewhere)
  double* d;     // diagonal of T
  double* e;     // off-diagonal of T (N - 1)
  double* tau;   // tau of reflector k
  double* pbuf;  // two N-vectors: p of the current and the next step
  EighHdr* hdr;
};

__device__ __forceinline__ void store_peer(double* at, uint32_t rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(mapa_shared(smem_u32(at), rank)), "d"(v)
               : "memory");
}

// R rows of up to 32 Q columns per row warp in registers.  An FP64 instruction of a warp holds its
// scheduler's FP64 unit for 64 clocks, whatever its active lanes, and takes as long.  A column is a
// chain of two sums over the vector, a square root, a division and a barrier; at 120 that chain (7700
// of 16700 clocks left) is all of it, at 1200 the rows' three operations per element and the vector's
// five on every SM are half of the 15700 clocks (8 rows a CTA, two a scheduler).  So the row warps
// work while the scalar warp runs the chain, and rows stay in registers: reading and writing them
// through L2 with the updates between the chain's parts took 1046 us at 120 and 12.9 ms at 1200,
// this 410 us and 8.8 ms.
template <int R, int Q, bool CL>
__global__ void __launch_bounds__(kTriThreads, 1) k_tridiag(TriArgs a) {
  extern __shared__ double sm[];
  __shared__ double red[2][kTriWarps];  // the warps' parts of the step's two sums
  __shared__ double sh[4];              // tau, beta, scale of the reflector; alpha
  __shared__ int s_flag;
  const int N = a.N, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int G = gridDim.x;
  const int W = N < 32 * Q ? 32 * Q : N;  // width of the vectors, zero past N
  double* v = sm;           // reflector of the current step (indices k+1 .. N-1)
  double* x = sm + W;       // next column, then its reflector
  double* p = sm + 2 * W;   // p = tau A v of the current step
  double* pb = sm + 3 * W;  // CL: p of the current and the next step, written by their owners
  double* rb = pb + 2 * N;  // CL: row k+1 of the current and the next step
  constexpr int kVec = CL ? 1 : kTriVec;
  double* A = a.A;
  const bool writer = blockIdx.x == 0;
  if (N <= 2) {
    if (writer && tid == 0) {
      a.d[0] = __ldcg(A);
      if (N == 2) {
        a.e[0] = __ldcg(A + 1);
        a.d[1] = __ldcg(A + 3);
      }
    }
    return;
  }
  // rows are dealt to CTAs cyclically (row i to CTA i mod G), then to the CTA's row warps, so
  // the shrinking trailing matrix stays spread over every CTA; with N <= G * kRowWarps * R each row
  // warp owns R rows at most and keeps them in registers.  The last warp owns no row: it adds the
  // warps' sums and forms the reflectors' scalars meanwhile.
  const bool row_warp = wid < kRowWarps;
  auto row_of = [&](int t) { return blockIdx.x + G * (wid + kRowWarps * t); };
  const bool reg_rows = CL || (N <= 32 * Q && N <= G * kRowWarps * R);
  int myrow[R];
#pragma unroll
  for (int t = 0; t < R; ++t) myrow[t] = row_warp ? row_of(t) : N;
  unsigned bar = 0;
  auto arrive = [&]() {
    if (CL) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    else grid_arrive(a.hdr);
  };
  auto wait = [&]() {
    if (!CL) return grid_wait(a.hdr, (++bar) * G, &s_flag);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    __syncthreads();  // what the CTA wrote behind its arrival
    return true;
  };
  for (int j = N + tid; j < W; j += kTriThreads) v[j] = x[j] = p[j] = 0.0;
  if (CL) cluster_sync_all();  // every CTA's shared memory exists

  // by the scalar warp: reflector of x[k0..N) from the warps' parts of xn2 = sum over j > k0 of
  // x_j^2: tau, beta and the scale of u's tail (0 when the column is already reduced: u = e_k0);
  // lane 0 divides for tau, lane 1 for the scale, in one division of the warp
  auto hh_scalars = [&](int k0, const double* parts) {
    const double xn2 = warps_sum_d(parts);
    if (lane < 2) {
      const double al = x[k0];
      double q = 0.0, b = al;
      if (xn2 != 0.0) {
        b = -copysign(sqrt(fma(al, al, xn2)), al);
        q = (lane == 0 ? b - al : 1.0) / (lane == 0 ? b : al - b);
      }
      sh[lane == 0 ? 0 : 2] = q;
      if (lane == 0) sh[1] = b;
    }
  };
  // after a barrier: x[k0+1..) scaled into u's tail, x[k0] = 1; CTA 0 also stores u as row
  // `refl` of Yr
  auto hh_apply = [&](int k0, int refl) {
    const double sc = sh[2];
    double* Yk = a.Yr + (size_t)refl * N;
    for (int j = k0 + tid; j < N; j += kTriThreads) {
      const double u = j == k0 ? 1.0 : x[j] * sc;
      x[j] = u;
      if (writer) Yk[j] = u;
    }
  };

  // reflector 0 from row 0 (column 0)
  double xn = 0.0;
  for (int j = tid; j < N; j += kTriThreads) {
    const double xj = __ldcg(A + j);
    x[j] = xj;
    if (j >= 2) xn = fma(xj, xj, xn);
  }
  xn = warp_sum_d(xn);
  if (lane == 0) red[1][wid] = xn;
  __syncthreads();
  if (!row_warp) hh_scalars(1, red[1]);
  __syncthreads();
  double tau_c = sh[0], beta = sh[1];
  if (writer && tid == 0) {
    a.d[0] = x[0];
    a.e[0] = beta;
    a.tau[0] = tau_c;
  }
  hh_apply(1, 0);
  __syncthreads();
  if (row_warp) {
    for (int t = 0;; ++t) {
      const int i = row_of(t);
      if (i >= N) break;
      if (i < 1) continue;
      const double* Ar = A + (size_t)i * N;
      double acc = 0.0;
#pragma unroll 4
      for (int j = 1 + lane; j < N; j += 32) acc = fma(__ldcg(Ar + j), x[j], acc);
      acc = warp_sum_d(acc);
      if (CL) {
        if (lane < G) store_peer(pb + i, lane, tau_c * acc);
      } else if (lane == 0) {
        a.pbuf[i] = tau_c * acc;
      }
    }
  }
  if (CL)
    for (int j = tid; j < N; j += kTriThreads) rb[j] = __ldcg(A + N + j);
  // the own rows, column lane + 32 q in rr[.][q], are kept in registers from here on
  double rr[R][Q];
#pragma unroll
  for (int t = 0; t < R; ++t)
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int j = lane + 32 * q;
      rr[t][q] = reg_rows && myrow[t] < N && j < N ? __ldcg(A + (size_t)myrow[t] * N + j) : 0.0;
    }
  arrive();
  if (!wait()) return;
  {
    double* t = v;
    v = x;
    x = t;
  }

  for (int k = 0; k <= N - 3; ++k) {
    const double* pk = a.pbuf + (size_t)(k & 1) * N;
    const double* Ak1 = A + (size_t)(k + 1) * N;
    const bool last = k + 1 == N - 2;
    // the loads of the step at once: p_k and row k+1
    double pr[kVec], ar[kVec];
#pragma unroll
    for (int r = 0; r < kVec; ++r) {
      const int j = k + 1 + tid + kTriThreads * r;
      pr[r] = 0.0;
      ar[r] = 0.0;
      if (j < N) {
        pr[r] = CL ? pb[(k & 1) * N + j] : __ldcg(pk + j);
        ar[r] = CL ? rb[(k & 1) * N + j] : __ldcg(Ak1 + j);
      }
    }
    bool has_row[R];
#pragma unroll
    for (int t = 0; t < R; ++t) has_row[t] = reg_rows && myrow[t] < N && myrow[t] >= k + 2;
    double acc = 0.0;
#pragma unroll
    for (int r = 0; r < kVec; ++r) {
      const int j = k + 1 + tid + kTriThreads * r;
      if (j < N) acc = fma(pr[r], v[j], acc);
    }
    for (int j = k + 1 + tid + kTriThreads * kVec; j < N; j += kTriThreads)
      acc = fma(__ldcg(pk + j), v[j], acc);
#pragma unroll
    for (int r = 0; r < kVec; ++r) {
      const int j = k + 1 + tid + kTriThreads * r;
      if (j < N) p[j] = pr[r];
    }
    for (int j = k + 1 + tid + kTriThreads * kVec; j < N; j += kTriThreads)
      p[j] = __ldcg(pk + j);
    if (k + 1 + 32 * wid < N) acc = warp_sum_d(acc);  // (a warp past the end: zeros)
    if (lane == 0) red[0][wid] = acc;
    __syncthreads();
    // alpha = (tau_k / 2)(p_k . v_k); with w = p - alpha v the update A - v w^T - w v^T is
    // A_ij - v_i p_j - (p_i - 2 alpha v_i) v_j, formed from p and v alone.  While the scalar warp
    // forms alpha, the row warps apply the part that does not need it (not at the last step, whose
    // 2 x 2 block is formed from the rows as they stand)
    double vi[R];
#pragma unroll
    for (int t = 0; t < R; ++t) vi[t] = has_row[t] ? v[myrow[t]] : 0.0;
    if (!row_warp) {
      const double t = warps_sum_d(red[0]);
      if (lane == 0) sh[3] = 0.5 * tau_c * t;
    } else if (!last) {
#pragma unroll
      for (int t = 0; t < R; ++t)
        if (has_row[t]) {
#pragma unroll
          for (int q0 = 0; q0 < Q; q0 += kRowGroup) {
            if (32 * (q0 + kRowGroup) <= k + 2 || 32 * q0 >= N) continue;
#pragma unroll
            for (int q = q0; q < q0 + kRowGroup && q < Q; ++q)
              rr[t][q] = fma(-vi[t], p[lane + 32 * q], rr[t][q]);
          }
        }
    }
    __syncthreads();
    const double al = sh[3];
    // row k+1 of the updated matrix (v[k+1] = 1): its column k+1 below the diagonal
    const double ck1 = fma(-2.0, al, p[k + 1]);
    xn = 0.0;
#pragma unroll
    for (int r = 0; r < kVec; ++r) {
      const int j = k + 1 + tid + kTriThreads * r;
      if (j < N) {
        const double xj = fma(-ck1, v[j], ar[r] - pr[r]);
        x[j] = xj;
        if (j >= k + 3) xn = fma(xj, xj, xn);
      }
    }
    for (int j = k + 1 + tid + kTriThreads * kVec; j < N; j += kTriThreads) {
      const double xj = fma(-ck1, v[j], __ldcg(Ak1 + j) - p[j]);
      x[j] = xj;
      if (j >= k + 3) xn = fma(xj, xj, xn);
    }
    if (k + 1 + 32 * wid < N) xn = warp_sum_d(xn);
    if (lane == 0) red[1][wid] = xn;
    __syncthreads();
    if (last) {  // the last 2 x 2 block
      if (writer && tid == 0) {
        a.d[N - 2] = x[N - 2];
        a.e[N - 2] = x[N - 1];
        const double vl = v[N - 1], cl = fma(-2.0 * al, vl, p[N - 1]);
        a.d[N - 1] = __ldcg(A + (size_t)(N - 1) * N + N - 1) - vl * p[N - 1] - cl * vl;
      }
      break;
    }
    // the scalar warp forms the next reflector while the row warps finish their row's update and
    // take its dot with the unscaled column (u_{k+2} = 1, u_j = sc x_j beyond).  The sums run over
    // the columns k+3+l, k+35+l, ..., whichever lane holds them, and the shuffle tree pairs the
    // same sums in every rotation of the lanes.  Row k+2 (at the end also the last) is published.
    // The rows' loops skip groups of columns that are done with (a few columns of a group are
    // updated for nothing: a test for each costs more), so that nothing but FP64 work is left
    double rawdot[R], r0[R];
#pragma unroll
    for (int t = 0; t < R; ++t) rawdot[t] = r0[t] = 0.0;
    if (!row_warp) {
      hh_scalars(k + 2, red[1]);
    } else {
#pragma unroll
      for (int t = 0; t < R; ++t) {
        if (!has_row[t]) continue;
        const double ci = fma(-2.0 * al, vi[t], p[myrow[t]]);
#pragma unroll
        for (int q0 = 0; q0 < Q; q0 += kRowGroup) {
          if (32 * (q0 + kRowGroup) <= k + 2 || 32 * q0 >= N) continue;
#pragma unroll
          for (int q = q0; q < q0 + kRowGroup && q < Q; ++q)
            rr[t][q] = fma(-ci, v[lane + 32 * q], rr[t][q]);
          if (32 * q0 <= k + 2) {  // the group that holds column k+2
#pragma unroll
            for (int q = q0; q < q0 + kRowGroup && q < Q; ++q) {
              const int j = lane + 32 * q;
              if (j == k + 2) r0[t] = rr[t][q];
              if (j > k + 2) rawdot[t] = fma(rr[t][q], x[j], rawdot[t]);
            }
          } else {
#pragma unroll
            for (int q = q0; q < q0 + kRowGroup && q < Q; ++q)
              rawdot[t] = fma(rr[t][q], x[lane + 32 * q], rawdot[t]);
          }
        }
        if ((!CL && myrow[t] == k + 2) || k == N - 4) {
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const int j = lane + 32 * q;
            if (j >= k + 2 && j < N) A[(size_t)myrow[t] * N + j] = rr[t][q];
          }
        }
        if (CL && myrow[t] == k + 2) {
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const int j = lane + 32 * q;
            if (j >= k + 2 && j < N)
              for (int c = 0; c < G; ++c) store_peer(rb + ((k + 1) & 1) * N + j, c, rr[t][q]);
          }
        }
        rawdot[t] = warp_sum_d(rawdot[t]);
      }
    }
    __syncthreads();
    const double tau_n = sh[0], sc = sh[2];
    beta = sh[1];
    if (writer && tid == 0) {
      a.d[k + 1] = x[k + 1];
      a.e[k + 1] = beta;
      a.tau[k + 1] = tau_n;
    }
    // p_{k+1} = tau A u over the own rows i >= k+2
    double* pn = a.pbuf + (size_t)((k + 1) & 1) * N;
    if (reg_rows) {
#pragma unroll
      for (int t = 0; t < R; ++t) {
        if (!has_row[t]) continue;  // (uniform over the warp)
        const double pi = tau_n * fma(sc, rawdot[t], r0[t]);  // in the lane that holds r0
        if (CL) {
          const double pv = __shfl_sync(0xffffffffu, pi, (k + 2) & 31);
          if (lane < G) store_peer(pb + ((k + 1) & 1) * N + myrow[t], lane, pv);
        } else if (lane == ((k + 2) & 31)) {
          pn[myrow[t]] = pi;
        }
      }
      arrive();
      hh_apply(k + 2, k + 1);
    } else {
      hh_apply(k + 2, k + 1);
      __syncthreads();  // the scaled reflector
      for (int t = 0; row_warp; ++t) {
        const int i = row_of(t);
        if (i >= N) break;
        if (i < k + 2) continue;
        double* Ar = A + (size_t)i * N;
        const double vr = v[i], ci = fma(-2.0 * al, vr, p[i]);
        double acc2 = 0.0;
        int j = k + 2 + lane;
        for (; j + 96 < N; j += 128) {
          const double a0 = __ldcg(Ar + j), a1 = __ldcg(Ar + j + 32), a2 = __ldcg(Ar + j + 64),
                       a3 = __ldcg(Ar + j + 96);
          const double b0 = fma(-ci, v[j], fma(-vr, p[j], a0));
          const double b1 = fma(-ci, v[j + 32], fma(-vr, p[j + 32], a1));
          const double b2 = fma(-ci, v[j + 64], fma(-vr, p[j + 64], a2));
          const double b3 = fma(-ci, v[j + 96], fma(-vr, p[j + 96], a3));
          Ar[j] = b0;
          Ar[j + 32] = b1;
          Ar[j + 64] = b2;
          Ar[j + 96] = b3;
          acc2 = fma(b0, x[j], acc2);
          acc2 = fma(b1, x[j + 32], acc2);
          acc2 = fma(b2, x[j + 64], acc2);
          acc2 = fma(b3, x[j + 96], acc2);
        }
        for (; j < N; j += 32) {
          const double b0 = fma(-ci, v[j], fma(-vr, p[j], __ldcg(Ar + j)));
          Ar[j] = b0;
          acc2 = fma(b0, x[j], acc2);
        }
        acc2 = warp_sum_d(acc2);
        if (lane == 0) pn[i] = tau_n * acc2;
      }
      arrive();
    }
    if (!wait()) return;
    double* t = v;
    v = x;
    x = t;
    tau_c = tau_n;
  }
}

// ---------------------------------------------------------------------------
// 2. splitting, Gershgorin bounds, bisection.  From here on T is scaled by the power of two
//    ts = 2^-ceil(log2 ||T||_inf), so that ||T||_inf <= 1 (exact), and every kernel reads the
//    scaled arrays.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool dbl_is_zero(double x) {
  return ((unsigned long long)__double_as_longlong(x) << 1) == 0ull;
}
__device__ __forceinline__ int dbl_biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int dbl_sign(double x) { return (int)((unsigned)__double2hiint(x) >> 31); }

// One CTA.  ||T||_inf and the scale ts; the split off-diagonal (es, es^2) and the diagonal
// scaled by ts (double and float copies); the blocks (bstart/bend of every row, from a bit mask of
// the rows that end one); each block's Gershgorin interval (at its first row, one warp
// per block); the twisted factorisations' pivot floor.
__global__ void __launch_bounds__(256) k_tri_prep(int N, const double* __restrict__ d,
                                                  const double* __restrict__ e, EighHdr* h,
                                                  double* ds, double* es, double* e2, float* df,
                                                  float* e2f, int* bstart, int* bend,
                                                  double* glo, double* ghi) {
  extern __shared__ int sflag[];  // [N]: row i ends a block; then the list of block starts
  int* blist = sflag + N;
  __shared__ double red[8];
  __shared__ int s_nb;
  double tn = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const double r = fabs(d[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0) + (i < N - 1 ? fabs(e[i]) : 0.0);
    tn = fmax(tn, r);
  }
  for (int o = 16; o; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = tn;
  __syncthreads();
  tn = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tn = fmax(tn, red[i]);
  if (!(tn > 0.0) || !isfinite(tn)) tn = 1.0;  // T = 0 (or not finite: NaN eigenvalues follow)
  int ex = 0;
  frexp(tn, &ex);  // tn = f 2^ex, f in [1/2, 1)
  const double ts = ldexp(1.0, -ex);
  const double thresh = 16.0 * N * DBL_EPSILON * tn;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const double di = d[i] * ts;
    ds[i] = di;
    df[i] = (float)di;
    int end = i == N - 1 ? 1 : 0;
    if (i < N - 1) {
      const double ei = fabs(e[i]) <= thresh ? 0.0 : e[i] * ts;
      es[i] = ei;
      e2[i] = ei * ei;
      e2f[i] = (float)(ei * ei);
      end = dbl_is_zero(ei) ? 1 : end;
    }
    sflag[i] = end;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    h->tnorm = tn * ts;
    h->tscale = ts;
    h->pivmin = 0x1p-100;
  }
  // the rows that end a block, a bit each; a row's block lies between the bits around it
  const int nwd = (N + 31) / 32;
  unsigned* ends = (unsigned*)(sflag + 2 * N);
  for (int i = threadIdx.x; i < nwd * 32; i += blockDim.x) {
    const unsigned m = __ballot_sync(0xffffffffu, i < N && sflag[i]);
    if ((threadIdx.x & 31) == 0) ends[i / 32] = m;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    int wd = i / 32;
    unsigned m = ends[wd] >> (i & 31) << (i & 31);
    while (!m) m = ends[++wd];  // (the last row ends a block)
    bend[i] = 32 * wd + __ffs(m);
    wd = i / 32;
    m = ends[wd] & ((1u << (i & 31)) - 1u);
    while (!m && wd > 0) m = ends[--wd];
    const int s0 = m ? 32 * wd + 32 - __clz(m) : 0;
    bstart[i] = s0;
    if (s0 == i) {
      int b = __popc(ends[i / 32] & ((1u << (i & 31)) - 1u));
      for (int q = 0; q < i / 32; ++q) b += __popc(ends[q]);
      blist[b] = i;
    }
    if (i == N - 1) {
      int b = 0;
      for (int q = 0; q < nwd; ++q) b += __popc(ends[q]);
      s_nb = b;
    }
  }
  __syncthreads();
  const int nb = s_nb, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int b = threadIdx.x >> 5; b < nb; b += nw) {
    const int s0 = blist[b], s1 = b + 1 < nb ? blist[b + 1] : N;
    if (s1 - s0 < 2) continue;  // a 1 x 1 block needs no bisection
    double lo = 0.0, hi = 0.0;
    bool any = false;
    for (int i = s0 + lane; i < s1; i += 32) {
      const double el = i > s0 ? fabs(es[i - 1]) : 0.0;
      const double er = i < s1 - 1 ? fabs(es[i]) : 0.0;
      const double l = ds[i] - el - er, u = ds[i] + el + er;
      lo = any ? fmin(lo, l) : l;
      hi = any ? fmax(hi, u) : u;
      any = true;
    }
    if (!any) {  // lanes beyond the block: neutral values
      lo = ds[s0];
      hi = ds[s0];
    }
    for (int o = 16; o; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      glo[s0] = lo;
      ghi[s0] = hi;
    }
  }
}

// Number of eigenvalues of the (scaled) block [s0, s1) below sig in float: the ratio form
// q_i = (d_i - sig) - e_{i-1}^2 / q_{i-1}, |q_i| floored at piv (a zero pivot counts negative).
// t holds (d_i, e_{i-1}^2).  The signs are shifted into a word, counted every eight rows.
__device__ __forceinline__ int sturm_count_f32(const float2* __restrict__ t, int s0, int s1,
                                               float sig) {
  constexpr float piv = 1e-30f;
  float q = t[s0].x - sig;
  if (fabsf(q) < piv) q = -piv;
  int cnt = q < 0.0f ? 1 : 0;
  int i = s0 + 1;
  for (; i + 8 <= s1; i += 8) {
    unsigned neg = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float2 r = t[i + u];
      q = (r.x - sig) - __fdividef(r.y, q);
      if (fabsf(q) < piv) q = -piv;
      neg = __funnelshift_l(__float_as_uint(q), neg, 1);
    }
    cnt += __popc(neg);
  }
  for (; i < s1; ++i) {
    const float2 r = t[i];
    q = (r.x - sig) - __fdividef(r.y, q);
    if (fabsf(q) < piv) q = -piv;
    cnt += q < 0.0f ? 1 : 0;
  }
  return cnt;
}

// The same count in double: sign changes of the leading minors
// p_i = (d_i - sig) p_{i-1} - e_{i-1}^2 p_{i-2} (a zero minor counts as a tiny negative ratio),
// the pair (p_{i-1}, p_i) rescaled by 2^-+300 after every eighth row when its larger magnitude
// has left [2^-300, 2^300] (with ||T||_inf <= 1 and the split threshold, eight rows move it by
// at most 2^13 up or 2^-616 down).  Eight rows at a time: their minors' signs go into a word, and a
// zero among them is only noted and its rows done again, so that a row is three FP64 operations,
// one of them in the chain, and little else.
__device__ __forceinline__ int sturm_count_f64(const double2* __restrict__ t, int s0, int s1,
                                               double sig) {
  double p0 = 1.0, p1 = t[s0].x - sig;
  if (dbl_is_zero(p1)) p1 = -0x1p-60;
  int cnt = dbl_sign(p1);
  for (int i = s0 + 1; i < s1; i += 8) {
    const double b0 = p0, b1 = p1;
    unsigned low = 0;
    if (i + 8 <= s1) {
      unsigned neg = (unsigned)dbl_sign(p1);  // signs of the minors, the last one in bit 0
      low = 0xffffffffu;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double2 r = t[i + u];
        const double p2 = fma(r.x - sig, p1, -(r.y * p0));
        const unsigned hi = (unsigned)__double2hiint(p2);
        neg = __funnelshift_l(hi, neg, 1);
        low = min(low, hi << 1);
        p0 = p1;
        p1 = p2;
      }
      if (low) cnt += __popc((neg ^ (neg >> 1)) & 0xffu);
    }
    if (!low) {  // the last rows, or a zero (or nearly) among the eight
      p0 = b0;
      p1 = b1;
      const int iend = min(i + 8, s1);
      for (int j = i; j < iend; ++j) {
        const double2 r = t[j];
        double p2 = fma(r.x - sig, p1, -(r.y * p0));
        if (dbl_is_zero(p2)) p2 = -p1 * 0x1p-60;
        cnt += dbl_sign(p2) ^ dbl_sign(p1);
        p0 = p1;
        p1 = p2;
      }
    }
    const int ex = max(dbl_biased_exp(p0), dbl_biased_exp(p1));
    if (ex > 1023 + 300 || ex < 1023 - 300) {  // (a branch: the FP64 pipe is what counts here)
      asm volatile("");
      const double f = ex > 1023 ? 0x1p-300 : 0x1p300;
      p0 *= f;
      p1 *= f;
    }
  }
  return cnt;
}

// Eigenvalue k = s - bstart[s] of the block holding row s, by multisection: a half-warp per
// eigenvalue, its 16 lanes counting at 16 points of the bracket per round.  Five float rounds
// (brackets of ~2^-20 ||T||), the bracket widened by 4e-6 ||T|| (the float counts are exact
// for a matrix within a few float roundings of T) and its ends checked by double counts (the
// Gershgorin interval again if either fails), then double rounds to the width eps ||T||.
// The nine double rounds are bound by the FP64 pipe, three operations of 64 clocks a row (with
// rescaling by selects and a test on every row, and four warps on an SM at small N: 275 us at 120
// and 2.6 ms at 1200; now 170 us and 1.56 ms).
constexpr int kBisThreads = 128;
__global__ void __launch_bounds__(kBisThreads) k_bisect(int N, const double* __restrict__ ds,
                                                        const double* __restrict__ e2,
                                                        const float* __restrict__ df,
                                                        const float* __restrict__ e2f,
                                                        const int* __restrict__ bstart,
                                                        const int* __restrict__ bend,
                                                        const double* __restrict__ glo,
                                                        const double* __restrict__ ghi,
                                                        const EighHdr* h, double* lam) {
  extern __shared__ double2 sb[];
  double2* sd = sb;  // (d_i, e_{i-1}^2)
  float2* sdf = (float2*)(sb + N);
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    sd[i] = make_double2(ds[i], i > 0 ? e2[i - 1] : 0.0);
    sdf[i] = make_float2(df[i], i > 0 ? e2f[i - 1] : 0.0f);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, j = lane & 15;
  const unsigned hm = 0xffffu << (lane & 16);
  const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  if (s >= N) return;  // uniform over the half-warp
  if (h->abort) {
    if (j == 0) lam[s] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  const int s0 = bstart[s], s1 = bend[s], k = s - s0;
  if (s1 - s0 == 1) {
    if (j == 0) lam[s] = sd[s0].x;
    return;
  }
  const double tn = h->tnorm;
  const double pad = 2.0 * N * DBL_EPSILON * tn;
  const double glo_s = glo[s0] - pad, ghi_s = ghi[s0] + pad;
  double lo = glo_s, hi = ghi_s;
  // narrow [lo, hi] to the points of the lanes: jh the first lane whose count exceeds k, jl
  // the last lane before it whose count does not
  auto narrow = [&](bool above, double base, double step, int off) {
    const unsigned ab = (__ballot_sync(hm, above) >> (lane & 16)) & 0xffffu;
    const unsigned be = (__ballot_sync(hm, !above) >> (lane & 16)) & 0xffffu;
    const int jh = ab ? __ffs(ab) - 1 : 16;
    const unsigned bl = be & ((1u << jh) - 1u);
    const int jl = bl ? 31 - __clz(bl) : -1;
    const double nhi = jh < 16 ? base + (jh + off) * step : hi;
    const double nlo = jl >= 0 ? base + (jl + off) * step : lo;
    hi = nhi;
    lo = nlo;
  };
  for (int r = 0; r < 5; ++r) {
    const double step = (hi - lo) * (1.0 / 17.0);
    const double sg = lo + (j + 1) * step;
    narrow(sturm_count_f32(sdf, s0, s1, (float)sg) > k, lo, step, 1);
  }
  lo -= 4e-6 * tn;
  hi += 4e-6 * tn;
  {  // 16 points from lo to hi inclusive: the ends verify the float bracket
    const double step = (hi - lo) * (1.0 / 15.0);
    const double sg = lo + j * step;
    const int c = sturm_count_f64(sd, s0, s1, sg);
    const int clo = __shfl_sync(hm, c, lane & 16), chi = __shfl_sync(hm, c, (lane & 16) + 15);
    if (clo <= k && chi > k) {
      narrow(c > k, lo, step, 0);
    } else {
      lo = glo_s;
      hi = ghi_s;
    }
  }
  for (int r = 0; r < 40; ++r) {
    if (!(hi - lo > fmax(DBL_EPSILON * tn, 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi))))) break;
    const double step = (hi - lo) * (1.0 / 17.0);
    const double sg = lo + (j + 1) * step;
    narrow(sturm_count_f64(sd, s0, s1, sg) > k, lo, step, 1);
  }
  if (j == 0) lam[s] = 0.5 * (lo + hi);
}

// Order-preserving integer key of a double (NaN above everything).
__device__ __forceinline__ long long dbl_key(double x) {
  const long long u = __double_as_longlong(x);
  return u >= 0 ? u : (u ^ 0x7fffffffffffffffll);
}

// Rank of every eigenvalue (integer keys, ties by slot), eigenvalues of A in ascending order;
// CTA 0 also lists the clusters: runs of a block's consecutive eigenvalues closer than
// kClusterTol ||T|| (the gaps tested in parallel, the runs found by one thread).
constexpr int kRankLanes = 8;  // threads per eigenvalue
__global__ void __launch_bounds__(256) k_rank_plan(int N, const double* __restrict__ lam,
                                                   const int* __restrict__ bend, EighHdr* h,
                                                   int* col, double* w_out, int* incl, int* cl,
                                                   int* cj, const int* __restrict__ bstart) {
  extern __shared__ long long skey[];
  int* sgap = (int*)(skey + N);
  for (int i = threadIdx.x; i < N; i += blockDim.x) skey[i] = dbl_key(lam[i]);
  __syncthreads();
  const double unscale = 1.0 / (h->tscale * h->scale);  // a power of two
  const int s = (blockIdx.x * blockDim.x + threadIdx.x) / kRankLanes;
  const int part = threadIdx.x % kRankLanes;
  {
    const long long ks = s < N ? skey[s] : 0;
    int r = 0;
    for (int t = part; t < N; t += kRankLanes) {
      const long long kt = skey[t];
      r += (kt < ks || (kt == ks && t < s)) ? 1 : 0;
    }
#pragma unroll
    for (int o = kRankLanes / 2; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (s < N && part == 0) {
      const double ls = lam[s];
      if (ls != ls) r = s;  // NaN (a failed reduction): its own slot
      col[s] = r;
      w_out[r] = ls * unscale;
    }
  }
  if (blockIdx.x != 0) return;
  const double tol = kClusterTol * h->tnorm;
  for (int i = threadIdx.x; i < N; i += blockDim.x)
    sgap[i] = (i + 1 < bend[i] && lam[i + 1] - lam[i] < tol) ? 1 : 0;
  __syncthreads();
  // no cluster anywhere, and the rows where one starts, a bit each
  const int nw = (N + 31) / 32;
  unsigned* first = (unsigned*)(sgap + N);
  for (int i = threadIdx.x; i < nw * 32; i += blockDim.x) {
    if (i < N) incl[i] = cj[i] = 0;
    const bool st = i < N && sgap[i] && (i == 0 || !sgap[i - 1]);
    const unsigned m = __ballot_sync(0xffffffffu, st);
    if ((threadIdx.x & 31) == 0) first[i / 32] = m;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int ncl = 0, maxcl = 0, off = 0;
  for (int wd = 0; wd < nw; ++wd)
    for (unsigned m0 = first[wd]; m0; m0 &= m0 - 1) {
      const int s0 = 32 * wd + __ffs(m0) - 1;
      int t = s0;
      while (sgap[t]) ++t;  // sgap[bend - 1] = 0 ends every run inside its block
      const int m = t - s0 + 1;
      for (int u = s0; u <= t; ++u) {
        incl[u] = ncl + 1;  // cluster id + 1
        cj[u] = u - s0;     // member index
      }
      const int a0 = bstart[s0], L = bend[s0] - a0;
      int* c = cl + kClDesc * ncl;
      c[0] = s0;
      c[1] = m;
      c[2] = a0;
      c[3] = L;
      c[4] = off;
      if (m > kSmallCl) off += m * L;  // large clusters keep their vectors in the scratch
      maxcl = max(maxcl, m);
      ++ncl;
    }
  h->ncl = ncl;
  h->maxcl = maxcl;
}

// ---------------------------------------------------------------------------
// 3. eigenvectors of T
// ---------------------------------------------------------------------------
// 1/x to double precision by Newton's iteration r <- r (2 - x r) from a float seed (the error
// squares each step: 2^-23, 2^-46, then rounding); 2^-126 < |x| < 2^126.
__device__ __forceinline__ double rcp_nr(double x) {
  double r = (double)__frcp_rn((float)x);
  double t = fma(-x, r, 1.0);
  r = fma(r, t, r);
  t = fma(-x, r, 1.0);
  return fma(r, t, r);
}
// a pivot of magnitude below 2^-100 (||T|| <= 1) becomes -2^-100
__device__ __forceinline__ double pivot_floor(double v) {
  return dbl_biased_exp(v) < 1023 - 100 ? -0x1p-100 : v;
}

// Twisted factorisation of T_b - lambda I for an eigenvalue outside the clusters, two threads
// per eigenvalue.  Thread 0 of the pair runs the forward pivots D+_i (stored in Z's column,
// their reciprocals in Wp), thread 1 the backward pivots D-_i (reciprocals in Wd); then
// gamma_i = D+_i - e_i^2 / D-_{i+1} (each thread half the rows), the twist r where |gamma_r|
// is smallest (first such row), z_r = 1, and thread 0 forms z_i = -e_i z_{i+1} / D+_i above r
// while thread 1 forms z_i = -e_{i-1} z_{i-1} / D-_i below it; normalised to unit length.
// Z[i][col] (row-major, column = rank of the eigenvalue), zero outside the block.  Bound by the
// chain of a row's pivot and reciprocal (five FP64 operations, three conversions), which both
// threads run in one stream of instructions; in the other passes a row's loads are ahead of the
// chain.  (The sides one after the other and each load in the chain: 157 us at 120 and 1.93 ms at
// 1200; now 87 us and 0.90 ms.)
__global__ void __launch_bounds__(32) k_twisted(int N, const double* __restrict__ ds,
                                                const double* __restrict__ es,
                                                const double* __restrict__ e2,
                                                const int* __restrict__ bstart,
                                                const int* __restrict__ bend,
                                                const double* __restrict__ lam,
                                                const int* __restrict__ col,
                                                const int* __restrict__ incl, double* Z,
                                                double* Wp, double* Wd) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = t >> 1, side = t & 1, lane = threadIdx.x;
  const unsigned pm = 3u << (lane & ~1);
  if (s >= N) return;  // uniform over the pair
  const int s0 = bstart[s], s1 = bend[s], c = col[s];
  const size_t ld = (size_t)N;
  if (s1 - s0 == 1) {
    if (side == 0) Z[s0 * ld + c] = 1.0;
    return;
  }
  if (incl[s]) return;
  const double lm = lam[s];
  {  // both threads' pivots in one stream of instructions: row i0 + dir t
    const int dir = side == 0 ? 1 : -1, i0 = side == 0 ? s0 : s1 - 1, eo = side == 0 ? -1 : 0;
    double* W = side == 0 ? Wp : Wd;
    double pv = pivot_floor(ds[i0] - lm), rv = rcp_nr(pv);
    if (side == 0) Z[i0 * ld + c] = pv;
    W[i0 * ld + c] = rv;
#pragma unroll 4
    for (int t = 1; t < s1 - s0; ++t) {
      const int i = i0 + dir * t;
      pv = pivot_floor(fma(-e2[i + eo], rv, ds[i] - lm));
      rv = rcp_nr(pv);
      if (side == 0) Z[i * ld + c] = pv;
      W[i * ld + c] = rv;
    }
  }
  __syncwarp(pm);
  // twist: thread 0 the rows [s0, mid), thread 1 [mid, s1)
  const int mid = (s0 + s1) >> 1;
  const int a = side == 0 ? s0 : mid, b = side == 0 ? mid : s1;
  double best = 0.0;
  int r = -1;
#pragma unroll 8
  for (int i = a; i < b; ++i) {
    const double g = i < s1 - 1 ? fabs(fma(-e2[i], Wd[(i + 1) * ld + c], Z[i * ld + c]))
                                : fabs(Z[i * ld + c]);
    if (r < 0 || g < best) {
      best = g;
      r = i;
    }
  }
  {
    const double ob = __shfl_xor_sync(pm, best, 1);
    const int orr = __shfl_xor_sync(pm, r, 1);
    // the lower rows win ties; an empty half (r < 0) never wins
    const bool take_other = orr >= 0 && (r < 0 || ob < best || (ob == best && orr < r));
    if (take_other) {
      best = ob;
      r = orr;
    }
  }
  __syncwarp(pm);
  // z: thread 0 upwards from r, thread 1 downwards; rescaled by 2^-500 when above 2^500.  kZ rows'
  // factors are loaded ahead of the chain of products that uses them
  constexpr int kZ = 8;
  int nres = 0;
  const int step = side == 0 ? -1 : 1, n_z = side == 0 ? r - s0 : s1 - 1 - r;
  const double* W = side == 0 ? Wp : Wd;
  if (side == 0) Z[r * ld + c] = 1.0;
  {
    double z = 1.0;
    for (int q0 = 0; q0 < n_z; q0 += kZ) {
      double ev[kZ], wv[kZ];
#pragma unroll
      for (int u = 0; u < kZ; ++u) {
        const int i = r + step * (q0 + u + 1);
        const bool in = q0 + u < n_z;
        ev[u] = in ? es[side == 0 ? i : i - 1] : 0.0;
        wv[u] = in ? W[i * ld + c] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kZ; ++u) {
        if (q0 + u >= n_z) break;
        const int i = r + step * (q0 + u + 1);
        z = -ev[u] * z * wv[u];
        if (fabs(z) > 0x1p500) {
          const int v0 = side == 0 ? i + 1 : r + 1, v1 = side == 0 ? r + 1 : i;
          for (int v = v0; v < v1; ++v) Z[v * ld + c] *= 0x1p-500;
          z *= 0x1p-500;
          ++nres;
        }
        Z[i * ld + c] = z;
      }
    }
  }
  __syncwarp(pm);
  // bring both halves to the same scale, then normalise
  const int lo_i = side == 0 ? s0 : r + 1, hi_i = side == 0 ? r + 1 : s1;
  const int other = __shfl_xor_sync(pm, nres, 1);
  for (int q = nres; q < other; ++q)
    for (int i = lo_i; i < hi_i; ++i) Z[i * ld + c] *= 0x1p-500;
  double n2 = 0.0;
#pragma unroll 8
  for (int i = lo_i; i < hi_i; ++i) {
    const double zi = Z[i * ld + c];
    n2 = fma(zi, zi, n2);
  }
  n2 += __shfl_xor_sync(pm, n2, 1);
  const double sc = 1.0 / sqrt(n2);
  for (int i0 = lo_i; i0 < hi_i; i0 += kZ) {
    double zv[kZ];
#pragma unroll
    for (int u = 0; u < kZ; ++u) zv[u] = i0 + u < hi_i ? Z[(i0 + u) * ld + c] : 0.0;
#pragma unroll
    for (int u = 0; u < kZ; ++u)
      if (i0 + u < hi_i) Z[(i0 + u) * ld + c] = zv[u] * sc;
  }
}

__device__ __forceinline__ double hash_uniform(unsigned long long key) {
  // splitmix64 (Steele, Lea and Flood, 2014), mapped to [-1, 1)
  unsigned long long z = key + 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  z ^= z >> 31;
  return (double)(z >> 11) * 0x1p-52 - 1.0;
}

// Clusters.  Every member first gets two steps of inverse iteration of its own, all members at
// once (a thread each): (T_b - lambda I) = L D L^T without pivoting (pivots floored at 2^-100
// as in the twisted factorisations), from a pseudo-random start, normalised after each step.
// The vectors of a small cluster go to Z's columns and are orthonormalised by one warp (modified
// Gram-Schmidt, twice); those of a large cluster go to rows of a scratch matrix and are
// orthonormalised in panels of 32 (block classical Gram-Schmidt and a Cholesky QR of the
// panel, each twice) on the GEMM kernel, then scattered to Z.  With shifts accurate to eps ||T||
// a member's vector is its eigenvector up to (eps / gap)^2 of its neighbours, so the
// orthonormalisation only mixes members whose eigenvalues are equal at working precision.
__global__ void __launch_bounds__(32) k_cluster_vectors(
    int N, const double* __restrict__ ds, const double* __restrict__ es,
    const int* __restrict__ bstart, const int* __restrict__ bend, const double* __restrict__ lam,
    const int* __restrict__ col, const int* __restrict__ incl, const int* __restrict__ cj,
    const int* __restrict__ cl, double* Z, double* Yc, double* Wrp, double* Wl) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= N || incl[t] == 0) return;
  const int* c = cl + kClDesc * (incl[t] - 1);
  const int a0 = bstart[t], L = bend[t] - a0, j = cj[t];
  const size_t ld = (size_t)N;
  const bool large = c[1] > kSmallCl;
  double* y = large ? Yc + (size_t)c[4] + (size_t)j * L : Z + (size_t)a0 * ld + col[t];
  const size_t ys = large ? 1 : ld;
  double* rp = Wrp + (size_t)t * ld;  // reciprocal pivots
  double* lm_ = Wl + (size_t)t * ld;  // multipliers
  const double lm = lam[t];
  double r = rcp_nr(pivot_floor(ds[a0] - lm));
  rp[0] = r;
  for (int i = 0; i + 1 < L; ++i) {
    const double li = es[a0 + i] * r;
    lm_[i] = li;
    r = rcp_nr(pivot_floor(fma(-li, es[a0 + i], ds[a0 + i + 1] - lm)));
    rp[i + 1] = r;
  }
  for (int i = 0; i < L; ++i)
    y[i * ys] = hash_uniform(((unsigned long long)t << 32) + (unsigned long long)i);
  for (int it = 0; it < 2; ++it) {
    // L u = x (in place), w = D^-1 u, L^T y = w
    double u = y[0];
    for (int i = 1; i < L; ++i) {
      u = fma(-lm_[i - 1], u, y[i * ys]);
      y[i * ys] = u;
    }
    double yy = y[(L - 1) * ys] * rp[L - 1];
    y[(L - 1) * ys] = yy;
    double amax = fabs(yy);
    for (int i = L - 2; i >= 0; --i) {
      yy = fma(-lm_[i], yy, y[i * ys] * rp[i]);
      y[i * ys] = yy;
      amax = fmax(amax, fabs(yy));
    }
    const double sa = amax > 0.0 && isfinite(amax) ? 1.0 / amax : 1.0;
    double n2 = 0.0;
    for (int i = 0; i < L; ++i) {
      const double v = y[i * ys] * sa;
      n2 = fma(v, v, n2);
    }
    const double sc = sa / sqrt(n2);
    for (int i = 0; i < L; ++i) y[i * ys] *= sc;
  }
}

// Small clusters (at most kSmallCl members): modified Gram-Schmidt over the members in order,
// twice, on Z's columns; one warp per cluster.
__global__ void __launch_bounds__(32) k_cluster_small(int N, const int* __restrict__ col,
                                                      const int* __restrict__ cl,
                                                      const EighHdr* h, double* Z) {
  const int ncl = h->ncl, lane = threadIdx.x;
  const size_t ld = (size_t)N;
  for (int q = blockIdx.x; q < ncl; q += gridDim.x) {
    const int* c = cl + kClDesc * q;
    const int s = c[0], m = c[1], a0 = c[2], L = c[3];
    if (m > kSmallCl) continue;
    for (int pass = 0; pass < 2; ++pass) {
      for (int j = 0; j < m; ++j) {
        double* zj = Z + (size_t)a0 * ld + col[s + j];
        for (int jj = 0; jj < j; ++jj) {
          const double* zk = Z + (size_t)a0 * ld + col[s + jj];
          double dot = 0.0;
          for (int i = lane; i < L; i += 32) dot = fma(zk[i * ld], zj[i * ld], dot);
          dot = __shfl_sync(0xffffffffu, warp_sum_d(dot), 0);
          for (int i = lane; i < L; i += 32) zj[i * ld] = fma(-dot, zk[i * ld], zj[i * ld]);
          __syncwarp();
        }
        double n2 = 0.0;
        for (int i = lane; i < L; i += 32) n2 = fma(zj[i * ld], zj[i * ld], n2);
        n2 = __shfl_sync(0xffffffffu, warp_sum_d(n2), 0);
        const double sc = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
        for (int i = lane; i < L; i += 32) zj[i * ld] *= sc;
        __syncwarp();
      }
    }
  }
}

// A panel of b <= 32 rows of length L (row-major, leading dimension L): the Cholesky factor
// R^T R of its Gram matrix G (b x b, formed by the GEMM), computed by every CTA, then each
// CTA's columns replaced by R^-T times them (the panel's rows become orthonormal).  A pivot
// that is not positive (a dependent row) is raised to 1e-300 of the diagonal.
__global__ void __launch_bounds__(128) k_chol_apply(int b, int L, const double* __restrict__ G,
                                                    double* P) {
  __shared__ double R[32][33];
  const int tid = threadIdx.x;
  for (int i = tid; i < b * b; i += blockDim.x) R[i / b][i % b] = G[i];
  __syncthreads();
  for (int k = 0; k < b; ++k) {  // right-looking Cholesky, R upper triangular in place
    if (tid == 0) {
      double d = R[k][k];
      if (!(d > 1e-300 * fabs(G[k * b + k]))) d = fmax(1e-300 * fabs(G[k * b + k]), 1e-300);
      R[k][k] = sqrt(d);
    }
    __syncthreads();
    const double rk = R[k][k];
    for (int jj = k + 1 + tid; jj < b; jj += blockDim.x) R[k][jj] /= rk;
    __syncthreads();
    for (int idx = tid; idx < b * b; idx += blockDim.x) {
      const int i = idx / b, jj = idx % b;
      if (i > k && jj >= i) R[i][jj] = fma(-R[k][i], R[k][jj], R[i][jj]);
    }
    __syncthreads();
  }
  const int cidx = blockIdx.x * blockDim.x + tid;
  if (cidx >= L) return;
  double y[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) y[i] = i < b ? P[(size_t)i * L + cidx] : 0.0;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    if (i < b) {
      double v = y[i];
#pragma unroll
      for (int k = 0; k < i; ++k) v = fma(-R[k][i], y[k], v);
      y[i] = v / R[i][i];
    }
  }
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i < b) P[(size_t)i * L + cidx] = y[i];
}

// The rows of a large cluster's scratch into Z's columns.
__global__ void k_cluster_scatter(int N, int s, int m, int a0, int L,
                                  const double* __restrict__ Y, const int* __restrict__ col,
                                  double* Z) {
  const long long tot = (long long)m * L;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(i / L), r = (int)(i % L);
    Z[(size_t)(a0 + r) * N + col[s + j]] = Y[i];
  }
}

// ---------------------------------------------------------------------------
// 4. back-transformation V = Q Z, Q = H_0 ... H_{nref-1} in blocks of kNb reflectors
// ---------------------------------------------------------------------------
// Gram matrices G_b = Y_b^T Y_b of every block, Y_b's column c the reflector k0 + c: grid (nblk,
// kNb / 16, kNb / 16) of 16 x 16 sub-tiles, the upper ones formed and mirrored.
__global__ void __launch_bounds__(256) k_gram(int N, int nref, const double* __restrict__ Yr,
                                              double* G) {
  const int b = blockIdx.x, tr = blockIdx.y, tc = blockIdx.z;
  if (tr > tc) return;
  __shared__ double Ys[2][16][65];
  const int k0 = b * kNb;
  const int m = nref - k0 < kNb ? nref - k0 : kNb;
  const int r = threadIdx.x / 16, c = threadIdx.x % 16;
  const int gr = tr * 16 + r, gc = tc * 16 + c;
  double acc = 0.0;
  for (int j0 = k0 + 1; j0 < N; j0 += 64) {
    for (int idx = threadIdx.x; idx < 2 * 16 * 64; idx += 256) {
      const int which = idx / 1024, rr = (idx / 64) % 16, jj = idx % 64;
      const int refl = (which == 0 ? tr : tc) * 16 + rr;
      const int j = j0 + jj;
      Ys[which][rr][jj] = (refl < m && j < N) ? Yr[(size_t)(k0 + refl) * N + j] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int jj = 0; jj < 64; ++jj) acc += Ys[0][r][jj] * Ys[1][c][jj];
    __syncthreads();
  }
  G[(size_t)b * kNb * kNb + gr * kNb + gc] = acc;
  if (tr < tc) G[(size_t)b * kNb * kNb + gc * kNb + gr] = acc;
}

// Triangular factors T_b (upper): T^-1 = diag(1 / tau) + the strictly upper part of G, so column
// j solves T_jj = tau_j, T_ij = -tau_i sum_{c = i+1}^{j} G_ic T_cj upwards from i = j - 1: a warp
// per column, lane l with the sums of rows l and l + 32, to which every new T_ij is added at once (G
// is symmetric: its row i holds the factors).  Bound by the chain of a product, a broadcast and an
// addition per row.  (Dots over the lanes: 39 us;
// this: 20 us.)
constexpr int kTfWarps = 4;
__global__ void __launch_bounds__(32 * kTfWarps) k_tfactor(int nref, const double* __restrict__ tau,
                                                           const double* __restrict__ G,
                                                           double* T) {
  const int b = blockIdx.x, lane = threadIdx.x & 31;
  const int k0 = b * kNb, j = blockIdx.y * kTfWarps + (threadIdx.x >> 5);
  const int m = nref - k0 < kNb ? nref - k0 : kNb;
  const double* Gb = G + (size_t)b * kNb * kNb;
  double* Tb = T + (size_t)b * kNb * kNb;
  const double t0 = lane < m ? -tau[k0 + lane] : 0.0, t1 = lane + 32 < m ? -tau[k0 + lane + 32] : 0.0;
  double s0 = 0.0, s1 = 0.0;  // sums, then (rows >= i) the entries of T
  if (j < m) {
    // T_jj as if -tau_j times a sum of -1
    if (lane == (j & 31)) (j < 32 ? s0 : s1) = -1.0;
#pragma unroll 4
    for (int i = j; i >= 0; --i) {
      const double g0 = lane < i ? Gb[i * kNb + lane] : 0.0;
      const double g1 = lane + 32 < i ? Gb[i * kNb + lane + 32] : 0.0;
      const double e = i < 32 ? t0 * s0 : t1 * s1;  // of use in lane i mod 32
      const double t = __shfl_sync(0xffffffffu, e, i & 31);
      if (lane == (i & 31)) (i < 32 ? s0 : s1) = t;
      if (lane < i) s0 = fma(g0, t, s0);
      if (i > 32 && lane + 32 < i) s1 = fma(g1, t, s1);
    }
  }
  Tb[(size_t)lane * kNb + j] = lane <= j ? s0 : 0.0;
  Tb[(size_t)(lane + 32) * kNb + j] = lane + 32 <= j ? s1 : 0.0;
}

struct DevInfo {
  int sms = 0;
};
std::mutex g_dev_mu;
std::map<int, DevInfo> g_dev;

int device_sms(int* sms) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DONOF_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_dev_mu);
  auto it = g_dev.find(dev);
  if (it == g_dev.end()) {
    DevInfo di;
    if (cudaDeviceGetAttribute(&di.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return DONOF_ERR_CUDA;
    it = g_dev.emplace(dev, di).first;
  }
  *sms = it->second.sms;
  return DONOF_OK;
}

// The largest cluster of CTAs of the cluster form that the device takes (asked once per device).
int tridiag_cluster_max() {
  static std::atomic<int> known[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= 64) return 0;
  int c = known[dev].load();
  if (c > 0) return c - 1;
  int best = 0;
  if (cudaFuncSetAttribute(k_tridiag<kClRows, kClCols / 32, true>,
                           cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    for (int size = kClCtas; size >= 1 && best == 0; size /= 2) {
      cudaLaunchAttribute at{};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = size;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(size);
      cfg.blockDim = dim3(kTriThreads);
      cfg.dynamicSmemBytes = ((size_t)7 * kClCols) * 8;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_tridiag<kClRows, kClCols / 32, true>, &cfg) ==
              cudaSuccess && n > 0)
        best = size;
    }
  }
  cudaGetLastError();  // a size that the device does not take is no error of the call
  known[dev].store(best + 1);
  return best;
}

cudaError_t launch_tridiag(TriArgs a, int sms, cudaStream_t s) {
  int size = 1;
  while (size * kRowWarps < a.N && size < kClCtas) size *= 2;
  // One cluster while a row warp has one row and the vector few pieces (all of donof_eigh, grid ->
  // cluster: 24: 278 -> 268 us, 64: 552 -> 509, 120: 962 -> 891; with two rows a warp 160: 1288 ->
  // 1298, 256: 2286 -> 2490).  Fewer CTAs for the grid form change nothing (1 to 8 rows a CTA)
  if (a.N <= kClCols && size <= tridiag_cluster_max()) {
    if (size > 8) {  // (each time: the context may be another one since the device was asked)
      const cudaError_t e = cudaFuncSetAttribute(
          k_tridiag<kClRows, kClCols / 32, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = size;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(kTriThreads);
    cfg.dynamicSmemBytes = ((size_t)3 * kClCols + 4 * a.N) * 8;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tridiag<kClRows, kClCols / 32, true>, a);
  }
  const auto kern = k_tridiag<1, kTriRowRegs, false>;
  const size_t smem = (size_t)3 * (a.N < 32 * kTriRowRegs ? 32 * kTriRowRegs : a.N) * 8;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kTriThreads, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidValue;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(sms), dim3(kTriThreads), args, smem, s);
}

}  // namespace

size_t eigh_workspace_bytes(int N) { return eigh_layout(N).total; }

EighScratch eigh_scratch(int N, char* ws) {
  const EighLayout L = eigh_layout(N);
  EighHdr* hdr = (EighHdr*)(ws + L.hdr);
  return EighScratch{ws + L.A, &hdr->abort_code, &hdr->abort};
}

int eigh_run(int N, const double* A, double* V, double* w, char* ws, cudaStream_t s) {
  if (N < 1 || N > kEighMaxN || !A || !V || !w || !ws) return DONOF_ERR_INVALID_ARG;
  const EighLayout L = eigh_layout(N);
  EighHdr* hdr = (EighHdr*)(ws + L.hdr);
  double* Aw = (double*)(ws + L.A);
  double* Yr = (double*)(ws + L.Yr);
  double* Wd = (double*)(ws + L.Wd);
  double* Wp = (double*)(ws + L.Wp);
  double* d = (double*)(ws + L.d);
  double* e = (double*)(ws + L.e);
  double* ds = (double*)(ws + L.ds);
  double* es = (double*)(ws + L.es);
  double* e2 = (double*)(ws + L.e2);
  float* df = (float*)(ws + L.df);
  float* e2f = (float*)(ws + L.e2f);
  double* tau = (double*)(ws + L.tau);
  double* lam = (double*)(ws + L.lam);
  double* glo = (double*)(ws + L.glo);
  double* ghi = (double*)(ws + L.ghi);
  int* col = (int*)(ws + L.col);
  int* bstart = (int*)(ws + L.bstart);
  int* bend = (int*)(ws + L.bend);
  int* incl = (int*)(ws + L.incl);
  int* cl = (int*)(ws + L.cl);
  int* cj = (int*)(ws + L.cj);
  double* T = (double*)(ws + L.T);
  double* G = (double*)(ws + L.G);
  double* W1 = (double*)(ws + L.W1);
  double* W2 = (double*)(ws + L.W2);
  double* part = (double*)(ws + L.part);
  const long long nn = (long long)N * N;
  const size_t nnb = (size_t)nn * 8;
  auto ok = [](cudaError_t e) { return e == cudaSuccess; };

  if (!ok(cudaMemsetAsync(hdr, 0, sizeof(EighHdr), s))) return DONOF_ERR_CUDA;
  const int gcopy = (int)((nn + 255) / 256 < 152 * 4 ? (nn + 255) / 256 : 152 * 4);
  k_eigh_amax<<<gcopy, 256, 0, s>>>(A, nn, hdr);
  k_eigh_scale_copy<<<gcopy, 256, 0, s>>>(A, nn, hdr, Aw);
  count_launch(2);
  // V may share A's storage: it is written only after the scaled copy
  if (!ok(cudaMemsetAsync(Yr, 0, nnb, s)) || !ok(cudaMemsetAsync(V, 0, nnb, s)))
    return DONOF_ERR_CUDA;

  // 1. tridiagonal reduction, one CTA per SM, co-resident (cooperative launch)
  int sms = 0;
  int rc = device_sms(&sms);
  if (rc != DONOF_OK) return rc;
  TriArgs ta{N, Aw, Yr, d, e, tau, (double*)(ws + L.pbuf), hdr};
  if (!ok(launch_tridiag(ta, sms, s))) return DONOF_ERR_CUDA;
  count_launch(1);

  // 2. eigenvalues (of T scaled to ||T||_inf <= 1)
  const size_t prep_smem = (size_t)2 * N * 4 + (size_t)(N + 31) / 32 * 4;
  if (!ok(cudaFuncSetAttribute(k_tri_prep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)prep_smem)))
    return DONOF_ERR_CUDA;
  k_tri_prep<<<1, 256, prep_smem, s>>>(N, d, e, hdr, ds, es, e2, df, e2f, bstart, bend, glo, ghi);
  const size_t bis_smem = (size_t)N * 24;
  if (!ok(cudaFuncSetAttribute(k_bisect, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)bis_smem)))
    return DONOF_ERR_CUDA;
  // a warp (two eigenvalues) per CTA while that spreads them over more SMs
  const int bis_threads = N <= 2 * sms ? 32 : kBisThreads;
  k_bisect<<<(N * 16 + bis_threads - 1) / bis_threads, bis_threads, bis_smem, s>>>(
      N, ds, e2, df, e2f, bstart, bend, glo, ghi, hdr, lam);
  const size_t rank_smem = (size_t)N * 12 + (size_t)(N + 31) / 32 * 4;
  if (!ok(cudaFuncSetAttribute(k_rank_plan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)rank_smem)))
    return DONOF_ERR_CUDA;
  k_rank_plan<<<(N * kRankLanes + 255) / 256, 256, rank_smem, s>>>(N, lam, bend, hdr, col, w, incl, cl, cj,
                                                      bstart);
  // 3. eigenvectors of T (into V)
  k_twisted<<<(2 * N + 31) / 32, 32, 0, s>>>(N, ds, es, e2, bstart, bend, lam, col, incl, V, Wp,
                                            Wd);
  count_launch(4);
  if (!ok(cudaGetLastError())) return DONOF_ERR_CUDA;
  // clusters: the plan is read on the host (one wait for the stream)
  int hp[2] = {0, 0};
  if (!ok(cudaMemcpyAsync(hp, &hdr->ncl, sizeof(hp), cudaMemcpyDeviceToHost, s)) ||
      !ok(cudaStreamSynchronize(s)))
    return DONOF_ERR_CUDA;
  if (hp[0] > 0) {
    // the scratch: Aw (free after the reduction) for the large clusters' vectors, Wd and Wp rows
    // for the members' factorisations (free after the twisted factorisations)
    k_cluster_vectors<<<(N + 31) / 32, 32, 0, s>>>(N, ds, es, bstart, bend, lam, col, incl, cj, cl,
                                                   V, Aw, Wd, Wp);
    k_cluster_small<<<kFixCTAs, 32, 0, s>>>(N, col, cl, hdr, V);
    count_launch(2);
    if (!ok(cudaGetLastError())) return DONOF_ERR_CUDA;
  }
  if (hp[1] > kSmallCl) {
    std::vector<int> hcl((size_t)kClDesc * hp[0]);
    if (!ok(cudaMemcpyAsync(hcl.data(), cl, hcl.size() * 4, cudaMemcpyDeviceToHost, s)) ||
        !ok(cudaStreamSynchronize(s)))
      return DONOF_ERR_CUDA;
    double* Cc = W1;  // r0 x 32 overlaps of a panel with the rows before it
    double* Gp = W2;  // 32 x 32 Gram matrix of a panel
    for (int q = 0; q < hp[0]; ++q) {
      const int* c = &hcl[(size_t)kClDesc * q];
      const int m = c[1], L = c[3];
      if (m <= kSmallCl) continue;
      double* Y = Aw + c[4];
      for (int r0 = 0; r0 < m; r0 += 32) {
        const int b = m - r0 < 32 ? m - r0 : 32;
        double* P = Y + (size_t)r0 * L;
        for (int pass = 0; pass < 2; ++pass) {
          if (r0 > 0) {
            // Cc = Y[0:r0] P^T, then P -= Cc^T Y[0:r0]
            if (!ok(cudaMemsetAsync(Cc, 0, (size_t)r0 * b * 8, s)) ||
                !ok(launch_dgemm(split_k_args(r0, b, L, Y, L, 1, P, 1, L, Cc, b, 1, part), s)))
              return DONOF_ERR_CUDA;
            DgemmArgs u{};
            u.M = b; u.N = L; u.K = r0; u.KB = 1; u.batch = 1; u.ksplit = 1;
            u.A = Cc; u.sAm = 1; u.sAk = b;
            u.B = Y; u.sBk = L; u.sBn = 1;
            u.C = P; u.sCm = L; u.sCn = 1;
            u.alpha = -1.0; u.beta = 1.0;
            if (!ok(launch_dgemm(u, s))) return DONOF_ERR_CUDA;
          }
          if (!ok(cudaMemsetAsync(Gp, 0, (size_t)b * b * 8, s)) ||
              !ok(launch_dgemm(split_k_args(b, b, L, P, L, 1, P, 1, L, Gp, b, 1, part), s)))
            return DONOF_ERR_CUDA;
          k_chol_apply<<<(L + 127) / 128, 128, 0, s>>>(b, L, Gp, P);
          count_launch(1);
        }
      }
      k_cluster_scatter<<<152 * 4, 256, 0, s>>>(N, c[0], m, c[2], L, Y, col, V);
      count_launch(1);
      if (!ok(cudaGetLastError())) return DONOF_ERR_CUDA;
    }
  }

  // 4. V = Q Z
  if (L.nblk > 0) {
    k_gram<<<dim3(L.nblk, kNb / 16, kNb / 16), 256, 0, s>>>(N, L.nref, Yr, G);
    k_tfactor<<<dim3(L.nblk, kNb / kTfWarps), 32 * kTfWarps, 0, s>>>(L.nref, tau, G, T);
    count_launch(2);
    if (!ok(cudaGetLastError()) ||
        !ok(digit_reflect(N, L.nref, Yr, T, V, ws + L.A, &hdr->abort_code, &hdr->abort, s)))
      return DONOF_ERR_CUDA;
  }
  return ok(cudaGetLastError()) ? DONOF_OK : DONOF_ERR_CUDA;
}

}  // namespace donof

using namespace donof;

extern "C" int donof_eigh_workspace_size(int32_t n, size_t* bytes) {
  if (n < 1 || n > kEighMaxN || !bytes) return DONOF_ERR_INVALID_ARG;
  *bytes = eigh_workspace_bytes(n);
  return DONOF_OK;
}

extern "C" int donof_eigh(int32_t n, const double* A, double* V, double* w, void* workspace,
                          size_t workspace_bytes, void* stream) {
  if (n < 1 || n > kEighMaxN || !A || !V || !w) return DONOF_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < eigh_workspace_bytes(n) ||
      ((uintptr_t)workspace % kAlign) != 0)
    return DONOF_ERR_WORKSPACE;
  return eigh_run(n, A, V, w, (char*)workspace, (cudaStream_t)stream);
}

extern "C" int donof_eigh_read_status(const void* workspace, int32_t* status, void* stream) {
  if (!workspace || !status) return DONOF_ERR_INVALID_ARG;
  EighHdr h{};
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemcpyAsync(&h, workspace, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return DONOF_ERR_CUDA;
  *status = h.abort ? DONOF_ERR_TIMEOUT : (h.nonfinite ? DONOF_ERR_NONFINITE : DONOF_OK);
  return DONOF_OK;
}
