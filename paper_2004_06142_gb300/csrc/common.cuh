// Internal declarations shared by the CUDA translation units of libdonof.
// Nothing here is part of the C ABI (include/donof.h is).
#pragma once

#include <utility>
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/donof.h"

namespace donof {

// ---------------------------------------------------------------------------
// Device-resident header at the start of every workspace.
// ---------------------------------------------------------------------------
struct DevHeader {
  int32_t status;      // DONOF_OK or the first DONOF_ERR_* raised on the device
  int32_t e3;          // output exponent of the G split partials (0: true units)
  int32_t zero_exp;    // always 0 (epilogue exponent of raw partial sums)
  int32_t abort_flag;  // set when a bounded device wait gives up; cleared per build
  double E;            // energy of the last build
  double sC2;          // bound on ||C_act||_2^2 (Gershgorin on C_act^T C_act)
};

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }
__host__ __device__ inline int round_up_int(int x, int a) { return (x + a - 1) / a * a; }

// Derived sizes of one problem.
struct Dims {
  int N, Q, A, Ap, Np, npair, ncwo, ng, pb, nblk, functional, layout, precision;
  int nsingle;  // singly occupied orbitals (Omega_I) at npair .. npair + nsingle - 1
  int splits;  // split-K factor of the G contraction (mixed path)
  int digit;   // FP64: the contractions as exact digit products on the tensor cores (digits.cu)
  size_t ws_total;  // bytes of the workspace (at least; FP64)
};

// Byte offsets of every buffer inside the workspace.
struct Layout {
  size_t header;
  // shared by both precisions
  size_t n, sqn, phi, dn, dsq, dphi, Acoef, Bcoef, Hd, hC, J, K, G, dEdg, Epart;
  size_t skp;  // deterministic split-K partials of the FP64 N x A products
  // FP64 path
  size_t X64, b64, Y64, Bun;
  // FP64 path on digit products: largest biased exponents of B's rows (eRow, from
  // prepare), of C's columns, h's rows and G's columns, of X per (P, q) and per mu, of b and
  // w, and Y's columns; the stage images of C_act (then of G) and of Y; w^P; the AO indices' scales
  // (KScale) of B and, for a build's end without a B, of h
  size_t eRow, eC64, eH64, eG64, exq, exm, bmax, wmax, exend, eY64, Cimg, Yimg, W64, sB, sH;
  // mixed path
  // integer + fraction planes (h, f) of the tensor-core operands and their per-row
  // exponents: B (Bhi/Blo, eB), C_act^T (Chi/Clo, eC), X^T for b (Xthi/Xtlo, eXt), X for G
  // (Xhi/Xlo, eX3 per split), Y (Yhi/Ylo, eY per split); the exponents of C^T and G^T for
  // lambda (eCf, eG; their planes share the buffers of h C_act below)
  size_t Bhi, Blo, eB, L1max, Chi, Clo, eC, cnorm, Xhi, Xlo, Xthi, Xtlo, eXt, b32, Yhi, Ylo,
      Gpart, D, rn2, spOf, eX3, eY, eCf, eG;
  // symmetric storage of the split B: per-AO scale exponents s, their source (max over P of
  // the row norms), per-slice maxima of the scaled row norms, and the split of
  // (diag 2^s C_act)^T that multiplies it
  size_t eS, rnmax, tmax, ChiS, CloS, eCs;
  size_t gram;  // per-chunk parts of the Gram matrix of C_act (fp32)
  // between the b and G contractions: w^P (fp32), per-split K and J partials (double),
  // fp32 copies of the J and K coefficient matrices ([Ap][Ap])
  size_t W, Ksp, Jsp, AcF, BcF;
  // h C_act and lambda = C^T G on the tensor cores: the split of h (then of C^T) extended
  // by its residual (four K-block planes per slot, hAH/hAF, exponents eh), the same planes
  // of C_act^T (then of G^T) (cPH/cPF), and the fp32 products of the four blocks (hpart)
  size_t hAH, hAF, cPH, cPF, eh, hpart;
  size_t total;
};

Dims make_dims(const donof_problem* p);

// Storage of the split B for the half transform.  N > kDenseMaxN: lower-triangle tile
// storage, row tiles of 128 AO indices (T of them), the last one stored with its rows rounded
// up to a multiple of 64; tile (i, j), j <= i, holds rows of tile i and columns of tile j as
// chunks of 64 columns, each chunk [R_i rows][64] with the 16-byte pieces of row r at
// piece ^ (r % 8).  N <= kDenseMaxN (dense): every slice whole, [N][ld] with ld = N rounded up
// to 8 (a tensor-map row pitch of 16-byte multiples), read through a 3-D tensor map whose
// zero fill pads the 128-row tiles and 64-wide K steps; at these sizes the tiles' padding
// would cost more bytes than the dense copy of the upper triangle.
constexpr int kDenseMaxN = 256;
struct SymTiles {
  int T, Rlast;
  long long perP;  // elements per slice and plane
  int dense, ld;   // dense storage and its row pitch (elements)
};
__host__ __device__ inline int sym_R(const SymTiles& t, int i) { return i < t.T - 1 ? 128 : t.Rlast; }
__host__ __device__ inline long long sym_tile_off(const SymTiles& t, int i, int j) {
  return 16384LL * i * (i + 1) / 2 + (long long)sym_R(t, i) * 128 * j;
}
__host__ __device__ inline SymTiles sym_tiles(int N) {
  SymTiles t;
  t.T = (N + 127) / 128;
  const int last = N - 128 * (t.T - 1);
  t.Rlast = (last + 63) / 64 * 64;
  t.dense = N <= kDenseMaxN ? 1 : 0;
  t.ld = (N + 7) / 8 * 8;
  t.perP = t.dense ? (long long)N * t.ld
                   : sym_tile_off(t, t.T - 1, 0) + (long long)t.Rlast * (128LL * (t.T - 1) + t.Rlast);
  return t;
}

// ---------------------------------------------------------------------------
// Chained launches (programmatic dependent launch).  A build is a chain of some 25 kernels, most
// of them a few microseconds long on the small molecules, and between two of them a plain launch
// leaves the chip idle while the first one drains and the next one is set up.  A chained kernel is
// set up while the one before it runs: every kernel of the chain lets its successor be launched as
// soon as its own CTAs are resident (the contractions: as they leave, because CTAs parked beside
// one slow it down), and waits before its first access to memory until the kernel before it is
// complete and its writes are visible.  The wait is transitive, as each kernel completes only after
// its own wait.  A call's first kernel is launched plainly, so that nothing is assumed of the
// caller's kernels; behind a copy or a memset a chained launch is a plain one.  The tridiagonal
// reduction, whose CTAs wait on one another, takes no part.  24 / 96 / 10 orbitals, mixed: 157 ->
// 115 us a build and adjoint; 97 / 331 / 19, double, with integrals: 216 -> 183.
//
// Only grids of up to kChainCtas CTAs (two per SM) are chained: the CTAs of a chained kernel are
// placed where the kernel before leaves room, unevenly, which costs wide kernels more than the gap
// (500 / 2000 / 80: J, K and Y with 785 and 1216 CTAs 86 us plainly, 154 chained).  The same holds
// for the fp16 contractions that fill the chip, which find the units of their neighbours in L2
// (launch_tc).  Grouped launches are wide and stay plain (64 instances: 1778 us, 1820 chained).
// ---------------------------------------------------------------------------
// First statement of a chained kernel (a plainly launched one passes through).  Returns 0, through
// the wait: loads through read-only pointers may be moved over a memory clobber, so that every such
// load has to take its address from this value (the block's coordinates, Blk::zero).
__device__ __forceinline__ int chain_begin() {
  int z;
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;\n\tmov.u32 %0, 0;"
               : "=r"(z)
               :
               : "memory");
  return z;
}
// The same for a kernel whose successor is launched only as its CTAs leave.
__device__ __forceinline__ int chain_wait() {
  int z;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(z) : : "memory");
  return z;
}
constexpr int kChainCtas = 304;
template <class... P, class... Args>
cudaError_t launch_chained_to(int max_ctas, void (*kernel)(P...), dim3 grid, dim3 block,
                              size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = (long long)grid.x * grid.y * grid.z <= max_ctas ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <class... P, class... Args>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t s, Args&&... args) {
  return launch_chained_to(kChainCtas, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------------------
// Grouped launches (batch.cu): one launch runs a kernel for every instance of a batch.  A
// kernel body takes its block coordinates as a Blk (the native ones for a single instance);
// in a grouped launch instance i owns the blocks [start[i], start[i+1]) of the flat grid,
// laid out as its own grid of dims[3i .. 3i+2].
// ---------------------------------------------------------------------------
struct Blk {
  int x, y, z, gx, gy, gz;
  int zero;  // 0, known only once the kernels before are complete (chain_begin)
};
__device__ __forceinline__ Blk native_blk() {
  const int z = chain_begin();
  return Blk{(int)blockIdx.x + z, (int)blockIdx.y + z, (int)blockIdx.z + z,
             (int)gridDim.x,      (int)gridDim.y,      (int)gridDim.z,      z};
}
// One instance of a batch: its sizes, workspace carving and pointers.
struct InstRec {
  Dims d;
  Layout L;
  char* ws;
  const double *h, *B, *C, *gamma;
  const int32_t* pm;
  double *E, *lam, *dEdg, *dEdC;
  const double* Ebar;  // upstream gradient of the adjoint (1.0)
};
struct GroupLaunch {
  const InstRec* inst;
  const int* start;  // [ninst + 1]
  const int* dims;   // [3 ninst]
  int ninst;
};
// The instance of this block and its coordinates in that instance's grid.
__device__ __forceinline__ int group_locate(const GroupLaunch& g, Blk& b) {
  const int bid = (int)blockIdx.x;
  int lo = 0, hi = g.ninst - 1;
  while (lo < hi) {  // the last instance whose first block is at or before bid
    const int mid = (lo + hi + 1) >> 1;
    if (g.start[mid] <= bid) lo = mid;
    else hi = mid - 1;
  }
  const int l = bid - g.start[lo];
  const int gx = g.dims[3 * lo], gy = g.dims[3 * lo + 1], gz = g.dims[3 * lo + 2];
  b.x = l % gx;
  b.y = (l / gx) % gy;
  b.z = l / (gx * gy);
  b.gx = gx;
  b.gy = gy;
  b.gz = gz;
  b.zero = 0;
  return lo;
}

// What a build accumulates into or writes only in part, cleared by spare CTAs of its first kernel
// (a memset each was a launch and broke the chain; 24 / 96 / 10 orbitals, mixed: 115 -> 109 us a
// build and adjoint).
struct ZeroJob {
  int* flag;          // one word, may be null
  double* p[4];       // n[i] doubles each (0: none)
  long long n[4];
  __host__ void add(void* at, size_t bytes) {
    for (int i = 0; i < 4; ++i)
      if (n[i] == 0) {
        p[i] = (double*)at;
        n[i] = (long long)(bytes / 8);
        return;
      }
  }
};
__device__ __forceinline__ void zero_ranges(const ZeroJob& z, int cta, int ctas) {
  if (z.flag && cta == 0 && threadIdx.x == 0) *z.flag = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    for (long long i = cta * (long long)blockDim.x + threadIdx.x; i < z.n[r];
         i += (long long)ctas * blockDim.x)
      z.p[r][i] = 0.0;
}

// The K and J partials' entries (q, p0..p0+3) on and below the diagonal (p0 <= q, p0 a
// multiple of 4), row by row: rows 4k .. 4k+3 have k + 1 such quads each, so the rows before
// 4k hold 2k(k+1) of them.
__host__ __device__ inline int kpart_quads(int A) {
  const int kb = A / 4;
  return 2 * kb * (kb + 1) + (A % 4) * (kb + 1);
}

// Entries of K and J per CTA of k_jk_eY's sums (mid.cu).
constexpr int kJkEntries = 64;
// Tiles of k_diag_w (mid.cu): a CTA per 32 slices and 64 columns.
constexpr int kDiagWTileSlices = 32, kDiagWTileCols = 64;

// The grouped launches of one batched build, in order (batch.cu builds their grids).
enum GroupKind {
  GK_ZERO, GK_OCC, GK_COEF, GK_SPLIT_C, GK_TC_HC, GK_SUM_HC, GK_GRAM_PART, GK_GRAM_FINAL,
  GK_HDIAG, GK_XEXP, GK_TC_HALF, GK_TC_B, GK_DIAGW, GK_KPART, GK_JKEY, GK_YQUANT, GK_TC_G,
  GK_REDUCEG, GK_EROWS, GK_EFINAL, GK_SPLIT_L, GK_TC_LAM, GK_SUM_L, GK_BWD, GK_COUNT
};
// Host launchers of the grouped kernels (blocks: the flat grid; threads, smem per block).
cudaError_t launch_fp64_group(int kind, const GroupLaunch& g, int blocks, int threads,
                              size_t smem, cudaStream_t s);
cudaError_t launch_mid_group(int kind, const GroupLaunch& g, int blocks, dim3 threads,
                             cudaStream_t s);
cudaError_t launch_tc_small_group(int kind, const GroupLaunch& g, int blocks, int threads,
                                  cudaStream_t s);
// Grouped tensor-core contractions (kind GK_TC_*; tc.cu): their argument and tensor-map
// records are opaque here, byte records of tc_args_bytes() and tc_maps_bytes() each (maps
// 64-byte aligned).  Setup fills instance records on the host and counts its work units;
// finish writes the kernel-wide settings into all records and returns the launch's shared
// memory and its numeric mode (cat: the planes of B concatenated, for narrow tiles); the
// launch reads the records from device memory.
bool tc_group_setup(int kind, const Dims& d, char* ws, const Layout& L, void* a_rec,
                    void* m_rec, int& units);
size_t tc_group_finish(int kind, void* a_recs, int ninst, int* status, int* abort_flag,
                       int& cat);
cudaError_t launch_tc_group(int kind, const void* args_dev, const void* maps_dev,
                            const int* ustart, int ninst, int units, size_t smem, int cat,
                            cudaStream_t s);
size_t tc_args_bytes();
size_t tc_maps_bytes();

// Tracing (api.cu): no-ops unless donof_profile_enable(1) was called.
void prof_begin(int phase, cudaStream_t s);
void prof_end(int phase, cudaStream_t s);
void count_launch(int n);
Layout make_layout(const Dims& d);

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------
__device__ inline void set_status(DevHeader* h, int code) {
  atomicCAS(&h->status, 0, code);
}

// Integer + fraction split of the tensor-core operands.  A vector x of K elements is
// 2^e (h + f) with y = x / 2^e, h = rint(y) rounded to fp16 (exact up to 2048, even
// integers up to 4096) and f = fp16(y - h).  e is the smallest exponent with
// ||y||_2 < T = 2^12 - sqrt(K)/2 - 2: then at most three elements exceed 2048, so
// |h - y| <= 1/2 elementwise except there (<= 3/2), ||h - y||_2 <= sqrt(K)/2 + 2 and
// ||h||_2 < 2^12.  For two such vectors every partial sum of h_a h_b is an integer below
// 2^24 in magnitude (Cauchy-Schwarz), so the integer products accumulate exactly in fp32.
// `nrm` must bound ||x||_2.
// 1/T rounded up (relative 2^-50), so that nrm * intfrac_inv_target(K) >= nrm / T after
// rounding: the exponent below never comes out too small.  Computed once per launch (the
// FP64 square root and division are slow on this GPU).
__host__ __device__ inline double intfrac_inv_target(double K) {
  double T = 4096.0 - 0.5 * sqrt(K) - 2.0;
  if (T < 1024.0) T = 1024.0;  // K above 3.7e7: exactness no longer guaranteed, values still
                               // represented to within the fp16 fraction
  return (1.0 / T) * (1.0 + 0x1p-50);
}
__host__ __device__ inline int intfrac_exponent_inv(double nrm, double invT) {
  if (!(nrm > 0.0)) return 0;
  int e;
  frexp(nrm * invT, &e);  // nrm / T <= nrm * invT < 2^e
  return e;
}
__host__ __device__ inline int intfrac_exponent(double nrm, double K) {
  return intfrac_exponent_inv(nrm, intfrac_inv_target(K));
}
// Exponent of a row from its squared norm, without the FP64 square root: the smallest e
// with sqrt(nrm2) / T < 2^e, from x = nrm2 * invT2 (invT2 >= 1/T^2 after rounding):
// x < 2^e2 gives sqrt(nrm2) / T <= sqrt(x) < 2^(e2/2) <= 2^ceil(e2/2).
__host__ __device__ inline double intfrac_inv_target_sq(double K) {
  const double i = intfrac_inv_target(K);
  return (i * i) * (1.0 + 0x1p-50);
}
__host__ __device__ inline int intfrac_exponent_sq(double nrm2, double invT2) {
  if (!(nrm2 > 0.0)) return 0;
  int e2;
  frexp(nrm2 * invT2, &e2);
  return e2 >= 0 ? (e2 + 1) / 2 : -((-e2) / 2);  // ceil(e2 / 2)
}
// 2^e as a double, exact for -1022 <= e <= 1023 (the exponents here are far inside)
__device__ inline double pow2d(int e) {
  e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
  return __longlong_as_double((long long)(e + 1023) << 52);
}
// The integer + fraction split (and its residual) of y = v 2^k for a double v, formed in
// fp32 (this GPU's FP64 pipe is narrow): v as the two-float vh + vl (vh = fl32(v), vl =
// fl32(v - vh), within 2^-48 |v|); both scaled by 2^k exactly; h = fp16(rint(yh)) (even
// above 2048), dh = yh - h (exact: |yh| < 2^12), f = fp16(dh + yl), r = fp16((dh - f) + yl).  The same h and f as the
// double split up to rounding ties (h may then be the other neighbour of y, |y - h| a few
// units of 2^-24 above 1/2), r to about 2^-36 of the unit of h.  Outside the normal range of
// a float scale (|k| > 120) the double arithmetic is used.
__device__ inline void intfrac_split_v(double v, int k, __half& h, __half& f, __half& r) {
  if (k < -120 || k > 120) {
    const double y = v * __longlong_as_double((long long)(k + 1023) << 52);
    const float hf = (float)rint(y);
    h = __float2half_rn(hf);
    f = __float2half_rn((float)(y - (double)__half2float(h)));
    r = __double2half((y - (double)__half2float(h)) - (double)__half2float(f));
    return;
  }
  const float vh = __double2float_rn(v);
  const float vl = __double2float_rn(v - (double)vh);
  const float sc = __int_as_float((k + 127) << 23);
  const float yh = vh * sc, yl = vl * sc;
  h = __float2half_rn(rintf(yh));
  const float dh = yh - __half2float(h);  // h as stored (even above 2048): exact
  f = __float2half_rn(dh + yl);
  r = __float2half_rn((dh - __half2float(f)) + yl);
}
__device__ inline void intfrac_split(double y, __half& h, __half& f) {
  const float hf = (float)rint(y);  // exact: |y| < 4096
  h = __float2half_rn(hf);
  f = __float2half_rn((float)(y - (double)__half2float(h)));
}
__device__ inline void intfrac_split(float y, __half& h, __half& f) {
  h = __float2half_rn(rintf(y));
  f = __float2half_rn(y - __half2float(h));  // exact difference: |y| < 4096
}

// ---------------------------------------------------------------------------
// Kernel launchers (host side), implemented in fp64.cu and tc.cu.
// All return a cudaError_t of the launch.
// ---------------------------------------------------------------------------

// C[b](m, n) = alpha * sum_{kb, k} A(m, kb, k) B(kb, k, n) + beta * C[b](m, n)
// with A(m, kb, k) = A[b*sAb + m*sAm + kb*sAkb + k*sAk] and
//      B(kb, k, n) = B[b*sBb + kb*sBkb + k*sBk + n*sBn];
// Ktot > 0 limits the flattened contraction index kb*K + k to [0, Ktot) (used to split one
// long contraction into KB chunks of K that ksplit CTAs share).
// Output tile width of k_dgemm: 32 where it pads the width less than 64 does.
inline int dgemm_tile_n(int N) { return (N + 31) / 32 * 32 < (N + 63) / 64 * 64 ? 32 : 64; }
// ksplit > 1 (batch 1 only): each CTA stores its partial product alpha * A B over its share
// of the kb range in part[ks][M][N], and a second kernel adds the ksplit partials to C in
// order of ks (C += sum, so beta must be 1): the result does not depend on scheduling.
struct DgemmArgs {
  int M, N, K, KB, batch, ksplit, Ktot;
  const double* A; long long sAb, sAm, sAk, sAkb;
  const double* B; long long sBb, sBk, sBn, sBkb;
  double* C; long long sCb, sCm, sCn;
  double alpha, beta;
  double* part;  // ksplit x M x N scratch when ksplit > 1
};
cudaError_t launch_dgemm(const DgemmArgs& a, cudaStream_t s);

// Powers of two taken off one operand of a contraction, along its k, and put on the other: info =
// {whether any s is not zero, the largest s}, s >= 0, kp = s 2^20, kn = -s 2^20, padded with zeros
// to kscale_pad (digits.cu).
struct KScale {
  const int* info;
  const uint32_t *kp, *kn;
};
__host__ __device__ inline int kscale_pad(int K) { return (K + 31) / 32 * 32; }
inline size_t kscale_bytes(int K) { return 256 + (size_t)2 * kscale_pad(K) * 4; }
inline KScale kscale_at(char* p, int K) {
  const uint32_t* w = (const uint32_t*)(p + 256);
  return KScale{(const int*)p, w, w + kscale_pad(K)};
}
// Products of doubles as exact digit products on the tensor cores (digits.cu).
struct DigitArgs {
  // A(m, k): row m = b Mb + r at A + b sAb + r sAm; k = kb Kpad + q at kb sAkb + q sAk
  // (q < Kin; Kpad a multiple of 8 pads each kb with zeros)
  const double* A;
  long long sAb, sAm, sAk, sAkb;
  int M, Mb, Kin, Kpad, KB;
  const int* eA;        // per row: the largest biased exponent in it, or a larger one; null: 1023
  // when set (KB 1): A(m, k) is taken times 2^-s_k, ks the words of KScale; where *ks_on is 0, s = 0
  const uint32_t* ks;
  const int* ks_on;
  const __half* Bimg;   // stage images of B (k_digit_planes)
  const int* eB;        // per column, as eA
  int N, NT, ntiles, mtiles, nstages, splits;
  int imgNT;            // columns of the images' tiles, a multiple of NT
  // C(m, n) at C + split sCs + (m / Mb) sCb + (m % Mb) sCm + n
  double* C;
  long long sCs, sCb, sCm;
  // when set: the largest biased exponents of the result, per (m / Mb, n) in exq[.. exq_ld + n]
  // and per m % Mb in exm (atomic maxima; zeroed by the caller); exq's of the result times
  // 2^-row_s[m % Mb]
  int *exq, *exm;
  int exq_ld;
  const uint32_t* row_s;  // as kp
  int sub;              // C -= A B
  int vecA, vecC;       // 16-byte loads of A / stores of C are aligned
  int *status, *abort_flag;
  uint32_t k64;         // the half2 word 1024, an argument so that it stays in a register
};
// Tiling of an operand B of N columns over a contraction of K (padded) elements: column tiles of
// NT (a multiple of 16, at most 64, as even as the width allows), stages of 32 elements, and
// the bytes of its stage images.
struct DigitShape {
  int NT, ntiles, nstages;
  size_t bytes;
};
inline DigitShape digit_shape(int N, long long K) {
  DigitShape t;
  const int c = (N + 15) / 16;
  t.ntiles = (c + 3) / 4;
  t.NT = 16 * ((c + t.ntiles - 1) / t.ntiles);
  t.nstages = (int)((K + 31) / 32);
  t.bytes = (size_t)t.ntiles * t.nstages * 8 * t.NT * 64;
  return t;
}
// Splits of the G contraction (about one unit per SM, at least four stages and at most 64
// chunks of 256 elements each, so that group 0 stays below 2^30) and of the
// sums over slices of J and K (about 300 CTAs, at least 8 slices each).
inline int g_splits_digit(int N, int A, int np) {
  const DigitShape t = digit_shape(A, (long long)np * round_up_int(A, 8));
  const int tiles = t.ntiles * ((N + 127) / 128);
  int sp = 152 / tiles;
  if (sp > t.nstages / 4) sp = t.nstages / 4;
  const int least = (t.nstages + 511) / 512;
  return sp < least ? least : sp;
}
inline int jk_splits64(int A, int np) {
  const int nb = (A * (A + 1) / 2 + 255) / 256;
  int sp = (300 + nb - 1) / nb;
  if (sp > (np + 7) / 8) sp = (np + 7) / 8;
  return sp < 1 ? 1 : sp;
}
// C = A B (M x N, C's rows ldc apart; A(m, k) at m sAm + k sAk, B(k, n) at k sBk + n sBn, one
// stride of each 1; K <= 16384) with the operands' exponents and B's digits in `scratch`
// (digit_product_bytes, 256-byte aligned); status and abort_flag: device words of the bounded
// waits.
size_t digit_product_bytes(int M, int N, int K);
cudaError_t digit_product(int M, int N, int K, const double* A, long long sAm, long long sAk,
                          const double* B, long long sBk, long long sBn, double* C, long long ldc,
                          char* scratch, int* status, int* abort_flag, cudaStream_t s);
// V = Q Z for Q = H_0 .. H_{nref-1} in blocks of 64 reflectors (rows of Yr, unit first element,
// zeros before it; T: the blocks' triangular factors, 64 x 64 each), Z = V in place, its elements
// at most 1: per block W = T Y^T Z and Z -= Y W as digit products.  img holds
// digit_reflect_bytes(N) bytes.
size_t digit_reflect_bytes(int N);
cudaError_t digit_reflect(int N, int nref, const double* Yr, const double* T, double* V, char* img,
                          int* status, int* abort_flag, cudaStream_t s);
// The FP64 path's parts on digit products: the exponents of B's rows, h C_act, one block of
// slices (X, b, J, K, G; Bblk: its slices, dense), lambda.
cudaError_t digit_prepare_B(const Dims& d, const double* B, char* ws, const Layout& L,
                            cudaStream_t s);
// (prepared: the workspace holds a B, whose scales of the AO indices are taken; else h's)
cudaError_t digit_hc(const Dims& d, const double* h, const double* C, bool prepared, char* ws,
                     const Layout& L, ZeroJob zero, cudaStream_t s);
int digit_block(const Dims& d, const double* Bblk, int p0, int np, char* ws, const Layout& L,
                cudaStream_t s);
cudaError_t digit_lambda(const Dims& d, const double* C, bool prepared, char* ws, const Layout& L,
                         double* lam, cudaStream_t s);
// The split count split_k_args uses for an M x N output with contraction length K.
int splitk_count(int M, int N, int K);
// Symmetric FP64 eigensolver (eigh.cu): A (N x N, row-major, symmetric; not modified) =
// V diag(w) V^T with w ascending and V row-major (column j = eigenvector j).  V may share
// A's storage.  Workspace: eigh_workspace_bytes(N), 256-byte aligned, its first bytes the
// solver's device header.
constexpr int kEighMaxN = 4096;
size_t eigh_workspace_bytes(int N);
int eigh_run(int N, const double* A, double* V, double* w, char* ws, cudaStream_t s);
// The part of the solver's workspace that is free between its calls, at least
// digit_product_bytes(N, N, N), with the status and abort words of bounded waits.
struct EighScratch {
  char* mem;
  int *status, *abort_flag;
};
EighScratch eigh_scratch(int N, char* ws);
int g_splits_fp64(int N, int A, int np);
// C(m, n) += sum_k A(m, k) B(k, n) with the contraction cut into 64-wide (or 16-wide) chunks
// shared by enough CTAs to fill the GPU; `part` holds splitk_count(M, N, K) x M x N doubles
// (C must be initialised).
DgemmArgs split_k_args(int M, int N, int K, const double* A, long long sAm, long long sAk,
                       const double* B, long long sBk, long long sBn, double* C, long long sCm,
                       long long sCn, double* part);

// (the Jacobians are zero already)
cudaError_t launch_occupations(const Dims& d, const double* gamma, const int32_t* pair_map,
                               char* ws, const Layout& L, cudaStream_t s);
cudaError_t launch_coefficients(const Dims& d, const int32_t* pair_map, char* ws, const Layout& L,
                                cudaStream_t s);
cudaError_t launch_unpack_B(const Dims& d, const double* Bp, int p0, int np, double* out,
                            cudaStream_t s);
// H_pp = C_p^T h C_p and G = n o (h C_act) (one_electron_G), or G = 0 (the partial sums of
// one shard of a sharded build carry only the two-electron part).
cudaError_t launch_hdiag_ginit(const Dims& d, const double* C, char* ws, const Layout& L,
                               bool one_electron_G, cudaStream_t s);
// y += x over n doubles.
cudaError_t launch_add(double* y, const double* x, long long n, cudaStream_t s);
cudaError_t launch_jk_accumulate_f64(const Dims& d, const double* b, int np, int ld, char* ws,
                                     const Layout& L, cudaStream_t s);

cudaError_t launch_build_Y_f64(const Dims& d, const double* b, double* Y, int np, char* ws,
                               const Layout& L, cudaStream_t s);

// Mixed path between the b and G contractions (mid.cu): J, K and the Y operand split.
cudaError_t launch_mid_mixed(const Dims& d, int np, int splits, char* ws, const Layout& L,
                             cudaStream_t s);

cudaError_t launch_energy(const Dims& d, const int32_t* pair_map, char* ws, const Layout& L,
                          double* E_out, double* dEdg_out, cudaStream_t s);
cudaError_t launch_backward(const Dims& d, const double* Ebar, const char* ws, const Layout& L,
                            double* dE_dC, double* dE_dgamma, cudaStream_t s);

// mixed path
cudaError_t launch_prepare_split_B(const Dims& d, const double* B, char* ws, const Layout& L,
                                   cudaStream_t s);
// The splits of C_act^T (for b and for h C_act), of diag(2^s) C_act (half transform) and of
// h (for h C_act), in two launches.
// with_half_transform = false leaves out the operand of the half transform (its exponents
// come from the prepared B), for a build that runs no contraction over B.
cudaError_t launch_split_C(const Dims& d, const double* C, const double* h, char* ws,
                           const Layout& L, bool with_half_transform, const ZeroJob& zero,
                           cudaStream_t s);
// hC = h C_act on the tensor cores from the planes written by launch_split_C (mixed path).
int run_hc_tc(const Dims& d, char* ws, const Layout& L, cudaStream_t s);
cudaError_t launch_reduce_G(const Dims& d, char* ws, const Layout& L, cudaStream_t s);
cudaError_t launch_gram_bound(const Dims& d, const double* C, char* ws, const Layout& L,
                              cudaStream_t s);
// The three tensor-core contractions of one block of np auxiliary slices starting at p0.
int run_tc_block(const Dims& d, int p0, int np, char* ws, const Layout& L, cudaStream_t s);
// lambda = C^T G on the tensor cores with residual-extended operands (mixed path).
int run_lambda_tc(const Dims& d, const double* C, char* ws, const Layout& L, double* lam,
                  cudaStream_t s);

}  // namespace donof
