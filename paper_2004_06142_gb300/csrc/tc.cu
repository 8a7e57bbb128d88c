// Tensor-core (tcgen05 + TMEM + TMA) contractions of the mixed-precision build.
//
// The large contractions of one build (DF form of Eqs. JKpq / Gpmn and of the orbital
// gradient of Eqs. lowdin, Vee-s, Vee-d), all on one warp-specialised kernel:
//   (1) X[P][mu][q] = sum_nu B[P][mu][nu] C[nu][q]    unit = (slice, 128-row tile); A from
//       the lower-triangle tile storage of the split B (B symmetric), N = Ap, K = N
//   (2) b[P][p][q]  = sum_mu C[mu][p] X[P][mu][q]     M = np*Ap (rows (P, q)), N = Ap, K = N
//   (3) G[mu][p]   += sum_P sum_q X[P][mu][q] Y[P][q][p]   M = N, N = Ap, K = np*Ap (split)
//   (4) h C_act and lambda = C^T G                    M = N, N = Ap, K = 4 blocks of N:
//       residual-extended operands (see SplitJob), near double precision
// Operands are integer + fraction pairs (kIntFrac below): four products per K step, the
// integer products exact in one TMEM accumulator, the others in a second, fp32.  A and B
// are staged by TMA (or bulk copies for the tile storage of B) with 128-byte (BK = 64) or
// 64-byte (BK = 32) swizzling; A may also be MN-major (transposed tiles of B) or K-major
// interleaved by 8 (X in the G contraction).
//
// CTA roles (384 threads): warp 0 lane 0 issues TMA, warp 1 lane 0 issues tcgen05.mma,
// warp 2 owns the TMEM allocation, warps 4..11 drain the accumulator (one TMEM lane per
// thread, two warps per lane quadrant, each with half of the columns).  When two accumulator
// sets fit in TMEM the epilogue of one tile overlaps the MMAs of the next; with three
// regions in rotation (144 or 160 columns) the next tile waits for half of the drain;
// otherwise the epilogue releases TMEM as soon as the accumulators are in registers.
// Persistent grid: one CTA per SM, units handed out round-robin.  With CTA pairs (clusters
// of two, cta_group::2) each 256-row tile is split between two SMs: the even CTA issues the
// MMAs, each CTA stages its 128 rows of A and half of the B rows, the odd CTA's warp 3
// relays its landed stages to the even CTA.
#include <cuda.h>
#include <stdio.h>
#include <stdlib.h>

#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"
#include "tcptx.cuh"

namespace donof {
namespace {

constexpr int BM = 128;

// ------------------------------------------------------------------ kernel
// Operand numerics.
//   kSplit3: every operand x is s * (hi + lo), hi = fp16(x / s), lo = fp16(x / s - hi), with one
//            power-of-two s per matrix; D = hi*hi + hi*lo + lo*hi in one fp32 accumulator
//            (the building block exposed by the test hook; the build itself uses kIntFrac).
//   kIntFrac: every operand row r is u_r * (h + f) with u_r = 2^e_r chosen from (a bound on)
//            the row's L2 norm so that ||h||_2 < 2^12 (intfrac_exponent), h an integer
//            exact in fp16 and f = fp16(x / u_r - h).  For any two rows |sum_k h_a h_b| <
//            2^24 (Cauchy-Schwarz, every partial sum included), so the integer products
//            accumulate exactly in fp32 -- the tensor core's truncating accumulation
//            cannot bias them.  h*h goes to accumulator 0, h*f + f*h + f*f to accumulator 1.
//            The representation error is about 2^-13 u_r per element, so the norm target
//            is kept as close to 2^12 as the rounding of h allows.
constexpr int kSplit3 = 0;
constexpr int kIntFrac = 1;
// kIntFracCat: kIntFrac for narrow tiles (2 Nn <= 128, no CTA pair): the two planes of B,
// staged back to back, form one operand of 2 Nn rows, so that a K step is two MMAs,
// h_A [h_B | f_B] and f_A [h_B | f_B], each reading its A plane from shared memory once
// (half the operand traffic of four N = Nn MMAs, which bounds narrow tiles): accumulators of
// 2 Nn columns, the first with the exact h_A h_B in its left half
constexpr int kIntFracCat = 2;
constexpr int kMaxRegCols = 160;  // epilogue keeps up to this many columns per row in registers
constexpr int kEpiGroups = 2;     // epilogue warps per TMEM lane quadrant (each half the columns)
constexpr int kThreads = 128 + 128 * kEpiGroups;  // producer, MMA, TMEM, relay warps + epilogue
// per epilogue warp, the column factors of its chunks (up to 256 columns split between the
// groups), one float2 per column, in shared memory after the barriers
constexpr int kTabCols = 256 / kEpiGroups;
constexpr int kMaxSets = 8;  // TMEM accumulator sets at most (narrow tiles)
constexpr int kMaxStages = 8;  // shared-memory stages at most (16 measured no faster)
constexpr int kBarTail = 2 * kMaxSets + 4;  // barriers after full/empty, then the TMEM slot
constexpr int kTabBytes = 4 * kEpiGroups * kTabCols * 8;

struct TcArgs {
  int mode;        // 1: X stores (integer + fraction X^T for b, X for G); 2: fp32
  int M;           // valid output rows per z
  int Nn;          // output columns = B box rows (multiple of 16, <= 256)
  int m_tiles, z_count, splits;
  int kt_per_kb, nkb;
  int a_z_kb;      // A tile z coordinate = kb (else a_z_unit ? the unit's z : 0)
  int a_z_unit;
  // dense half transform whose last row tile holds at most 64 AO indices: the last tiles of
  // slices 2p and 2p + 1 share a unit (rows 0-63 and 64-127, A through the 64-row maps ah2,
  // al2), after the z_count x (m_tiles - 1) units of the full tiles
  int pack2;
  int b_z_mode;    // 0: 0, 1: z, 2: kb
  int stages;
  int nbuf;        // TMEM accumulator sets: 1, 2, 4, 8, or 3 (three regions in rotation, below)
  int epi_alt;     // 1: the two epilogue warp groups take alternate tiles (nbuf even)
  int region;      // nbuf 3: columns of each region (at least Nn)
  int nb_stage;    // B rows a shared-memory stage holds (at least this CTA's share of Nn)
  int buf_stride;  // TMEM columns per accumulator set
  int tmem_cols;
  // per-row / per-column exponents (kIntFrac): value = 2^(eA[row] + eB[col]) * acc, with
  // eA indexed by z * eA_zstride + split * eA_sstride + row (eB likewise by column)
  const int* eA; long long eA_zstride, eA_sstride;
  const int* eB; long long eB_zstride, eB_sstride;
  const int* glob_exp;  // extra power of two applied to every output (mode 2)
  // symmetric half transform: the lower-triangle tile storage of the split B (see sym below)
  const __half* a_tiled_h;
  const __half* a_tiled_f;
  int a_mn;  // 1: A operand MN-major (BK = 64): its map is [K][M], two 64-wide M boxes
  // 1: A operand interleaved by 8 along K, [z][K/8][rows][8], loaded without swizzle as
  // core matrices (4-D map of 8-row groups, coordinates {0, row/8, k/8, z})
  int a_il8;
  // symmetric half transform (BK = 64): A from the lower-triangle tile storage of the split
  // B at a_tiled_h/f + z * st.perP; unit = (slice z, row tile mt); its K steps visit the tile
  // columns in a round-robin order in which row tiles i and j of a slice read their shared
  // stored tile (i, j) in the same round (K-major for the larger index, MN-major transposed
  // for the smaller); output row mt * 128 + r is AO index mu of slice z
  int sym;
  SymTiles st;
  int grid;  // CTAs (CTA pairs) to launch (0: one per SM (pair of SMs), at most one per unit)
  // mode 1 outputs, X[row][c] with row = P * Nmu + mu (mu < Nrow valid): integer +
  // fraction X for the G contraction, interleaved by 8 along c as [P][c/8][mu < Np][8]
  // (exponent eX3[spOf[P]][mu], common to the slices of one G split) and X^T[P][c][mu]
  // (exponent eXt[P][c]) for b = C^T X; the row exponents eA are indexed by P * Nrow + mu
  int Nmu, Nrow, Ap, Np;
  __half *xhi, *xlo, *xth, *xtf;
  const int* eXt;
  const int* spOf;
  const int* eX3;
  // mode 2 output
  float* out;
  long long out_ld, out_zstride;
  // mode 2, rows (P, q) of slices of Ap rows: when set, the diagonal b^P_qq (q < diag_A) is
  // also written to diag[P * diag_A + q]
  float* diag;
  int diag_A;
  int* status;
  int* abort_flag;
};

// The operand maps of one contraction (integer and fraction planes of A and B; ah2, al2: A
// in boxes of 64 rows, for pack2).
struct TcMaps {
  CUtensorMap ah, al, bh, bl, ah2, al2;
};

// Work units of one problem (PAIR: units of a CTA pair).
__host__ __device__ inline int tc_units(const TcArgs& A, int pair) {
  if (A.pack2) return A.z_count * (A.m_tiles - 1) + (A.z_count + 1) / 2;
  const int zu = (pair && A.sym) ? (A.z_count + 1) / 2 : A.z_count;
  const int mu = (pair && !A.sym) ? (A.m_tiles + 1) / 2 : A.m_tiles;
  return zu * mu * A.splits;
}

// Round-robin (circle method) schedule over the T row tiles of a slice: in round r row
// tile i works on tile column rr_partner(i, r, T), an involution, so both row tiles that
// share a stored tile read it in the same round; every tile column once in T rounds (the
// diagonal tile in the round with no partner).
__device__ __forceinline__ int rr_partner(int i, int r, int T) {
  if ((T & 1) == 0 && r == T - 1) return i;  // even T: the round of the diagonal tiles
  const int n = T + (T & 1);                 // participants (a dummy when T is odd)
  int p;
  if (i == n - 1) p = r;
  else if (i == r) p = n - 1;
  else {
    p = 2 * r - i;  // mod n - 1, within (-(n - 1), 2 (n - 1))
    if (p < 0) p += n - 1;
    if (p >= n - 1) p -= n - 1;
  }
  return p >= T ? i : p;
}

// intfrac_split of two values at once (paired conversions; the same results)
__device__ __forceinline__ void intfrac_split2(float y0, float y1, __half2& h, __half2& f) {
  h = __floats2half2_rn(rintf(y0), rintf(y1));
  const float2 hb = __half22float2(h);
  f = __floats2half2_rn(y0 - hb.x, y1 - hb.y);
}

__device__ __forceinline__ float pow2f(int e) {
  e = e < -126 ? -126 : (e > 127 ? 127 : e);
  return __int_as_float((e + 127) << 23);
}

// The kernel body over a table of problems: problem i has the arguments targs[i] and the
// tensor maps tmaps[i] and owns the work units [ustart[i], ustart[i + 1]) of the grid's
// unit sequence (ustart null: one problem).  The kernel-wide settings (stages, TMEM layout,
// the rows of B a stage holds, the status and abort words) are those of targs[0].
template <int BK, int NUM, int PAIR>
__device__ __forceinline__ void tc_body(const TcArgs* __restrict__ targs,
                                        const TcMaps* __restrict__ tmaps,
                                        const int* __restrict__ ustart, int ninst) {
  const TcArgs& a0 = targs[0];
  constexpr int SWZ = BK * 2;  // bytes per tile row
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem =
      (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int S = a0.stages;
  // PAIR: the two CTAs of a cluster compute one M = 256 tile with cta_group::2 MMAs issued by
  // the even CTA: each CTA stages its own 128 rows of A and half of the B rows (the output
  // columns), and holds its 128 rows of the accumulator in its own TMEM
  const int nb_rows = a0.nb_stage;  // B rows a stage holds (this CTA's share, widest problem)
  const uint32_t a_bytes = BM * BK * 2;
  const uint32_t b_bytes = (uint32_t)nb_rows * BK * 2;
  const uint32_t stage_bytes = 2 * a_bytes + 2 * b_bytes;
  uint64_t* bars = (uint64_t*)(smem + (size_t)S * stage_bytes);
  // barriers: full[S], empty[S], tfull[kMaxSets], tempty[kMaxSets], drain, trel[2]; then the
  // TMEM address and the epilogue's factor tables
  const int kFull = 0, kEmpty = S, kTfull = 2 * S, kTempty = 2 * S + kMaxSets,
            kDrain = 2 * S + 2 * kMaxSets, kTrel = 2 * S + 2 * kMaxSets + 1;
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * S + kBarTail - 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  int* status = a0.status;
  int* abort_flag = a0.abort_flag;
  // kernel-wide settings in registers (the asm statements' memory clobbers would otherwise
  // reload them from the argument table after every MMA and TMEM access)
  const int nbuf = a0.nbuf;
  constexpr bool bcat = NUM == kIntFracCat && !PAIR;
  const bool nbuf3 = !bcat && nbuf == 3;  // three TMEM regions (never with bcat: Nn <= 64)
  const bool epi_alt = a0.epi_alt != 0;
  const uint32_t region = (uint32_t)a0.region, buf_stride = (uint32_t)a0.buf_stride;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int cl = PAIR ? (int)cluster_id_x() : (int)blockIdx.x;   // this CTA's work stream
  const int ncl = PAIR ? (int)ncluster_x() : (int)gridDim.x;
  // epilogue threads that release TMEM (of both CTAs of a pair)
  // epi_alt: the epilogue groups take alternate tiles (all columns), otherwise they split the
  // columns of every tile
  const uint32_t rel_count = (PAIR ? 2u : 1u) * 128u * (epi_alt ? 1u : (uint32_t)kEpiGroups);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      // PAIR: the even CTA's full barrier also waits for the odd CTA's relayed arrival
      mbar_init(bar(kFull + i), (PAIR && rank == 0) ? 2 : 1);
      mbar_init(bar(kEmpty + i), 1);
    }
    for (int i = 0; i < kMaxSets; ++i) {
      mbar_init(bar(kTfull + i), 1);
      mbar_init(bar(kTempty + i), rel_count);
    }
    mbar_init(bar(kDrain), 1);
    mbar_init(bar(kTrel + 0), rel_count);
    mbar_init(bar(kTrel + 1), rel_count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) tmem_alloc<PAIR>(smem_u32(tmem_slot), a0.tmem_cols);
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();  // the peer's barriers are initialised before any remote use
  tc_fence_after();
  const uint32_t tmem_base = *(volatile uint32_t*)tmem_slot;
  // all of the above while the kernel before runs (it holds no TMEM: one CTA of this kind per SM);
  // no load below goes through a read-only pointer
  chain_wait();

  // work units: (z, row tile, split) of each problem; PAIR: a unit is the M = 256 tile of the
  // cluster, rows of slice pair (2 zp, 2 zp + 1) in the symmetric mode, row tiles
  // (2 mu, 2 mu + 1) otherwise
  // the symmetric mode is per problem (a table may mix it with dense half transforms)
  auto sym_of = [&](const TcArgs& A) { return BK == 64 && A.sym; };
  auto z_units = [&](const TcArgs& A) {
    return (PAIR && sym_of(A)) ? (A.z_count + 1) / 2 : A.z_count;
  };
  auto m_units = [&](const TcArgs& A) {
    return (PAIR && !sym_of(A)) ? (A.m_tiles + 1) / 2 : A.m_tiles;
  };
  const int units = ustart ? ustart[ninst] : tc_units(a0, PAIR);
  // the problem of unit u and the unit's index lu among that problem's units: every role
  // walks its units in increasing order, so the problem index only moves forward
  struct Walk {
    int inst, lo, hi;
  };
  auto walk0 = [&]() { return Walk{0, 0, ustart ? ustart[1] : 0x7fffffff}; };
  auto locate = [&](Walk& w, int u, int& lu) {
    while (u >= w.hi && w.inst < ninst - 1) {
      ++w.inst;
      w.lo = w.hi;
      w.hi = ustart[w.inst + 1];
    }
    lu = u - w.lo;
    return w.inst;
  };
  // consecutive units share the split (and so the B tiles of one K range, which then come
  // from L2 for all M tiles of that split)
  auto decode = [&](const TcArgs& A, int u, int& z, int& mt, int& sp, int& half) {
    half = 0;
    if (A.pack2) {  // full tiles, then the shared last tiles of slice pairs
      const int nf = A.z_count * (A.m_tiles - 1);
      sp = 0;
      if (u < nf) {
        z = u / (A.m_tiles - 1);
        mt = u % (A.m_tiles - 1);
      } else {
        z = 2 * (u - nf);
        mt = A.m_tiles - 1;
        half = 1;
      }
      return;
    }
    const int mu_n = m_units(A);
    const int zu = u / (mu_n * A.splits);
    const int r = u % (mu_n * A.splits);
    sp = r / mu_n;
    const int mu = r % mu_n;
    z = (PAIR && sym_of(A)) ? 2 * zu + (int)rank : zu;
    mt = (PAIR && !sym_of(A)) ? 2 * mu + (int)rank : mu;
  };
  auto unit_iters = [&](const TcArgs& A, int sp) {
    if (sym_of(A)) return 2 * (A.st.T - 1) + A.st.Rlast / 64;
    const int kb0 = (int)((long long)A.nkb * sp / A.splits);
    const int kb1 = (int)((long long)A.nkb * (sp + 1) / A.splits);
    return (kb1 - kb0) * A.kt_per_kb;
  };
  // bytes of B a stage receives for a problem (its own rows)
  auto b_bytes_of = [&](const TcArgs& A) { return (uint32_t)(PAIR ? A.Nn / 2 : A.Nn) * BK * 2; };

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------ TMA producer (both CTAs of a pair)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    long long issued = 0;  // stages filled so far
    const int b_row0 = (int)rank * nb_rows;
    Walk wk = walk0();
    // the current problem's arguments, copied into registers when the problem changes (the
    // table is in global memory, and every asm statement's memory clobber would reload them)
    int cur = -1;
    TcArgs acur;
    for (int u = cl; u < units && ok; u += ncl) {
      int lu;
      const int inst = locate(wk, u, lu);
      if (inst != cur) {
        acur = targs[inst];
        cur = inst;
      }
      const TcArgs& args = acur;
      const TcMaps& maps = tmaps[inst];
      const uint32_t bu = b_bytes_of(args);
      const uint32_t bl_off = bcat ? bu : b_bytes;  // the fraction plane of B
      int z, mt, sp, half;
      decode(args, lu, z, mt, sp, half);
      if (sym_of(args)) {
        const SymTiles st = args.st;
        const bool a_valid = z < args.z_count;  // PAIR: the odd slice of an odd count is absent
        const int i = mt, Ri = sym_R(st, i);
        const size_t zoff = (size_t)z * st.perP;
        for (int r = 0; r < st.T && ok; ++r) {
          const int j = rr_partner(i, r, st.T);
          const int nch = j < st.T - 1 ? 2 : st.Rlast / 64;
          for (int c = 0; c < nch; ++c) {
            if (!mbar_wait(bar(kEmpty + stage), phase ^ 1u, status, abort_flag)) {
              ok = false;
              break;
            }
            const uint32_t fb = bar(kFull + stage);
            const uint32_t base = smem_u32(smem + (size_t)stage * stage_bytes);
            if (!a_valid) {
              mbar_expect_tx(fb, 2 * bu);
            } else if (j <= i) {  // stored tile (i, j), chunk c: Ri rows of 128 bytes, K-major
              const uint32_t ab = (uint32_t)Ri * 128u;
              mbar_expect_tx(fb, 2 * ab + 2 * bu);
              const size_t off = zoff + sym_tile_off(st, i, j) + (size_t)c * Ri * 64;
              bulk_load_once(base, args.a_tiled_h + off, ab, fb);
              bulk_load_once(base + a_bytes, args.a_tiled_f + off, ab, fb);
            } else {  // stored tile (j, i), rows 64c..64c+63 of both its chunks: MN-major
              const int Rj = sym_R(st, j);
              mbar_expect_tx(fb, 2 * a_bytes + 2 * bu);
#pragma unroll
              for (int m = 0; m < 2; ++m) {
                const size_t off =
                    zoff + sym_tile_off(st, j, i) + ((size_t)m * Rj + 64 * c) * 64;
                bulk_load_once(base + m * 8192, args.a_tiled_h + off, 8192, fb);
                bulk_load_once(base + a_bytes + m * 8192, args.a_tiled_f + off, 8192, fb);
              }
            }
            tma_load_3d(base + 2 * a_bytes, &maps.bh, fb, 128 * j + 64 * c, b_row0, 0);
            tma_load_3d(base + 2 * a_bytes + bl_off, &maps.bl, fb, 128 * j + 64 * c, b_row0, 0);
            ++issued;
            if (++stage == S) { stage = 0; phase ^= 1u; }
          }
        }
        continue;
      }
      const int kb0 = (int)((long long)args.nkb * sp / args.splits);
      const int kb1 = (int)((long long)args.nkb * (sp + 1) / args.splits);
      const bool il8 = args.a_il8 != 0, amn = BK == 64 && args.a_mn != 0;
      const bool az_kb = args.a_z_kb != 0, az_unit = args.a_z_unit != 0;
      const int bzm = args.b_z_mode, ktn = args.kt_per_kb;
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        const int az = az_kb ? kb : (az_unit ? z : 0);
        const int bz = bzm == 1 ? z : (bzm == 2 ? kb : 0);
        for (int kt = 0; kt < ktn; ++kt) {
          if (!mbar_wait(bar(kEmpty + stage), phase ^ 1u, status, abort_flag)) { ok = false; break; }
          const uint32_t fb = bar(kFull + stage);
          const uint32_t base = smem_u32(smem + (size_t)stage * stage_bytes);
          mbar_expect_tx(fb, 2 * a_bytes + 2 * bu);
          if (il8) {
            tma_load_4d(base, &maps.ah, fb, 0, mt * BM / 8, kt * BK / 8, az);
            tma_load_4d(base + a_bytes, &maps.al, fb, 0, mt * BM / 8, kt * BK / 8, az);
          } else if (half) {  // the last row tiles of slices z and z + 1, 64 rows each
            tma_load_3d(base, &maps.ah2, fb, kt * BK, mt * BM, z);
            tma_load_3d(base + a_bytes / 2, &maps.ah2, fb, kt * BK, mt * BM, z + 1);
            tma_load_3d(base + a_bytes, &maps.al2, fb, kt * BK, mt * BM, z);
            tma_load_3d(base + a_bytes + a_bytes / 2, &maps.al2, fb, kt * BK, mt * BM, z + 1);
          } else if (amn) {
            tma_load_3d(base, &maps.ah, fb, mt * BM, kt * BK, az);
            tma_load_3d(base + a_bytes / 2, &maps.ah, fb, mt * BM + 64, kt * BK, az);
            tma_load_3d(base + a_bytes, &maps.al, fb, mt * BM, kt * BK, az);
            tma_load_3d(base + a_bytes + a_bytes / 2, &maps.al, fb, mt * BM + 64, kt * BK, az);
          } else {
            tma_load_3d(base, &maps.ah, fb, kt * BK, mt * BM, az);
            tma_load_3d(base + a_bytes, &maps.al, fb, kt * BK, mt * BM, az);
          }
          tma_load_3d(base + 2 * a_bytes, &maps.bh, fb, kt * BK, b_row0, bz);
          tma_load_3d(base + 2 * a_bytes + bl_off, &maps.bl, fb, kt * BK, b_row0, bz);
          ++issued;
          if (++stage == S) { stage = 0; phase ^= 1u; }
        }
      }
    }
    // after an abort, every load already issued lands before the CTA leaves: stages below
    // `stage` were filled in this lap of the ring, the others in the previous one (if any)
    if (*(volatile int*)abort_flag != 0) {
      for (int s = 0; s < S; ++s) {
        if (s < stage) mbar_wait_quiet(bar(kFull + s), phase, kDrainLimitNs);
        else if (issued >= S) mbar_wait_quiet(bar(kFull + s), phase ^ 1u, kDrainLimitNs);
      }
    }
  } else if (PAIR && rank == 1 && warp == 3 && lane == 0) {
    // ------------------------------------------------ relay (odd CTA of a pair): each stage
    // of this CTA that has landed is announced on the even CTA's full barrier
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    Walk wk = walk0();
    // the current problem's arguments, copied into registers when the problem changes (the
    // table is in global memory, and every asm statement's memory clobber would reload them)
    int cur = -1;
    TcArgs acur;
    for (int u = cl; u < units && ok; u += ncl) {
      int lu;
      const int inst = locate(wk, u, lu);
      if (inst != cur) {
        acur = targs[inst];
        cur = inst;
      }
      const TcArgs& args = acur;
      int z, mt, sp, half;
      decode(args, lu, z, mt, sp, half);
      const int iters = unit_iters(args, sp);
      for (int it = 0; it < iters; ++it) {
        if (!mbar_wait(bar(kFull + stage), phase, status, abort_flag)) { ok = false; break; }
        mbar_arrive_remote(mapa_shared(bar(kFull + stage), 0));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1 && lane == 0 && rank == 0) {
    // ------------------------------------------------ MMA issuer (even CTA of a pair)
    // MN-major A (BK = 64): the two 64-wide M chunks 8 KB apart (leading byte offset),
    // 8-row K groups 1 KB apart (stride byte offset)
    const uint32_t mn_lbo = 8192u, mn_sbo = 1024u;
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    int local = 0;
    Walk wk = walk0();
    // the current problem's arguments, copied into registers when the problem changes (the
    // table is in global memory, and every asm statement's memory clobber would reload them)
    int cur = -1;
    TcArgs acur;
    for (int u = cl; u < units && ok; u += ncl, ++local) {
      int lu;
      const int inst = locate(wk, u, lu);
      if (inst != cur) {
        acur = targs[inst];
        cur = inst;
      }
      const TcArgs& args = acur;
      const int nn = args.Nn;
      const bool il8 = args.a_il8 != 0, amn = args.a_mn != 0;
      const uint32_t idesc =
          idesc_f16(PAIR ? 2 * BM : BM, bcat ? 2 * nn : nn) | (amn ? (1u << 15) : 0u);
      const int T = args.st.T, rl64 = args.st.Rlast / 64;
      int z, mt, sp, half;
      decode(args, lu, z, mt, sp, half);
      // the accumulator pair (d0: h*h, d1: the cross products) of this unit
      uint32_t d0, d1;
      int tf;
      if (nbuf3) {
        // three regions of Nn columns, X = [0, Nn), Y = [Nn, 2 Nn), Z = [2 Nn, 3 Nn): d1 is
        // always Y, d0 alternates X, Z; the epilogue releases Y first, so the next unit
        // waits for half of the drain only
        tf = 0;
        if (!mbar_wait(bar(kTempty + 0), (uint32_t)(local & 1) ^ 1u, status, abort_flag)) break;
        if (!mbar_wait(bar(kTrel + (local & 1)), (uint32_t)((local / 2) & 1) ^ 1u, status,
                       abort_flag))
          break;
        d1 = tmem_base + region;
        d0 = tmem_base + ((local & 1) ? 2 * region : 0u);
      } else {
        const int acc = local % nbuf;
        const uint32_t acc_phase = (uint32_t)((local / nbuf) & 1);
        if (!mbar_wait(bar(kTempty + acc), acc_phase ^ 1u, status, abort_flag)) break;
        tf = acc;
        d0 = tmem_base + (uint32_t)acc * buf_stride;
        d1 = d0 + (uint32_t)((bcat ? 2 : 1) * nn);  // second accumulator (kIntFrac)
      }
      tc_fence_after();
      // symmetric mode: the K steps in the producer's order, K-major or transposed
      const int iters = unit_iters(args, sp);
      const bool sym = sym_of(args);
      int rr = 0, cc = 0, jj = 0, nch = 0;
      if (sym) {
        jj = rr_partner(mt, 0, T);
        nch = jj < T - 1 ? 2 : rl64;
      }
      for (int it = 0; it < iters; ++it) {
        if (!mbar_try(bar(kFull + stage), phase) &&
            !mbar_wait(bar(kFull + stage), phase, status, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t base = smem_u32(smem + (size_t)stage * stage_bytes) >> 4;  // in 16 bytes
        const bool tr = amn || (sym && jj > mt);
        const uint32_t id = tr ? (idesc | (1u << 15)) : idesc;
        // the words of the descriptors and their step per 16 of k
        constexpr uint32_t kHi = sdesc_hi(8 * SWZ, SWZ == 128 ? 2 : 4);
        uint32_t a_lo = base, a_hi, a_step;
        if (il8) {  // two K-adjacent core-matrix columns (BM rows x 16 B) per step
          a_lo |= (uint32_t)(BM * 16 >> 4) << 16;
          a_hi = sdesc_hi(128, 0);
          a_step = 2 * BM * 16 >> 4;
        } else if (tr) {
          a_lo |= (mn_lbo >> 4) << 16;
          a_hi = sdesc_hi(mn_sbo, 2);
          a_step = 2048 >> 4;
        } else {
          a_lo |= 1u << 16;
          a_hi = kHi;
          a_step = 32 >> 4;
        }
        const uint32_t b_lo = (base + (2 * a_bytes >> 4)) | 1u << 16;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) {
          const uint32_t ah = a_lo + (uint32_t)k * a_step, al = ah + (a_bytes >> 4);
          const uint32_t bh = b_lo + (uint32_t)k * 2, bl = bh + (b_bytes >> 4);
          const uint32_t first = (it > 0 || k > 0) ? 1u : 0u;
          auto mma = [&](uint32_t d, uint32_t a, uint32_t b, uint32_t acc) {
            mma_f16_words<PAIR>(d, a, a_hi, b, kHi, id, acc);
          };
          if (NUM == kSplit3) {
            mma(d0, ah, bh, first);
            mma(d0, ah, bl, 1u);
            mma(d0, al, bh, 1u);
          } else if (bcat) {  // bh: the 2 Nn rows of both planes
            mma(d0, ah, bh, first);  // [h h | h f]
            mma(d1, al, bh, first);  // [f h | f f]
          } else {
            mma(d0, ah, bh, first);  // integer x integer: exact
            mma(d1, ah, bl, first);
            mma(d1, al, bh, 1u);
            mma(d1, al, bl, 1u);
          }
        }
        mma_commit<PAIR>(bar(kEmpty + stage));  // frees the stage in both CTAs of a pair
        if (++stage == S) { stage = 0; phase ^= 1u; }
        if (sym && ++cc == nch) {
          cc = 0;
          if (++rr < T) {
            jj = rr_partner(mt, rr, T);
            nch = jj < T - 1 ? 2 : rl64;
          }
        }
      }
      if (!ok) break;
      mma_commit<PAIR>(bar(kTfull + tf));
    }
    // after an abort, the MMAs already issued complete before the TMEM is freed
    if (*(volatile int*)abort_flag != 0) {
      mma_commit_local<PAIR>(bar(kDrain));
      mbar_wait_quiet(bar(kDrain), 0u, kDrainLimitNs);
    }
  } else if (warp >= 4) {
    // ------------------------------------------------ epilogue: TMEM -> registers -> global
    // warp 4 + ew reads TMEM lane quadrant q = ew % 4 (the quadrant a warp may access is its
    // index mod 4) and the column chunks of group ew / 4
    const int ew = warp - 4;
    const int q = ew & 3, eg = ew >> 2;
    // this warp's table of column factors
    float2* ctab = (float2*)(bars + 2 * S + kBarTail) + ew * kTabCols;
    // a release of TMEM: on the even CTA's barrier (remotely from the odd CTA of a pair)
    auto release = [&](int i) {
      tc_fence_before();
      if (PAIR && rank == 1) mbar_arrive_remote(mapa_shared(bar(i), 0));
      else mbar_arrive(bar(i));
    };
    int local = 0;
    Walk wk = walk0();
    for (int u = cl; u < units; u += ncl, ++local) {
      if (epi_alt && (local % kEpiGroups) != eg) continue;  // another group's tile
      int lu;
      const TcArgs& args = targs[locate(wk, u, lu)];
      const int glob = args.glob_exp ? *args.glob_exp : 0;
      // this group's 16-column chunks [ch0, ch1)
      const int nch = args.Nn / 16;
      const int hch = epi_alt ? nch : (nch + kEpiGroups - 1) / kEpiGroups;
      const int ch0 = epi_alt ? 0 : eg * hch, ch1 = ch0 + hch < nch ? ch0 + hch : nch;
      int z, mt, sp, half;
      decode(args, lu, z, mt, sp, half);
      int tf;
      uint32_t tf_phase, c0off, c1off;
      if (nbuf3) {
        tf = 0;
        tf_phase = (uint32_t)(local & 1);
        c0off = (local & 1) ? 2 * region : 0u;
        c1off = region;
      } else {
        tf = local % nbuf;
        tf_phase = (uint32_t)((local / nbuf) & 1);
        c0off = (uint32_t)tf * buf_stride;
        c1off = c0off + (uint32_t)((bcat ? 2 : 1) * args.Nn);
      }
      // everything that needs no accumulator (exponents, the factor table) is looked up
      // before waiting for it, while the tile's MMAs run
      // a shared unit (half): lane quadrants 0, 1 hold slice z, quadrants 2, 3 slice z + 1
      const int zq = (half && q >= 2) ? z + 1 : z;
      const int row = half ? mt * BM + (q & 1) * 32 + lane : mt * BM + q * 32 + lane;
      // mode 1: slice and AO index of this row, the exponent of its X row in the G
      // contraction and the row of X^T exponents, looked up once per tile
      int rP = 0, rmu = 0;
      bool valid = row < args.M && z < args.z_count;
      if (args.sym || args.a_z_unit) {  // the unit is one slice zq
        rP = zq;
        rmu = row;
        valid = row < args.Nrow && zq < args.z_count;
      } else if (args.mode == 1) {
        rP = row / args.Nmu;
        rmu = row % args.Nmu;
        valid = valid && rmu < args.Nrow;
      }
      const int erow_i = (args.mode == 1 || args.sym) ? rP * args.Nrow + rmu : row;
      const uint32_t lane_off = (uint32_t)(q * 32) << 16;
      const uint32_t t0 = tmem_base + c0off + lane_off;
      const uint32_t t1 = tmem_base + c1off + lane_off;
      const int erow = (NUM != kSplit3 && valid)
                           ? args.eA[z * args.eA_zstride + sp * args.eA_sstride + erow_i]
                           : 0;
      // every output is the accumulator times powers of two: a row factor 2^erow (and for X
      // 2^-eX3 of its G split) and a column factor, 2^(ecol - eXt) for X^T and 2^ecol for X
      // (mode 1), 2^(ecol + glob) (mode 2); the column factors of this warp's chunks are
      // tabulated once per tile
      const bool zvalid = zq < args.z_count;
      const int* ecol =
          (NUM != kSplit3) ? args.eB + z * args.eB_zstride + sp * args.eB_sstride : nullptr;
      __syncwarp();  // every lane is done with the previous tile's table
      if (zvalid) {
        const int* exz = args.mode == 1 ? args.eXt + (size_t)zq * args.Ap : nullptr;
        for (int k = lane; k < (ch1 - ch0) * 16; k += 32) {
          const int c = ch0 * 16 + k;
          const int ec = NUM != kSplit3 ? ecol[c] : 0;
          ctab[k] = args.mode == 1 ? make_float2(pow2f(ec - exz[c]), pow2f(ec))
                                   : make_float2(pow2f(ec + glob), 0.f);
        }
      }
      __syncwarp();
      const float rT = pow2f(erow);
      float rX = 0.f;
      if (args.mode == 1 && valid)
        rX = rT * pow2f(-args.eX3[(size_t)args.spOf[rP] * args.Nrow + rmu]);
      // the diagonal entry of this row (mode 2 with diag): its column, -1 for none
      int dq = -1;
      long long drow = 0;
      if (args.mode == 2 && args.diag && valid) {
        const int qd = row % args.Nn;
        if (qd < args.diag_A) {
          dq = qd;
          drow = (long long)(row / args.Nn) * args.diag_A + qd;
        }
      }

      bool ok = mbar_wait(bar(kTfull + tf), tf_phase, status, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();

      // one 16-column chunk: raw accumulator values -> outputs
      auto emit = [&](int c0, const float (&a)[16]) {
        if (!valid) return;
        const float2* tb = ctab + (c0 - ch0 * 16);
        if (args.mode == 1) {
          const size_t to = ((size_t)rP * args.Ap + c0) * args.Np + rmu;
          __align__(16) __half2 hi[8], lo[8];
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const float2 t0 = tb[j], t1 = tb[j + 1];
            __half2 h, f;
            // X^T for b = C^T X (exponent of its row (P, q))
            intfrac_split2(a[j] * rT * t0.x, a[j + 1] * rT * t1.x, h, f);
            args.xth[to + (size_t)j * args.Np] = __low2half(h);
            args.xth[to + (size_t)(j + 1) * args.Np] = __high2half(h);
            args.xtf[to + (size_t)j * args.Np] = __low2half(f);
            args.xtf[to + (size_t)(j + 1) * args.Np] = __high2half(f);
            // X for the G contraction (exponent of its row (split, mu))
            intfrac_split2(a[j] * rX * t0.y, a[j + 1] * rX * t1.y, hi[j / 2], lo[j / 2]);
          }
          // X interleaved by 8 along c, [P][c/8][mu][8]: the lanes (consecutive mu) of one
          // store write 512 contiguous bytes
          const size_t o0 = (((size_t)rP * (args.Ap / 8) + c0 / 8) * args.Np + rmu) * 8;
          const size_t o1 = o0 + (size_t)args.Np * 8;
          *(uint4*)(args.xhi + o0) = ((uint4*)hi)[0];
          *(uint4*)(args.xhi + o1) = ((uint4*)hi)[1];
          *(uint4*)(args.xlo + o0) = ((uint4*)lo)[0];
          *(uint4*)(args.xlo + o1) = ((uint4*)lo)[1];
        } else {
          float v[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = a[j] * rT * tb[j].x;
          float* o = args.out + (long long)(z * args.splits + sp) * args.out_zstride +
                     (long long)row * args.out_ld + c0;
#pragma unroll
          for (int j = 0; j < 16; j += 4) *(float4*)(o + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
          if (dq >= c0 && dq < c0 + 16) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if (c0 + j == dq) args.diag[drow] = v[j];
          }
        }
      };
      // bcat (Nn <= 64, so always drained through registers below): the value is
      // h h + ((h f + f h) + f f), columns c of the left halves and Nn + c of the right halves
      // of the two accumulators
      const uint32_t nnc = (uint32_t)args.Nn;
      auto load = [&](int c0, float (&a)[16]) {
        uint32_t r[16];
        tmem_ld16(t0 + (uint32_t)c0, r);
#pragma unroll
        for (int j = 0; j < 16; ++j) a[j] = __uint_as_float(r[j]);
        if (NUM != kSplit3) {
          tmem_ld16(t1 + (uint32_t)c0, r);
#pragma unroll
          for (int j = 0; j < 16; ++j) a[j] += __uint_as_float(r[j]);
        }
      };

      // chunks held (bcat: Nn <= 64, four chunks at most)
      constexpr int kKeep = bcat ? 4 : (kMaxRegCols / 16 + kEpiGroups - 1) / kEpiGroups;
      if (bcat || args.Nn <= kMaxRegCols) {
        // drain the accumulators into registers, hand TMEM back, then write.  nbuf 3: the
        // cross products (region Y) first, all in flight together, then Y is released and the
        // integer products (X or Z) are added chunk by chunk; otherwise both accumulators
        // chunk by chunk
        float keep[kKeep * 16];
        if (nbuf3) {
#pragma unroll
          for (int k = 0; k < kKeep; ++k)
            if (ch0 + k < ch1) tmem_ld16_nowait(t1 + (uint32_t)((ch0 + k) * 16), keep + k * 16);
          tmem_wait_ld();
          release(kTempty + 0);
        }
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
          if (ch0 + k < ch1) {
            const uint32_t c = (uint32_t)((ch0 + k) * 16);
            if (nbuf3) {
              float tmp[16];
              tmem_ld16_nowait(t0 + c, tmp);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 16; ++j) keep[k * 16 + j] = tmp[j] + keep[k * 16 + j];
            } else if (NUM == kSplit3) {
              tmem_ld16_nowait(t0 + c, keep + k * 16);
            } else {
              // the cross products, then the exact h h added last: t0 + t1, or with the
              // planes of B concatenated h h + ((h f + f h) + f f)
              float tmp[16];
              const bool cat = bcat;
              tmem_ld16_nowait((cat ? t0 + nnc : t1) + c, keep + k * 16);
              if (cat) {
                tmem_ld16_nowait(t1 + c, tmp);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) keep[k * 16 + j] += tmp[j];
                tmem_ld16_nowait(t1 + nnc + c, tmp);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) keep[k * 16 + j] += tmp[j];
              }
              tmem_ld16_nowait(t0 + c, tmp);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 16; ++j) keep[k * 16 + j] = tmp[j] + keep[k * 16 + j];
            }
          }
        }
        tmem_wait_ld();
        release(nbuf3 ? kTrel + (local & 1) : kTempty + tf);
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
          if (ch0 + k < ch1) {
            float a[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) a[j] = keep[k * 16 + j];
            emit((ch0 + k) * 16, a);
          }
        }
      } else {
        for (int c = ch0; c < ch1; ++c) {
          float a[16];
          load(c * 16, a);
          emit(c * 16, a);
        }
        release(kTempty + tf);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();  // no CTA frees its TMEM while the pair's MMAs may write it
  if (warp == 2) {
    tc_fence_after();
    tmem_dealloc<PAIR>(tmem_base, a0.tmem_cols);
  }
}

template <int BK, int NUM, int PAIR>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm(const __grid_constant__ TcMaps maps, const __grid_constant__ TcArgs args) {
  tc_body<BK, NUM, PAIR>(&args, &maps, nullptr, 1);
}

// Grouped launch: the work units of every problem of a batch in one grid.
template <int BK, int NUM>
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm_group(const TcArgs* targs, const TcMaps* tmaps, const int* ustart, int ninst) {
  tc_body<BK, NUM, 0>(targs, tmaps, ustart, ninst);
}

// ------------------------------------------------------------------ host: tile tuning
// Launch variant per contraction kind and shape, chosen by donof_autotune from timed builds;
// optional persistence in the file named by the DONOF_TUNE_CACHE environment variable (lines
// "kind N Ap np code").  A code is bk + 1000 pair + 2000 full: the K-tile width (BK, 32 or
// 64 elements), whether a CTA pair computes each 256-row tile with cta_group::2 MMAs, and
// (half transform) whether the grid takes every SM pair rather than a whole number of
// slices' row tiles at once.
struct TuneKey {
  int kind, N, Ap, np;
  bool operator<(const TuneKey& o) const {
    return std::tie(kind, N, Ap, np) < std::tie(o.kind, o.N, o.Ap, o.np);
  }
};
struct TuneCode {
  int bk, pair, full;
};
TuneCode decode_tune(int code) { return TuneCode{code % 1000, (code / 1000) & 1, code >= 2000}; }
bool valid_tune(int code) {
  const TuneCode t = decode_tune(code);
  return (t.bk == 32 || t.bk == 64) && code >= 0 && code < 4000 && !(t.pair && t.bk != 64) &&
         !(t.full && !t.pair);
}
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tune;
bool g_tune_loaded = false;

void tune_load_locked() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = getenv("DONOF_TUNE_CACHE");
  if (!path) return;
  FILE* f = fopen(path, "r");
  if (!f) return;
  TuneKey k;
  int bk;
  while (fscanf(f, "%d %d %d %d %d", &k.kind, &k.N, &k.Ap, &k.np, &bk) == 5)
    if (valid_tune(bk)) g_tune[k] = bk;
  fclose(f);
}

void tune_save_locked() {
  const char* path = getenv("DONOF_TUNE_CACHE");
  if (!path) return;
  FILE* f = fopen(path, "w");
  if (!f) return;
  for (const auto& kv : g_tune)
    fprintf(f, "%d %d %d %d %d\n", kv.first.kind, kv.first.N, kv.first.Ap, kv.first.np, kv.second);
  fclose(f);
}

// kinds: 1 = half transform, 2 = b, 3 = G.  Defaults (the fastest measured at the large
// workload): single CTAs, BK 64 for the half transform (a whole number of slices at once)
// and b, BK 32 for G.
TuneCode tuned_variant(int kind, int N, int Ap, int np) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  tune_load_locked();
  auto it = g_tune.find(TuneKey{kind, N, Ap, np});
  if (it != g_tune.end()) return decode_tune(it->second);
  return decode_tune(kind == 3 ? 32 : 64);
}

// ------------------------------------------------------------------ host: tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = (EncodeTiledFn)p;
  }
  return fn;
}

// 3-D fp16 map: x (contiguous, extent dx), y (extent dy, pitch sy bytes), z (extent dz,
// pitch sz bytes); box {bx, by, 1}.  Reads past an extent return zeros, so the x extent
// of every map is the true contraction length (row padding is never read).
bool make_map(CUtensorMap* m, const void* base, uint64_t dx, uint64_t dy, uint64_t dz, uint64_t sy,
              uint64_t sz, uint32_t bx, uint32_t by) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {dx, dy, dz};
  cuuint64_t strides[2] = {sy, sz};
  cuuint32_t box[3] = {bx, by, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUtensorMapSwizzle sw = (bx * 2 == 128) ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides,
                   box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// 4-D fp16 map of an operand interleaved by 8 along K: [nz][K/8][rows][8] (K and rows
// multiples of 8), viewed with 8-row groups as its innermost 64-element (128-byte) rows so
// that TMA moves whole 128-byte lines: dims {64, rows/8, K/8, nz}, box {64, box_rows/8,
// bk/8, 1}, no swizzle; in shared memory the same [K/8][rows][8] order (core matrices of 8
// rows x 16 bytes).
bool make_map_il8(CUtensorMap* m, const void* base, uint64_t K, uint64_t rows, uint64_t nz,
                  uint32_t bk, uint32_t box_rows) {
  EncodeTiledFn enc = get_encode();
  if (!enc || K % 8 != 0 || rows % 8 != 0) return false;
  cuuint64_t dims[4] = {64, rows / 8, K / 8, nz};
  cuuint64_t strides[3] = {128, rows * 16, (K / 8) * rows * 16};
  cuuint32_t box[4] = {64, box_rows / 8, bk / 8, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(base), dims, strides,
                   box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

int num_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// TMEM use of a launch whose widest tile has nn columns (per_set: the columns of one set of
// accumulators).  Narrow tiles (nn <= 80, all of a tile's columns fit one epilogue warp's
// registers): as many sets as fit, up to kMaxSets (a power of two), the two epilogue groups on
// alternate tiles, so that the epilogue's per-tile latency overlaps and the MMAs run several
// tiles ahead.  Wider: two sets if they fit, else (kIntFrac, up to kMaxRegCols columns) three
// regions in rotation, else one set; the groups split every tile's columns.  Returns false
// when a set does not fit.
bool tmem_plan(int nn, int per_set, bool intfrac, int& nbuf, int& stride, int& epi_alt) {
  epi_alt = 0;
  if (nn <= 80 && 2 * per_set <= 512) {
    nbuf = 2;
    while (2 * nbuf <= kMaxSets && 2 * nbuf * per_set <= 512) nbuf *= 2;
    stride = 512 / nbuf;
    epi_alt = 1;
  } else if (2 * per_set <= 512) {
    nbuf = 2;
    stride = 256;
    if (per_set > 256) return false;
  } else if (intfrac && 3 * nn <= 512 && nn <= kMaxRegCols) {
    nbuf = 3;
    stride = 0;
  } else {
    nbuf = 1;
    stride = 0;
  }
  return per_set <= 512;
}

template <int BK, int NUM, int PAIR>
cudaError_t launch_tc(const TcMaps& m, TcArgs a, cudaStream_t s) {
  if constexpr (NUM == kIntFrac && !PAIR) {
    if (2 * a.Nn <= 128) return launch_tc<BK, kIntFracCat, 0>(m, a, s);
  }
  const size_t a_bytes = (size_t)BM * BK * 2, b_bytes = (size_t)(PAIR ? a.Nn / 2 : a.Nn) * BK * 2;
  const size_t stage_bytes = 2 * a_bytes + 2 * b_bytes;
  // the 227 KB opt-in limit, less alignment, barriers and the epilogue's factor tables
  const size_t budget = 232448 - 1024 - 512 - kTabBytes;
  int stages = (int)(budget / stage_bytes);
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages < 2) stages = 2;
  a.stages = stages;
  // TMEM: one or two accumulators per set (kIntFrac keeps h*h apart; of 2 Nn columns each
  // with the planes of B concatenated), sets as tmem_plan says
  const int per_set = (NUM != kSplit3 ? 2 : 1) * (NUM == kIntFracCat ? 2 : 1) * a.Nn;
  a.tmem_cols = 512;
  if (!tmem_plan(a.Nn, per_set, NUM != kSplit3, a.nbuf, a.buf_stride, a.epi_alt))
    return cudaErrorInvalidValue;
  a.region = a.Nn;
  a.nb_stage = PAIR ? a.Nn / 2 : a.Nn;
  size_t smem = 1024 + (size_t)stages * stage_bytes + (2 * stages + kBarTail) * 8 + kTabBytes;
  if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA per SM: the TMEM allocation never waits
  cudaError_t e = cudaFuncSetAttribute(k_tc_gemm<BK, NUM, PAIR>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int units = tc_units(a, PAIR);
  int work = a.grid > 0 ? a.grid : (PAIR ? num_sms() / 2 : num_sms());  // CTAs or CTA pairs
  if (work > units) work = units;
  if (work < 1) work = 1;
  if (PAIR) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * work);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_tc_gemm<BK, NUM, PAIR>, m, a);
    count_launch(1);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  // chained while it leaves SMs free (500 / 2000 / 80: 989 us a build with no contraction chained,
  // 960 with the small ones, 991 with all)
  launch_chained_to(num_sms() - 1, k_tc_gemm<BK, NUM, PAIR>, work, kThreads, smem, s, m, a);
  count_launch(1);
  return cudaGetLastError();
}

template <int NUM>
cudaError_t launch_tc_bk(int bk, const TcMaps& m, TcArgs a, cudaStream_t s) {
  return bk == 32 ? launch_tc<32, NUM, 0>(m, a, s) : launch_tc<64, NUM, 0>(m, a, s);
}

// The launch of a tuned variant (the B maps must have boxes of Nn / 2 rows for a pair).
template <int NUM>
cudaError_t launch_tc_variant(const TuneCode& t, const TcMaps& m, TcArgs a, cudaStream_t s) {
  if (t.pair) return launch_tc<64, NUM, 1>(m, a, s);
  return launch_tc_bk<NUM>(t.bk, m, a, s);
}

// ------------------------------------------------------------------ split / scale kernels
__device__ inline void atomic_max_nonneg(unsigned long long* a, double v) {
  atomicMax(a, (unsigned long long)__double_as_longlong(v));
}


__device__ inline double load_B_elem(const double* __restrict__ B, int layout, long long P,
                                     long long r, int mu, int nu, int N, long long npk) {
  if (layout == DONOF_B_DENSE) return B[r * N + nu];
  const int a = mu > nu ? mu : nu, b = mu > nu ? nu : mu;
  return B[P * npk + (long long)a * (a + 1) / 2 + b];
}

// The passes over B below work in fp32 on elements scaled by a power of two per slice (this
// GPU's FP64 pipe gives 1.6 operations per clock and SM, its double-to-float conversion 100): a
// CTA per slice finds the largest (scaled) exponent, then sums elements brought to at most 2.
// The double (hi, lo), within a normal float's range, cut to a float's 24 bits.  From the bits: the
// conversion instruction holds the FP64 unit of its scheduler for 64 clocks, as any FP64 one does
// (k_p_scale of 1103 packed slices of 301: 336 us with it, 281 so).
__device__ __forceinline__ float float_of_top(uint32_t hi, uint32_t lo) {
  const uint32_t t = __funnelshift_l(lo, hi, 3) + ((127u - 1023u) << 23);
  return __uint_as_float((t & 0x7fffffffu) | (hi & 0x80000000u));
}
// two_floats: v 2^k (biased exponent e of v, e + k within a float's range) as xh + xl, xh the
// upper 24 bits rounded half up, xl the lower 29 bits (rounded to 24), from the bits alone.
__device__ __forceinline__ void two_floats(double v, int k, float& xh, float& xl) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu) + k;
  const bool tiny = (hi & 0x7ff00000u) == 0 || e < 1023 - 120;  // taken as zero
  uint32_t h2 = hi + ((uint32_t)k << 20), l2 = lo;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(l2), "+r"(h2) : "r"(0x10000000u));
  xh = tiny ? 0.f : float_of_top(h2, l2);
  // the lower bits as a signed number of 2^-3: weight 2^(e - 1023 - 52 - 3)
  const float w = __int_as_float(max(e - 1078 + 127, 0) << 23);
  const float r = (float)(int)(lo << 3) * w;
  xl = tiny ? 0.f : ((int)hi < 0 ? -r : r);
}
// |v| 2^k rounded (half up) to a float, for sums that a few roundings do not matter to.
__device__ __forceinline__ float one_float(double v, int k) {
  const uint32_t hi = (uint32_t)__double2hiint(v);
  const int e = (int)((hi >> 20) & 0x7ffu) + k;
  const bool tiny = (hi & 0x7ff00000u) == 0 || e < 1023 - 120;
  uint32_t h2 = (hi & 0xfffffu) | ((uint32_t)e << 20), l2 = (uint32_t)__double2loint(v);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(l2), "+r"(h2) : "r"(0x10000000u));
  return tiny ? 0.f : float_of_top(h2, l2);
}
// s + c += p, the rounding of s kept in c (Knuth's two-sum)
__device__ __forceinline__ void add_comp(float& s, float& c, float p) {
  const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
  c += __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
}
// What elements too small for their square to be a float can add to a row's sum, per element.
constexpr double kStatsLost = 0x1p-118;

constexpr int kFlatN = 46000;  // slices below it are walked by 32-bit offsets
constexpr int kBoundSlack = 64;
// How a slice is walked: dense rows; a packed lower triangle's stored rows; or its whole rows, the
// part above the diagonal gathered from the columns (packed slices whose sums of columns have no
// room in shared memory).
enum SliceForm { kSliceDense = 0, kSlicePacked = 1, kSliceGathered = 2 };
// Row sums of slice P (N x N, symmetric) over its elements times 2^(-s_mu - s_nu) (s null: 0) in
// units of 2^top: row(mu, squares, magnitudes), called by one thread per row.  EXACT: compensated
// sums, to about 2^-40; otherwise squares only, to sum_margin.  Whole rows: a warp per row.  Packed: a
// warp per stored row, whose elements also count for their columns (partial sums per warp in
// shared memory, added in the order of the warps).  bound: 4096 + an upper bound of the largest
// scaled biased exponent, less than kBoundSlack above it, the largest over the threads; negative: it
// is found first.  Returns top, the bound or the exponent itself (above 4096: a NaN or an infinity).
// All threads of the CTA call it; sh holds kSums N floats per warp and once more (packed), red 33
// ints.
template <SliceForm FORM, bool EXACT, class Row>
__device__ __forceinline__ int slice_row_sums(const double* __restrict__ B, int N,
                                              const int* __restrict__ s, float* sh, int* red,
                                              int bound, const Row& row) {
  constexpr bool PACKED = FORM == kSlicePacked;
  constexpr int kSums = EXACT ? 4 : 1;  // squares, their compensation, magnitudes, theirs
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int m = bound < 0 ? 0 : bound;  // biased; 0: the slice is zero
  if (bound < 0 && !s && N < kFlatN) {  // the exponents alone: the slice from end to end, eight loads in flight
    const int per = FORM != kSliceDense ? N * (N + 1) / 2 : N * N;  // (N below kFlatN)
    for (int i0 = threadIdx.x; i0 < per; i0 += 8 * blockDim.x) {
      int h[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = i0 + j * blockDim.x;
        h[j] = i < per ? __double2hiint(B[i]) : 0;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int e = (h[j] >> 20) & 0x7ff;
        if (e > 0) m = max(m, e == 2047 ? 1 << 20 : e + 4096);
      }
    }
  }
  // A row at a time, kBatch loads of a lane ahead of their use, over the ends of rows too (bound by
  // the latency of the loads otherwise: a row is a few of them per lane): at(mu, nu, v) for every
  // element in order, end(mu) after a row
  constexpr int kBatch = 4;
  auto walk = [&](auto at, auto end) {
    auto row_at = [&](int mu) {
      return B + (FORM != kSliceDense ? (long long)mu * (mu + 1) / 2 : (long long)mu * N);
    };
    int mu = w, n0 = 0;  // the batch in v: row mu, elements n0 + lane + 32 u
    double v[kBatch];
    auto load = [&](int r, int c0, double (&x)[kBatch]) {
      const int n = PACKED ? r + 1 : N;
      const double* p = row_at(r);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int nu = c0 + lane + 32 * u;
        if (FORM == kSliceGathered && nu > r)
          x[u] = r < N && nu < n ? B[(long long)nu * (nu + 1) / 2 + r] : 0.0;
        else
          x[u] = r < N && nu < n ? p[nu] : 0.0;
      }
    };
    if (mu < N) load(mu, 0, v);
    while (mu < N) {
      const int n = PACKED ? mu + 1 : N;
      int r2 = mu, c2 = n0 + 32 * kBatch;
      if (c2 >= n) {
        r2 += nw;
        c2 = 0;
      }
      double x[kBatch];
      load(r2, c2, x);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int nu = n0 + lane + 32 * u;
        if (nu < n) at(mu, nu, v[u]);
      }
      if (r2 != mu) end(mu);
      mu = r2;
      n0 = c2;
#pragma unroll
      for (int u = 0; u < kBatch; ++u) v[u] = x[u];
    }
  };
  if (bound < 0 && (s || N >= kFlatN))
    walk([&](int mu, int nu, double v) {
      const int e = (__double2hiint(v) >> 20) & 0x7ff;
      if (e > 0) m = max(m, e == 2047 ? 1 << 20 : e + 4096 - (s ? s[mu] + s[nu] : 0));
    }, [](int) {});
  m = __reduce_max_sync(0xffffffffu, m);
  __syncthreads();  // red and sh are free
  if (lane == 0) red[w] = m;
  if (PACKED)
    for (int i = threadIdx.x; i < kSums * N * nw; i += blockDim.x) sh[i] = 0.f;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < nw ? red[threadIdx.x] : 0;
    m = __reduce_max_sync(0xffffffffu, m);
    if (threadIdx.x == 0) red[32] = m;
  }
  __syncthreads();
  const int top = red[32] - 4096;  // the largest scaled biased exponent
  float* cs = sh + kSums * N * w;  // this warp's partial sums of the columns
  float ss = 0.f, sc = 0.f, l1 = 0.f, lc = 0.f;
  const int k0 = 1023 - top;
  walk([&](int mu, int nu, double v) {
    const int k = k0 - (s ? s[mu] + s[nu] : 0);
    if (EXACT) {
      float xh, xl;
      two_floats(v, k, xh, xl);
      const float q = __fmul_rn(xh, xh);
      const float qe = fmaf(2.f * xh, xl, fmaf(xh, xh, -q)), a = fabsf(xh);
      const float al = xh < 0.f ? -xl : xl;
      add_comp(ss, sc, q);
      sc += qe;
      add_comp(l1, lc, a);
      lc += al;
      if (PACKED && nu < mu) {
        float ts = cs[nu], tc = cs[N + nu], tl = cs[2 * N + nu], td = cs[3 * N + nu];
        add_comp(ts, tc, q);
        add_comp(tl, td, a);
        cs[nu] = ts;
        cs[N + nu] = tc + qe;
        cs[2 * N + nu] = tl;
        cs[3 * N + nu] = td + al;
      }
    } else {
      const float x = one_float(v, k);
      ss = fmaf(x, x, ss);
      if (PACKED && nu < mu) cs[nu] = fmaf(x, x, cs[nu]);
    }
  }, [&](int mu) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (EXACT) {
        const float c2 = __shfl_xor_sync(0xffffffffu, sc, o), d2 = __shfl_xor_sync(0xffffffffu, lc, o);
        add_comp(ss, sc, __shfl_xor_sync(0xffffffffu, ss, o));
        add_comp(l1, lc, __shfl_xor_sync(0xffffffffu, l1, o));
        sc += c2;
        lc += d2;
      } else {
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
      }
    }
    if (lane == 0) {
      if (PACKED) {  // the row's own part, behind the warps' column sums
        float* o = sh + kSums * N * nw + mu;
        o[0] = ss;
        if (EXACT) {
          o[N] = sc;
          o[2 * N] = l1;
          o[3 * N] = lc;
        }
      } else {
        row(mu, (double)ss + (double)sc, (double)l1 + (double)lc);
      }
    }
    ss = sc = l1 = lc = 0.f;
  });
  if (PACKED) {
    __syncthreads();
    for (int mu = threadIdx.x; mu < N; mu += blockDim.x) {
      float t[4] = {0.f, 0.f, 0.f, 0.f};
      for (int i = 0; i <= nw; ++i) {
        const float* c = sh + kSums * N * i + mu;
        if (EXACT) {
          add_comp(t[0], t[1], c[0]);
          add_comp(t[2], t[3], c[2 * N]);
          t[1] += c[N];
          t[3] += c[3 * N];
        } else {
          t[0] += c[0];
        }
      }
      row(mu, (double)t[0] + (double)t[1], (double)t[2] + (double)t[3]);
    }
  }
  return top;
}
// The largest of the threads' non-negative doubles, in every thread (red: 33 64-bit words).
__device__ __forceinline__ double block_max(double v, unsigned long long* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (unsigned long long)__double_as_longlong(v);
  __syncthreads();
  unsigned long long t = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = max(t, red[i]);
  return __longlong_as_double((long long)t);
}
// Warps of a slice's CTA and its shared memory.  Packed slices whose sums of columns leave a CTA
// fewer than two warps are gathered by rows (5000 functions, 152 slices: 154 ms with one warp).
constexpr int kPackedStatsMaxN = 4266;
inline SliceForm slice_form(bool packed, int N) {
  return !packed ? kSliceDense : N <= kPackedStatsMaxN ? kSlicePacked : kSliceGathered;
}
inline int slice_warps(SliceForm form, int N) {
  int nw = 8;
  while (form == kSlicePacked && nw > 1 && (size_t)(nw + 1) * 16 * N > 200 * 1024) --nw;
  return nw;
}
constexpr int kSliceSmemMax = 224 * 1024;
inline size_t slice_smem(SliceForm form, int N) {
  return form == kSlicePacked ? (size_t)(slice_warps(form, N) + 1) * 16 * N : 0;  // (k_b_stats)
}

// Per row (P, mu) of B: its squared L2 norm (rn2, fp32 rounded up, for the exponents of X in the
// G contraction), the slice's largest row L1 norm (L1max, the bound on X^T rows) and the AO
// index's largest row norm over the slices (rnmax, for the symmetric scaling); any
// non-finite element raises DONOF_ERR_NONFINITE.  Bound by its instructions (54 float additions an
// element, for two compensated sums over its row and over its column).  1103 packed slices of 301:
// 0.28 ms (with a row's loads behind the reduction of the row before: 0.39; in double, every element
// gathered twice: 1.18).
template <SliceForm FORM>
__global__ void __launch_bounds__(256) k_b_stats(const double* __restrict__ B, int Q, int N,
                                                 DevHeader* hdr, double* L1max, float* rn2,
                                                 unsigned long long* rnmax_bits) {
  extern __shared__ float sh_f[];
  __shared__ int red[33];
  __shared__ unsigned long long redl[33];
  const long long per = FORM != kSliceDense ? (long long)N * (N + 1) / 2 : (long long)N * N;
  constexpr double kUp = 1.0 + 0x1p-36;  // above the compensated sums' error
  const double lost = N * kStatsLost;
  for (int P = blockIdx.x; P < Q; P += gridDim.x) {
    double mx = 0.0;
    float* out = rn2 + (size_t)P * N;
    // the slice's scale is known to every thread only after the call: the rows are scaled by
    // the exponent that the call found, which it leaves in red
    const int top = slice_row_sums<FORM, true>(
        B + P * per, N, nullptr, sh_f, red, -1, [&](int mu, double ss, double l1) {
          const int t = red[32] - 4096;
          if (t > 4096) {
            out[mu] = __int_as_float(0x7fc00000);
            return;
          }
          const double sc = pow2d(t - 1023);
          out[mu] = __double2float_ru((ss * kUp + lost) * sc * sc);
          atomic_max_nonneg(rnmax_bits + mu, sqrt(ss) * sc);
          mx = fmax(mx, l1);
        });
    const double l1 = block_max(mx, redl);
    if (threadIdx.x == 0) {
      if (top > 4096) {
        set_status(hdr, DONOF_ERR_NONFINITE);
        L1max[P] = __longlong_as_double(0x7ff8000000000000ll);
      } else {
        L1max[P] = (l1 * kUp + lost) * pow2d(top - 1023);
      }
    }
  }
}

// Per slice: t_P, the exponent of the largest row norm of Bt^P without t_P.  Where the fp32 sums
// cannot tell on which side of a power of two the norm lies, the slice's sums are taken in
// double.  1103 packed slices of 301: 0.13 ms (with a pass for the largest element first: 0.20; with
// the loads of a row behind the row before too: 0.28; in double, with an ldexp per element: 1.35).
template <SliceForm FORM>
__global__ void __launch_bounds__(256) k_p_scale(const double* __restrict__ B, int Q, int N,
                                                 const int* __restrict__ eS, int s_in_smem,
                                                 double invT, const float* __restrict__ rn2,
                                                 int* tP) {
  constexpr bool PACKED = FORM == kSlicePacked;
  extern __shared__ float sh_f[];
  __shared__ int red[33];
  __shared__ unsigned long long redl[33];
  const long long npk = (long long)N * (N + 1) / 2;
  const long long per = FORM != kSliceDense ? npk : (long long)N * N;
  // rounding of the sums: N / 32 terms a lane, N / nw in a warp's sum of a column, the tree over
  // lanes, the warps' sums, every term rounded before
  const int nw = blockDim.x >> 5;
  int* sh_s = (int*)(sh_f + (PACKED ? (nw + 1) * N : 0));  // the scale exponents, behind the sums
  const int* sS = s_in_smem ? sh_s : eS;
  int lo = 1 << 20, hi = -(1 << 20);
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const int e = eS[i];
    if (s_in_smem) sh_s[i] = e;
    lo = min(lo, e);
    hi = max(hi, e);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = lo;
    red[16 + (threadIdx.x >> 5)] = hi;
  }
  __syncthreads();
  for (int i = 0; i < nw; ++i) {
    lo = min(lo, red[i]);
    hi = max(hi, red[16 + i]);
  }
  const double mg = (N / 32 + (PACKED ? N / nw : 0) + 32) * 0x1p-24;
  for (int P = blockIdx.x; P < Q; P += gridDim.x) {
    const double* Bp = B + P * per;
    double mx = 0.0;
    // the scale of the sums from the rows' norms: |B_mu,nu| 2^(-s_mu - s_nu) < 2^(b - s_mu - min s),
    // 4^b > the row's squared norm.  Not for norms near a float's range or scales that differ
    // by more than the sums bear
    int bound = 0, far = hi - lo > kBoundSlack - 24 ? 1 : 0;
    for (int mu = threadIdx.x; mu < N; mu += blockDim.x) {
      const int e = (__float_as_int(rn2[(size_t)P * N + mu]) >> 23) & 0x1ff;  // (with the sign)
      if (e < 27 || e > 227) far = 1;
      bound = max(bound, ((e - 125) >> 1) - sS[mu] - lo + 1022 + 4096);
    }
    if (__syncthreads_or(far)) bound = -1;
    const int top = slice_row_sums<FORM, false>(
        Bp, N, sS, sh_f, red, bound, [&](int, double ss, double) { mx = fmax(mx, ss); });
    const double ss = block_max(mx, redl);
    const double sc = pow2d(top - 1023);
    const int e0 = intfrac_exponent_inv(sqrt(ss * (1.0 - mg)) * sc, invT);
    const int e1 = intfrac_exponent_inv(sqrt(ss * (1.0 + mg)) * sc, invT);
    if (e0 == e1) {  // (the same in every thread)
      if (threadIdx.x == 0) tP[P] = top > 4096 ? 0 : e0;
      continue;
    }
    double t2 = 0.0;
    for (int mu = threadIdx.x >> 5; mu < N; mu += nw) {
      double t = 0.0;
      for (int nu = threadIdx.x & 31; nu < N; nu += 32) {
        const double v = ldexp(load_B_elem(Bp, FORM != kSliceDense ? DONOF_B_PACKED : DONOF_B_DENSE,
                                           0, mu, mu, nu, N, npk),
                               -eS[mu] - eS[nu]);
        t = fma(v, v, t);
      }
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      t2 = fmax(t2, t);
    }
    const double exact = block_max(sqrt(t2), redl);
    if (threadIdx.x == 0) tP[P] = intfrac_exponent_inv(exact, invT);
  }
}

// The same two passes for a B of few slices, whose CTAs would leave most of the chip idle: a warp per
// row (P, mu) of the whole B, in double, the part above a packed row's diagonal gathered.  L1max and
// tmax start at zero; k_t_exps then gives t_P.
__global__ void __launch_bounds__(256) k_b_stats_rows(const double* __restrict__ B, int layout,
                                                      long long Q, int N, DevHeader* hdr,
                                                      unsigned long long* L1max_bits, float* rn2,
                                                      unsigned long long* rnmax_bits) {
  const long long rows = Q * N, npk = (long long)N * (N + 1) / 2;
  const int lane = threadIdx.x % 32;
  bool bad = false;
  for (long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32; row < rows;
       row += (long long)gridDim.x * blockDim.x / 32) {
    const long long P = row / N;
    const int mu = (int)(row % N);
    double ss = 0.0, l1 = 0.0;
    for (int nu = lane; nu < N; nu += 32) {
      const double v = load_B_elem(B, layout, P, row, mu, nu, N, npk);
      ss = fma(v, v, ss);
      l1 += fabs(v);
    }
    for (int o = 16; o > 0; o >>= 1) {
      ss += __shfl_xor_sync(0xffffffffu, ss, o);
      l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    const double nr = sqrt(ss);
    if (lane == 0) {
      rn2[row] = __double2float_ru(ss);
      atomic_max_nonneg(L1max_bits + P, l1);
      atomic_max_nonneg(rnmax_bits + mu, nr);
    }
    bad = bad || !isfinite(nr);
  }
  if (lane == 0 && bad) set_status(hdr, DONOF_ERR_NONFINITE);
}
__global__ void __launch_bounds__(256) k_p_scale_rows(const double* __restrict__ B, int layout,
                                                      long long Q, int N,
                                                      const int* __restrict__ eS,
                                                      unsigned long long* tmax_bits) {
  const long long rows = Q * N, npk = (long long)N * (N + 1) / 2;
  const int lane = threadIdx.x % 32;
  for (long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32; row < rows;
       row += (long long)gridDim.x * blockDim.x / 32) {
    const long long P = row / N;
    const int mu = (int)(row % N);
    double ss = 0.0;
    for (int nu = lane; nu < N; nu += 32) {
      const double v = ldexp(load_B_elem(B, layout, P, row, mu, nu, N, npk), -eS[mu] - eS[nu]);
      ss = fma(v, v, ss);
    }
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) atomic_max_nonneg(tmax_bits + P, sqrt(ss));
  }
}
__global__ void k_t_exps(const double* __restrict__ tmax, int Q, double invT, int* tP) {
  for (int P = blockIdx.x * blockDim.x + threadIdx.x; P < Q; P += gridDim.x * blockDim.x)
    tP[P] = intfrac_exponent_inv(tmax[P], invT);
}
// Whether the passes go by rows: a slice's CTA takes about 1.1 ns an element, the chip by rows 15 ps.
// Both measured (donof_prepare_B, ms, slices / rows): 1200 dense, 16 slices 2.52 / 0.47, 64 slices
// 2.61 / 1.63; 1200 packed, 16 1.27 / 0.47, 64 1.48 / 1.64; 3000 packed, 64 19.1 / 8.8, 152 20 / 21;
// 200 dense, 16 0.140 / 0.085, 64 0.149 / 0.143; 5000 gathered, 64 50 / 24, 152 50 / 56.
inline bool slices_by_rows(SliceForm form, int Q, int N) {
  const int few = form == kSliceDense ? 80 : form == kSliceGathered ? 130 : 384 / slice_warps(form, N);
  return N > 1 && Q < few;
}

// Symmetric scaling of B: B^P_{mu nu} = 2^(t_P + s_mu + s_nu) Bt^P_{mu nu} keeps Bt^P
// symmetric, so one stored triangle serves both operand orders of the half transform.
// s equilibrates the AO indices: with a_mu = max_P ||B^P_{mu .}||_2, a rank-one-like
// |B_{mu nu}| ~ d_mu d_nu has a_mu = d_mu ||d||, ||d||^4 = sum_mu a_mu^2, so
// 2^s_mu = d_mu rounded to a power of two.  One CTA.
__global__ void __launch_bounds__(1024) k_sym_scale(const double* __restrict__ rnmax, int N,
                                                    int* eS) {
  __shared__ double red[32];
  double ss = 0.0;
  for (int mu = threadIdx.x; mu < N; mu += blockDim.x) ss += rnmax[mu] * rnmax[mu];
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += red[w];
    red[0] = t;
  }
  __syncthreads();
  const double norm_d = sqrt(sqrt(red[0]));
  for (int mu = threadIdx.x; mu < N; mu += blockDim.x) {
    const double dmu = rnmax[mu] / norm_d;
    eS[mu] = (dmu > 0.0 && norm_d > 0.0) ? (int)rint(log2(dmu)) : 0;
  }
}

// eA[P][mu] = t_P + s_mu: the exponent of output row (P, mu) of the half transform.
__global__ void k_sym_exps(const int* __restrict__ tP, const int* __restrict__ eS,
                           long long Q, int N, int* eA) {
  const long long tot = Q * N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)gridDim.x * blockDim.x)
    eA[i] = tP[i / N] + eS[i % N];
}

// The integer + fraction split of y = v 2^k, |y| < 4096, as the double split forms it (h =
// fp16(rint(y)), f = fp16(fl32(y - h))), without an FP64 operation: y = yh + yl (two_floats); rint(y)
// is rint(yh) except where yh lies half-way between two integers and yl decides; y - h =
// (yh - h) + yl with an exact difference.
__device__ __forceinline__ void intfrac_split_scaled(double v, int k, __half& h, __half& f) {
  float yh, yl;
  two_floats(v, k, yh, yl);
  float t = rintf(yh);
  const float d = yh - t;
  t += (d == 0.5f && yl > 0.f) ? 1.f : ((d == -0.5f && yl < 0.f) ? -1.f : 0.f);
  h = __float2half_rn(t);
  f = __float2half_rn((yh - __half2float(h)) + yl);
}

// Bt^P 2^-t_P -> integer + fraction planes in the lower-triangle tile storage (SymTiles).  A CTA per
// 8 stored rows of a slice (rows of the last tile padded to Rlast), their pieces of 8 consecutive
// stored elements dealt over its threads; the columns reach to the end of the rows' tile.  Bound by
// its integer instructions, so that pieces past the matrix are only zeroed and no lane is left
// over at the ends of rows (1103 packed slices of 301, a warp per row and zeros converted like
// all others: 299 us; this: 214).  Off: the offsets within a slice, 64 bits from kFlatN on.
template <class Off>
__global__ void __launch_bounds__(256) k_split_B_sym(const double* __restrict__ B, int layout,
                                                     int Q, int N, SymTiles st,
                                                     const int* __restrict__ eS,
                                                     const int* __restrict__ tP, __half* H,
                                                     __half* F) {
  const bool dense = layout == DONOF_B_DENSE;
  const size_t per = dense ? (size_t)N * N : (size_t)N * (N + 1) / 2;
  const int rows = 128 * (st.T - 1) + st.Rlast;  // stored rows (= columns) per slice
  const int rb = rows / 8, tot = Q * rb;
  for (int u = blockIdx.x; u < tot; u += gridDim.x) {  // 8 rows of a slice per CTA
    const int P = u / rb, mu0 = (u - P * rb) * 8;
    const int ti = mu0 >> 7, Ri = sym_R(st, ti), tp = tP[P];
    const double* Bp = B + (size_t)P * per;
    const size_t base = (size_t)P * st.perP;
    const int n8 = 16 * ti + (ti == st.T - 1 ? st.Rlast : 128) / 8;  // pieces of a row
    const uint32_t inv = 0xffffffffu / (uint32_t)n8 + 1;  // 2^32 / n8 upwards (8 n8^2 < 2^32)
    for (int it = threadIdx.x; it < 8 * n8; it += blockDim.x) {
      const int r8 = (int)__umulhi((uint32_t)it, inv), c8 = it - r8 * n8, mu = mu0 + r8;
      const int r = mu & 127, nu0 = 8 * c8;
      __align__(16) __half hv[8], fv[8];
      if (mu < N && nu0 < N) {
        const int k0 = -tp - eS[mu];
        double v[8];
        int k[8];
        // element nu0 + j: in mu's row up to the diagonal, above it in row nu0 + j
        const double* Br = dense ? Bp + (size_t)mu * N : Bp;
        const Off row = dense ? (Off)nu0 : (Off)mu * (mu + 1) / 2 + nu0;
        const int diag = dense ? 8 : mu - nu0;  // the last j of the row
        Off col = dense ? 0 : (Off)nu0 * (nu0 + 1) / 2 + mu;
        if (nu0 + 8 <= N) {
          *(int4*)k = *(const int4*)(eS + nu0);
          *(int4*)(k + 4) = *(const int4*)(eS + nu0 + 4);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            v[j] = __ldg(Br + (j <= diag ? row + j : col));
            col += nu0 + j + 1;
            k[j] = k0 - k[j];
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool in = nu0 + j < N;
            v[j] = in ? __ldg(Br + (j <= diag ? row + j : col)) : 0.0;
            col += nu0 + j + 1;
            k[j] = in ? k0 - eS[nu0 + j] : 0;
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) intfrac_split_scaled(v[j], k[j], hv[j], fv[j]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) hv[j] = fv[j] = __float2half_rn(0.f);
      }
      const int tj = c8 >> 4, c = (c8 >> 3) & 1, j8 = c8 & 7;
      const size_t o = base + sym_tile_off(st, ti, tj) + ((size_t)c * Ri + r) * 64 +
                       (size_t)((j8 ^ (r & 7)) * 8);
      *(uint4*)(H + o) = *(const uint4*)hv;
      *(uint4*)(F + o) = *(const uint4*)fv;
    }
  }
}

// Bt^P 2^-t_P -> integer + fraction planes in the dense storage, [P][mu][ld] (columns
// nu >= N zero).  A lane per 8 consecutive stored elements of a row; the rows of a slice share
// a warp when they are short.
__global__ void __launch_bounds__(256) k_split_B_dense(const double* __restrict__ B, int layout,
                                                       long long Q, int N, int ld,
                                                       const int* __restrict__ eS,
                                                       const int* __restrict__ tP, __half* H,
                                                       __half* F) {
  const long long npk = (long long)N * (N + 1) / 2;
  const int n8 = ld / 8, per = N * n8;  // 8-element pieces of a slice (N <= 256)
  const int ctas = (per + 255) / 256;
  for (long long u = blockIdx.x; u < Q * ctas; u += gridDim.x) {
    const int P = (int)(u / ctas), i = (int)(u - (long long)P * ctas) * 256 + threadIdx.x;
    if (i >= per) continue;
    const int mu = i / n8, j8 = i - mu * n8;
    const int k0 = -tP[P] - eS[mu];
    const double* Bp = B + (layout == DONOF_B_DENSE ? (size_t)P * N * N : (size_t)P * npk);
    __align__(16) __half hv[8], fv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int nu = j8 * 8 + j;
      const double v = nu < N ? load_B_elem(Bp, layout, 0, mu, mu, nu, N, npk) : 0.0;
      intfrac_split_scaled(v, nu < N ? k0 - eS[nu] : 0, hv[j], fv[j]);
    }
    const size_t o = ((size_t)P * N + mu) * ld + (size_t)j8 * 8;
    *(uint4*)(H + o) = *(const uint4*)hv;
    *(uint4*)(F + o) = *(const uint4*)fv;
  }
}

// One transposed integer + fraction split: S (N rows, leading dimension ld), output rows
// c < nrows_out of the split of S^T (zero for c >= ncols), optionally of diag(2^eS) S.
//
// Residual planes (planes != 0) serve a product U V^T that must come out to near double
// precision from the integer + fraction kernel.  With y = h + f + r per element (r, the
// residual of the split, rounded to fp16) the product is taken as four K blocks, block k
// with operands (PH[k], PF[k]) on each side; the kernel forms PH_U PH_V exactly in one
// accumulator and PH_U PF_V + PF_U PH_V + PF_U PF_V in the other, and each block is kept
// as its own output, so that no block sums an exact part with a rounded one:
//   block 0: U (h, 0), V (h, 0)  ->  h_U h_V                 (exact)
//   block 1: U (0, h), V (r, f)  ->  h_U (r_V + f_V)
//   block 2: U (0, f), V (h, f)  ->  f_U (h_V + f_V)
//   block 3: U (0, r), V (h, f)  ->  r_U (h_V + f_V)
// together (h_U + f_U + r_U)(h_V + f_V + r_V) less f_U r_V and r_U r_V, the two smallest
// terms.  planes = 1 writes the U side, planes = 2 the V side ([4][nrows_out][Np] each).
struct SplitJob {
  const double* S;
  long long ld;
  int N, ncols, nrows_out;
  const int* eS;  // may be null
  int* e;         // per-row exponents of the output
  double* norm;   // may be null: receives the column norms
  __half* H;      // may be null (planes only)
  __half* F;
  int planes;     // 0, 1 (U side) or 2 (V side)
  __half* PH;
  __half* PF;
};
struct SplitJobs {
  SplitJob j[3];  // blockIdx.y (norms) or blockIdx.z (splits) selects the job
  int count;
};

// Column norms of job.S -> exponents of the integer + fraction split of S^T: e[c] for
// c < nrows_out.  A CTA of (at least) columns x G threads per kNormCols columns (32 where the split
// follows), G = norm_groups(N) (row groups enough for the columns' length): thread (c, g < G) sums rows g, g + G, ...
// (coalesced across c, four loads in flight, in order of mu), the G partial sums of a column
// are then added in order.
__host__ __device__ inline int norm_groups(int N) { return N > 256 ? 32 : 8; }
__device__ __forceinline__ double colnorm_partial(const SplitJob& jb, int c, int g, int G) {
  double ss = 0.0;
  if (c >= jb.ncols) return ss;
  const double* __restrict__ S = jb.S;
  const int* __restrict__ eS = jb.eS;
  const long long ld = jb.ld;
  const int N = jb.N;
  int mu = g;
  for (; mu + 3 * G < N; mu += 4 * G) {
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = S[(size_t)(mu + G * u) * ld + c];
      if (eS) v[u] *= pow2d(eS[mu + G * u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) ss = fma(v[u], v[u], ss);
  }
  for (; mu < N; mu += G) {
    double v = S[(size_t)mu * ld + c];
    if (eS) v *= pow2d(eS[mu]);
    ss = fma(v, v, ss);
  }
  return ss;
}
// the column's exponent (and norm) from the partial sums red[0..G)[tx]
__device__ __forceinline__ int colnorm_finish(const SplitJob& jb, int c, const double (*red)[33],
                                              int tx, int G, double invT, DevHeader* hdr) {
  double t = 0.0;
  for (int g = 0; g < G; ++g) t += red[g][tx];
  const double nr = sqrt(t);
  if (!isfinite(nr)) set_status(hdr, DONOF_ERR_NONFINITE);
  const int e = intfrac_exponent_inv(nr, invT);
  jb.e[c] = e;
  if (jb.norm) jb.norm[c] = nr;
  return e;
}
// kNormCols columns a CTA: the FP64 work of a CTA is what bounds it (64 clocks a warp instruction
// and scheduler), so that many narrow CTAs beat few of whole lines (500 columns of 500: 14.5 us by
// 32 columns, 11.2 by 8).
constexpr int kNormCols = 8;
__device__ __forceinline__ void k_colnorms_body(const Blk& B_, SplitJobs jobs, double invT, DevHeader* hdr) {
  const SplitJob& jb = jobs.j[B_.y];
  if ((int)B_.x * kNormCols >= jb.nrows_out) return;  // uniform over the CTA
  __shared__ double red[32][33];
  const int tx = threadIdx.x % kNormCols, ty = threadIdx.x / kNormCols;
  const int G = norm_groups(jb.N);
  const int c = B_.x * kNormCols + tx;
  if (ty < G) red[ty][tx] = colnorm_partial(jb, c, ty, G);
  __syncthreads();
  if (ty == 0 && c < jb.nrows_out) colnorm_finish(jb, c, red, tx, G, invT, hdr);
}
// The row of CTAs behind the jobs', if any, clears `zero`.
__global__ void __launch_bounds__(32 * kNormCols) k_colnorms(SplitJobs jobs, double invT, DevHeader* hdr,
                                                   const ZeroJob zero) {
  const Blk b = native_blk();
  if (b.y == jobs.count) {
    zero_ranges(zero, b.x, b.gx);
    return;
  }
  k_colnorms_body(b, jobs, invT, hdr);
}

// The split itself, as rows c < nrows_out of Np halves (zero for c >= ncols or mu >= N):
// element (c, mu) is 2^e[c] (h + f) of S[mu][c] (times 2^eS[mu] when eS is given), and the
// residual planes when asked for.  32 x 32 tiles through shared memory, so that both the
// reads and the writes are coalesced.
__device__ __forceinline__ void k_split_T_body(const Blk& B_, SplitJobs jobs, int Np) {
  const SplitJob& jb = jobs.j[B_.z];
  const int mu0 = B_.x * 32, c0 = B_.y * 32;
  if (c0 >= jb.nrows_out) return;  // uniform over the CTA
  __shared__ double tile[32][33];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int mu = mu0 + ty + 8 * j, c = c0 + tx;
    tile[ty + 8 * j][tx] = (mu < jb.N && c < jb.ncols) ? jb.S[(size_t)mu * jb.ld + c] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = c0 + ty + 8 * j, mu = mu0 + tx;
    if (c < jb.nrows_out && mu < Np) {
      const size_t o = (size_t)c * Np + mu;
      const int k = ((jb.eS && mu < jb.N) ? jb.eS[mu] : 0) - jb.e[c];
      __half h, f, r;
      intfrac_split_v(tile[tx][ty + 8 * j], k, h, f, r);
      if (jb.H) {
        jb.H[o] = h;
        jb.F[o] = f;
      }
      if (jb.planes) {
        const size_t ps = (size_t)jb.nrows_out * Np;
        // the planes' zero blocks (U side: h's blocks 1-3, f's block 0; V side: f's block 0)
        // are cleared once when B is prepared and never written
        if (jb.planes == 1) {
          jb.PH[o] = h;
          jb.PF[ps + o] = h; jb.PF[2 * ps + o] = f; jb.PF[3 * ps + o] = r;
        } else {
          jb.PH[o] = h; jb.PH[ps + o] = r; jb.PH[2 * ps + o] = h; jb.PH[3 * ps + o] = h;
          jb.PF[ps + o] = f; jb.PF[2 * ps + o] = f; jb.PF[3 * ps + o] = f;
        }
      }
    }
  }
}
__global__ void __launch_bounds__(256) k_split_T(SplitJobs jobs, int Np) {
  k_split_T_body(native_blk(), jobs, Np);
}

// Column norms and split at once (grouped launches): a CTA of 32 x (at least the row groups)
// threads per 32 columns cb of one job (the grouped grid runs over the jobs' column blocks in
// turn, so that no block is idle): the norms as k_colnorms forms them (same order), the
// exponents kept in shared memory, then the split of those columns as k_split_T forms it,
// warp w writing pairs of mu 64 w, 64 (w + warps), ... (the columns come from L1 after the
// norms).
__device__ __forceinline__ void k_colsplit_body(const SplitJob& jb, int cb, double invT,
                                                DevHeader* hdr, int Np) {
  const int c0 = cb * 32;
  if (c0 >= jb.nrows_out) return;  // uniform over the CTA
  __shared__ double red[32][33];
  __shared__ int ecol[32];
  const double* __restrict__ S = jb.S;
  const int* __restrict__ eS = jb.eS;
  const long long ld = jb.ld;
  const int N = jb.N;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  {
    const int c = c0 + tx;
    const int G = norm_groups(N);
    if (ty < G) red[ty][tx] = colnorm_partial(jb, c, ty, G);
    __syncthreads();
    if (ty == 0) ecol[tx] = c < jb.nrows_out ? colnorm_finish(jb, c, red, tx, G, invT, hdr) : 0;
    __syncthreads();
  }
  // two consecutive mu per thread (Np is even), 4-byte stores of both
  const int ncl = min(32, jb.nrows_out - c0);
  const int np2 = Np / 2;
  for (int m2 = ty * 32 + tx; m2 - tx < np2; m2 += (int)blockDim.x) {
    if (m2 >= np2) continue;
    const int mu0 = 2 * m2, mu1 = mu0 + 1;
    const int s0 = (eS && mu0 < N) ? eS[mu0] : 0;
    const int s1 = (eS && mu1 < N) ? eS[mu1] : 0;
    for (int cc = 0; cc < ncl; ++cc) {
      const int c = c0 + cc;
      const bool cin = c < jb.ncols;
      const double v0 = (mu0 < N && cin) ? S[(size_t)mu0 * ld + c] : 0.0;
      const double v1 = (mu1 < N && cin) ? S[(size_t)mu1 * ld + c] : 0.0;
      __half h0, f0, r0, h1, f1, r1;
      intfrac_split_v(v0, s0 - ecol[cc], h0, f0, r0);
      intfrac_split_v(v1, s1 - ecol[cc], h1, f1, r1);
      const size_t o = (size_t)c * Np + mu0;
      const __half2 h2 = __halves2half2(h0, h1), f2 = __halves2half2(f0, f1);
      if (jb.H) {
        *(__half2*)(jb.H + o) = h2;
        *(__half2*)(jb.F + o) = f2;
      }
      if (jb.planes) {
        const __half2 r2 = __halves2half2(r0, r1);
        const size_t ps = (size_t)jb.nrows_out * Np;
        __half2* PH = (__half2*)(jb.PH + o);
        __half2* PF = (__half2*)(jb.PF + o);
        const size_t p2 = ps / 2;  // a plane in half2 units (ps is even)
        // zero blocks as in k_split_T: cleared when B is prepared
        if (jb.planes == 1) {
          PH[0] = h2;
          PF[p2] = h2; PF[2 * p2] = f2; PF[3 * p2] = r2;
        } else {
          PH[0] = h2; PH[p2] = r2; PH[2 * p2] = h2; PH[3 * p2] = h2;
          PF[p2] = f2; PF[2 * p2] = f2; PF[3 * p2] = f2;
        }
      }
    }
  }
}

// The splits of a build's prep phase: C_act^T for b (and its residual planes, the V side of
// h C_act), diag(2^s) C_act for the symmetric half transform (with_half_transform), and
// h^T = h (the U side of h C_act).
__host__ __device__ inline SplitJob split_c_job(const Dims& d, const Layout& L, char* ws,
                                               const double* C, const double* h, int k) {
  if (k == 0)
    return SplitJob{C, d.N, d.N, d.A, d.Ap, nullptr, (int*)(ws + L.eC),
                    (double*)(ws + L.cnorm), (__half*)(ws + L.Chi), (__half*)(ws + L.Clo),
                    2, (__half*)(ws + L.cPH), (__half*)(ws + L.cPF)};
  if (k == 1)
    return SplitJob{C, d.N, d.N, d.A, d.Ap, (const int*)(ws + L.eS), (int*)(ws + L.eCs),
                    nullptr, (__half*)(ws + L.ChiS), (__half*)(ws + L.CloS),
                    0, nullptr, nullptr};
  return SplitJob{h, d.N, d.N, d.N, d.N, nullptr, (int*)(ws + L.eh), nullptr, nullptr,
                  nullptr, 1, (__half*)(ws + L.hAH), (__half*)(ws + L.hAF)};
}
__host__ __device__ inline SplitJobs split_c_jobs(const Dims& d, const Layout& L, char* ws,
                                                  const double* C, const double* h,
                                                  bool with_half_transform) {
  SplitJobs jobs{};
  jobs.j[0] = split_c_job(d, L, ws, C, h, 0);
  jobs.j[1] = split_c_job(d, L, ws, C, h, with_half_transform ? 1 : 2);
  jobs.j[2] = split_c_job(d, L, ws, C, h, 2);
  jobs.count = with_half_transform ? 3 : 2;
  return jobs;
}
// The splits of lambda = C^T G: the residual planes of C^T (all N columns of C, U side) and of
// G^T (V side), in the buffers of h C_act (free by then).
__host__ __device__ inline SplitJob lambda_job(const Dims& d, const Layout& L, char* ws,
                                               const double* C, int k) {
  const int N = d.N, A = d.A;
  if (k == 0)
    return SplitJob{C, N, N, N, N, nullptr, (int*)(ws + L.eCf), nullptr, nullptr, nullptr,
                    1, (__half*)(ws + L.hAH), (__half*)(ws + L.hAF)};
  return SplitJob{(const double*)(ws + L.G), A, N, A, d.Ap, nullptr, (int*)(ws + L.eG),
                  nullptr, nullptr, nullptr, 2, (__half*)(ws + L.cPH), (__half*)(ws + L.cPF)};
}
__host__ __device__ inline SplitJobs lambda_jobs(const Dims& d, const Layout& L, char* ws,
                                                 const double* C) {
  SplitJobs jobs{};
  jobs.j[0] = lambda_job(d, L, ws, C, 0);
  jobs.j[1] = lambda_job(d, L, ws, C, 1);
  jobs.count = 2;
  return jobs;
}

// All jobs' norms, then all splits: two launches.  `first`: the first of a call (launched plainly).
cudaError_t launch_split_jobs(const SplitJobs& jobs, int Np, double invT, DevHeader* hdr,
                              const ZeroJob& zero, bool first, cudaStream_t s) {
  int rmax = 0;
  for (int k = 0; k < jobs.count; ++k)
    if (jobs.j[k].nrows_out > rmax) rmax = jobs.j[k].nrows_out;
  const bool clear = zero.flag || zero.n[0] > 0;
  launch_chained_to(first ? 0 : kChainCtas, k_colnorms,
                    dim3((rmax + kNormCols - 1) / kNormCols, jobs.count + (clear ? 1 : 0)),
                    kNormCols * norm_groups(jobs.j[0].N), 0, s, jobs, invT, hdr, zero);
  launch_chained(k_split_T, dim3((Np + 31) / 32, (rmax + 31) / 32, jobs.count), 256, 0, s, jobs, Np);
  count_launch(2);
  return cudaGetLastError();
}

// s_C^2 >= ||C_act||_2^2: Gershgorin bound max_i sum_j |(C_act^T C_act)_ij| of the Gram
// matrix, formed in fp32 with a relative safety margin of 1e-4 far above its rounding
// error.  k_gram_part: one CTA per (chunk of 32 AO indices mu, block of 16 rows i): the
// chunk of C_act in shared memory (fp32), thread (i, j0) forms entries (i, j0 + 16 k) with
// the chunk's mu in order; k_gram_final: one CTA per row, the chunks summed in order.
constexpr int kGramChunk = 32;
__device__ __forceinline__ void k_gram_part_body(const Blk& B_, const double* __restrict__ C, int N, int A,
                                                   float* part) {
  __shared__ float cs[kGramChunk][256];  // A <= 256
  const int ch = B_.x, i0 = B_.y * 16;
  const int mu0 = ch * kGramChunk, nmu = min(kGramChunk, N - mu0);
  for (int t = threadIdx.x; t < kGramChunk * A; t += blockDim.x) {
    const int m = t / A, j = t % A;
    cs[m][j] = m < nmu ? (float)C[(size_t)(mu0 + m) * N + j] : 0.f;
  }
  __syncthreads();
  const int i = i0 + threadIdx.x / 16, jl = threadIdx.x % 16;
  if (i >= A) return;
  float g[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) g[k] = 0.f;
  for (int m = 0; m < kGramChunk; ++m) {
    const float ci = cs[m][i];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int j = jl + 16 * k;
      if (j < A) g[k] = fmaf(ci, cs[m][j], g[k]);
    }
  }
  float* out = part + ((size_t)ch * A + i) * A;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int j = jl + 16 * k;
    if (j < A) out[j] = g[k];
  }
}
__global__ void __launch_bounds__(256) k_gram_part(const double* __restrict__ C, int N, int A,
                                                   float* part) {
  k_gram_part_body(native_blk(), C, N, A, part);
}

__device__ __forceinline__ void k_gram_final_body(const Blk& B_, const float* __restrict__ part, int nch,
                                                    int A, DevHeader* hdr) {
  const int i = B_.x;
  const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
  float rs = 0.f;
  for (int j = threadIdx.x; j < A; j += blockDim.x) {
    float t = 0.f;
    for (int ch = 0; ch < nch; ++ch) t += part[((size_t)ch * A + i) * A + j];
    rs += fabsf(t);
  }
  __shared__ float red[8];
  for (int o = 16; o > 0; o >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, o);
  if (lane == 0) red[w] = rs;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int k = 0; k < 8; ++k) t += red[k];
    atomic_max_nonneg((unsigned long long*)&hdr->sC2, (double)t * (1.0 + 1e-4));
  }
}
__global__ void __launch_bounds__(256) k_gram_final(const float* __restrict__ part, int nch,
                                                    int A, DevHeader* hdr) {
  k_gram_final_body(native_blk(), part, nch, A, hdr);
}

// The per-block exponents of the two X splits written by the half transform (blocks with
// blockIdx.y = 0 and 1 respectively):
//  * X^T rows (P, q) for b: ||X[P][:][q]||_2 = ||B^P C_q||_2 <= ||B^P||_inf ||C_q||_2 (B^P
//    symmetric, so ||B^P||_2 <= ||B^P||_inf);
//  * X rows (split, mu) for G: the row runs over the split's slices and q, and its squared
//    norm sum_P ||B^P_mu C_act||^2 <= s_C^2 sum_P ||B^P_mu||^2 (s_C^2 the Gram bound).
__device__ __forceinline__ void k_x_exponents_body(const Blk& B_, const double* __restrict__ L1max, const double* __restrict__ cnorm,
                              int Ap, double invT, int* eXt, const float* __restrict__ rn2,
                              const DevHeader* hdr, int np, int splits, int N, double invT2,
                              int* spOf, int* eX3) {
  if (B_.y == 0) {  // a thread per (P, q)
    for (long long i = B_.x * (long long)blockDim.x + threadIdx.x; i < (long long)np * Ap;
         i += (long long)B_.gx * blockDim.x)
      eXt[i] = intfrac_exponent_inv(L1max[i / Ap] * cnorm[i % Ap], invT);
    return;
  }
  const double sC2 = hdr->sC2;
  const long long tot = (long long)splits * N;
  for (long long i = B_.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)B_.gx * blockDim.x) {
    const int sp = (int)(i / N), mu = (int)(i % N);
    const int P0 = (int)((long long)np * sp / splits), P1 = (int)((long long)np * (sp + 1) / splits);
    // fp32 sum of the rounded-up row norms, in order of P; the 2^-16 margin covers its
    // rounding (at most 64 slices a split, 2^-24 an addition)
    float r2 = 0.f;
    int P = P0;
    for (; P + 8 <= P1; P += 8) {  // eight loads in flight, summed in order of P
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = rn2[(size_t)(P + u) * N + mu];
#pragma unroll
      for (int u = 0; u < 8; ++u) r2 += v[u];
    }
    if (P < P1) {
      float v[7];
#pragma unroll
      for (int u = 0; u < 7; ++u) v[u] = P + u < P1 ? rn2[(size_t)(P + u) * N + mu] : 0.f;
#pragma unroll
      for (int u = 0; u < 7; ++u) r2 += v[u];
    }
    if (mu == 0)
      for (int Q = P0; Q < P1; ++Q) spOf[Q] = sp;
    eX3[i] = intfrac_exponent_sq(sC2 * (double)r2 * (1.0 + 0x1p-16), invT2);
  }
}
__global__ void k_x_exponents(const double* __restrict__ L1max, const double* __restrict__ cnorm,
                              int Ap, double invT, int* eXt, const float* __restrict__ rn2,
                              const DevHeader* hdr, int np, int splits, int N, double invT2,
                              int* spOf, int* eX3) {
  k_x_exponents_body(native_blk(), L1max, cnorm, Ap, invT, eXt, rn2, hdr, np, splits, N, invT2, spOf, eX3);
}




// G[mu][p] += 2^e3 * sum_s Gpart[s][mu][p]: groups of eight partials summed in fp32 (the
// FP64 pipe of this GPU is narrow), the groups in double, in order of s; four consecutive p
// per thread.
__device__ __forceinline__ void k_reduce_G_body(const Blk& B_, const float* __restrict__ Gp, int S, int N, int A, int Ap,
                           const DevHeader* hdr, double* G) {
  const double sc = ldexp(1.0, hdr->e3);
  const int r4 = Ap / 4;
  const long long tot = (long long)N * r4;
  const float4* G4 = (const float4*)Gp;
  for (long long i = B_.x * (long long)blockDim.x + threadIdx.x; i < tot;
       i += (long long)B_.gx * blockDim.x) {
    const long long mu = i / r4;
    const int p0 = (int)(i % r4) * 4;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int k = 0;
    for (; k + 8 <= S; k += 8) {  // groups of eight partials in fp32, double across groups
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = G4[(size_t)(k + u) * tot + i];
      float4 g = v[0];
#pragma unroll
      for (int u = 1; u < 8; ++u) {
        g.x += v[u].x;
        g.y += v[u].y;
        g.z += v[u].z;
        g.w += v[u].w;
      }
      s0 += g.x;
      s1 += g.y;
      s2 += g.z;
      s3 += g.w;
    }
    if (k < S) {  // the rest, its loads in flight together too
      float4 v[7];
#pragma unroll
      for (int u = 0; u < 7; ++u)
        v[u] = k + u < S ? G4[(size_t)(k + u) * tot + i] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 7; ++u) {
        if (k + u >= S) break;
        s0 += v[u].x;
        s1 += v[u].y;
        s2 += v[u].z;
        s3 += v[u].w;
      }
    }
    double* g = G + mu * A + p0;
    const double sv[4] = {s0, s1, s2, s3};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (p0 + j < A) g[j] += sc * sv[j];
  }
}
__global__ void k_reduce_G(const float* __restrict__ Gp, int S, int N, int A, int Ap,
                           const DevHeader* hdr, double* G) {
  k_reduce_G_body(native_blk(), Gp, S, N, A, Ap, hdr, G);
}

}  // namespace

// ---------------------------------------------------------------------------
cudaError_t launch_prepare_split_B(const Dims& d, const double* B, char* ws, const Layout& L,
                                   cudaStream_t s) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const cudaError_t e0 = cudaMemsetAsync(ws + L.rnmax, 0, (size_t)d.N * sizeof(double), s);
  if (e0 != cudaSuccess) return e0;
  int* tP = (int*)(ws + L.tmax);
  const int* eS = (const int*)(ws + L.eS);
  const double invT = intfrac_inv_target(d.N);
  const SliceForm form = slice_form(d.layout == DONOF_B_PACKED, d.N);
  const size_t smem = slice_smem(form, d.N);
  const bool by_rows = slices_by_rows(form, d.Q, d.N);
  const int s_in_smem = smem / 4 + (size_t)d.N * 4 <= kSliceSmemMax ? 1 : 0;
  const size_t smem2 = smem / 4 + (s_in_smem ? (size_t)d.N * 4 : 0);
  const int threads = 32 * slice_warps(form, d.N), ctas = d.Q < num_sms() * 8 ? d.Q : num_sms() * 8;
  auto stats = form == kSliceDense    ? k_b_stats<kSliceDense>
               : form == kSlicePacked ? k_b_stats<kSlicePacked>
                                      : k_b_stats<kSliceGathered>;
  auto scale = form == kSliceDense    ? k_p_scale<kSliceDense>
               : form == kSlicePacked ? k_p_scale<kSlicePacked>
                                      : k_p_scale<kSliceGathered>;
  // the 48 KB that need no attribute are for the kernels' static shared memory too; one limit for
  // every size, so that calls from several threads don't lower each other's
  auto raise = [](const void* fn, size_t bytes) {
    return bytes <= 47 * 1024 ? cudaSuccess
                              : cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     kSliceSmemMax);
  };
  double* L1max = (double*)(ws + L.L1max);
  float* rn2 = (float*)(ws + L.rn2);
  auto* rnmax = (unsigned long long*)(ws + L.rnmax);
  double* tmax = (double*)(ws + L.eB);  // by rows: in the space of the exponents made from it
  if (by_rows) {
    cudaError_t e = cudaMemsetAsync(L1max, 0, (size_t)d.Q * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(tmax, 0, (size_t)d.Q * 8, s);
    if (e != cudaSuccess) return e;
    k_b_stats_rows<<<num_sms() * 8, 256, 0, s>>>(B, d.layout, d.Q, d.N, hdr,
                                                 (unsigned long long*)L1max, rn2, rnmax);
  } else {
    cudaError_t e = raise((const void*)stats, smem);
    if (e == cudaSuccess) e = raise((const void*)scale, smem2);
    if (e != cudaSuccess) return e;
    stats<<<ctas, threads, smem, s>>>(B, d.Q, d.N, hdr, L1max, rn2, rnmax);
  }
  k_sym_scale<<<1, 1024, 0, s>>>((const double*)(ws + L.rnmax), d.N, (int*)(ws + L.eS));
  if (by_rows) {
    k_p_scale_rows<<<num_sms() * 8, 256, 0, s>>>(B, d.layout, d.Q, d.N, eS,
                                                 (unsigned long long*)tmax);
    k_t_exps<<<1, 256, 0, s>>>(tmax, d.Q, invT, tP);
    count_launch(1);
  } else {
    scale<<<ctas, threads, smem2, s>>>(B, d.Q, d.N, eS, s_in_smem, invT, rn2, tP);
  }
  k_sym_exps<<<num_sms() * 4, 256, 0, s>>>(tP, eS, d.Q, d.N, (int*)(ws + L.eB));
  const SymTiles st = sym_tiles(d.N);
  if (st.dense)
    k_split_B_dense<<<num_sms() * 8, 256, 0, s>>>(B, d.layout, d.Q, d.N, st.ld, eS, tP,
                                                  (__half*)(ws + L.Bhi), (__half*)(ws + L.Blo));
  else
    (d.N < kFlatN ? k_split_B_sym<int> : k_split_B_sym<long long>)<<<num_sms() * 8, 256, 0, s>>>(
        B, d.layout, d.Q, d.N, st, eS, tP, (__half*)(ws + L.Bhi), (__half*)(ws + L.Blo));
  count_launch(5);
  return cudaGetLastError();
}

cudaError_t launch_split_C(const Dims& d, const double* C, const double* h, char* ws,
                           const Layout& L, bool with_half_transform, const ZeroJob& zero,
                           cudaStream_t s) {
  return launch_split_jobs(split_c_jobs(d, L, ws, C, h, with_half_transform), d.Np,
                           intfrac_inv_target(d.N), (DevHeader*)(ws + L.header), zero, true, s);
}

cudaError_t launch_gram_bound(const Dims& d, const double* C, char* ws, const Layout& L,
                              cudaStream_t s) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int nch = (d.N + kGramChunk - 1) / kGramChunk;
  float* part = (float*)(ws + L.gram);
  launch_chained(k_gram_part, dim3(nch, (d.A + 15) / 16), 256, 0, s, C, d.N, d.A, part);
  launch_chained(k_gram_final, d.A, 256, 0, s, part, nch, d.A, hdr);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t launch_reduce_G(const Dims& d, char* ws, const Layout& L, cudaStream_t s) {
  // small CTAs, so that a small product's threads reach every SM (500 x 80 over 76 splits: 24.5 us in
  // 40 CTAs of 256 threads, and its last loads one by one, 15 in 157 of 64)
  const int nb = (int)(((long long)d.N * (d.Ap / 4) + 63) / 64);
  launch_chained(k_reduce_G, nb, 64, 0, s, (const float*)(ws + L.Gpart), d.splits, d.N, d.A, d.Ap,
                                           (const DevHeader*)(ws + L.header), (double*)(ws + L.G));
  count_launch(1);
  return cudaGetLastError();
}

// out[r * ld + c] = sum_s part[s][r][c] (r < M, c < ncols): the four K blocks of a
// residual-extended product added in double in block order.
__device__ __forceinline__ void k_sum_blocks_body(const Blk& B_, const float* __restrict__ part, int M, int ncols, int Ap,
                             double* out, long long ld) {
  const long long tot = (long long)M * ncols;
  const size_t ps = (size_t)M * Ap;
  for (long long i = threadIdx.x + (long long)B_.x * blockDim.x; i < tot;
       i += (long long)blockDim.x * B_.gx) {
    const int r = (int)(i / ncols), c = (int)(i - (long long)r * ncols);
    const size_t o = (size_t)r * Ap + c;
    out[(size_t)r * ld + c] = (((double)part[o] + (double)part[ps + o]) +
                               (double)part[2 * ps + o]) + (double)part[3 * ps + o];
  }
}
__global__ void k_sum_blocks(const float* __restrict__ part, int M, int ncols, int Ap,
                             double* out, long long ld) {
  k_sum_blocks_body(native_blk(), part, M, ncols, Ap, out, ld);
}

// Arguments and maps of U V^T (M x Ap, fp32 block outputs in hpart) from the residual planes
// of U (M rows, in hAH/hAF, exponents eU) and V (Ap rows, in cPH/cPF, exponents eV) over
// K = N: the four K blocks as four splits.
bool ext_setup(const Dims& d, int M, const int* eU, const int* eV, char* ws, const Layout& L,
               TcArgs& a, TcMaps& m) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, Ap = d.Ap, Np = d.Np;
  const size_t h2 = sizeof(__half);
  if (!make_map(&m.ah, ws + L.hAH, N, M, 4, Np * h2, (uint64_t)M * Np * h2, 64, BM) ||
      !make_map(&m.al, ws + L.hAF, N, M, 4, Np * h2, (uint64_t)M * Np * h2, 64, BM) ||
      !make_map(&m.bh, ws + L.cPH, N, Ap, 4, Np * h2, (uint64_t)Ap * Np * h2, 64, Ap) ||
      !make_map(&m.bl, ws + L.cPF, N, Ap, 4, Np * h2, (uint64_t)Ap * Np * h2, 64, Ap))
    return false;
  a = TcArgs{};
  a.mode = 2; a.M = M; a.Nn = Ap;
  a.m_tiles = (M + BM - 1) / BM; a.z_count = 1;
  a.splits = 4;  // one K block per split
  a.kt_per_kb = (N + 63) / 64; a.nkb = 4; a.a_z_kb = 1; a.b_z_mode = 2;
  a.eA = eU; a.eA_sstride = 0;
  a.eB = eV; a.eB_sstride = 0;
  a.out = (float*)(ws + L.hpart); a.out_ld = Ap; a.out_zstride = (long long)M * Ap;
  a.glob_exp = &hdr->zero_exp;
  a.status = &hdr->status; a.abort_flag = &hdr->abort_flag;
  return true;
}

// out = U V^T (M x ncols, row stride ld): the four K blocks as four splits of one launch,
// each with its own fp32 output (block 0 exact, the others to the fp32 rounding of terms
// 2^-12 and smaller relative to the row norms), added in double by k_sum_blocks.
int run_extended_product(const Dims& d, int M, const int* eU, const int* eV, int ncols,
                         double* out, long long ld, char* ws, const Layout& L, cudaStream_t s) {
  TcArgs a;
  TcMaps m;
  if (!ext_setup(d, M, eU, eV, ws, L, a, m)) return DONOF_ERR_CUDA;
  if (launch_tc<64, kIntFrac, 0>(m, a, s) != cudaSuccess)
    return DONOF_ERR_CUDA;
  const long long nb = ((long long)M * ncols + 255) / 256;
  launch_chained(k_sum_blocks, (int)(nb < num_sms() * 8 ? nb : num_sms() * 8), 256, 0, s,
      (const float*)(ws + L.hpart), M, ncols, d.Ap, out, ld);
  count_launch(1);
  return cudaGetLastError() == cudaSuccess ? DONOF_OK : DONOF_ERR_CUDA;
}

// hC = h C_act (h symmetric: its rows are the rows of h^T) from the planes written by
// launch_split_C.
int run_hc_tc(const Dims& d, char* ws, const Layout& L, cudaStream_t s) {
  return run_extended_product(d, d.N, (const int*)(ws + L.eh), (const int*)(ws + L.eC), d.A,
                              (double*)(ws + L.hC), d.A, ws, L, s);
}

// lambda[q][p] = sum_mu C[mu][q] G[mu][p] (q < N, p < nact), row stride N, from the planes
// of C^T (all N columns of C) and G^T; the planes and block outputs of h C_act are free by
// now and are reused.
int run_lambda_tc(const Dims& d, const double* C, char* ws, const Layout& L, double* lam,
                  cudaStream_t s) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, A = d.A;
  ZeroJob zero{};
  zero.add(lam, (size_t)N * N * 8);
  if (launch_split_jobs(lambda_jobs(d, L, ws, C), d.Np, intfrac_inv_target(N), hdr, zero, false,
                        s) != cudaSuccess)
    return DONOF_ERR_CUDA;
  return run_extended_product(d, N, (const int*)(ws + L.eCf), (const int*)(ws + L.eG), A, lam,
                              N, ws, L, s);
}

// Arguments and maps of (1) X = B C_act for slices p0 .. p0+np-1: A operand the split B in
// its symmetric tile storage (bulk copies) or dense (TMA), BK = 64, B operand
// (diag(2^s) C_act)^T; unit = (slice, row tile of 128 AO indices); outputs the X and X^T
// splits (mode 1).
bool half_setup(const Dims& d, int p0, int np, const TuneCode& tv, char* ws, const Layout& L,
                TcArgs& a, TcMaps& m) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, Ap = d.Ap, Np = d.Np;
  const size_t h2 = sizeof(__half);
  const SymTiles st = sym_tiles(N);
  const int bk = 64;  // the stored tiles are laid out for it
  const uint32_t brows = tv.pair ? Ap / 2 : Ap;  // B rows staged per CTA
  if (!make_map(&m.bh, ws + L.ChiS, N, Ap, 1, Np * h2, (uint64_t)Ap * Np * h2, bk, brows) ||
      !make_map(&m.bl, ws + L.CloS, N, Ap, 1, Np * h2, (uint64_t)Ap * Np * h2, bk, brows))
    return false;
  a = TcArgs{};
  a.mode = 1; a.Nn = Ap;
  a.m_tiles = st.T; a.z_count = np; a.splits = 1;
  a.nkb = 1; a.a_z_kb = 0; a.b_z_mode = 0;
  a.st = st;
  const int work = tv.pair ? num_sms() / 2 : num_sms();
  if (st.dense) {
    // dense slices: A through a 3-D map [np][N][ld] with boxes of 64 x 128 (zero fill past N
    // in both directions); unit = (slice, row tile), K steps of 64 in order
    const char* bh = ws + L.Bhi + (size_t)p0 * st.perP * h2;
    const char* bl = ws + L.Blo + (size_t)p0 * st.perP * h2;
    if (!make_map(&m.ah, bh, N, N, np, (uint64_t)st.ld * h2, (uint64_t)st.perP * h2, bk, BM) ||
        !make_map(&m.al, bl, N, N, np, (uint64_t)st.ld * h2, (uint64_t)st.perP * h2, bk, BM))
      return false;
    a.M = N;
    a.kt_per_kb = (N + bk - 1) / bk;
    a.sym = 0; a.a_z_unit = 1;
    a.grid = work;
    // a last row tile of at most 64 AO indices: two slices' last tiles share a unit
    a.pack2 = (!tv.pair && N - BM * (st.T - 1) <= 64) ? 1 : 0;
    if (a.pack2 &&
        (!make_map(&m.ah2, bh, N, N, np, (uint64_t)st.ld * h2, (uint64_t)st.perP * h2, bk, 64) ||
         !make_map(&m.al2, bl, N, N, np, (uint64_t)st.ld * h2, (uint64_t)st.perP * h2, bk, 64)))
      return false;
  } else {
    m.ah = m.bh;  // unused: the A tiles come from the bulk copies
    m.al = m.bl;
    a.M = st.T * BM;
    a.kt_per_kb = 1;
    a.sym = 1;
    // whole slices at once (the partner row tiles of a slice read their shared stored tile
    // in the same round, so the second read can hit L2); a pair takes two slices' row tiles
    a.grid = (tv.full || work < st.T) ? work : work / st.T * st.T;
  }
  a.a_tiled_h = (const __half*)(ws + L.Bhi) + (size_t)p0 * st.perP;
  a.a_tiled_f = (const __half*)(ws + L.Blo) + (size_t)p0 * st.perP;
  a.eA = (const int*)(ws + L.eB) + (size_t)p0 * N; a.eA_zstride = 0;
  a.eB = (const int*)(ws + L.eCs); a.eB_zstride = 0;
  a.glob_exp = &hdr->zero_exp;  // not applied in mode 1
  a.Nmu = N; a.Nrow = N; a.Ap = Ap; a.Np = Np;
  a.xhi = (__half*)(ws + L.Xhi); a.xlo = (__half*)(ws + L.Xlo);
  a.xth = (__half*)(ws + L.Xthi); a.xtf = (__half*)(ws + L.Xtlo); a.eXt = (const int*)(ws + L.eXt);
  a.spOf = (const int*)(ws + L.spOf); a.eX3 = (const int*)(ws + L.eX3);
  a.status = &hdr->status; a.abort_flag = &hdr->abort_flag;
  return true;
}

// (2) b[P] = C_act^T X[P] for the np slices of the block: one GEMM over all of them, rows
// (P, q) of X^T flattened into M, C_act^T rows as N; b[(P, q)][p] = b^P[q][p] is b^P
// (symmetric) in the [P][Ap][Ap] layout; the epilogue also writes the diagonal d^P.
bool b_setup(const Dims& d, int np, const TuneCode& tv, char* ws, const Layout& L, TcArgs& a,
             TcMaps& m) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, Ap = d.Ap, Np = d.Np;
  const size_t h2 = sizeof(__half);
  const uint64_t rows = (uint64_t)np * Ap;
  const int bk = tv.bk;
  const uint32_t brows = tv.pair ? Ap / 2 : Ap;
  if (!make_map(&m.ah, ws + L.Xthi, N, rows, 1, Np * h2, rows * Np * h2, bk, BM) ||
      !make_map(&m.al, ws + L.Xtlo, N, rows, 1, Np * h2, rows * Np * h2, bk, BM) ||
      !make_map(&m.bh, ws + L.Chi, N, Ap, 1, Np * h2, (uint64_t)Ap * Np * h2, bk, brows) ||
      !make_map(&m.bl, ws + L.Clo, N, Ap, 1, Np * h2, (uint64_t)Ap * Np * h2, bk, brows))
    return false;
  a = TcArgs{};
  a.mode = 2; a.M = (int)rows; a.Nn = Ap;
  a.m_tiles = (int)((rows + BM - 1) / BM); a.z_count = 1; a.splits = 1;
  a.kt_per_kb = (N + bk - 1) / bk; a.nkb = 1; a.a_z_kb = 0; a.b_z_mode = 0;
  a.eA = (const int*)(ws + L.eXt); a.eA_zstride = 0;
  a.eB = (const int*)(ws + L.eC); a.eB_zstride = 0;
  a.glob_exp = &hdr->zero_exp;
  a.out = (float*)(ws + L.b32); a.out_ld = Ap; a.out_zstride = 0;
  a.diag = (float*)(ws + L.D); a.diag_A = d.A;  // d^P for the mid section
  a.status = &hdr->status; a.abort_flag = &hdr->abort_flag;
  return true;
}

// (3) Gpart[s] = sum_{P in split s} X[P] Y[P] (integer + fraction operands, exponents
//     common to the slices of a split); X interleaved by 8 along q.
bool g_setup(const Dims& d, int np, int splits3, const TuneCode& tv, char* ws, const Layout& L,
             TcArgs& a, TcMaps& m) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, Ap = d.Ap, Np = d.Np;
  const size_t h2 = sizeof(__half);
  const int bk = tv.bk;
  const uint32_t brows = tv.pair ? Ap / 2 : Ap;
  if (!make_map_il8(&m.ah, ws + L.Xhi, Ap, Np, np, bk, BM) ||
      !make_map_il8(&m.al, ws + L.Xlo, Ap, Np, np, bk, BM) ||
      !make_map(&m.bh, ws + L.Yhi, Ap, Ap, np, Ap * h2, (uint64_t)Ap * Ap * h2, bk, brows) ||
      !make_map(&m.bl, ws + L.Ylo, Ap, Ap, np, Ap * h2, (uint64_t)Ap * Ap * h2, bk, brows))
    return false;
  a = TcArgs{};
  a.mode = 2; a.M = N; a.Nn = Ap;
  a.m_tiles = (N + BM - 1) / BM; a.z_count = 1;
  a.splits = splits3;
  a.kt_per_kb = (Ap + bk - 1) / bk; a.nkb = np; a.a_z_kb = 1; a.b_z_mode = 2;
  a.a_il8 = 1;
  a.eA = (const int*)(ws + L.eX3); a.eA_sstride = N;
  a.eB = (const int*)(ws + L.eY); a.eB_sstride = Ap;
  a.out = (float*)(ws + L.Gpart); a.out_ld = Ap; a.out_zstride = (long long)N * Ap;
  a.glob_exp = &hdr->zero_exp;
  a.status = &hdr->status; a.abort_flag = &hdr->abort_flag;
  return true;
}

// The tensor-core part of one block of np auxiliary slices (slices p0 .. p0+np-1).
int run_tc_block(const Dims& d, int p0, int np, char* ws, const Layout& L, cudaStream_t s) {
  DevHeader* hdr = (DevHeader*)(ws + L.header);
  const int N = d.N, Ap = d.Ap;
  TcArgs a;
  TcMaps m;
  // exponents of the X splits (for b and for the G contraction)
  const int splits3 = d.splits < np ? d.splits : np;  // splits of the G contraction
  // the G contraction's rows run over (slices of a split) x Ap: the largest split's length
  const double invT2 = intfrac_inv_target_sq((double)((np + splits3 - 1) / splits3) * Ap);
  const int gx3 = (splits3 * N + 255) / 256;
  const long long gx1 = std::min(((long long)np * Ap + 255) / 256, num_sms() * 4ll);
  launch_chained(
      k_x_exponents, dim3((unsigned)std::max<long long>(gx3, gx1), 2), 256, 0, s,
      (const double*)(ws + L.L1max) + p0, (const double*)(ws + L.cnorm), Ap,
      intfrac_inv_target(N), (int*)(ws + L.eXt), (const float*)(ws + L.rn2) + (size_t)p0 * N,
      (const DevHeader*)hdr, np, splits3, N, invT2, (int*)(ws + L.spOf), (int*)(ws + L.eX3));
  count_launch(1);
  // (1) X = B C_act
  prof_begin(DONOF_PHASE_HALF_TRANSFORM, s);
  {
    const TuneCode tv = tuned_variant(1, N, Ap, np);
    if (!half_setup(d, p0, np, tv, ws, L, a, m)) return DONOF_ERR_CUDA;
    if (launch_tc_variant<kIntFrac>(tv, m, a, s) != cudaSuccess)
      return DONOF_ERR_CUDA;
  }
  prof_end(DONOF_PHASE_HALF_TRANSFORM, s);
  // (2) b = C_act^T X
  prof_begin(DONOF_PHASE_MO_3INDEX, s);
  {
    const TuneCode tv = tuned_variant(2, N, Ap, np);
    if (!b_setup(d, np, tv, ws, L, a, m)) return DONOF_ERR_CUDA;
    if (launch_tc_variant<kIntFrac>(tv, m, a, s) != cudaSuccess)
      return DONOF_ERR_CUDA;
  }
  prof_end(DONOF_PHASE_MO_3INDEX, s);
  // J, K and Y from b
  prof_begin(DONOF_PHASE_JK_Y, s);
  if (launch_mid_mixed(d, np, splits3, ws, L, s) != cudaSuccess) return DONOF_ERR_CUDA;
  prof_end(DONOF_PHASE_JK_Y, s);
  // (3) the G contraction and the sum of its split partials
  prof_begin(DONOF_PHASE_G_BUILD, s);
  {
    const TuneCode tv = tuned_variant(3, N, Ap, np);
    if (!g_setup(d, np, splits3, tv, ws, L, a, m)) return DONOF_ERR_CUDA;
    if (launch_tc_variant<kIntFrac>(tv, m, a, s) != cudaSuccess)
      return DONOF_ERR_CUDA;
    Dims d2 = d;
    d2.splits = a.splits;
    if (launch_reduce_G(d2, ws, L, s) != cudaSuccess) return DONOF_ERR_CUDA;
  }
  prof_end(DONOF_PHASE_G_BUILD, s);
  return DONOF_OK;
}

}  // namespace donof

// ---------------------------------------------------------------------------
// Grouped launches over a batch (one block of np = naux slices per instance).
// ---------------------------------------------------------------------------
namespace donof {
namespace {
__device__ __forceinline__ int grp_splits(const Dims& d) { return d.splits < d.Q ? d.splits : d.Q; }
__global__ void __launch_bounds__(1024) k_colsplit_group(const GroupLaunch g, int which) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  const Dims& d = I.d;
  const int nC = (d.Ap + 31) / 32, nN = (d.N + 31) / 32;
  const double invT = intfrac_inv_target(d.N);
  DevHeader* hdr = (DevHeader*)(I.ws + I.L.header);
  if (which == 0) {  // blocks: C_act^T (nC), diag(2^s) C_act (nC), h (nN)
    const int k = b.x < nC ? 0 : (b.x < 2 * nC ? 1 : 2);
    k_colsplit_body(split_c_job(d, I.L, I.ws, I.C, I.h, k), b.x - k * nC, invT, hdr, d.Np);
  } else {  // blocks: C (nN), G (nC)
    const int k = b.x < nN ? 0 : 1;
    k_colsplit_body(lambda_job(d, I.L, I.ws, I.C, k), b.x - k * nN, invT, hdr, d.Np);
  }
}
__global__ void __launch_bounds__(256) k_gram_part_group(const GroupLaunch g) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  k_gram_part_body(b, I.C, I.d.N, I.d.A, (float*)(I.ws + I.L.gram));
}
__global__ void __launch_bounds__(256) k_gram_final_group(const GroupLaunch g) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  k_gram_final_body(b, (const float*)(I.ws + I.L.gram), (I.d.N + kGramChunk - 1) / kGramChunk,
                    I.d.A, (DevHeader*)(I.ws + I.L.header));
}
__global__ void k_x_exponents_group(const GroupLaunch g) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  const Dims& d = I.d;
  const Layout& L = I.L;
  char* ws = I.ws;
  const int np = d.Q, sp3 = grp_splits(d);
  const double invT2 = intfrac_inv_target_sq((double)((np + sp3 - 1) / sp3) * d.Ap);
  k_x_exponents_body(b, (const double*)(ws + L.L1max), (const double*)(ws + L.cnorm), d.Ap,
                     intfrac_inv_target(d.N), (int*)(ws + L.eXt), (const float*)(ws + L.rn2),
                     (const DevHeader*)(ws + L.header), np, sp3, d.N, invT2, (int*)(ws + L.spOf),
                     (int*)(ws + L.eX3));
}
__global__ void k_reduce_G_group(const GroupLaunch g) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  const Dims& d = I.d;
  char* ws = I.ws;
  k_reduce_G_body(b, (const float*)(ws + I.L.Gpart), grp_splits(d), d.N, d.A, d.Ap,
                  (const DevHeader*)(ws + I.L.header), (double*)(ws + I.L.G));
}
__global__ void k_sum_blocks_group(const GroupLaunch g, int which) {
  Blk b;
  const InstRec& I = g.inst[group_locate(g, b)];
  const Dims& d = I.d;
  if (which == 0)
    k_sum_blocks_body(b, (const float*)(I.ws + I.L.hpart), d.N, d.A, d.Ap,
                      (double*)(I.ws + I.L.hC), d.A);
  else
    k_sum_blocks_body(b, (const float*)(I.ws + I.L.hpart), d.N, d.A, d.Ap, I.lam, d.N);
}
}  // namespace

// Arguments and maps of instance (d, ws, L) for a grouped tensor-core contraction (one block
// of all naux slices), and its number of work units.  The launch settings are those of the
// single launches' defaults: BK 64 (32 for the G contraction), single CTAs.
bool tc_group_setup(int kind, const Dims& d, char* ws, const Layout& L, void* a_rec,
                    void* m_rec, int& units) {
  TcArgs& a = *(TcArgs*)a_rec;
  TcMaps& m = *(TcMaps*)m_rec;
  const int np = d.Q, sp3 = d.splits < np ? d.splits : np;
  bool ok = false;
  switch (kind) {
    case GK_TC_HC:
      ok = ext_setup(d, d.N, (const int*)(ws + L.eh), (const int*)(ws + L.eC), ws, L, a, m);
      break;
    case GK_TC_LAM:
      ok = ext_setup(d, d.N, (const int*)(ws + L.eCf), (const int*)(ws + L.eG), ws, L, a, m);
      break;
    case GK_TC_HALF: ok = half_setup(d, 0, np, TuneCode{64, 0, 0}, ws, L, a, m); break;
    case GK_TC_B: ok = b_setup(d, np, TuneCode{64, 0, 0}, ws, L, a, m); break;
    case GK_TC_G: ok = g_setup(d, np, sp3, TuneCode{32, 0, 0}, ws, L, a, m); break;
    default: return false;
  }
  units = tc_units(a, 0);
  return ok;
}

// Kernel-wide settings of a grouped contraction from its widest instance (as launch_tc sets
// them for one), written into every instance's arguments together with the batch's status
// and abort words; returns the dynamic shared memory of the launch.
size_t tc_group_finish(int kind, void* a_recs, int ninst, int* status, int* abort_flag,
                       int& cat) {
  TcArgs* a = (TcArgs*)a_recs;
  const int BK = kind == GK_TC_G ? 32 : 64;
  int nn = 16;
  for (int i = 0; i < ninst; ++i) nn = a[i].Nn > nn ? a[i].Nn : nn;
  const size_t a_bytes = (size_t)BM * BK * 2, b_bytes = (size_t)nn * BK * 2;
  const size_t stage_bytes = 2 * a_bytes + 2 * b_bytes;
  int stages = (int)((232448 - 1024 - 512 - kTabBytes) / stage_bytes);
  stages = stages > kMaxStages ? kMaxStages : (stages < 2 ? 2 : stages);
  int nbuf, stride, epi_alt;
  cat = 2 * nn <= 128 ? 1 : 0;  // kIntFracCat for every instance of the launch
  tmem_plan(nn, (cat ? 4 : 2) * nn, true, nbuf, stride, epi_alt);
  for (int i = 0; i < ninst; ++i) {
    a[i].stages = stages;
    a[i].tmem_cols = 512;
    a[i].nbuf = nbuf;
    a[i].buf_stride = stride;
    a[i].epi_alt = epi_alt;
    a[i].region = nn;
    a[i].nb_stage = nn;
    a[i].status = status;
    a[i].abort_flag = abort_flag;
  }
  size_t smem = 1024 + (size_t)stages * stage_bytes + (2 * stages + kBarTail) * 8 + kTabBytes;
  return smem < 120 * 1024 ? 120 * 1024 : smem;
}

template <int BK, int NUM>
cudaError_t launch_group_bk(const TcArgs* targs, const TcMaps* tmaps, const int* ustart,
                            int ninst, int grid, size_t smem, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_tc_gemm_group<BK, NUM>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_tc_gemm_group<BK, NUM><<<grid, kThreads, smem, s>>>(targs, tmaps, ustart, ninst);
  count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_tc_group(int kind, const void* args_dev, const void* maps_dev,
                            const int* ustart, int ninst, int units, size_t smem, int cat,
                            cudaStream_t s) {
  const TcArgs* targs = (const TcArgs*)args_dev;
  const TcMaps* tmaps = (const TcMaps*)maps_dev;
  int grid = num_sms();
  if (grid > units) grid = units;
  if (grid < 1) grid = 1;
  if (kind == GK_TC_G)
    return cat ? launch_group_bk<32, kIntFracCat>(targs, tmaps, ustart, ninst, grid, smem, s)
               : launch_group_bk<32, kIntFrac>(targs, tmaps, ustart, ninst, grid, smem, s);
  return cat ? launch_group_bk<64, kIntFracCat>(targs, tmaps, ustart, ninst, grid, smem, s)
             : launch_group_bk<64, kIntFrac>(targs, tmaps, ustart, ninst, grid, smem, s);
}

size_t tc_args_bytes() { return sizeof(TcArgs); }
size_t tc_maps_bytes() { return sizeof(TcMaps); }

cudaError_t launch_tc_small_group(int kind, const GroupLaunch& g, int blocks, int threads,
                                  cudaStream_t s) {
  switch (kind) {
    case GK_SPLIT_C: k_colsplit_group<<<blocks, threads, 0, s>>>(g, 0); break;
    case GK_SPLIT_L: k_colsplit_group<<<blocks, threads, 0, s>>>(g, 1); break;
    case GK_GRAM_PART: k_gram_part_group<<<blocks, threads, 0, s>>>(g); break;
    case GK_GRAM_FINAL: k_gram_final_group<<<blocks, threads, 0, s>>>(g); break;
    case GK_XEXP: k_x_exponents_group<<<blocks, threads, 0, s>>>(g); break;
    case GK_REDUCEG: k_reduce_G_group<<<blocks, threads, 0, s>>>(g); break;
    case GK_SUM_HC: k_sum_blocks_group<<<blocks, threads, 0, s>>>(g, 0); break;
    case GK_SUM_L: k_sum_blocks_group<<<blocks, threads, 0, s>>>(g, 1); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch(1);
  return cudaGetLastError();
}
}  // namespace donof

// ---------------------------------------------------------------------------
// Autotuner: time each tensor-core contraction of a build in each of its launch variants (K
// tile, single CTAs or CTA pairs, grid; CUDA events through the tracing phases) and keep the
// fastest per contraction and shape.
namespace donof {
int autotune_build(const donof_problem* prob, const double* h, const double* B, const double* C,
                   const double* gamma, const int32_t* pair_map, void* ws, size_t bytes,
                   cudaStream_t s) {
  const Dims d = make_dims(prob);
  const int np = d.pb < d.Q ? d.pb : d.Q;
  // candidates per contraction (codes of decode_tune); the half transform always runs with
  // BK = 64 (its pre-tiled operand is laid out for it): single CTAs or CTA pairs, the grid a
  // whole number of slices' row tiles or every SM pair
  const int phases[3] = {DONOF_PHASE_HALF_TRANSFORM, DONOF_PHASE_MO_3INDEX, DONOF_PHASE_G_BUILD};
  constexpr int kCand = 3;
  const int cand[3][kCand] = {{64, 1064, 3064}, {64, 32, 1064}, {32, 64, 1064}};
  double best_ms[3] = {1e300, 1e300, 1e300};
  int best_code[3] = {64, 64, 32};
  double* E = nullptr;
  if (cudaMallocAsync((void**)&E, sizeof(double), s) != cudaSuccess) return DONOF_ERR_CUDA;
  int rc = DONOF_OK;
  for (int c = 0; c < kCand && rc == DONOF_OK; ++c) {
    {
      std::lock_guard<std::mutex> lk(g_tune_mu);
      tune_load_locked();
      for (int k = 0; k < 3; ++k) g_tune[TuneKey{k + 1, d.N, d.Ap, np}] = cand[k][c];
    }
    rc = donof_energy_lagrangian(prob, h, B, C, gamma, pair_map, ws, bytes, E, nullptr, nullptr,
                                 s);  // warm-up
    if (rc != DONOF_OK) break;
    donof_profile_enable(1);
    for (int r = 0; r < 2 && rc == DONOF_OK; ++r)
      rc = donof_energy_lagrangian(prob, h, B, C, gamma, pair_map, ws, bytes, E, nullptr, nullptr,
                                   s);
    for (int k = 0; k < 3 && rc == DONOF_OK; ++k) {
      double ms = 0.0;
      int n = 0;
      if (donof_profile_read(phases[k], &ms, &n) != DONOF_OK || n == 0) continue;
      if (ms / n < best_ms[k]) {
        best_ms[k] = ms / n;
        best_code[k] = cand[k][c];
      }
    }
    donof_profile_enable(0);
  }
  cudaFreeAsync(E, s);
  std::lock_guard<std::mutex> lk(g_tune_mu);
  for (int k = 0; k < 3; ++k) g_tune[TuneKey{k + 1, d.N, d.Ap, np}] = best_code[k];
  tune_save_locked();
  return rc;
}
}  // namespace donof

extern "C" int donof_autotune(const donof_problem* prob, const double* h, const double* B,
                              const double* C, const double* gamma, const int32_t* pair_map,
                              void* workspace, size_t workspace_bytes, void* stream) {
  if (!prob || prob->precision != DONOF_MIXED) return DONOF_OK;  // nothing to tune
  return donof::autotune_build(prob, h, B, C, gamma, pair_map, workspace, workspace_bytes,
                               (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// Test hook (include/donof_testing.h): one plain split-product GEMM.
// ---------------------------------------------------------------------------
#include "../../include/donof_testing.h"

namespace donof {
namespace {
__device__ int g_test_words[4];  // [0] zero exponent, [1] status, [2] abort flag
}  // namespace
}  // namespace donof

extern "C" int donof_testing_tc_gemm_ex(const uint16_t* A_hi, const uint16_t* A_lo,
                                        const uint16_t* B_hi, const uint16_t* B_lo, float* D,
                                        int32_t M, int32_t N, int32_t K, int32_t layout,
                                        int32_t pair, void* stream) {
  using namespace donof;
  if (!A_hi || !A_lo || !B_hi || !B_lo || !D) return DONOF_ERR_INVALID_ARG;
  if (M < 1 || K < 8 || K % 8 != 0 || N < 16 || N > 256 || N % 16 != 0)
    return DONOF_ERR_INVALID_ARG;
  if (layout < 0 || layout > 2 || pair < 0 || pair > 1) return DONOF_ERR_INVALID_ARG;
  if ((layout == 1 && M % 64 != 0) || (layout == 2 && M % 8 != 0))
    return DONOF_ERR_INVALID_ARG;
  int* words = nullptr;
  if (cudaGetSymbolAddress((void**)&words, g_test_words) != cudaSuccess) return DONOF_ERR_CUDA;
  CUtensorMap ah, al, bh, bl;
  const uint64_t h2 = 2;
  bool ok;
  if (layout == 1)  // A as [K][M]: x = M (contiguous), y = K; box 64 x 64
    ok = make_map(&ah, A_hi, M, K, 1, M * h2, (uint64_t)M * K * h2, 64, 64) &&
         make_map(&al, A_lo, M, K, 1, M * h2, (uint64_t)M * K * h2, 64, 64);
  else if (layout == 2)
    ok = make_map_il8(&ah, A_hi, K, M, 1, 64, BM) && make_map_il8(&al, A_lo, K, M, 1, 64, BM);
  else
    ok = make_map(&ah, A_hi, K, M, 1, K * h2, (uint64_t)M * K * h2, 64, BM) &&
         make_map(&al, A_lo, K, M, 1, K * h2, (uint64_t)M * K * h2, 64, BM);
  const uint32_t brows = pair ? N / 2 : N;  // B rows staged per CTA
  ok = ok && make_map(&bh, B_hi, K, N, 1, K * h2, (uint64_t)N * K * h2, 64, brows) &&
       make_map(&bl, B_lo, K, N, 1, K * h2, (uint64_t)N * K * h2, 64, brows);
  if (!ok) return DONOF_ERR_CUDA;
  TcArgs a{};
  a.mode = 2; a.M = M; a.Nn = N;
  a.m_tiles = (M + BM - 1) / BM; a.z_count = 1; a.splits = 1;
  a.kt_per_kb = (K + 63) / 64; a.nkb = 1; a.a_z_kb = 0; a.b_z_mode = 0;
  a.a_mn = layout == 1;
  a.a_il8 = layout == 2;
  a.out = D; a.out_ld = N; a.out_zstride = 0;
  a.glob_exp = words + 0; a.status = words + 1; a.abort_flag = words + 2;
  if (cudaMemsetAsync(words + 2, 0, sizeof(int), (cudaStream_t)stream) != cudaSuccess)
    return DONOF_ERR_CUDA;
  const TcMaps m{ah, al, bh, bl, {}, {}};
  const cudaError_t e = pair ? launch_tc<64, kSplit3, 1>(m, a, (cudaStream_t)stream)
                             : launch_tc<64, kSplit3, 0>(m, a, (cudaStream_t)stream);
  return e == cudaSuccess ? DONOF_OK : DONOF_ERR_CUDA;
}

extern "C" int donof_testing_tc_gemm(const uint16_t* A_hi, const uint16_t* A_lo,
                                     const uint16_t* B_hi, const uint16_t* B_lo, float* D,
                                     int32_t M, int32_t N, int32_t K, void* stream) {
  return donof_testing_tc_gemm_ex(A_hi, A_lo, B_hi, B_lo, D, M, N, K, 0, 0, stream);
}

extern "C" int donof_testing_tc_gemm_mn(const uint16_t* A_hi, const uint16_t* A_lo,
                                        const uint16_t* B_hi, const uint16_t* B_lo, float* D,
                                        int32_t M, int32_t N, int32_t K, void* stream) {
  return donof_testing_tc_gemm_ex(A_hi, A_lo, B_hi, B_lo, D, M, N, K, 1, 0, stream);
}

extern "C" int donof_testing_tc_gemm_il8(const uint16_t* A_hi, const uint16_t* A_lo,
                                         const uint16_t* B_hi, const uint16_t* B_lo, float* D,
                                         int32_t M, int32_t N, int32_t K, void* stream) {
  return donof_testing_tc_gemm_ex(A_hi, A_lo, B_hi, B_lo, D, M, N, K, 2, 0, stream);
}

namespace donof {
namespace {
// Two roles wait on mbarriers that nothing completes: warp 0 with a short limit, warp 1
// with a long one; warp 0's time-out must raise the abort flag and end warp 1's wait too.
__global__ void k_test_wait(unsigned long long limit_a, unsigned long long limit_b, int* words) {
  __shared__ __align__(8) uint64_t bars[2];
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bars[0]), 1);
    mbar_init(smem_u32(&bars[1]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0 && warp < 2)
    mbar_wait(smem_u32(&bars[warp]), 0, words + 1, words + 2, warp == 0 ? limit_a : limit_b);
  __syncthreads();
}
}  // namespace
}  // namespace donof

extern "C" int donof_testing_wait_timeout(int64_t limit_a_ns, int64_t limit_b_ns, void* stream) {
  using namespace donof;
  if (limit_a_ns <= 0 || limit_b_ns <= 0 || limit_a_ns > 2000000000LL ||
      limit_b_ns > 20000000000LL)
    return DONOF_ERR_INVALID_ARG;
  int* words = nullptr;
  if (cudaGetSymbolAddress((void**)&words, g_test_words) != cudaSuccess) return DONOF_ERR_CUDA;
  if (cudaMemsetAsync(words + 2, 0, sizeof(int), (cudaStream_t)stream) != cudaSuccess)
    return DONOF_ERR_CUDA;
  k_test_wait<<<1, 64, 0, (cudaStream_t)stream>>>((unsigned long long)limit_a_ns,
                                                  (unsigned long long)limit_b_ns, words);
  count_launch(1);
  return cudaGetLastError() == cudaSuccess ? DONOF_OK : DONOF_ERR_CUDA;
}

extern "C" int donof_testing_status(void* stream) {
  using namespace donof;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return DONOF_ERR_CUDA;
  int* words = nullptr;
  if (cudaGetSymbolAddress((void**)&words, g_test_words) != cudaSuccess) return DONOF_ERR_CUDA;
  int st = 0;
  if (cudaMemcpy(&st, words + 1, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return DONOF_ERR_CUDA;
  const int zero = 0;
  if (cudaMemcpy(words + 1, &zero, sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess)
    return DONOF_ERR_CUDA;
  return st;
}
