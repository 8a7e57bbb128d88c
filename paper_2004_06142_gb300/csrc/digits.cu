// Double-precision matrix products on the tensor cores by exact digit products.
//
// This GPU's FP64 pipe gives about 1 TFLOP/s (2 FMA per clock and SM), its fp16 tensor cores
// 1.9 PFLOP/s.  A product C(m, n) = sum_k A(m, k) B(k, n) of doubles is taken in fixed point
// instead: with |a| < 2^EA over a row of A and |b| < 2^EB over a column of B, every element is
// an integer F = a 2^(57 - EA) of at most 57 bits and a sign, written in kD = 8 balanced digits,
//   F = sum_i d_i 2^(7 (7 - i)),   |d_0| <= 256,  -64 <= d_i <= 63 (i > 0),
// which are exact in fp16.  The digit products of equal weight, i + j = g, go to one fp32
// accumulator in TMEM, g = 0 .. 7 (36 of the 64 products; those left out weigh 2^-58 and less
// relative to 2^(EA + EB)).  Over kChunk = 256 elements of k no partial sum of a group exceeds
//   256 * 256^2 = 2^24 (g = 0),  256 (2 * 256 * 64 + (g - 1) 64^2) <= 14.7e6 (g > 0),
// so every accumulation is exact whatever the tensor core's rounding; after each chunk the
// groups are added up in integers (group 0 in 32 bits: at most 127 chunks; contractions are cut at
// 64, K <= 16384), and the sum, cut to its leading 62 bits, is rounded once, to the double that is
// stored.  (Splitting operands so that products of low precision are exact: Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication".)
//
// Error: elements within 2^4 of their row's (column's) largest are represented exactly, smaller
// ones to 2^-57 of it; the digit products left out add about 2^-57 sqrt(K) of the product of the
// two maxima.  A chain of K double FMAs rounds its running sum K times, relative to the terms:
// as much or more where the terms are of one size (tests/test_gpu_digits.py), but less where small
// elements of one operand meet large ones of the other.  In a build that is so when the AO
// functions' norms differ, and there the scales of k_scales take it off (tests/
// test_gpu_ao_scaling.py).  Rows or columns that hold a NaN or an infinity give NaN; elements below
// 2^-958 (scaled) count as zero.
//
// The B operand's digits are written once per product, as the images of the shared-memory
// stages (k_digit_planes); the digits of A are formed on the way into shared memory from the
// doubles themselves (8 bytes per element read once per column tile instead of 16 of digits
// written and read).
//
// CTA (one per SM: 16 worker warps, an MMA warp, a copying warp and, for wide tiles, two idle ones
// that leave their registers to the workers): a unit is a 128 x NT output tile (NT <= 64) and a range
// of 32-wide K stages.  Per stage each worker thread turns 8
// doubles (fetched one stage ahead) into 8 x 8 digits in shared memory; the MMA warp multiplies A's
// digit i with B's stacked digits 0 .. 7 - i, whose products land in the neighbouring
// accumulators i .. 7, so a digit of A is read once per 256 columns; the copying warp fetches B's
// digits.  The flush of a chunk follows the splitting of the next stage, so the MMAs drain
// meanwhile; carries go back to TMEM, so that only group 0 needs registers between the chunks of a
// unit.
//
// Measured: about 2850 clocks per stage of a 128 x 48 tile, 1.5 us, and some 10000 per unit for the
// conversion of its result; X = B C at N 500, 80 orbitals, 2000 slices: 3.14 ms (78.9 ms on the FP64
// pipe).  What bounds it: the workers' integer instructions (about 400 per warp and stage, the
// integer ALU at half rate, 2000 clocks), with four warps to a scheduler to hide their latencies;
// the MMAs' shared-memory reads (100 KB per 16 of k at 128 bytes a clock, 1600 clocks per stage)
// run beside them.  Tried and dropped: the double-to-integer conversion for the split (10 %
// slower), A's digits in TMEM (the MMAs are faster, but NT is 48 at most and the stores cost the
// workers as much), stages of 16 (slower), loops instead of unrolled columns in the conversion
// of the results (what they keep in local memory costs 20 %), waits that sleep (1 % slower).
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "tcptx.cuh"

namespace donof {
namespace {

constexpr int kD = 8;             // digits of an operand
constexpr int kStageK = 32;       // elements of k per stage (64-byte rows, 64-byte swizzle)
constexpr int kChunkStages = 8;   // stages per exact accumulation (256 elements)
constexpr int kWorkers = 16;      // worker warps
// Registers a thread of the wide tiles once the roles part: the launch's 96 (five warps on a
// scheduler) leave the workers' elements and columns spilled, which the scales' words make worse (a
// build of 500 / 2000 / 80 4.75 ms without the scales, 5.12 with them, 4.45 so; narrow tiles do not
// spill, and a short product pays about 0.5 us for the exchange).
constexpr int kWorkerRegs = 112, kOtherRegs = 32;
constexpr bool split_regs(int NT) { return NT >= 48; }
constexpr int dig_threads(int NT) { return 32 * (kWorkers + (split_regs(NT) ? 4 : 2)); }
constexpr int kTileM = 128;
constexpr uint32_t kABytes = kD * kTileM * kStageK * 2;  // a stage of A digits
// sum_{i > 0} 64 2^(7 (7 - i)) + 256 2^49: makes every digit's field non-negative
constexpr long long kBias = 64ll * (((1ll << 49) - 1) / 127) + (256ll << 49);

// The biased exponent of x; of a NaN or an infinity kNanMark, above every finite (and scaled) one.
constexpr int kNanMark = 1 << 14;
__device__ __forceinline__ int exp_of(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 2047 ? kNanMark : e;
}
// The exponent word of a row (or column) whose largest biased exponent is em, for its products'
// scale (a row with a NaN or an infinity: far above every finite scale, which marks its results).
constexpr int kNanExp = 1 << 20;
__device__ __forceinline__ int scale_exp(int em) {
  return em >= kNanMark / 2 ? kNanExp : (em < 64 ? 64 : em);
}
// ... and as split_exp, (em + 7) << 20, for the shift of its elements' mantissas.
__device__ __forceinline__ uint32_t split_exp(int em) { return (uint32_t)((em < 64 ? 64 : em) + 7) << 20; }

// x in fixed point relative to its row (e20 = split_exp), with kBias added so that every digit's
// field is non-negative: bits l, h, and v, bits 4..35.  (Integer shifts: the conversion
// instruction, 14 per clock and SM, made the split 10 % slower.)
struct Fixed {
  uint32_t l, h, v;
};
__device__ __forceinline__ Fixed to_fixed(double x, uint32_t e20) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t sh = (e20 - (hi & 0x7ff00000u)) >> 20;
  // the mantissa, left-justified with its hidden bit in bit 63
  unsigned long long f =
      ((unsigned long long)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
  asm("shr.u64 %0, %1, %2;" : "=l"(f) : "l"(f), "r"(sh));  // 0 for shifts of 64 and more
  const long long sg = (long long)((int)hi >> 31);
  f = (f ^ (unsigned long long)sg) + (unsigned long long)(kBias - sg);
  Fixed r;
  r.l = (uint32_t)f;
  r.h = (uint32_t)(f >> 32);
  r.v = __funnelshift_r(r.l, r.h, 4);
  return r;
}

// Digit D of two neighbouring elements as a half2 (element 0 in the low half): the 16-bit
// windows of the two numbers that hold the field at bit s <= 3, masked into the mantissa of
// fp16(1024 + u 2^s), then u - 64 (u - 256 for digit 0) by one multiply-add, exactly.
template <int D>
__device__ __forceinline__ uint32_t digit_pair(const Fixed& a, const Fixed& b, uint32_t k64) {
  constexpr uint32_t kSel = D == 7 || D == 6 || D == 2 ? 0x5410u
                            : D == 5 || D == 1         ? 0x6521u
                            : D == 3                   ? 0x7733u
                                                       : 0x7632u;
  constexpr int s = D == 7 || D == 3 || D == 0 ? 0 : D == 6 || D == 2 ? 3 : D == 5 || D == 1 ? 2 : 1;
  constexpr uint32_t kField = (D == 0 ? 0x3ffu : 0x7fu) << s;
  const uint32_t x = D == 7 ? a.l : D >= 3 ? a.v : a.h, y = D == 7 ? b.l : D >= 3 ? b.v : b.h;
  uint32_t u = __byte_perm(x, y, kSel);
  if (D == 0) u >>= 1;  // its ten bits start at bit 1 of the window
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;"  // (window & mask) | 0x64006400
      : "=r"(u)
      : "r"(u), "n"(kField | (kField << 16)), "r"(k64));
  const __half2 h = *reinterpret_cast<const __half2*>(&u);
  const __half2 d = s == 0 ? __hsub2(h, __float2half2_rn(D == 0 ? 1280.0f : 1088.0f))
                           : __hfma2(h, __float2half2_rn(1.0f / (1 << s)),
                                     __float2half2_rn(-1024.0f / (1 << s) - 64.0f));
  return *reinterpret_cast<const uint32_t*>(&d);
}
// The digits of 8 consecutive elements of k, one 16-byte word per digit.
struct Fixed8 {
  Fixed f[8];
  uint32_t k64;
};
__device__ __forceinline__ void to_fixed8(const double (&x)[8], uint32_t e20, uint32_t k64,
                                          Fixed8& r) {
#pragma unroll
  for (int j = 0; j < 8; ++j) r.f[j] = to_fixed(x[j], e20);
  r.k64 = k64;
}
// The same with the elements scaled by the powers of two of their k (ks: KScale's words of the 8).
__device__ __forceinline__ void to_fixed8(const double (&x)[8], uint32_t e20,
                                          const uint32_t* __restrict__ ks, uint32_t k64, Fixed8& r) {
  const uint4 a = __ldg((const uint4*)ks), b = __ldg((const uint4*)ks + 1);
  const uint32_t k[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
  for (int j = 0; j < 8; ++j) r.f[j] = to_fixed(x[j], e20 + k[j]);
  r.k64 = k64;
}
template <int D = 0, class Put>
__device__ __forceinline__ void store_digits(const Fixed8& r, const Put& put) {
  if constexpr (D < kD) {
    put(D, digit_pair<D>(r.f[0], r.f[1], r.k64), digit_pair<D>(r.f[2], r.f[3], r.k64),
        digit_pair<D>(r.f[4], r.f[5], r.k64), digit_pair<D>(r.f[6], r.f[7], r.k64));
    store_digits<D + 1>(r, put);
  }
}

// Byte offset of (row, 8-element chunk) in a tile of 64-byte rows with the 64-byte swizzle.
__device__ __forceinline__ uint32_t sw64(int row, int chunk) {
  return (uint32_t)(row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4));
}

// mbar_wait without a call: a call saves the caller's registers, among them the elements of A that
// are still on their way from memory, and so waits for them (a build of 500 / 2000 / 80: 5.73 ms
// with calls, 5.68 without).
__device__ __forceinline__ bool wait_for(uint32_t bar, uint32_t parity, const DigitArgs& a) {
  uint32_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 255u) != 255u) continue;
    if (*(volatile int*)a.abort_flag != 0) return false;
    const uint32_t t = (uint32_t)globaltimer();
    if (it == 255u) t0 = t;
    if (t - t0 > (uint32_t)kWaitLimitNs) {
      atomicExch(a.abort_flag, 1);
      atomicCAS(a.status, 0, (int)DONOF_ERR_TIMEOUT);
      return false;
    }
  }
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const float (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr),
               "r"(__float_as_uint(r[0])), "r"(__float_as_uint(r[1])), "r"(__float_as_uint(r[2])),
               "r"(__float_as_uint(r[3]))
               : "memory");
}

// The sum hi 2^28 + lo, lo in [0, 2^28), as a double whose bit t has the biased exponent
// t + ee: its leading 62 bits (or all of it) converted, then scaled by an addition to the
// exponent.  Results below the normal range are flushed to zero; ee from a kNanExp gives NaN.
// Free of branches: a thread converts many elements side by side.
__device__ __forceinline__ double fixed_to_double(long long hi, uint32_t lo, int ee) {
  const uint32_t hl = (uint32_t)hi, hh = (uint32_t)((unsigned long long)hi >> 32);
  const int k = min(28, __clz((int)(hh ^ (uint32_t)((int)hh >> 31))) - 2);  // |hi| < 2^62
  const uint32_t vh = __funnelshift_l(hl, hh, k), vl = (hl << k) | (lo >> (28 - k));
  const double d = __ll2double_rn((long long)(((unsigned long long)vh << 32) | vl));
  const uint32_t dh = (uint32_t)__double2hiint(d);
  const int adj = ee + 28 - k - 1023, eb = (int)((dh >> 20) & 0x7ffu) + adj;
  const bool zero = (dh << 1) == 0;  // (d is an integer: zero or at least 1)
  const bool special = (uint32_t)(eb - 1) >= 2046u || zero;
  const uint32_t sv = ee > kNanExp / 2 ? 0x7ff80000u : (eb < 1 || zero ? 0u : 0x7ff00000u);
  const uint32_t rh = special ? (dh & 0x80000000u) | sv : dh + ((uint32_t)adj << 20);
  return __hiloint2double((int)rh, special ? 0 : __double2loint(d));
}
// acc + v 2^k for an integer v held in a float
template <int K>
__device__ __forceinline__ void add_group(long long& acc, uint32_t v) {
  asm("mad.wide.s32 %0, %1, %2, %0;"
      : "+l"(acc)
      : "r"(__float2int_rn(__uint_as_float(v))), "n"(1 << K));
}

// Position of a worker thread in the sequence of (unit, stage) of its CTA: a row of A and the 8
// elements of k it fetches next.  k contiguous in memory (KC): four neighbouring threads per
// row; otherwise neighbouring threads on neighbouring rows (one block of k only).
template <bool KC>
struct Cursor {
  int u, st, st_end;
  int left;        // elements of this block of k from here on (0 and less: zeros)
  uint32_t e20;    // split_exp of the row
  const double* p;
  int kb;
  __device__ __forceinline__ Cursor(const DigitArgs& a, int units, int zero) {
    u = (int)blockIdx.x;  // (warp-uniform; the addresses of the first loads carry `zero`)
    st = st_end = 0;
    if (u < units) enter(a, zero);
  }
  __device__ __forceinline__ void enter(const DigitArgs& a, int zero = 0) {
    const int m = (u / a.ntiles) % a.mtiles, sp = u / (a.ntiles * a.mtiles);
    st = (int)((long long)a.nstages * sp / a.splits);
    st_end = (int)((long long)a.nstages * (sp + 1) / a.splits);
    const int tid = (int)threadIdx.x + zero;
    const int row = m * kTileM + (KC ? tid >> 2 : tid & 127);
    const long long kk = (long long)st * kStageK + 8 * (KC ? tid & 3 : tid >> 7);
    kb = (int)(kk / a.Kpad);
    const int q = (int)(kk - (long long)kb * a.Kpad);
    e20 = split_exp(2047);
    left = -(1 << 30);
    p = a.A;
    if (row < a.M) {
      e20 = split_exp(a.eA ? __ldg(a.eA + row) : 1023);
      const int b = row / a.Mb, r = row - b * a.Mb;
      p = a.A + (long long)b * a.sAb + (long long)r * a.sAm + (long long)kb * a.sAkb +
          (long long)q * a.sAk;
      if (kb < a.KB) left = a.Kin - q;
    }
  }
  __device__ __forceinline__ bool last() const { return st + 1 == st_end; }
  __device__ __forceinline__ void next(const DigitArgs& a, int units) {
    if (++st == st_end) {
      u += (int)gridDim.x;
      if (u < units) enter(a);
      return;
    }
    left -= kStageK;
    p += kStageK * a.sAk;
    while (left <= a.Kin - a.Kpad && left > -(1 << 29)) {  // on to the next block of k
      p += a.sAkb - a.Kpad * a.sAk;
      left = ++kb < a.KB ? left + a.Kpad : -(1 << 30);
    }
  }
  __device__ __forceinline__ void load(const DigitArgs& a, double (&x)[8]) const {
    if (KC && a.vecA && left >= 8) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double2 v = __ldg((const double2*)p + j);
        x[2 * j] = v.x;
        x[2 * j + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = j < left ? __ldg(p + (KC ? j : j * a.sAk)) : 0.0;
    }
  }
};

__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r));
  return r;
}
// mma_f16<0> by the lanes with lead != 0, the descriptors given as their low words (start address
// and leading byte offset); the high word is that of 64-byte rows.
__device__ __forceinline__ void mma_f16_if(uint32_t lead, uint32_t dtmem, uint32_t a, uint32_t b,
                                           uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
      "mov.b64 da, {%1, %6};\n\t"
      "mov.b64 db, {%2, %6};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(dtmem),
      "r"(a), "r"(b), "r"(idesc), "r"(accumulate), "r"(lead), "n"(sdesc_hi(8 * 64, 4))
      : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const __half* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"((unsigned long long)src), "r"(bytes), "r"(bar)
      : "memory");
}

// Whether a contraction's k are scaled: the word is loaded before the chain's wait (it is written
// before the first kernel of a call, which is launched plainly) and looked at behind it, by adding the
// wait's zero.
__device__ __forceinline__ int scales_word(const int* info) {
  return info ? *(const volatile int*)info : 0;
}

template <bool KC, int NT>
__global__ void __launch_bounds__(dig_threads(NT), 1)
    k_digit_gemm(const __grid_constant__ DigitArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr uint32_t b_bytes = (uint32_t)kD * NT * kStageK * 2;
  constexpr uint32_t stage_bytes = kABytes + b_bytes;
  uint64_t* bars = (uint64_t*)(smem + 2 * (size_t)stage_bytes);
  // barriers: A digits written [2], B digits landed [2], stage free [2], accumulators complete,
  // accumulators read, clean-up
  enum { kAFull = 0, kBFull = 2, kEmpty = 4, kAccFull = 6, kAccEmpty = 7, kClean = 8 };
  uint32_t* tmem_slot = (uint32_t*)(bars + 9);
  const int tid = threadIdx.x, lane = tid % 32;
  const int warp = __shfl_sync(0xffffffffu, tid / 32, 0);
  const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u, bar0 = smem0 + 2 * stage_bytes;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int units = a.mtiles * a.ntiles * a.splits;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(kAFull + i), kWorkers);
      mbar_init(bar(kBFull + i), 1);
      mbar_init(bar(kEmpty + i), 1);
    }
    mbar_init(bar(kAccFull), 1);
    mbar_init(bar(kAccEmpty), kWorkers);
    mbar_init(bar(kClean), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kWorkers) tmem_alloc<0>(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's: they start at column 0
  const int scales = scales_word(a.ks_on);
  // all of the above while the kernel before runs
  const int zero = chain_wait();
  const bool scaled = scales + zero != 0;

  if (warp >= kWorkers) {
    if constexpr (split_regs(NT)) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (warp == kWorkers) {  // ---------------------------------------- MMA issuer
      // The whole warp walks the stages and one elected lane issues, so that the descriptors are
      // computed in the uniform registers the MMAs take them from (a branch of one lane moves
      // them there, eight moves an MMA: a build of 500 / 2000 / 80 5.68 ms, so 5.19)
      uint32_t it = 0, chunk = 0;
      const uint32_t lead = elect_one();
      bool ok = true;
      constexpr int per = 256 / NT < kD ? 256 / NT : kD;  // digits of B per MMA
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int sp = u / (a.ntiles * a.mtiles);
        const int s0 = (int)((long long)a.nstages * sp / a.splits);
        const int s1 = (int)((long long)a.nstages * (sp + 1) / a.splits);
        for (int st = s0; st < s1; ++st, ++it) {
          const int c = (st - s0) % kChunkStages;
          const uint32_t buf = it & 1u, ph = (it >> 1) & 1u;
          bool ready = c > 0 || wait_for(bar(kAccEmpty), (chunk & 1u) ^ 1u, a);
          ready = ready && wait_for(bar(kBFull + buf), ph, a) && wait_for(bar(kAFull + buf), ph, a);
          if (!__all_sync(0xffffffffu, ready)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t ad0 = ((smem0 + buf * stage_bytes) >> 4) | 1u << 16;
          const uint32_t bd0 = ad0 + (kABytes >> 4);
#pragma unroll
          for (int k = 0; k < kStageK / 16; ++k) {
            const uint32_t acc = (st > s0 || k > 0) ? 1u : 0u;
#pragma unroll
            for (int i = 0; i < kD; ++i) {
#pragma unroll
              for (int j = 0; j < kD - i; j += per) {
                const int n = kD - i - j < per ? kD - i - j : per;
                // descriptors: the start address counts 16 bytes; the first products of every
                // accumulator are those of digit 0 of A
                mma_f16_if(lead, tmem + (uint32_t)((i + j) * NT),
                           ad0 + (uint32_t)((i * (kTileM * 64) + k * 32) >> 4),
                           bd0 + (uint32_t)((j * NT * 64 + k * 32) >> 4),
                           idesc_f16(kTileM, n * NT), i == 0 ? acc : 1u);
              }
            }
          }
          if (lead) mma_commit<0>(bar(kEmpty + buf));
          if (c == kChunkStages - 1 || st == s1 - 1) {
            if (lead) mma_commit<0>(bar(kAccFull));
            ++chunk;
          }
        }
      }
      // after an abort, MMAs in flight complete before TMEM is freed
      if (__any_sync(0xffffffffu, *(volatile int*)a.abort_flag != 0)) {
        if (lead) mma_commit_local<0>(bar(kClean));
        __syncwarp();
        mbar_wait_quiet(bar(kClean), 0u, kDrainLimitNs);
      }
      __syncwarp();
    } else if (warp == kWorkers + 1) {  // ------------------------------- copies of B's digits
      // (a warp of its own: one of the workers, whose arrivals all wait for, held up every stage: a
      // build of 500 / 2000 / 80 5.19 ms, so 4.78)
      if (lane == 0) {
        uint32_t it = 0, issued[2] = {0, 0};
        bool ok = true;
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
          const int sp = u / (a.ntiles * a.mtiles);
          const int s0 = (int)((long long)a.nstages * sp / a.splits);
          const int s1 = (int)((long long)a.nstages * (sp + 1) / a.splits);
          const int n0 = u % a.ntiles * NT;
          const size_t img_stage = (size_t)kD * a.imgNT * kStageK;
          // NT rows of every digit's rows (a multiple of 16: the swizzle's phase is theirs)
          const __half* img = a.Bimg + ((size_t)(n0 / a.imgNT) * a.nstages + s0) * img_stage +
                              n0 % a.imgNT * kStageK;
          for (int st = s0; st < s1; ++st, ++it, img += img_stage) {
            const uint32_t buf = it & 1u, ph = (it >> 1) & 1u;
            if (!wait_for(bar(kEmpty + buf), ph ^ 1u, a)) {
              ok = false;
              break;
            }
            const uint32_t dst = smem0 + buf * stage_bytes + kABytes;
            mbar_expect_tx(bar(kBFull + buf), b_bytes);
            if (a.imgNT == NT) {
              bulk_copy(dst, img, b_bytes, bar(kBFull + buf));
            } else {
#pragma unroll
              for (int d = 0; d < kD; ++d)
                bulk_copy(dst + (uint32_t)d * (NT * kStageK * 2),
                          img + (size_t)d * a.imgNT * kStageK, NT * kStageK * 2, bar(kBFull + buf));
            }
            ++issued[buf];
          }
        }
        // the copies issued land before the CTA leaves, after an abort too
        for (int i = 0; i < 2; ++i)
          if (issued[i]) mbar_wait_quiet(bar(kBFull + i), (issued[i] - 1) & 1u, kDrainLimitNs);
      }
      __syncwarp();
    }
  } else {  // --------------------------------------------------------- workers
    if constexpr (split_regs(NT)) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kWorkerRegs));
    // group 0 of this thread's row (TMEM lane) and a quarter of the columns, over the chunks of a
    // unit so far (the other groups stay in TMEM)
    constexpr int kCols = NT / 4;
    const int q4 = warp & 3, c0 = (warp >> 2) * kCols;
    int top[kCols];
#pragma unroll
    for (int j = 0; j < kCols; ++j) top[j] = 0;
    Cursor<KC> cur(a, units, zero);
    double x[8];
    if (cur.u < units) cur.load(a, x);
    uint32_t it = 0, nflush = 0;

    // After a chunk: group 0 is moved to `top`, the carries of the other groups to their
    // neighbours, exactly in fp32 (a group is below 2^24 - 2^17, its carry at most 2^17), which
    // leaves at most 64 in each, so that the next chunk accumulates onto them without rounding.
    // After the last chunk of a unit: everything to doubles in C.
    auto flush = [&](int u, bool last) -> bool {
      if (!wait_for(bar(kAccFull), nflush & 1u, a)) return false;
      ++nflush;
      __syncwarp();
      tc_fence_after();
      const uint32_t t0 = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0;
      if (!last) {
#pragma unroll
        for (int h = 0; h < kCols; h += 4) {
          uint32_t r[kD][4];
#pragma unroll
          for (int g = 0; g < kD; ++g) tmem_ld4(t0 + (uint32_t)(g * NT + h), r[g]);
          tmem_wait_ld();
          float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int g = kD - 1; g > 0; --g) {
            float d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float v = __uint_as_float(r[g][j]) + c[j];
              c[j] = (fmaf(v, 0x1p-7f, 12582912.f)) - 12582912.f;  // rint(v / 128)
              d[j] = fmaf(c[j], -128.f, v);
            }
            tmem_st4(t0 + (uint32_t)(g * NT + h), d);
          }
          const float zero[4] = {0.f, 0.f, 0.f, 0.f};
          tmem_st4(t0 + (uint32_t)h, zero);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            top[h + j] += __float2int_rn(__uint_as_float(r[0][j])) + __float2int_rn(c[j]);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kAccEmpty));
        return true;
      }
      const int n0 = (u % a.ntiles) * NT + c0;
      const int m = (u / a.ntiles) % a.mtiles, sp = u / (a.ntiles * a.mtiles);
      const int row = m * kTileM + q4 * 32 + lane;
      const bool rv = row < a.M;
      const int b = rv ? row / a.Mb : 0, r = rv ? row - b * a.Mb : 0;
      const int ea = (rv ? (a.eA ? scale_exp(__ldg(a.eA + row)) : 1023) : 0) - 1086;
      double* Crow = a.C + (long long)sp * a.sCs + (long long)b * a.sCb + (long long)r * a.sCm + n0;
      int rmax = 0;
      // exponents of the result per (b, column), its rows scaled as the k of the next product that
      // they are: the lanes of a warp span one or two b when a b has at least 32 rows
      const int rs = rv && a.row_s ? (int)(__ldg(a.row_s + r) >> 20) : 0;
      const int b_lo = __shfl_sync(0xffffffffu, b, 0);
      const bool wide = a.Mb >= 32;
      const bool two = __any_sync(0xffffffffu, rv && b != b_lo);
      int mx0 = 0, mx1 = 0;
#pragma unroll
      for (int h = 0; h < kCols; h += 4) {
        uint32_t r[kD][4];
#pragma unroll
        for (int g = 0; g < kD; ++g) tmem_ld4(t0 + (uint32_t)(g * NT + h), r[g]);
        tmem_wait_ld();
        if (h + 4 >= kCols) {  // everything is in registers: the next unit's MMAs may start
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(kAccEmpty));
        }
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int n = n0 + h + j;
          long long lo = 0, hi = 0;
          add_group<21>(lo, r[4][j]);
          add_group<14>(lo, r[5][j]);
          add_group<7>(lo, r[6][j]);
          add_group<0>(lo, r[7][j]);
          hi = (lo >> 28) + (long long)top[h + j] * (1ll << 21);
          add_group<21>(hi, r[0][j]);
          add_group<14>(hi, r[1][j]);
          add_group<7>(hi, r[2][j]);
          add_group<0>(hi, r[3][j]);
          top[h + j] = 0;
          // (columns past N, whose digits are zero, take the last column's exponent)
          v[j] = fixed_to_double(hi, (uint32_t)lo & 0x0fffffffu,
                                 ea + (a.eB ? scale_exp(__ldg(a.eB + (n < a.N ? n : a.N - 1))) : 1023));
          if (a.exq) {
            int e = rv ? exp_of(v[j]) : 0;
            rmax = max(rmax, e);
            e = max(e - rs, 0);
            if (wide) {
              const int r0 = __reduce_max_sync(0xffffffffu, b == b_lo ? e : 0);
              if (lane == h + j) mx0 = r0;
              if (two) {
                const int r1 = __reduce_max_sync(0xffffffffu, b != b_lo ? e : 0);
                if (lane == h + j) mx1 = r1;
              }
            } else if (rv && n < a.N) {
              atomicMax(a.exq + (size_t)b * a.exq_ld + n, e);
            }
          }
        }
        if (a.sub && rv) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (n0 + h + j < a.N) v[j] = Crow[h + j] - v[j];
        }
        if (rv) {
          if (a.vecC && n0 + h + 3 < a.N) {
            *(double2*)(Crow + h) = make_double2(v[0], v[1]);
            *(double2*)(Crow + h + 2) = make_double2(v[2], v[3]);
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (n0 + h + j < a.N) Crow[h + j] = v[j];
          }
        }
      }
      if (a.exq) {
        if (wide && lane < kCols && n0 + lane < a.N) {
          atomicMax(a.exq + (size_t)b_lo * a.exq_ld + n0 + lane, mx0);
          if (two) atomicMax(a.exq + (size_t)(b_lo + 1) * a.exq_ld + n0 + lane, mx1);
        }
        if (rv && rmax > __ldcg(a.exm + r)) atomicMax(a.exm + r, rmax);
      }
      return true;
    };

    bool pend = false, pend_last = false;
    int pend_u = 0, c = 0;
    const uint32_t dst = KC ? sw64(tid >> 2, tid & 3) : sw64(tid & 127, tid >> 7);
    const uint32_t* ks = a.ks + 8 * (KC ? tid & 3 : tid >> 7);
    // Wide tiles: the last flush behind the loop, a second copy of its code (units of 128 x 48 take
    // 7 % less so); narrow ones, whose products are short, in the loop's last turn.
    constexpr bool kTail = split_regs(NT);
    for (;;) {
      const bool more = cur.u < units;
      if (!more && (kTail || !pend)) break;
      const int u = cur.u;
      bool last = false;
      if (more) {
        const uint32_t buf = it & 1u, ph = (it >> 1) & 1u;
        if (!wait_for(bar(kEmpty + buf), ph ^ 1u, a)) {
          pend = false;
          break;
        }
        const uint32_t sa = smem0 + buf * stage_bytes;
        last = cur.last();
        Fixed8 f;
        if (scaled) to_fixed8(x, cur.e20, ks + cur.st * kStageK, a.k64, f);
        else to_fixed8(x, cur.e20, a.k64, f);
        cur.next(a, units);
        if (cur.u < units) cur.load(a, x);  // the next stage's elements, in flight over a stage
        store_digits(f, [&](int d, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(sa + dst + d * (kTileM * 64)),
                       "r"(w0), "r"(w1), "r"(w2), "r"(w3)
                       : "memory");
        });
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kAFull + buf));
        ++it;
      }
      if (pend) {
        pend = false;
        if (!flush(pend_u, pend_last)) break;
      }
      if (!more) break;
      if (last || ++c == kChunkStages) {
        pend = true;
        pend_u = u;
        pend_last = last;
        c = 0;
      }
    }
    if (kTail && pend) flush(pend_u, pend_last);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kWorkers) tmem_dealloc<0>(tmem, 512);
}

// ------------------------------------------------------------------ exponents and planes
// Largest biased exponents of the columns (by_col: atomic maxima into zeroed words) or of the
// rows of up to three matrices, their elements scaled by the powers of two of the contraction's k
// (columns: C, by 2^s of the row; rows: h, by 2^-s of the column; minus: G's columns by 2^-s).
struct ExpJob {
  const double* S;
  long long ld;
  long long rows;
  int cols, by_col;
  int* out;
  KScale k;
  int minus;
};
struct ExpJobs {
  ExpJob j[3];
};
constexpr int kExpRows = 64;  // rows of a column job per CTA

__device__ __forceinline__ int scale_of(const KScale& k, int i) { return (int)(k.kp[i] >> 20); }
// The exponent scaled by 2^s; of a zero 0.
__device__ __forceinline__ int exp_scaled(double x, int s) {
  const int e = exp_of(x);
  return e ? max(e + s, 1) : 0;
}
// The least exponent word of an operand scaled upwards, so that its zeros (which have no hidden bit)
// are shifted out whatever their scale.
__device__ __forceinline__ int least_up(const int* info) { return 64 + info[1]; }

__global__ void __launch_bounds__(256) k_exps(ExpJobs jobs) {
  const int scales = scales_word(jobs.j[blockIdx.y].k.info);
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  const bool s = scales + z != 0;
  const ExpJob jb = jobs.j[blockIdx.y + z];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  if (jb.by_col) {
    __shared__ int red[8][32];
    const int ncb = (jb.cols + 31) / 32;
    const long long tiles = (long long)ncb * ((jb.rows + kExpRows - 1) / kExpRows);
    const int least = s && !jb.minus ? least_up(jb.k.info) : 0;
    for (long long t = bx; t < tiles; t += gridDim.x) {
      const int c = (int)(t % ncb) * 32 + tx;
      const long long r0 = t / ncb * kExpRows;
      int m = least;
      if (c < jb.cols) {
#pragma unroll
        for (int i = 0; i < kExpRows / 8; ++i) {
          const long long r = r0 + ty + 8 * i;
          if (r < jb.rows) {
            const double v = jb.S[r * jb.ld + c];
            const int sr = s ? scale_of(jb.k, (int)r) : 0;
            m = max(m, s ? exp_scaled(v, jb.minus ? -sr : sr) : exp_of(v));
          }
        }
      }
      red[ty][tx] = m;
      __syncthreads();
      if (ty == 0 && c < jb.cols) {
#pragma unroll
        for (int i = 1; i < 8; ++i) m = max(m, red[i][tx]);
        atomicMax(jb.out + c, m);
      }
      __syncthreads();
    }
  } else {
    for (long long r = (long long)bx * 8 + ty; r < jb.rows; r += (long long)gridDim.x * 8) {
      const double* row = jb.S + r * jb.ld;
      int m = 0;
#pragma unroll 4
      for (int c = tx; c < jb.cols; c += 32) {
        const double v = __ldg(row + c);
        m = max(m, s ? exp_scaled(v, -scale_of(jb.k, c)) : exp_of(v));
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (tx == 0) jb.out[r] = m;
    }
  }
}

// ------------------------------------------------------------------ scales of the AO indices
// Fixed point relative to the largest element of a row loses the small ones, and rows of B (and
// columns of C) in an AO basis whose functions are of very different norm hold both: with B and h
// scaled by w_mu w_nu and C by 1 / w_nu, spread over 1e8, builds were off by 1e-10, in double by 1e-15
// whatever the spread.  So the contractions over AO indices take B, h, X and G times 2^-s and C
// times 2^s, exactly, in the exponents' subtraction that splits them (their scaled products are the
// same numbers).  s_mu is half the exponent of the largest B^P_mu,mu, or, where B's off-diagonal
// elements do not bear that out (|B_mu,nu| <= 2^(s_mu + s_nu) holds for integrals), what brings the
// row's largest element to the level of B's: it moves with the functions' norms, so that errors do
// not depend on them.  Where s spans no more than kEvenSpan it is taken as zero, and the operands
// and results are those of unscaled products.
constexpr int kEvenSpan = 3;
constexpr int kScaleMax = 1000;  // (the shifts stay below 4096)
// rm, dm: largest exponents of the rows and of the diagonal elements, `copies` of each, the first of
// which takes the others' maxima.  Leaves in k: info = {whether
// any s is not zero, the largest}; s >= 0; kp and kn, s 2^20 and -s 2^20, padded with zeros.
__global__ void __launch_bounds__(1024) k_scales(int* rm, int* dm, int copies, int N, int* info,
                                                 uint32_t* kp, uint32_t* kn) {
  __shared__ int red[32];
  auto all_max = [&](int v) {
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
    __syncthreads();
    v = red[threadIdx.x % 32];
    return __reduce_max_sync(0xffffffffu, v);
  };
  int R = 0;
  for (int i = threadIdx.x; i < N; i += 1024) {  // (a thread's own i throughout)
    int m = 0, e = 0;
#pragma unroll 4
    for (int c = 0; c < copies; ++c) {
      m = max(m, rm[(size_t)c * N + i]);
      e = max(e, dm[(size_t)c * N + i]);
    }
    rm[i] = m;
    dm[i] = e;
    if (m < kNanMark) R = max(R, m);
  }
  R = all_max(R);
  int least = -(1 << 20), most = -(1 << 20);  // of -s and s
  auto raw = [&](int i) { return max(dm[i], 2 * rm[i] - R) >> 1; };
  auto counts = [&](int i) { return rm[i] > 0 && rm[i] < kNanMark; };  // (a row of zeros: any s)
  for (int i = threadIdx.x; i < N; i += 1024)
    if (counts(i)) {
      least = max(least, -raw(i));
      most = max(most, raw(i));
    }
  const int lo = -all_max(least), span = all_max(most) - lo;
  const bool on = span > kEvenSpan;
  const int hi = span < kScaleMax ? span : kScaleMax;
  for (int i = threadIdx.x; i < kscale_pad(N); i += 1024) {
    const int v = on && i < N && counts(i) ? min(raw(i) - lo, hi) : 0;
    kp[i] = (uint32_t)v << 20;
    kn[i] = 0u - ((uint32_t)v << 20);
  }
  if (threadIdx.x == 0) {
    info[0] = on;
    info[1] = on ? hi : 0;
  }
}

// Rows of N elements (row r: AO index r mod N) of a B of whole rows, or of h: a warp per row.  FIRST:
// the largest exponents of the rows (into out, unless null), of the AO indices' rows and of their
// diagonal elements (atomic maxima into zeroed words, `copies` of them, which k_scales puts together:
// with one copy the first rows of all CTAs queued for the same few lines, 140 us instead of 95 for
// 4000 slices of 97).  The second pass: those of the rows scaled by
// 2^-s of the column, where any s is not zero.  TRI: rows of packed lower triangles, the part above
// the diagonal gathered.  Bound by memory: 2000 slices of 700 1.2 ms a pass.
template <bool TRI, bool FIRST>
__global__ void __launch_bounds__(256) k_row_exps(const double* __restrict__ B, long long rows, int N,
                                                  int* out, int* rm, int* dm, int copies, KScale k) {
  const int z = chain_begin();
  if (!FIRST && !k.info[z]) return;
  if (FIRST) {
    rm += (size_t)(blockIdx.x % copies) * N;
    dm += (size_t)(blockIdx.x % copies) * N;
  }
  const int tx = threadIdx.x % 32;
  const long long npk = (long long)N * (N + 1) / 2;
  for (long long r = blockIdx.x * 8 + threadIdx.x / 32 + z; r < rows; r += (long long)gridDim.x * 8) {
    const long long P = r / N;
    const int mu = (int)(r - P * N);
    const double* row = TRI ? B + P * npk + (long long)mu * (mu + 1) / 2 : B + r * N;
    const int own = TRI ? mu + 1 : N;
    int m = 0;
    auto take = [&](double v, int c) { m = max(m, FIRST ? exp_of(v) : exp_scaled(v, -scale_of(k, c))); };
#pragma unroll 4
    for (int c = tx; c < own; c += 32) take(__ldg(row + c), c);
    if (TRI) {
#pragma unroll 4
      for (int c = own + tx; c < N; c += 32)
        take(__ldg(B + P * npk + (long long)c * (c + 1) / 2 + mu), c);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (tx != 0) continue;
    if (out) out[r] = m;
    if (FIRST) {
      if (m > *(volatile int*)(rm + mu)) atomicMax(rm + mu, m);
      const int e = exp_of(__ldg(row + mu));
      if (e < kNanMark && e > *(volatile int*)(dm + mu)) atomicMax(dm + mu, e);
    }
  }
}

// The rows of symmetric slices stored as packed lower triangles, the passes of k_row_exps: one CTA
// per slice, the slice's maxima in shared memory, and its diagonal's (FIRST).
// (A wave of slices takes its CTAs' time however few they are: 1500 functions 2.1 ms for 500 slices as
// for 1000, by rows 1.6 and 3.2; 700 functions 0.51 and 0.53, by rows 0.30 and 0.6.)
constexpr int kPackedFewSlices = 700;
template <bool FIRST>
__global__ void __launch_bounds__(256) k_packed_exps(const double* __restrict__ Bp, int Q, int N,
                                                     int* out, int* rm, int* dm, int copies,
                                                     KScale k) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  extern __shared__ int ex[];
  if (!FIRST && !k.info[z]) return;
  if (FIRST) {
    rm += (size_t)(bx % copies) * N;
    dm += (size_t)(bx % copies) * N;
  }
  const long long npk = (long long)N * (N + 1) / 2;
  for (int P = bx; P < Q; P += gridDim.x) {
    for (int i = threadIdx.x; i < N; i += 256) ex[i] = 0;
    __syncthreads();
    const double* B = Bp + (size_t)P * npk;
    for (int mu = threadIdx.x / 32; mu < N; mu += 8) {
      const double* row = B + (long long)mu * (mu + 1) / 2;
      const int smu = FIRST ? 0 : scale_of(k, mu);
      int m = 0;
      for (int nu = threadIdx.x % 32; nu <= mu; nu += 32) {
        const double v = __ldg(row + nu);
        int e = (__double2hiint(v) >> 20) & 0x7ff, f = e;  // (marked at the end)
        if (!FIRST) {
          e = exp_scaled(v, -scale_of(k, nu));
          f = exp_scaled(v, -smu);
        }
        m = max(m, e);
        if (f > *(volatile int*)(ex + nu)) atomicMax(ex + nu, f);
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (threadIdx.x % 32 == 0) {
        atomicMax(ex + mu, m);
        if (FIRST) ex[N + mu] = exp_of(__ldg(row + mu));
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += 256) {
      const int e = FIRST && ex[i] == 2047 ? kNanMark : ex[i];
      out[(size_t)P * N + i] = e;
      if (FIRST) {
        const int ed = ex[N + i];
        if (e > *(volatile int*)(rm + i)) atomicMax(rm + i, e);
        if (ed < kNanMark && ed > *(volatile int*)(dm + i)) atomicMax(dm + i, ed);
      }
    }
    __syncthreads();
  }
}

// Address (in halves) of digit 0 of column n, elements 8 kc .. 8 kc + 7 of k in the stage
// images; digit d is d NT 32 halves behind it.
__device__ __forceinline__ size_t img_addr(int n, int kc, int NT, int nstages) {
  const int nt = n / NT, r = n - nt * NT;
  return (((size_t)nt * nstages + (kc >> 2)) * (size_t)(kD * NT * 64) + sw64(r, kc & 3)) / 2;
}
// ks: the words of the 8 elements' scales, or null.
__device__ __forceinline__ void put_planes(const double (&x)[8], int em, const uint32_t* ks,
                                           uint32_t k64, __half* img, size_t at, int NT) {
  Fixed8 f;
  if (ks) to_fixed8(x, split_exp(em), ks, k64, f);
  else to_fixed8(x, split_exp(em), k64, f);
  store_digits(f, [&](int d, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
    *(uint4*)(img + at + (size_t)d * NT * kStageK) = make_uint4(w0, w1, w2, w3);
  });
}

// Stage images of a matrix S[k sk + n sn]: a thread per column and 8 elements of k (columns past
// N and elements past K are zero; ex null: exponent 1023), scaled by 2^s of its k (minus: 2^-s).
constexpr int kZeroExp = 2047;  // the exponent word of the columns that are only padding
__global__ void __launch_bounds__(256) k_digit_planes(const double* __restrict__ S, long long sk,
                                                      long long sn, int K, int N, uint32_t k64,
                                                      const int* __restrict__ ex, KScale ksc,
                                                      int minus, __half* img, int NT, int ntiles,
                                                      int nstages) {
  const int scales = scales_word(ksc.info);
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  const bool on = scales + z != 0;
  const int W = NT * ntiles;
  const uint32_t* ks = !on ? nullptr : minus ? ksc.kp : ksc.kn;
  const long long tot = (long long)W * nstages * 4;
  for (long long i = bx * 256ll + threadIdx.x; i < tot; i += 256ll * gridDim.x) {
    const int kc = (int)(i / W), n = (int)(i - (long long)kc * W);
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = 8 * kc + j;
      x[j] = (n < N && k < K) ? S[(long long)k * sk + (long long)n * sn] : 0.0;
    }
    put_planes(x, n < N ? (ex ? ex[n] : 1023) : kZeroExp, ks ? ks + 8 * kc : nullptr, k64, img,
               img_addr(n, kc, NT, nstages), NT);
  }
}

// The same with the exponents found on the way, for K <= kFuseK: a CTA per 32 columns passes over
// them twice (the second time from L1 or L2), so that a short product needs one launch less, and the
// call no memsets; but few CTAs, each with all of K, take longer the larger K is (a whole build with
// separate launches / so: nbf 24 99 / 90 us, 100 134 / 123, 300 166 / 165, 500 253 / 263, 640 233 /
// 248, 1200 472 / 507);
// the CTAs from col_ctas on find the rows' exponents of a second matrix (R, rows of `rows_k`
// elements), a warp per row, and those behind them clear `zero`.
constexpr int kFuseK = 320;
__global__ void __launch_bounds__(256) k_exps_planes(const double* __restrict__ S, long long ld,
                                                     int K, int ncols, int N, uint32_t k64,
                                                     int* ex, KScale ksc, int minus, __half* img,
                                                     int NT, int nstages, int col_ctas, const double* __restrict__ R,
                                                     int rows, int rows_k, int* ex_rows,
                                                     int row_ctas, const ZeroJob zero) {
  const int scales = scales_word(ksc.info);
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  const bool on = scales + z != 0;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  if (bx >= col_ctas + row_ctas) {
    zero_ranges(zero, bx - col_ctas - row_ctas, (int)gridDim.x - col_ctas - row_ctas);
    return;
  }
  if (bx >= col_ctas) {
    for (int r = (bx - col_ctas) * 8 + ty; r < rows; r += row_ctas * 8) {
      int m = 0;
      for (int c0 = tx; c0 < rows_k; c0 += 128) {
        double v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          v[i] = c0 + 32 * i < rows_k ? __ldg(R + (long long)r * rows_k + c0 + 32 * i) : 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          int e = exp_of(v[i]);
          if (on && e) e = max(e - scale_of(ksc, c0 + 32 * i), 1);  // (not a zero: within the row)
          m = max(m, e);
        }
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (tx == 0) ex_rows[r] = m;
    }
    return;
  }
  __shared__ int red[8][32];
  const int n = bx * 32 + tx;  // columns past N: to the width of the images
  int m = 0;
  if (n < ncols) {
    for (int k0 = ty; k0 < K; k0 += 32) {
      double v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = k0 + 8 * i < K ? S[(long long)(k0 + 8 * i) * ld + n] : 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int e = exp_of(v[i]);
        if (on && e) {
          const int sk = scale_of(ksc, k0 + 8 * i);
          e = max(e + (minus ? -sk : sk), 1);
        }
        m = max(m, e);
      }
    }
  }
  if (on && !minus) m = max(m, least_up(ksc.info));
  red[ty][tx] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) m = max(m, red[i][tx]);
  if (ty == 0 && n < ncols) ex[n] = m;
  if (n >= (N + NT - 1) / NT * NT) return;  // (the images' width: every tile is NT columns)
  const uint32_t* ks = !on ? nullptr : minus ? ksc.kp : ksc.kn;
  for (int kc = ty; kc < nstages * 4; kc += 8) {
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = 8 * kc + j;
      x[j] = (n < N && k < K) ? S[(long long)k * ld + n] : 0.0;
    }
    put_planes(x, n < N ? m : kZeroExp, ks ? ks + 8 * kc : nullptr, k64, img,
               img_addr(n, kc, NT, nstages), NT);
  }
}

// ------------------------------------------------------------------ between b and G
// Two passes over b in one launch.  CTAs below w_ctas: w^P_p = sum_r Acoef_pr b^P_rr of their
// slices and the largest biased exponents of w.  The others: partial sums over the slices of one
// split of J_pq = sum_P b_pp b_qq and K_pq = sum_P b_pq^2 for the entries q <= p (256 of them a
// CTA), and the largest biased exponent of b_pq.
__global__ void __launch_bounds__(256) k_w_jk64(const double* __restrict__ b, int np, int A,
                                                const double* __restrict__ Ac, double* W,
                                                int* wmax, int w_ctas, int splits, double* part,
                                                int* bmax) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  extern __shared__ double dv[];
  if (bx < w_ctas) {
    for (int P = bx; P < np; P += w_ctas) {
      const double* bp = b + (size_t)P * A * A;
      for (int r = threadIdx.x; r < A; r += 256) dv[r] = bp[(size_t)r * A + r];
      __syncthreads();
      for (int p = threadIdx.x + z; p < A; p += 256) {
        double w[4] = {0.0, 0.0, 0.0, 0.0};  // four chains: the FP64 latency bounds this part
        const double* row = Ac + p;          // Acoef is symmetric: read down its columns
        int r = 0;
        for (; r + 4 <= A; r += 4)
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = fma(row[(size_t)(r + i) * A], dv[r + i], w[i]);
        for (; r < A; ++r) w[0] = fma(row[(size_t)r * A], dv[r], w[0]);
        const double t = (w[0] + w[1]) + (w[2] + w[3]);
        W[(size_t)P * A + p] = t;
        const int e = exp_of(t);
        if (e > *(volatile int*)(wmax + p)) atomicMax(wmax + p, e);
      }
      __syncthreads();
    }
    return;
  }
  const int cta = bx - w_ctas, split = cta % splits;
  const int tri = A * (A + 1) / 2, i = cta / splits * 256 + threadIdx.x;
  if (i >= tri) return;
  int p = (int)((sqrtf(8.0f * (float)i + 1.0f) - 1.0f) * 0.5f);
  while (p * (p + 1) / 2 > i) --p;
  while ((p + 1) * (p + 2) / 2 <= i) ++p;
  const int q = i - p * (p + 1) / 2;
  const int P0 = (int)((long long)np * split / splits);
  const int P1 = (int)((long long)np * (split + 1) / splits);
  double sj[2] = {0.0, 0.0}, sk[2] = {0.0, 0.0};
  int m = 0;
  const size_t AA = (size_t)A * A, opq = (size_t)p * A + q, op = (size_t)p * A + p,
               oq = (size_t)q * A + q;
  int P = P0;
  for (; P + 4 <= P1; P += 4) {
    double v[4], dp[4], dq[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double* bp = b + (size_t)(P + u) * AA;
      v[u] = bp[opq];
      dp[u] = bp[op];
      dq[u] = bp[oq];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      sj[u & 1] = fma(dp[u], dq[u], sj[u & 1]);
      sk[u & 1] = fma(v[u], v[u], sk[u & 1]);
      m = max(m, exp_of(v[u]));
    }
  }
  for (; P < P1; ++P) {
    const double* bp = b + (size_t)P * AA;
    const double v = bp[opq];
    sj[0] = fma(bp[op], bp[oq], sj[0]);
    sk[0] = fma(v, v, sk[0]);
    m = max(m, exp_of(v));
  }
  double* o = part + (size_t)split * 2 * tri;
  o[i] = sj[0] + sj[1];
  o[tri + i] = sk[0] + sk[1];
  atomicMax(bmax + i, m);
}

// J and K (both triangles) from the splits' partial sums, in order, and the exponent bounds of
// the columns of Y: |Y_qp| <= |Bcoef_qp| |b_qp| (+ |w_p| on the diagonal).
__global__ void __launch_bounds__(256) k_jk_final64(const double* __restrict__ part, int splits,
                                                    int A, const double* __restrict__ Bc,
                                                    const int* __restrict__ bmax,
                                                    const int* __restrict__ wmax, double* J,
                                                    double* K, int* eY, int jk_blocks,
                                                    int first) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  const int tri = A * (A + 1) / 2;
  if (bx < jk_blocks) {
    const int i = bx * 256 + threadIdx.x;
    if (i >= tri) return;
    int p = (int)((sqrtf(8.0f * (float)i + 1.0f) - 1.0f) * 0.5f);
    while (p * (p + 1) / 2 > i) --p;
    while ((p + 1) * (p + 2) / 2 <= i) ++p;
    const int q = i - p * (p + 1) / 2;
    double sj = 0.0, sk = 0.0;
#pragma unroll 4
    for (int s = 0; s < splits; ++s) {
      sj += part[(size_t)s * 2 * tri + i];
      sk += part[(size_t)s * 2 * tri + tri + i];
    }
    const double j = first ? sj : J[(size_t)p * A + q] + sj;
    const double k = first ? sk : K[(size_t)p * A + q] + sk;
    J[(size_t)p * A + q] = j;
    K[(size_t)p * A + q] = k;
    if (p != q) {
      J[(size_t)q * A + p] = j;
      K[(size_t)q * A + p] = k;
    }
    return;
  }
  const int p = (bx - jk_blocks) * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (p >= A) return;
  // 2^(f - 1022) bounds every |Y_qp|, f = e(Bcoef) + e(b) - 1022 for a product, one more for
  // the rounding of b_qp against b_pq and one for the sum with w
  int f = wmax[p];
  for (int q = lane; q < A; q += 32) {
    const int hi = p > q ? p : q, lw = p > q ? q : p;
    const int eb = bmax[hi * (hi + 1) / 2 + lw], ec = exp_of(Bc[(size_t)q * A + p]);
    f = max(f, eb >= kNanMark || ec >= kNanMark ? kNanMark : (ec && eb ? ec + eb - 1022 : 0));
  }
  f = __reduce_max_sync(0xffffffffu, f);
  if (lane == 0) eY[p] = f >= kNanMark ? kNanMark : (f + 2 > 2046 ? 2046 : f + 2);
}

// Stage images of Y over k = P Kpad + q: Y^P_qp = Bcoef_qp b^P_qp + delta_qp w^P_p, formed and
// split in one pass.
__global__ void __launch_bounds__(256) k_y_planes(const double* __restrict__ b, int np, int A,
                                                  int Kpad, uint32_t k64,
                                                  const double* __restrict__ Bc,
                                                  const double* __restrict__ W,
                                                  const int* __restrict__ eY, __half* img, int NT,
                                                  int ntiles, int nstages) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  const int Wd = NT * ntiles;
  const long long tot = (long long)Wd * nstages * 4;
  for (long long i = bx * 256ll + threadIdx.x; i < tot; i += 256ll * gridDim.x) {
    const int kc = (int)(i / Wd), n = (int)(i - (long long)kc * Wd);
    const int P = (int)(8ll * kc / Kpad), q0 = (int)(8ll * kc - (long long)P * Kpad);
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int q = q0 + j;
      x[j] = 0.0;
      if (n < A && q < A && P < np) {
        x[j] = Bc[(size_t)q * A + n] * b[((size_t)P * A + q) * A + n];
        if (q == n) x[j] += W[(size_t)P * A + n];
      }
    }
    put_planes(x, n < A ? eY[n] : kZeroExp, nullptr, k64, img, img_addr(n, kc, NT, nstages), NT);
  }
}

// C[i] += sum over the splits of part[s][i], i < tot: 8 threads per element take every eighth
// split, their sums added in order.
__global__ void __launch_bounds__(256) k_split_sum(const double* __restrict__ part, int splits,
                                                   long long tot, double* C) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  __shared__ double red[8][32];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const long long i = bx * 32ll + tx;
  double t = 0.0;
  if (i < tot) {
#pragma unroll 4
    for (int s = ty; s < splits; s += 8) t += part[(size_t)s * tot + i];
  }
  red[ty][tx] = t;
  __syncthreads();
  if (ty == 0 && i < tot) {
#pragma unroll
    for (int g = 1; g < 8; ++g) t += red[g][tx];
    C[i] += t;
  }
}

constexpr uint32_t kK64 = 0x64006400u;  // fp16 1024, twice

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  }();
  return n;
}
int grid_for(long long threads) {
  const long long nb = (threads + 255) / 256;
  return (int)(nb < 1 ? 1 : (nb < 152 * 16 ? nb : 152 * 16));
}

cudaError_t launch_exps(const ExpJob* jobs, int count, cudaStream_t s) {
  ExpJobs js{};
  long long nb = 1;
  for (int i = 0; i < count; ++i) {
    js.j[i] = jobs[i];
    const long long t = jobs[i].by_col ? (long long)((jobs[i].cols + 31) / 32) *
                                             ((jobs[i].rows + kExpRows - 1) / kExpRows)
                                       : (jobs[i].rows + 7) / 8;
    if (t > nb) nb = t;
  }
  launch_chained(k_exps, dim3((unsigned)(nb < 152 * 8 ? nb : 152 * 8), count), 256, 0, s, js);
  count_launch(1);
  return cudaGetLastError();
}

cudaError_t launch_planes(const double* S, long long sk, long long sn, int K, int N, const int* ex,
                          const KScale& k, int minus, void* img, cudaStream_t s) {
  const DigitShape sh = digit_shape(N, K);
  launch_chained(k_digit_planes, grid_for((long long)sh.NT * sh.ntiles * sh.nstages * 4), 256, 0, s,
      S, sk, sn, K, N, kK64, ex, k, minus, (__half*)img, sh.NT, sh.ntiles, sh.nstages);
  count_launch(1);
  return cudaGetLastError();
}

// ncols columns' exponents and the planes of the first N, K <= kFuseK; rows' exponents of R; zero
// cleared.  `first`: the first launch of a call.
cudaError_t launch_exps_planes(const double* S, long long ld, int K, int ncols, int N, int* ex,
                               const KScale& k, int minus, void* img, const double* R, int rows, int rows_k, int* ex_rows,
                               const ZeroJob& zero, bool first, cudaStream_t s) {
  const DigitShape sh = digit_shape(N, K);
  const int width = ncols > sh.NT * sh.ntiles ? ncols : sh.NT * sh.ntiles;
  const int cc = (width + 31) / 32, rc = (rows + 7) / 8;
  long long nz = 0;
  for (int i = 0; i < 4; ++i) nz += zero.n[i];
  const int zc = (int)(nz < 2048 * 32 ? (nz + 2047) / 2048 : 32);
  launch_chained_to(first ? 0 : kChainCtas, k_exps_planes, cc + rc + (zero.flag && !zc ? 1 : zc),
                    256, 0, s, S, ld, K, ncols, N, kK64, ex, k, minus, (__half*)img, sh.NT,
                    sh.nstages, cc, R, rows, rows_k, ex_rows, rc, zero);
  count_launch(1);
  return cudaGetLastError();
}

// Columns of a unit's tile: the width of the images' tiles or a divisor of it, whichever takes the
// units through the chip soonest.  Wide tiles split A less often; narrow ones fill more SMs and have
// less to do once the last stage is in.  Clocks measured per stage, per unit and (code not yet in the
// instruction caches) per launch, of tiles of 16, 32, 48 and 64.  With the images' width throughout:
// 120^3 27 us, 500 x 80 x 500 43, 640^3 65, 1200^3 194; by this rule 21, 35, 52, 194.
// (Measured before the wide tiles' registers, which make their stages a tenth shorter; that changes
// the choice in 9 of 1710 products tried, near ties.)
int tile_columns(int N, int imgNT, long long mtiles, int splits, int nstages) {
  constexpr int kStage[4] = {2400, 2800, 3150, 3850}, kUnit[4] = {3500, 6000, 10000, 13000},
                kCold[4] = {13000, 14000, 24000, 30000};
  const long long stages = (nstages + splits - 1) / splits;
  long long best = 0;
  int NT = imgNT;
  for (int w = imgNT; w >= 16; w -= 16) {
    if (imgNT % w) continue;
    const long long units = mtiles * ((N + w - 1) / w) * splits;
    const long long waves = (units + sm_count() - 1) / sm_count();
    const long long t =
        waves * (stages * kStage[w / 16 - 1] + kUnit[w / 16 - 1]) + kCold[w / 16 - 1];
    if (w == imgNT || t < best) {
      best = t;
      NT = w;
    }
  }
  return NT;
}

// Fills the tiling of `a` (its operands, K layout and output are set) and launches it.
cudaError_t launch_digit_gemm(DigitArgs a, long long K, cudaStream_t s) {
  const DigitShape sh = digit_shape(a.N, K);
  a.imgNT = sh.NT;
  a.nstages = sh.nstages;
  a.mtiles = (a.M + kTileM - 1) / kTileM;
  a.NT = tile_columns(a.N, sh.NT, a.mtiles, a.splits, sh.nstages);
  a.ntiles = (a.N + a.NT - 1) / a.NT;
  a.k64 = kK64;
  if (a.KB == 1) a.Kpad = sh.nstages * kStageK;
  auto even = [](long long v) { return (v & 1) == 0; };
  const bool kc = a.sAk == 1;
  a.vecA = kc && ((uintptr_t)a.A % 16) == 0 && even(a.sAb) && even(a.sAm) && even(a.sAkb);
  a.vecC = ((uintptr_t)a.C % 16) == 0 && even(a.sCs) && even(a.sCb) && even(a.sCm);
  size_t smem = 1024 + 2 * ((size_t)kABytes + (size_t)kD * a.NT * kStageK * 2) + 128;
  if (smem < 120 * 1024) smem = 120 * 1024;  // one CTA per SM: the TMEM allocation never waits
  if (!kc && a.KB != 1) return cudaErrorInvalidValue;
  using Fn = void (*)(const DigitArgs);
  static const Fn fns[2][4] = {
      {k_digit_gemm<false, 16>, k_digit_gemm<false, 32>, k_digit_gemm<false, 48>,
       k_digit_gemm<false, 64>},
      {k_digit_gemm<true, 16>, k_digit_gemm<true, 32>, k_digit_gemm<true, 48>,
       k_digit_gemm<true, 64>}};
  const Fn fn = fns[kc][a.NT / 16 - 1];
  const long long units = (long long)a.mtiles * a.ntiles * a.splits;
  const int grid = (int)(units < sm_count() ? units : sm_count());
  // The kernel's shared-memory limit is raised once per device; a launch that fails all the same
  // (the device was reset since) raises it again.
  static std::atomic<uint64_t> raised[2][4];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? 1ull << dev : 0;
  std::atomic<uint64_t>& mask = raised[kc][a.NT / 16 - 1];
  for (int attempt = 0; attempt < 2; ++attempt) {
    const bool raise = attempt > 0 || !(mask.load() & bit);
    if (raise) {
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      // the workers wait for the registers that they ask for: the launch has to hold the split's sum
      cudaFuncAttributes fa;
      e = cudaFuncGetAttributes(&fa, fn);
      if (e != cudaSuccess) return e;
      if (split_regs(a.NT) && fa.numRegs / 8 * 8 * dig_threads(a.NT) < 32 * (4 * kOtherRegs + kWorkers * kWorkerRegs))
        return cudaErrorInvalidConfiguration;
      mask |= bit;
    }
    launch_chained(fn, grid, dig_threads(a.NT), smem, s, a);
    e = cudaGetLastError();
    if (e == cudaSuccess || raise) break;
  }
  count_launch(1);
  return e;
}

#define CKE(x)                              \
  do {                                      \
    const cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_;       \
  } while (0)

}  // namespace

size_t digit_product_bytes(int M, int N, int K) {
  return align_up((size_t)M * 4) + align_up((size_t)N * 4) + digit_shape(N, K).bytes;
}

cudaError_t digit_product(int M, int N, int K, const double* A, long long sAm, long long sAk,
                          const double* B, long long sBk, long long sBn, double* C, long long ldc,
                          char* scratch, int* status, int* abort_flag, cudaStream_t s) {
  int* eA = (int*)scratch;
  int* eB = (int*)(scratch + align_up((size_t)M * 4));
  char* img = (char*)eB + align_up((size_t)N * 4);
  if (sAk != 1 || sBn == 1)  // a matrix read down its columns accumulates maxima
    CKE(cudaMemsetAsync(scratch, 0, (size_t)(img - scratch), s));
  ExpJob jobs[2] = {{B, sBk, K, N, 1, eB, {}, 0}, {A, sAm, M, K, 0, eA, {}, 0}};
  if (sBn != 1) jobs[0] = ExpJob{B, sBn, N, K, 0, eB, {}, 0};
  if (sAk != 1) jobs[1] = ExpJob{A, sAk, K, M, 1, eA, {}, 0};
  CKE(launch_exps(jobs, 2, s));
  CKE(launch_planes(B, sBk, sBn, K, N, eB, KScale{}, 0, img, s));
  DigitArgs a{};
  a.KB = 1; a.splits = 1;
  a.A = A; a.sAm = sAm; a.sAk = sAk; a.M = M; a.Mb = M; a.Kin = K; a.eA = eA;
  a.Bimg = (const __half*)img; a.eB = eB; a.N = N;
  a.C = C; a.sCm = ldc;
  a.status = status; a.abort_flag = abort_flag;
  return launch_digit_gemm(a, K, s);
}

// ------------------------------------------------------------------ reflectors
namespace {
constexpr int kRefBlk = 64;   // reflectors per block
constexpr int kRefCols = 4;   // columns of Z per CTA of k_reflect_w
// W = T (sum over the splits of part[s][n][c]) for the columns n of Z, c < 64 reflectors, and its
// stage images (k = c, two stages): the sums and W in shared memory, a thread per reflector and
// column; then a thread per column and 8 reflectors.  Bound by the FP64 units of a CTA's SM: 8
// columns a CTA and two a thread took 18.5 us at 120 columns, 21.4 at 1200; this 13.6 and 19.4.
__global__ void __launch_bounds__(256) k_reflect_w(const double* __restrict__ part, int splits,
                                                   int N, const double* __restrict__ T,
                                                   uint32_t k64, int* eW, __half* img, int NT,
                                                   int ntiles) {
  const int z = chain_begin(), bx = (int)blockIdx.x + z;
  __shared__ double Ts[kRefBlk][kRefBlk + 1];
  __shared__ double Ws[kRefCols][kRefBlk], Wt[kRefCols][kRefBlk];
  const int tid = threadIdx.x, n0 = bx * kRefCols;
  for (int i = tid; i < kRefBlk * kRefBlk; i += 256) Ts[i / kRefBlk][i % kRefBlk] = T[i + z];
  for (int i = tid; i < kRefCols * kRefBlk; i += 256) {
    const int n = n0 + i / kRefBlk, c = i % kRefBlk;
    double t = 0.0;
    if (n < N)
      for (int s = 0; s < splits; ++s) t += part[((size_t)s * N + n) * kRefBlk + c];
    Ws[i / kRefBlk][c] = t;
  }
  __syncthreads();
  {
    const int r = tid % kRefBlk, g = tid / kRefBlk;  // T is upper triangular
    double a0 = 0.0, a1 = 0.0;                       // two chains
    int c = r;
    for (; c + 1 < kRefBlk; c += 2) {
      a0 = fma(Ts[r][c], Ws[g][c], a0);
      a1 = fma(Ts[r][c + 1], Ws[g][c + 1], a1);
    }
    if (c < kRefBlk) a0 = fma(Ts[r][c], Ws[g][c], a0);
    Wt[g][r] = a0 + a1;
  }
  __syncthreads();
  if (tid < kRefCols * 8) {  // (a whole warp; 8 neighbouring lanes per column)
    const int j = tid / 8, kc = tid % 8, n = n0 + j;
    double x[8];
    int m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = Wt[j][8 * kc + i];
      m = max(m, exp_of(x[i]));
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (n < N && kc == 0) eW[n] = m;
    if (n < NT * ntiles) put_planes(x, n < N ? m : kZeroExp, nullptr, k64, img, img_addr(n, kc, NT, 2), NT);
  }
}
int reflect_splits(int N, int stages) {
  const int mt = (N + kTileM - 1) / kTileM;
  int sp = 152 / mt;
  if (sp > (stages + 1) / 2) sp = (stages + 1) / 2;
  return sp < 1 ? 1 : sp;
}
struct ReflectLayout {
  size_t y, w, eW, part, total;
};
ReflectLayout reflect_layout(int N) {
  ReflectLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = align_up(off + bytes);
    return o;
  };
  const DigitShape one = digit_shape(kRefBlk, N);
  L.y = take((size_t)((N + kRefBlk - 1) / kRefBlk) * one.bytes);
  L.w = take(digit_shape(N, kRefBlk).bytes);
  L.eW = take((size_t)N * 4);
  L.part = take((size_t)reflect_splits(N, one.nstages) * N * kRefBlk * 8);
  L.total = off;
  return L;
}
}  // namespace

size_t digit_reflect_bytes(int N) { return reflect_layout(N).total; }

cudaError_t digit_reflect(int N, int nref, const double* Yr, const double* T, double* V, char* img,
                          int* status, int* abort_flag, cudaStream_t s) {
  const ReflectLayout L = reflect_layout(N);
  const int nblk = (nref + kRefBlk - 1) / kRefBlk;
  // every block's reflectors as column tiles of one image over k = 0 .. N - 1 (|y| <= 1)
  const DigitShape ysh = digit_shape(kRefBlk, N);  // NT 64, one tile per block
  const int W = nblk * kRefBlk;
  launch_chained(k_digit_planes, grid_for((long long)W * ysh.nstages * 4), 256, 0, s,
      Yr, 1, N, N, nref, kK64, nullptr, KScale{}, 0, (__half*)(img + L.y), kRefBlk, nblk,
      ysh.nstages);
  count_launch(1);
  CKE(cudaGetLastError());
  const DigitShape wsh = digit_shape(N, kRefBlk);
  double* part = (double*)(img + L.part);
  int* eW = (int*)(img + L.eW);
  for (int b = nblk - 1; b >= 0; --b) {
    const int k0 = b * kRefBlk, R0 = k0 + 1;
    const int st0 = R0 / kStageK, Ra = st0 * kStageK;  // (the rows Ra .. R0 - 1 of Y are zero)
    const int stages = ysh.nstages - st0;
    // part[s][n][c] = sum over the split's rows of Z[j][n] Y[j][c]
    DigitArgs a{};
    a.KB = 1;
    a.splits = reflect_splits(N, stages);
    a.A = V + (size_t)Ra * N; a.sAm = 1; a.sAk = N; a.M = N; a.Mb = N; a.Kin = N - Ra;
    a.Bimg = (const __half*)(img + L.y) +
             ((size_t)b * ysh.nstages + st0) * (kD * kRefBlk * kStageK);
    a.N = kRefBlk;
    a.C = part; a.sCs = (long long)N * kRefBlk; a.sCm = kRefBlk;
    a.status = status; a.abort_flag = abort_flag;
    CKE(launch_digit_gemm(a, N - Ra, s));
    launch_chained(k_reflect_w, (wsh.NT * wsh.ntiles + kRefCols - 1) / kRefCols, 256, 0, s,
        part, a.splits, N, T + (size_t)b * kRefBlk * kRefBlk, kK64, eW, (__half*)(img + L.w), wsh.NT,
        wsh.ntiles);
    count_launch(1);
    CKE(cudaGetLastError());
    // Z[R0 ..] -= Y W
    DigitArgs u{};
    u.KB = 1;
    u.splits = 1;
    u.A = Yr + (size_t)k0 * N + R0; u.sAm = 1; u.sAk = N; u.M = N - R0; u.Mb = N - R0;
    u.Kin = nref - k0 < kRefBlk ? nref - k0 : kRefBlk;
    u.Bimg = (const __half*)(img + L.w); u.eB = eW; u.N = N;
    u.C = V + (size_t)R0 * N; u.sCm = N; u.sub = 1;
    u.status = status; u.abort_flag = abort_flag;
    CKE(launch_digit_gemm(u, kRefBlk, s));
  }
  return cudaSuccess;
}

namespace {
DigitArgs digit_args(char* ws, const Layout& L) {
  DigitArgs a{};
  a.KB = 1;
  a.splits = 1;
  a.status = &((DevHeader*)(ws + L.header))->status;
  a.abort_flag = &((DevHeader*)(ws + L.header))->abort_flag;
  return a;
}
}  // namespace

namespace {
// Scales of the AO indices from the exponents that the first pass left.
cudaError_t launch_scales(int* rm, int* dm, int copies, int N, const KScale& k, cudaStream_t s) {
  k_scales<<<1, 1024, 0, s>>>(rm, dm, copies, N, (int*)k.info, (uint32_t*)k.kp, (uint32_t*)k.kn);
  count_launch(1);
  return cudaGetLastError();
}
}  // namespace

cudaError_t digit_prepare_B(const Dims& d, const double* B, char* ws, const Layout& L,
                            cudaStream_t s) {
  int* out = (int*)(ws + L.eRow);
  const KScale k = kscale_at(ws + L.sB, d.N);
  // (X's space, free between builds, holds at least 8 N pb A bytes)
  const int copies = (long long)d.pb * d.A < 16 ? d.pb * d.A : 16;
  int *rm = (int*)(ws + L.X64), *dm = rm + (size_t)copies * d.N;
  CKE(cudaMemsetAsync(rm, 0, (size_t)2 * copies * d.N * 4, s));
  const int tri = d.layout == DONOF_B_PACKED;
  const long long rows = (long long)d.Q * d.N, nb = (rows + 7) / 8;
  const size_t smem = (size_t)d.N * 8;
  if (tri && smem > 47 * 1024) {  // (one limit for all sizes)
    CKE(cudaFuncSetAttribute(k_packed_exps<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             16384 * 8));
    CKE(cudaFuncSetAttribute(k_packed_exps<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             16384 * 8));
  }
  const dim3 slices(d.Q < 152 * 8 ? d.Q : 152 * 8), by_rows((unsigned)(nb < 152 * 8 ? nb : 152 * 8));
  for (int pass = 0; pass < 2; ++pass) {
    if (tri && d.Q >= kPackedFewSlices)
      (pass ? k_packed_exps<false> : k_packed_exps<true>)<<<slices, 256, smem, s>>>(
          B, d.Q, d.N, out, rm, dm, copies, k);
    else
      (tri ? (pass ? k_row_exps<true, false> : k_row_exps<true, true>)
           : (pass ? k_row_exps<false, false> : k_row_exps<false, true>))<<<by_rows, 256, 0, s>>>(
          B, rows, d.N, out, rm, dm, copies, k);
    count_launch(1);
    CKE(cudaGetLastError());
    if (pass == 0) CKE(launch_scales(rm, dm, copies, d.N, k, s));
  }
  return cudaSuccess;
}

cudaError_t digit_hc(const Dims& d, const double* h, const double* C, bool prepared, char* ws,
                     const Layout& L, ZeroJob zero, cudaStream_t s) {
  const int N = d.N;
  const KScale k = kscale_at(ws + (prepared ? L.sB : L.sH), N);
  if (!prepared) {  // no B in this workspace: the scales that h shows
    int *rm = (int*)(ws + L.eC64), *dm = (int*)(ws + L.exm);
    CKE(cudaMemsetAsync(ws + L.eC64, 0, L.exend - L.eC64, s));
    k_row_exps<false, true><<<(N + 7) / 8 < 152 * 8 ? (N + 7) / 8 : 152 * 8, 256, 0, s>>>(
        h, N, N, nullptr, rm, dm, 1, k);
    count_launch(1);
    CKE(cudaGetLastError());
    CKE(launch_scales(rm, dm, 1, N, k, s));
  }
  // exponents of C's columns (the operand planes, and lambda's rows) and of h's rows
  if (N <= kFuseK) {
    zero.add(ws + L.exq, L.exend - L.exq);
    CKE(launch_exps_planes(C, N, N, N, d.A, (int*)(ws + L.eC64), k, 0, ws + L.Cimg, h, N, N,
                           (int*)(ws + L.eH64), zero, true, s));
  } else {
    CKE(cudaMemsetAsync(ws + L.eC64, 0, L.exend - L.eC64, s));
    if (zero.flag) CKE(cudaMemsetAsync(zero.flag, 0, sizeof(int), s));
    for (int i = 0; i < 4; ++i)
      if (zero.n[i] > 0) CKE(cudaMemsetAsync(zero.p[i], 0, (size_t)zero.n[i] * 8, s));
    const ExpJob jobs[2] = {{C, N, N, N, 1, (int*)(ws + L.eC64), k, 0},
                            {h, N, N, N, 0, (int*)(ws + L.eH64), k, 0}};
    CKE(launch_exps(jobs, 2, s));
    CKE(launch_planes(C, N, 1, N, d.A, (const int*)(ws + L.eC64), k, 0, ws + L.Cimg, s));
  }
  DigitArgs a = digit_args(ws, L);
  a.A = h; a.sAm = N; a.sAk = 1; a.M = N; a.Mb = N; a.Kin = N;
  a.eA = (const int*)(ws + L.eH64);
  a.ks = k.kp; a.ks_on = k.info;
  a.Bimg = (const __half*)(ws + L.Cimg); a.eB = (const int*)(ws + L.eC64);
  a.N = d.A;
  a.C = (double*)(ws + L.hC); a.sCm = d.A;
  return launch_digit_gemm(a, N, s);
}

// X, b, J, K and G of the np slices from p0 on; Bblk: those slices, dense.
int digit_block(const Dims& d, const double* Bblk, int p0, int np, char* ws, const Layout& L,
                cudaStream_t s) {
#define CKI(x)                                    \
  do {                                            \
    if ((x) != cudaSuccess) return DONOF_ERR_CUDA; \
  } while (0)
  const int N = d.N, A = d.A;
  const KScale k = kscale_at(ws + L.sB, N);
  double* X = (double*)(ws + L.X64);
  double* b = (double*)(ws + L.b64);
  int* exq = (int*)(ws + L.exq);
  int* exm = (int*)(ws + L.exm);
  if (p0 > 0) CKI(cudaMemsetAsync(ws + L.exq, 0, L.exend - L.exq, s));
  {  // X[P][mu][q] = sum_nu B[P][mu][nu] C[nu][q]
    DigitArgs a = digit_args(ws, L);
    a.A = Bblk; a.sAb = (long long)N * N; a.sAm = N; a.sAk = 1;
    a.M = np * N; a.Mb = N; a.Kin = N;
    a.eA = (const int*)(ws + L.eRow) + (size_t)p0 * N;
    a.ks = k.kp; a.ks_on = k.info;
    a.Bimg = (const __half*)(ws + L.Cimg); a.eB = (const int*)(ws + L.eC64);
    a.N = A;
    a.C = X; a.sCb = (long long)N * A; a.sCm = A;
    a.exq = exq; a.exq_ld = A; a.exm = exm; a.row_s = k.kp;
    CKI(launch_digit_gemm(a, N, s));
  }
  prof_end(DONOF_PHASE_HALF_TRANSFORM, s);
  prof_begin(DONOF_PHASE_MO_3INDEX, s);
  {  // b[P][q][p] = sum_mu X[P][mu][q] C[mu][p]
    DigitArgs a = digit_args(ws, L);
    a.A = X; a.sAb = (long long)N * A; a.sAm = 1; a.sAk = A;
    a.M = np * A; a.Mb = A; a.Kin = N;
    a.eA = exq;
    a.ks = k.kp; a.ks_on = k.info;
    a.Bimg = (const __half*)(ws + L.Cimg); a.eB = (const int*)(ws + L.eC64);
    a.N = A;
    a.C = b; a.sCb = (long long)A * A; a.sCm = A;
    CKI(launch_digit_gemm(a, N, s));
  }
  prof_end(DONOF_PHASE_MO_3INDEX, s);
  prof_begin(DONOF_PHASE_JK_Y, s);
  const int tri = A * (A + 1) / 2, jb = (tri + 255) / 256;
  const int Kpad = round_up_int(A, 8);
  const DigitShape ys = digit_shape(A, (long long)np * Kpad);
  {
    double *W = (double*)(ws + L.W64), *part = (double*)(ws + L.skp);
    int *bmax = (int*)(ws + L.bmax), *wmax = (int*)(ws + L.wmax), *eY = (int*)(ws + L.eY64);
    const double *Ac = (const double*)(ws + L.Acoef), *Bc = (const double*)(ws + L.Bcoef);
    const int js = jk_splits64(A, np), wc = np < 152 * 4 ? np : 152 * 4;
    // (a slice's diagonal in shared memory: above 48 KB with the attribute, the largest there is, so
    // that calls of several sizes don't lower each other's)
    if ((size_t)A * 8 > 47 * 1024)
      CKI(cudaFuncSetAttribute(k_w_jk64, cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * 8));
    launch_chained(k_w_jk64, wc + jb * js, 256, (size_t)A * 8, s, b, np, A, Ac, W, wmax, wc, js,
                   part, bmax);
    launch_chained(k_jk_final64, jb + (A + 7) / 8, 256, 0, s, part, js, A, Bc, bmax, wmax,
                   (double*)(ws + L.J), (double*)(ws + L.K), eY, jb, p0 == 0 ? 1 : 0);
    launch_chained(k_y_planes, grid_for((long long)ys.NT * ys.ntiles * ys.nstages * 4), 256, 0, s,
        b, np, A, Kpad, kK64, Bc, W, eY, (__half*)(ws + L.Yimg), ys.NT, ys.ntiles, ys.nstages);
    count_launch(3);
    CKI(cudaGetLastError());
  }
  prof_end(DONOF_PHASE_JK_Y, s);
  prof_begin(DONOF_PHASE_G_BUILD, s);
  {  // G[mu][p] += sum_P sum_q X[P][mu][q] Y[P][q][p]
    DigitArgs a = digit_args(ws, L);
    a.A = X; a.sAm = A; a.sAk = 1; a.sAkb = (long long)N * A;
    a.M = N; a.Mb = N; a.Kin = A; a.Kpad = Kpad; a.KB = np;
    a.eA = exm;
    a.Bimg = (const __half*)(ws + L.Yimg); a.eB = (const int*)(ws + L.eY64);
    a.N = A;
    a.splits = g_splits_digit(N, A, np);
    a.C = (double*)(ws + L.skp); a.sCs = (long long)N * A; a.sCm = A;
    CKI(launch_digit_gemm(a, (long long)np * Kpad, s));
    launch_chained(k_split_sum, (unsigned)(((long long)N * A + 31) / 32), 256, 0, s,
        (const double*)(ws + L.skp), a.splits, (long long)N * A, (double*)(ws + L.G));
    count_launch(1);
    CKI(cudaGetLastError());
  }
  return DONOF_OK;
}

cudaError_t digit_lambda(const Dims& d, const double* C, bool prepared, char* ws, const Layout& L,
                         double* lam, cudaStream_t s) {
  const int N = d.N, A = d.A;
  const KScale k = kscale_at(ws + (prepared ? L.sB : L.sH), N);
  const double* G = (const double*)(ws + L.G);
  int* eG = (int*)(ws + L.eG64);
  // C's planes are done with
  if (N <= kFuseK) {
    ZeroJob zero{};
    zero.add(lam, (size_t)N * N * 8);
    CKE(launch_exps_planes(G, A, N, A, A, eG, k, 1, ws + L.Cimg, nullptr, 0, 0, nullptr, zero, false,
                           s));
  } else {
    CKE(cudaMemsetAsync(lam, 0, (size_t)N * N * 8, s));
    const ExpJob jobs[1] = {{G, A, N, A, 1, eG, k, 1}};
    CKE(launch_exps(jobs, 1, s));
    CKE(launch_planes(G, A, 1, N, A, eG, k, 1, ws + L.Cimg, s));
  }
  DigitArgs a = digit_args(ws, L);
  a.A = C; a.sAm = 1; a.sAk = N; a.M = N; a.Mb = N; a.Kin = N;
  a.eA = (const int*)(ws + L.eC64);
  a.ks = k.kn; a.ks_on = k.info;  // C's side of the scales
  a.Bimg = (const __half*)(ws + L.Cimg); a.eB = eG;
  a.N = A;
  a.C = lam; a.sCm = N;
  return launch_digit_gemm(a, N, s);
}

}  // namespace donof

#include "../../include/donof_testing.h"

extern "C" int donof_testing_digit_product(const double* A, int64_t sAm, int64_t sAk,
                                           const double* B, int64_t ldb, double* C, int64_t ldc,
                                           int32_t M, int32_t N, int32_t K, void* workspace,
                                           size_t workspace_bytes, void* stream) {
  using namespace donof;
  if (!A || !B || !C || M < 1 || N < 1 || K < 1 || K > 16384 || (sAm != 1 && sAk != 1))
    return DONOF_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < kAlign + digit_product_bytes(M, N, K) ||
      ((uintptr_t)workspace % kAlign) != 0)
    return DONOF_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  int* words = (int*)workspace;  // status, abort flag
  if (cudaMemsetAsync(words, 0, kAlign, s) != cudaSuccess ||
      digit_product(M, N, K, A, sAm, sAk, B, ldb, 1, C, ldc, (char*)workspace + kAlign, words,
                    words + 1, s) != cudaSuccess)
    return DONOF_ERR_CUDA;
  return DONOF_OK;
}
