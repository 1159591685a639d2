// Tensor-core (tcgen05 / TMEM) complex128 front GEMM:  C (128 x 32 tile) (+)= +-A B^T in 64-bit accuracy from exact
// integer products, after Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applications" (2012), for the Schur update F_BR -= (Z D^{-1}) Z^T
// and the two triangular multiplies of selective inversion (§2.2).
//
// Each row of an operand is scaled, per block of 128 k, by the power of two above its largest entry, and every real
// number becomes a 62-bit integer written with eight signed base-256 digits, most significant first (digits are
// exact in fp16).  The digit products a_i b_j of i + j = d share a weight; for each d = 0 .. 7 they are accumulated in
// FP32 in tensor memory, exactly: over 128 k a sum of d = 3 stays below 4 x 2 x 128 x 2^14 = 2^24, and the lower
// d (4 .. 7), which may pass it, weigh 2^-32 and less.  The eight sums are then combined in 64-bit integers, rounded
// once to 53 bits or at 2^-63 of the row scales' product, and added to C in FP64.
//
// Accuracy.  Products of i + j >= 8 are dropped: one real product loses up to 2^-59 of the row scales' product, the 256
// of an accumulation 2^-51 at worst and about 2^-59 on entries with random digits.  That is relative to the largest
// entries of two rows, so it is as good as 64-bit arithmetic only if those meet: before the rows are scaled, column k of A
// is multiplied and column k of B divided by a power of two that makes their largest entries equal (k_oz_colmax; the sum
// over k does not change).  Then C_ij's error is below 2^-51 sqrt(max_j' P_ij' max_i' P_i'j), P = |A| |B|^T, whatever
// the entries' sizes.  Measured against 80-bit products as the largest entry's error over that square root: on lens
// fronts 1e-16 (FP64 products: 2e-15), with PML amplitudes of 4e4 .. 4e6 or frequencies of 1e-4, whose pivots differ by
// many orders, 2e-16 (FP64: 2e-15; without the balance up to 5e-10).
//
// What bounds it: FP64 units do 2 DFMA per clock and SM, and the CUDA-core product (k_gemm) already ran them at 0.9 of
// their measured rate.  The 36 digit products are 72 fp16 MMAs of 128 x 64 x 16 per 16 k of a tile, at about 42 clocks
// each (48 by their shared-memory reads of 6 KB; 70 before their descriptors were unrolled to constants), and the
// blocks' way from L2 (88 KB per 16 k) is next: with a sixth of the MMAs the time falls to 0.57.  One CTA per SM over
// many tiles, so copies and MMAs of the next tile overlap this one's additions (one tile per CTA: 107 against 92 ms
// then).  The front products of an 80^3 lens setup: 860 ms with FP64 FMAs, 76 ms here plus 24 ms to write the digits
// and 3 ms for the columns' balance (the wide fronts' F_TL and inverse among them, psp_api.cu kOzBlock).
#include <cstdint>

#include "cplx.cuh"
#include "psp_internal.h"
#include "tcgen05.cuh"

namespace psp {

namespace {

constexpr int OM = 128, ON = 32, OK = 16;      // tile rows, tile columns, k per MMA step
constexpr int OKC = 128;                       // k per row scale and accumulation
constexpr int ND = 8;                          // digits
constexpr int A_PLANE = OM * OK * 2;           // 4 KB: 128 rows x 16 k of one digit, real or imaginary
constexpr int B_PLANE = 3 * ON * OK * 2;       // 3 KB: rows [-Im | Re | Im] of one digit
constexpr int A_BLOCK = ND * 2 * A_PLANE;      // 64 KB per 16 k
constexpr int B_BLOCK = ND * B_PLANE;          // 24 KB per 16 k
constexpr int STAGE = A_BLOCK + B_BLOCK;       // 88 KB
static_assert(OM == kOz.tile_m && ON == kOz.tile_n && OK == kOz.k && OKC == kOz.kc && A_BLOCK == kOz.a_block && B_BLOCK == kOz.b_block,
              "the planner's figures");
constexpr int NSTAGE = 2;
constexpr int SMEM = NSTAGE * STAGE + 1024;    // + barriers and the TMEM slot
constexpr uint32_t LBO = 128, SBO = 256;       // next core matrix (8 rows x 16 bytes) along k, next 8 rows
constexpr uint32_t TMEM_COLS = 512;            // ND sums x (32 real + 32 imaginary columns)
constexpr int EPI_THREADS = 256, THREADS = EPI_THREADS + 64;   // + the copying warp and the MMA warp
constexpr int kEmptyRow = -(1 << 16);          // exponent of a row of zeros
constexpr int kBadRow = 1 << 20;               // exponent of a row with an infinity or a NaN
constexpr int kFar = 1 << 12;                  // balance of a column whose partner is zero: past every exponent
constexpr int kNear = 4;                       // spread of two balances, in bits, over which one serves for the other

__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((LBO >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((SBO >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for tcgen05; layout type 0 = no swizzle
  return d;
}

// kind::f16 instruction descriptor: D f32, A and B fp16, both K-major, M = 128, N = 64 (32 real, 32 imaginary columns)
constexpr uint32_t kInstr = (1u << 4) | ((uint32_t)(2 * ON >> 3) << 17) | ((uint32_t)(OM >> 4) << 24);

__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(kInstr), "r"(acc));
}

// biased exponent of |x|: 0 for zero, 1 for denormals too, 2047 for infinities and NaN
__device__ __forceinline__ int exponent(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return (hi | __double2loint(x)) == 0 ? 0 : max(hi >> 20, 1);
}
__device__ __forceinline__ int exponent(double2 v) { return max(exponent(v.x), exponent(v.y)); }

// x as the 62-bit integer x 2^(62 - e), rounded, every base-256 digit biased by 128; emax = biased exponent of the
// row's largest entry (e = emax - 1022) in units of x
__device__ __forceinline__ unsigned long long biased_digits(double x, int emax) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(bits >> 52) & 0x7ff;
  unsigned long long m = (bits & 0xfffffffffffffull) | (e > 0 ? 0x10000000000000ull : 0ull);
  const int sh = emax - max(e, 1) - 9;
  if (sh <= 0) m <<= -sh;
  else m = sh < 56 ? (m + (1ull << (sh - 1))) >> sh : 0ull;
  if (bits >> 63) m = 0ull - m;
  return m + 0x8080808080808080ull;
}

// the digit at byte b of two biased integers as two fp16: 1024 + byte in each half, minus 1152 (negated: 1152 minus it)
__device__ __forceinline__ uint32_t digit_pair(unsigned long long x, unsigned long long y, int b, bool neg) {
  const uint32_t wx = b < 4 ? (uint32_t)x : (uint32_t)(x >> 32), wy = b < 4 ? (uint32_t)y : (uint32_t)(y >> 32);
  const uint32_t c = (uint32_t)(b & 3);
  const uint32_t h = (__byte_perm(wx, wy, c | (c << 4) | ((4 + c) << 8) | ((4 + c) << 12)) & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  const uint32_t bias = 0x64806480u;   // 1152 = 1024 + 128 in fp16, twice
  if (neg) asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(bias), "r"(h));
  else asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(bias));
  return r;
}

// acc +-= (h + rem 2^-14) 2^(e - 54), rounded to 53 bits or at 2^(e - 63), whichever is coarser: sums below 2^53 units take nine of
// the bits below a unit along.  A row with an infinity or a NaN gives NaN
__device__ __forceinline__ void add_scaled(double& acc, int64_t h, uint32_t rem, int e, bool neg) {
  const bool fine = (uint64_t)(h + (1ll << 53)) < (1ull << 54);
  double x = (double)(fine ? (h << 9) + (rem >> 5) : h);
  int ex = e + (fine ? 1023 - 63 : 1023 - 54);
  if ((unsigned)(ex - 1) >= 2046u) {   // a scale that is not a normal number: part of it goes to x first, exactly
    const int over = ex < 1 ? max(ex - 1, -1022) : min(ex - 2046, 900);
    x *= __hiloint2double((1023 + over) << 20, 0);
    ex = ex < 1 ? (ex - over < 1 ? 0 : 1) : 2046;
  }
  const int hi = e > kBadRow / 2 ? 0x7ff80000 : ex << 20;
  acc = fma(x, __hiloint2double(neg ? hi | (int)0x80000000 : hi, 0), acc);
}

__device__ __forceinline__ int64_t rounded_sum(const float v) { return (int64_t)__float2int_rn(v); }

}  // namespace

// entry (r, k) of an operand before its scale: r < R, k < K
template <typename Task>
__device__ __forceinline__ double2 operand_entry(const Task& tk, int r, int k) {
  if (tk.mode == TC_PACK_PLAIN) return tk.src[(int64_t)k * tk.ld + r];
  if (tk.mode == TC_PACK_TRANSPOSED) return tk.src[(int64_t)r * tk.ld + k];   // X[k, r]
  if (k == r) return make_double2(1.0, 0.0);
  if (tk.mode == TC_PACK_UNIT_LOWER) return k < r ? tk.src[(int64_t)k * tk.ld + r] : make_double2(0.0, 0.0);   // T[r, k]
  return k > r ? tk.src[(int64_t)r * tk.ld + k] : make_double2(0.0, 0.0);     // T[k, r], unit lower (transposed read)
}

// ---------------------------------------------------------------------------
// k_oz_colmax: exponent of the largest entry of 32 columns k of an operand, over its R rows.  Reads the operand once,
// 16 bytes an entry, contiguous over rows (a warp per column) or, for transposed operands, over k (a lane per column).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_oz_colmax(const OzColTask* __restrict__ tasks) {
  __shared__ int part[8][32];
  const OzColTask tk = tasks[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (tk.mode == TC_PACK_PLAIN || tk.mode == TC_PACK_UNIT_LOWER) {
    for (int k = tk.k0 + warp; k < min(tk.k0 + 32, tk.K); k += 8) {
      int em = 0;
#pragma unroll 4
      for (int r = (tk.mode == TC_PACK_PLAIN ? 0 : k) + lane; r < tk.R; r += 32) em = max(em, exponent(operand_entry(tk, r, k)));
      em = __reduce_max_sync(0xffffffffu, em);
      if (lane == 0) tk.out[k] = em;
    }
  } else {
    const int k = tk.k0 + lane, rend = tk.mode == TC_PACK_TRANSPOSED ? tk.R : min(tk.R, k + 1);
    int em = 0;
    if (k < tk.K)
#pragma unroll 4
      for (int r = warp; r < rend; r += 8) em = max(em, exponent(operand_entry(tk, r, k)));
    part[warp][lane] = em;
    __syncthreads();
    if (warp == 0 && k < tk.K) {
      for (int w = 1; w < 8; ++w) em = max(em, part[w][lane]);
      tk.out[k] = em;
    }
  }
}

// ---------------------------------------------------------------------------
// k_oz_pack: digits of 128 rows x 128 k of an operand (rows r0.., k from k0) per CTA, laid out as the MMAs read
// them from shared memory (K-major, 8-row x 16-byte core matrices).  Thread (row, half): k in [8 half, 8 half + 8) of
// every 16.  Two passes over the source (the second from L2): row exponents, then digits.  The balance 2^s(k) of a
// column is added to its entries' exponents.  16 bytes read and 32 (A) or 48 (B) written per entry, at 0.4 of DRAM's rate: the
// passes' latency and the digits' integer instructions bound it.
//
// Z D^-1 is an operand of the Schur update, balanced by its scale D^-1 alone, and of M_BL, balanced by that and the columns
// of Z and inv(L)^T.  Over 128 k the two balances differ by a constant, which the row exponents absorb, and by what the
// columns' sizes vary besides; where that stays within kNear bits M_BL takes the Schur update's balance and digits (four
// fifths of a 48^3 lens' front entries).  It costs up to those bits of the thirteen that the digits have beyond 64-bit
// sums (2^-59 against 2^-46 for 128 terms; measured, M_BL's error stays at 1.4e-16 where FP64 products have 2e-15).  80^3
// lens, k_oz_pack: 29.0 ms with Z D^-1 packed twice everywhere, 24.5 so (24.2 before products were balanced).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_oz_pack(const OzPackTask* __restrict__ tasks) {
  __shared__ int emax_s[2][OM], bal[OKC], least, most;
  const OzPackTask tk = tasks[blockIdx.x];
  const int row = threadIdx.x & (OM - 1), half = threadIdx.x >> 7;
  const int rg = tk.r0 + row;
  if (threadIdx.x == 0) {
    least = kFar;
    most = -kFar;
  }
  __syncthreads();
  int s = 0, scale_s = 0;   // balance of column threadIdx.x, and by the scale alone
  if (threadIdx.x < OKC) {
    const int k = tk.k0 + threadIdx.x;
    if (k < tk.K && (tk.ka || tk.kd)) {
      const int ea = tk.ka ? tk.ka[k] : 1, eb = tk.ka ? tk.kb[k] : 1, ed = tk.kd ? exponent(tk.kd[(int64_t)k * tk.ldk]) - 1023 : 0;
      s = ea == 0 ? kFar : eb == 0 ? -kFar : (eb - ea - ed) >> 1;
      scale_s = -ed >> 1;
      if (tk.near) {
        atomicMin(&least, s - scale_s);
        atomicMax(&most, s - scale_s);
      }
    }
  }
  __syncthreads();
  const bool near = tk.near && most - least <= kNear && most < kFar / 2 && least > -kFar / 2;
  if (near && (tk.near & OZ_KEEP)) return;
  if (threadIdx.x < OKC) bal[threadIdx.x] = (tk.rows_b ? -1 : 1) * (near ? scale_s : s);
  __syncthreads();
  auto load = [&](int k) {
    double2 v = make_double2(0.0, 0.0);
    if (rg < tk.R && k < tk.K) {
      v = operand_entry(tk, rg, k);
      if (tk.scale) v = cmul(v, tk.scale[(int64_t)k * tk.lds]);
    }
    return v;
  };
  const int nkb = min((tk.K - tk.k0 + OK - 1) / OK, OKC / OK);
  int em = 2 * kEmptyRow;
  for (int kb = 0; kb < nkb; ++kb)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int kk = kb * OK + half * 8 + q, e = exponent(load(tk.k0 + kk));
      if (e > 0) em = max(em, e == 0x7ff ? kBadRow : e + bal[kk]);
    }
  emax_s[half][row] = em;
  __syncthreads();
  em = max(emax_s[0][row], emax_s[1][row]);
  const int sub = tk.rows_b ? row >> 5 : 0;         // B: blocks of 32 rows
  const bool live = !tk.rows_b || tk.r0 + sub * ON < tk.R;
  if (half == 0 && live)
    tk.exps[tk.rows_b ? (int64_t)sub * tk.exp_stride + (row & 31) : row] =
        em == kBadRow ? kBadRow : (em < kEmptyRow ? kEmptyRow : em - 1022);
  if (!live) return;
  if (em < kEmptyRow) em = kBadRow;   // every digit zero
  for (int kb = 0; kb < nkb; ++kb) {
    unsigned long long re[8], im[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int kk = kb * OK + half * 8 + q;
      const double2 v = load(tk.k0 + kk);
      re[q] = biased_digits(v.x, em - bal[kk]);
      im[q] = biased_digits(v.y, em - bal[kk]);
    }
    unsigned char* dst = tk.dst + (int64_t)kb * (tk.rows_b ? B_BLOCK : A_BLOCK);
    if (tk.rows_b) dst += (int64_t)sub * tk.sub_stride;
    const int rr = tk.rows_b ? row & 31 : row;
    const uint32_t at = (uint32_t)((rr >> 3) * SBO + half * LBO + (rr & 7) * 16);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int b = ND - 1 - d;   // the most significant digit first
      uint32_t r[4], i[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        r[p] = digit_pair(re[2 * p], re[2 * p + 1], b, false);
        i[p] = digit_pair(im[2 * p], im[2 * p + 1], b, false);
      }
      if (!tk.rows_b) {
        *reinterpret_cast<uint4*>(dst + 2 * d * A_PLANE + at) = make_uint4(r[0], r[1], r[2], r[3]);
        *reinterpret_cast<uint4*>(dst + (2 * d + 1) * A_PLANE + at) = make_uint4(i[0], i[1], i[2], i[3]);
      } else {
        uint32_t n[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) n[p] = digit_pair(im[2 * p], im[2 * p + 1], b, true);
        unsigned char* pl = dst + d * B_PLANE + at;
        *reinterpret_cast<uint4*>(pl) = make_uint4(n[0], n[1], n[2], n[3]);
        *reinterpret_cast<uint4*>(pl + ON / 8 * SBO) = make_uint4(r[0], r[1], r[2], r[3]);
        *reinterpret_cast<uint4*>(pl + 2 * (ON / 8) * SBO) = make_uint4(i[0], i[1], i[2], i[3]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// k_oz_gemm: 128 x 32 output tiles, one CTA per SM over every gridDim.x-th tile, so that the next tile's copies and MMAs
// run while this one's sums are added to C (tiles of a small front spend more on that than on their MMAs).  Warp 8
// copies the operands' blocks of 16 k into two stages, warp 9 issues the MMAs (Re += Ar Br - Ai Bi and Im += Ar Bi + Ai Br as two N = 64 MMAs per digit pair: B's rows are stored as
// [-Im | Re | Im], so [Re | Im] and [-Im | Re] are windows of it), warps 0 - 7 combine the sums after every 128 k.
// Every wait is bounded; one that gives up records an error in status[1] and raises the CTA's abort flag.  The additions'
// tensor-memory reads are warp-wide instructions, so whether a warp goes on is one decision of the whole warp; after an
// abort the CTA's copies and MMAs in flight are waited for (bounded too) before its shared and tensor memory go back.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const OzGemmTask* __restrict__ tasks, int ntasks, int* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NSTAGE * STAGE);
  uint64_t* empty = full + NSTAGE;
  uint64_t* sums = empty + NSTAGE;       // the sums of 128 k are complete
  uint64_t* drained = sums + 1;          // ... and have been read
  uint64_t* quiet = drained + 1;         // after an abort: the MMAs issued have ended
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(quiet + 1);
  volatile int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(sums)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(drained)), "r"(EPI_THREADS) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(quiet)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *abort_flag = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  constexpr int PER = OKC / OK;          // blocks of 16 k per accumulation
  auto give_up = [&] {
    *abort_flag = 1;
    atomicCAS(status + 1, 0, 1);
  };

  int i = 0;   // warps 8 and 9: blocks of 16 k copied, consumed
  if (warp == 8) {
    if (lane == 0) {
      for (int t = blockIdx.x; t < ntasks && !*abort_flag; t += gridDim.x) {
        const OzGemmTask& tk = tasks[t];
        const unsigned char *A = tk.A, *B = tk.B;
        const int kb1 = tk.kb0 + tk.nkb;
        for (int kb = tk.kb0; kb < kb1; ++kb, ++i) {
          const int s = i & 1;
          if (i >= NSTAGE && !mbar_wait(smem_u32(&empty[s]), (uint32_t)(((i >> 1) - 1) & 1))) {
            give_up();
            break;
          }
          const uint32_t fb = smem_u32(&full[s]);
          const uint32_t dst = smem_u32(smem + s * STAGE);
          expect_tx(fb, STAGE);
          if (kb == tk.kb0 && (tk.flags & GF_TEST_STALL)) continue;   // announced, never copied
          bulk_copy(dst, A + (int64_t)kb * A_BLOCK, A_BLOCK, fb);
          bulk_copy(dst + A_BLOCK, B + (int64_t)kb * B_BLOCK, B_BLOCK, fb);
        }
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      int chunk = 0;   // accumulations made
      for (int t = blockIdx.x; t < ntasks && !*abort_flag; t += gridDim.x) {
        const int kb0 = tasks[t].kb0, kb1 = kb0 + tasks[t].nkb;
        for (int kb = kb0; kb < kb1; ++kb, ++i) {
          const int s = i & 1;
          const bool first = kb == kb0 || kb % PER == 0;   // the first block of an accumulation
          bool ok = !first || chunk == 0 || mbar_wait(smem_u32(drained), (uint32_t)((chunk - 1) & 1));
          if (ok) ok = mbar_wait(smem_u32(&full[s]), (uint32_t)((i >> 1) & 1));
          if (!ok) {
            give_up();
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          // fully unrolled: a descriptor is the stage's plus a constant (addresses count 16-byte units)
          const uint64_t a0 = make_desc(smem_u32(smem + s * STAGE)), b0 = make_desc(smem_u32(smem + s * STAGE + A_BLOCK));
          const uint32_t acc = first ? 0u : 1u;
#pragma unroll
          for (int d = 0; d < ND; ++d) {
#pragma unroll
            for (int p = 0; p <= d; ++p) {
              const uint64_t ap = a0 + (uint64_t)(2 * p * A_PLANE >> 4), bp = b0 + (uint64_t)((d - p) * B_PLANE >> 4);
              mma_f16(tmem + (uint32_t)(d * 2 * ON), ap, bp + (ON / 8 * SBO >> 4), p == 0 ? acc : 1u);   // Ar [Br | Bi]
              mma_f16(tmem + (uint32_t)(d * 2 * ON), ap + (A_PLANE >> 4), bp, 1u);                       // Ai [-Bi | Br]
            }
          }
          mma_commit(smem_u32(&empty[s]));
          if (kb + 1 == kb1 || (kb + 1) % PER == 0) {
            mma_commit(smem_u32(sums));
            ++chunk;
          }
        }
      }
    }
  } else {
    const int q = warp & 3, half = warp >> 2;
    const int row = 32 * q + lane, col0 = half * (ON / 2);
    constexpr int W = ON / 4;   // columns a thread combines at a time (two turns)
    int chunk = 0;
    for (int tile = blockIdx.x; tile < ntasks; tile += gridDim.x) {
      if (__any_sync(0xffffffffu, *abort_flag)) break;
      const OzGemmTask tk = tasks[tile];
      const bool neg = tk.flags & GF_NEG, beta0 = tk.flags & GF_BETA0;
      const int kb1 = tk.kb0 + tk.nkb;
      for (int kb = tk.kb0; kb < kb1; ++chunk) {
        const bool fresh = beta0 && kb == tk.kb0;
        const int kc = kb / PER;
        kb = (kc + 1) * PER;
        const int ea = row < tk.m ? __ldg(tk.ea + (int64_t)kc * OM + row) : kEmptyRow;
        bool ready = false;
        for (int turn = 0; turn < 2; ++turn) {
          const int c0 = col0 + turn * W;
          double2* cp = tk.C + (int64_t)c0 * tk.ldc + row;
          double2 v[W];   // C's entries are on their way while the MMAs finish
#pragma unroll
          for (int c = 0; c < W; ++c)
            v[c] = (row < tk.m && c0 + c < tk.n && row + tk.doff >= c0 + c && !fresh)
                       ? cp[(int64_t)c * tk.ldc]
                       : make_double2(0.0, 0.0);
          if (turn == 0) {
            ready = __all_sync(0xffffffffu, mbar_wait(smem_u32(sums), (uint32_t)(chunk & 1)));
            if (!ready) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          __syncwarp();
          const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0;
          int64_t hr[W], hi[W];
          uint32_t rem[W];   // what d = 5 .. 7 leave below a unit: 14 bits each, real | imaginary
          // weights (units of 2^(ea + eb - 54)): d = 0 .. 5: 2^42, 2^34, .. 2^2; d = 6, 7: 2^-6, 2^-14
#pragma unroll
          for (int d = ND - 1; d >= 0; --d) {
            uint32_t vr[W], vi[W];
            tmem_ld8(base + (uint32_t)(d * 2 * ON), vr);
            tmem_ld8(base + (uint32_t)(d * 2 * ON + ON), vi);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int c = 0; c < W; ++c) {
              const int64_t r = rounded_sum(__uint_as_float(vr[c])), i = rounded_sum(__uint_as_float(vi[c]));
              if (d == ND - 1) {
                hr[c] = r;
                hi[c] = i;
              } else if (d >= 5) {
                hr[c] += r << (8 * (ND - 1 - d));
                hi[c] += i << (8 * (ND - 1 - d));
                if (d == 5) {
                  rem[c] = (uint32_t)(hr[c] & 0x3fff) | (uint32_t)(hi[c] & 0x3fff) << 16;
                  hr[c] >>= 14;
                  hi[c] >>= 14;
                }
              } else {
                hr[c] += r << (42 - 8 * d);
                hi[c] += i << (42 - 8 * d);
              }
            }
          }
          if (turn == 1) {   // the sums have been read: the next 128 k may overwrite them
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(drained)) : "memory");
          }
          const int* ebp = tk.eb + (int64_t)kc * ON + c0;
#pragma unroll
          for (int c = 0; c < W; ++c) {
            if (row >= tk.m || c0 + c >= tk.n || row + tk.doff < c0 + c) continue;
            const int e = ea + __ldg(ebp + c);
            add_scaled(v[c].x, hr[c], rem[c] & 0xffffu, e, neg);
            add_scaled(v[c].y, hi[c], rem[c] >> 16, e, neg);
            cp[(int64_t)c * tk.ldc] = v[c];
          }
        }
        if (!ready) {
          give_up();
          break;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag) {   // nothing writes it any more
    if (warp == 8 && lane == 0) {
      for (int j = i > NSTAGE ? i - NSTAGE : 0; j < i; ++j) mbar_wait(smem_u32(&full[j & 1]), (uint32_t)((j >> 1) & 1));
    } else if (warp == 9 && lane == 0) {
      mma_commit(smem_u32(quiet));
      mbar_wait(smem_u32(quiet), 0u);
    }
    __syncthreads();
  }
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

void launch_oz_colmax(const OzColTask* tasks, int ntasks, cudaStream_t st) {
  if (ntasks > 0) k_oz_colmax<<<ntasks, 256, 0, st>>>(tasks);
}

void launch_oz_pack(const OzPackTask* tasks, int ntasks, cudaStream_t st) {
  if (ntasks > 0) k_oz_pack<<<ntasks, 256, 0, st>>>(tasks);
}

void launch_oz_gemm(const OzGemmTask* tasks, int ntasks, int* status, cudaStream_t st) {
  if (ntasks <= 0) return;
  cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  k_oz_gemm<<<ntasks < sms ? ntasks : sms, THREADS, SMEM, st>>>(tasks, ntasks, status);
}

}  // namespace psp
