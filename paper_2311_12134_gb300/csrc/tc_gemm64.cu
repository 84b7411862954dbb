// Trailing update of the complex128 LU, A22 -= L21 U12, on the 5th-generation
// tensor cores (tcgen05, sm_103a): the operands are rounded to bf16 digits (the Ozaki
// scheme), the digits' products summed exactly and rounded to FP64 once per panel.
//
// What bounds it.  GB300's FP64 pipe retires 2 multiply-adds per SM and clock, so
// the 128 of one complex element and panel (NB = 32) cost 64 clocks; as integer
// digit products the same update needs 0.9 clocks of the tensor pipe, and what is
// left is the epilogue (one FP64 conversion and one multiply-add per real value).
//
// Digits.  The operands become integers relative to a scale.  K column k of A (32 of
// them) is multiplied by 2^s_k and row k of B by 2^-s_k, an exact balance that makes
// the terms of a sum comparable (the LU takes s_k from the largest entries of L21's columns
// in the CTA's 128 rows, the solve from those of the solved block's rows); then row r of A is scaled by its largest exponent and
// column c of B by its own.  A scaled value |v| < 2^E becomes rint(v 2^(55 - E)) and its
// seven balanced base-256 digits,
//   v 2^(7 - E) = sum_{s=0..6} a_s 2^(-8 s) + rest,  -128 <= a_s <= 128,
//   |rest| <= 2^-49 (2^-56 of 2^E),
// taken with integer instructions (no FP64 operation) and exact in bf16.  The 34
// digit pairs s + t <= 7 run as bf16 products with FP32 accumulation in tensor
// memory, one accumulator per class g = s + t; a class holds at most 7 pairs of
// 2^14 per real K, so the 64 real K of a panel sum exactly (below 2^23).  The complex
// product is the real embedding
//   [Re C | Im C] -= [Re L | Im L] x [[Re U, Im U], [-Im U, Re U]].
// The B planes of the digits t = 0, 1, .. lie one after the other, so one
// instruction per digit s of A forms all its classes: N = 32 (8 - s) columns
// starting at class s (the eighth plane of B is zero: class 7 starts from zero with
// the others), and A is read 7 times per 16 K instead of 34.
//
// Error.  Per real term, with 2^E_r and 2^E_c the scales of its row and column: at most
// 2^-56 of 2^(E_r + E_c) for the rest of each operand and 5 x 2^-64 for the classes left
// out, and once per sum 2^-57 for the conversion; an FP64 sum rounds each term to
// 2^-53 of the partial sum.  That is a normwise statement: an entry formed only from
// terms far below its row's and column's scales keeps fewer bits, so it matters what the
// scales are.  Without the balance s_k one large entry of U (a large t^-1 pivoted into
// a row of order g) set the scale of its row, and tau's error grew with t^-1.  Measured
// against long double solutions (in brackets LAPACK's error, then without the balance
// and class 7): below 1e-14 (8e-16, 4.6e-13) at n = 320 and an f phase of 1e-6, below
// 8e-14 (1e-14, 5.9e-12) at n = 688, below 4e-13 (2e-14, 1.4e-4) with every channel's
// t^-1 scaled at random by 10^-12 .. 10^12.  In a restatement of both in NumPy the digits'
// error is 0.3 to 1 times that of FP64 updates on nearly all such matrices (1.1e-15 and
// 1.5e-15 at n = 688 with ordinary phase shifts), at most twice on any.
//
// Measured (216 matrices of n = 688, 21 panels): 15.2 ms (14.6 without class 7) against
// 165 ms for a register-tiled product on the FP64 pipe (0.98 of that pipe's rate).
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "tc_bf16.cuh"

namespace lsms {

namespace oz {

using namespace tb;  // descriptors, instructions, barriers

constexpr int NB = 32;                // complex panel width
constexpr int TM = 128;               // rows per CTA (TMEM lanes)
constexpr int NCC = 16;               // complex columns per tile
constexpr int NR = 2 * NCC;           // real accumulator columns per class: [Re | Im]
constexpr int NT = 512;               // threads: (row, 8-column chunk) of L21; (column, row) of a U12 tile
constexpr int ND = 7;                 // digits per operand
constexpr int NG = 8;                 // classes per accumulator
constexpr int PLANE_A = TM * 128;     // one digit of A: 64 real K x 2 bytes per row, 128-byte swizzle
constexpr int PLANE_B = NR * 128;
constexpr int STAGE_B = NG * PLANE_B;  // the last plane zero
constexpr int kGemmSmem = ND * PLANE_A + 2 * STAGE_B + 4 * TM * 4 + 4 * NCC * 4 + 4 * NB * 4 + 64 + 1024;
constexpr uint32_t ACC_COLS = NG * NR;  // columns of an accumulator (two of them)
constexpr uint32_t TMEM_COLS = 512;
static_assert(NT == TM * 4 && NT == NCC * NB && 2 * ACC_COLS == TMEM_COLS, "tile shape");

__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(taddr));
}

// One thread: the digit products (per 16 K, one instruction per digit of A) of a 128 x 16
// complex tile with 32 complex K, committed to an mbarrier.
__device__ __forceinline__ void issue_tile(uint32_t d, uint32_t a0, uint32_t b0, uint32_t mbar) {
#pragma unroll
  for (int s = 0; s < ND; ++s)
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
      mma_bf16(d + (uint32_t)(s * NR), make_desc(a0 + s * PLANE_A + ks * 32), make_desc(b0 + ks * 32),
               make_idesc(TM, NR * (NG - s)), (ks | s) ? 1u : 0u);
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

// Scale of class_sum's integers for the scales el, eu of the row and the column (exponent
// fields, the balance in them cancelled): class 0 weighs 2^(el + eu - 2 * 1022 - 14), the
// integers count 2^-42 of it.  NaN when one of the two stands for a non-finite value.
__device__ __forceinline__ double product_scale(int el, int eu) {
  const int ex = el + eu - 2 * 1022 - 14 - 42 + 1023;
  return __hiloint2double(ex <= 0 ? 0 : (ex >= 0x7ff ? 0x7ff80000 : ex << 20), 0);
}

constexpr int kNoExp = -4096;        // zero (subnormals count as zero: below 2^-1022)
constexpr int kNonFinite = 1 << 14;  // above every sum of fields: product_scale gives NaN

// Larger exponent field of a complex value's parts: 0 for zero, 0x7ff for a non-finite value.
__device__ __forceinline__ int exp_field(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff);
}
// the field as an exponent of the balance (0, below all others, unless finite and nonzero) and of a scale
__device__ __forceinline__ int balance_exp(int e) { return e == 0x7ff ? 0 : e; }
__device__ __forceinline__ int scale_exp(int e, int balance) {
  return e == 0x7ff ? kNonFinite : (e == 0 ? kNoExp : e + balance);
}

// rint(v 2^(55 - E)) plus 128 in each of its six low bytes, E = emax - 1022 (|v| < 2^E when v's
// exponent field is at most emax): the low bytes are digits 6 .. 1 plus 128, what is above them
// digit 0.
__device__ __forceinline__ long long biased_digits(double v, int emax) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const long long m = e ? ((b & 0xfffffffffffffll) | 0x10000000000000ll) : 0ll;
  const int sh = min(e - emax + 2, 2);  // m 2^(e - 1075) 2^(..): at most 2 to the left
  const int r = min(max(-sh, 0), 62);
  const long long half = r ? 1ll << (r - 1) : 0ll;
  const long long mag = ((m << max(sh, 0)) + half) >> r;
  return (b < 0 ? -mag : mag) + 0x0000808080808080ll;
}

// Digit s of a biased value as the bits of a float (an integer of at most 8 significant
// bits: its upper 16 bits are the bf16 value, exactly).
template <int s>
__device__ __forceinline__ uint32_t digit_bits(long long j) {
  const uint32_t hi = (uint32_t)((unsigned long long)j >> 32);
  if constexpr (s == 0) {  // the 16 bits above the bytes
    return __float_as_uint(__uint_as_float(__byte_perm(hi ^ 0x80000000u, 0x4B000000u, 0x7432)) - 8421376.f);
  } else {
    constexpr int byte = ND - 1 - s;
    const uint32_t w = byte >= 4 ? hi : (uint32_t)j;
    return __float_as_uint(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 + (byte & 3))) - 8388736.f);
  }
}

// One digit plane of A: the 8 columns of this thread's chunk, real parts to 16-byte unit
// `chunk` of its row, imaginary parts to unit 4 + chunk.
template <int s>
__device__ __forceinline__ void put_a(uint8_t* sA, int row, int chunk, const long long (&jr)[8], const long long (&ji)[8]) {
  uint4 re, im;
  uint32_t* pr = &re.x;
  uint32_t* pi = &im.x;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    pr[q] = __byte_perm(digit_bits<s>(jr[2 * q]), digit_bits<s>(jr[2 * q + 1]), 0x7632);
    pi[q] = __byte_perm(digit_bits<s>(ji[2 * q]), digit_bits<s>(ji[2 * q + 1]), 0x7632);
  }
  uint8_t* p = sA + s * PLANE_A + row * 128;
  *reinterpret_cast<uint4*>(p + ((chunk ^ (row & 7)) << 4)) = re;
  *reinterpret_cast<uint4*>(p + (((4 + chunk) ^ (row & 7)) << 4)) = im;
  if constexpr (s + 1 < ND) put_a<s + 1>(sA, row, chunk, jr, ji);
}

// One digit plane of B, U12(k, c): row c (real output) holds Re at K k and -Im at K 32 + k,
// row 16 + c (imaginary output) Im and Re.
template <int t>
__device__ __forceinline__ void put_b(uint8_t* sB, int c, int k, long long jr, long long ji) {
  const uint32_t re = digit_bits<t>(jr) >> 16, im = digit_bits<t>(ji) >> 16;
  const int u = k >> 3, off = (k & 7) * 2, x = c & 7;
  uint8_t* p = sB + t * PLANE_B + c * 128;
  uint8_t* q = p + NCC * 128;  // (16 + c) & 7 == c & 7
  *reinterpret_cast<unsigned short*>(p + ((u ^ x) << 4) + off) = (unsigned short)re;
  *reinterpret_cast<unsigned short*>(p + (((4 + u) ^ x) << 4) + off) = (unsigned short)(im ^ 0x8000u);
  *reinterpret_cast<unsigned short*>(q + ((u ^ x) << 4) + off) = (unsigned short)im;
  *reinterpret_cast<unsigned short*>(q + (((4 + u) ^ x) << 4) + off) = (unsigned short)re;
  if constexpr (t + 1 < ND) put_b<t + 1>(sB, c, k, jr, ji);
}

// Plane 7 of a stage of B, after the digits' planes: zero.
__device__ __forceinline__ void zero_plane(uint8_t* stage, int tid) {
  static_assert(PLANE_B % (NT * 8) == 0, "8 bytes per thread");
#pragma unroll
  for (int o = 0; o < PLANE_B; o += NT * 8) *reinterpret_cast<uint2*>(stage + ND * PLANE_B + o + tid * 8) = make_uint2(0, 0);
}

// The class sums of one real value as a number in units of 2^-42 of the class-0 weight (2^-56 of
// the two scales), the last two classes rounded to it, then to FP64.
__device__ __forceinline__ double class_sum(const float (&v)[NG]) {
  int i[NG];
#pragma unroll
  for (int g = 0; g < NG; ++g) i[g] = __float2int_rn(v[g]);
  const int a = i[0] * 256 + i[1];  // below 2^29
  const int b = i[2] * 256 + i[3];  // below 2^30
  const int c = i[4] * 256 + i[5];  // below 2^31
  const int d = i[6] * 256 + i[7];  // below 2^31 - 2^27
  return (double)(((long long)a << 34) + (long long)b * (1 << 18) + (long long)c * 4 + ((d + (1 << 13)) >> 14));
}

}  // namespace oz

// grid (row tiles of 128, n_units, column splits), block 512, dynamic smem
// oz::kGemmSmem (one CTA per SM).  One CTA per 128-row block of a unit's trailing
// matrix walks its share of the 16-column tiles: L21's digit planes are staged
// once; the digits of the next tile's U12 are staged and its product issued (into
// the other accumulator) before the epilogue of the current tile, which the
// tensor cores therefore overlap.  Waits on the tensor core are bounded
// (LSMS_UNIT_TIMEOUT).  A row or column with a non-finite value gives NaN.
__global__ void __launch_bounds__(oz::NT, 1) k_gemm64_tc(const Unit* __restrict__ units, char* fac_base, int k,
                                                         int32_t* stat) {
  using namespace oz;
  const Unit u = units[blockIdx.y];
  const int n = u.n;
  const int t0 = k + NB;
  const int mt = n - t0;
  if (mt <= 0) return;
  const int row0 = t0 + blockIdx.x * TM;
  if (row0 >= n) return;
  const int tiles = (mt + NCC - 1) / NCC;
  const int per = (tiles + gridDim.z - 1) / gridDim.z;
  const int j0 = blockIdx.z * per, j1 = min(tiles, j0 + per);
  if (j0 >= j1) return;
  double2* A = reinterpret_cast<double2*>(fac_base + u.fac_off);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = smem + ND * PLANE_A;
  int* sRexp = reinterpret_cast<int*>(sB + 2 * STAGE_B);   // [4][TM] exponent maxima of the row chunks
  int* sCexp = sRexp + 4 * TM;                             // [4][NCC] exponents of the tiles' columns
  int* sKexp = sCexp + 4 * NCC;                            // [4][NB] exponent maxima of L21's columns, by 32 rows
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sKexp + 4 * NB);  // [2], one per accumulator
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 2);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar + 1)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }

  // U12: warp = column of the tile, lane = row of the panel
  auto load_u = [&](int j) -> double2 {
    const int col = t0 + j * NCC + warp;
    return col < n ? A[(size_t)col * n + k + lane] : make_double2(0.0, 0.0);
  };
  int kexp = 0;  // largest exponent of the CTA's rows in column `lane` of L21: 2^kexp balances U12's row
  auto stage_u = [&](int j, double2 v) {
    const int e = __reduce_max_sync(0xffffffffu, scale_exp(exp_field(v), kexp));
    // (slots of 4: a slower warp may still read the exponents of tile j - 2)
    if (lane == 0) sCexp[(j & 3) * NCC + warp] = e;
    put_b<0>(sB + (j & 1) * STAGE_B, warp, lane, biased_digits(v.x, e - kexp), biased_digits(v.y, e - kexp));
  };
  double2 uv = load_u(j0);

  // L21: thread (row, chunk of 8 columns)
  const int ar = tid & (TM - 1), chunk = tid >> 7;
  zero_plane(sB, tid);
  zero_plane(sB + STAGE_B, tid);
  {
    const int row = row0 + ar;
    double2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      v[q] = row < n ? A[(size_t)(k + chunk * 8 + q) * n + row] : make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = __reduce_max_sync(0xffffffffu, balance_exp(exp_field(v[q])));
      if (lane == q) sKexp[(warp & 3) * NB + chunk * 8 + q] = e;
    }
    __syncthreads();
    kexp = max(max(sKexp[lane], sKexp[NB + lane]), max(sKexp[2 * NB + lane], sKexp[3 * NB + lane]));
    int e = kNoExp;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      e = max(e, scale_exp(exp_field(v[q]), -__shfl_sync(0xffffffffu, kexp, chunk * 8 + q)));
    sRexp[chunk * TM + ar] = e;
    __syncthreads();
    e = max(max(sRexp[ar], sRexp[TM + ar]), max(sRexp[2 * TM + ar], sRexp[3 * TM + ar]));
    long long jr[8], ji[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int eq = e + __shfl_sync(0xffffffffu, kexp, chunk * 8 + q);
      jr[q] = biased_digits(v[q].x, eq);
      ji[q] = biased_digits(v[q].y, eq);
    }
    put_a<0>(sA, ar, chunk, jr, ji);
  }

  // epilogue: TMEM lane (warp % 4) * 32 + lane = row, complex columns 4 (warp / 4) .. + 3
  const int er = (warp & 3) * 32 + lane, ec = (warp >> 2) * 4;
  const int crow = row0 + er;
  const int rexp = max(max(sRexp[er], sRexp[TM + er]), max(sRexp[2 * TM + er], sRexp[3 * TM + er]));

  // stage U12 of tile j (its buffer and accumulator free: tile j - 2 is done) and issue its product
  uint32_t tmem = 0;
  auto launch_tile = [&](int j) {
    stage_u(j - j0, uv);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem = *tslot;
    if (tid == 0) {
      const int b = (j - j0) & 1;
      issue_tile(tmem + (uint32_t)b * ACC_COLS, smem_u32(sA), smem_u32(sB + b * STAGE_B), smem_u32(mbar + b));
    }
    if (j + 1 < j1) uv = load_u(j + 1);
  };

  launch_tile(j0);
  bool ok = true;
  int issued = 0;
  for (int j = j0; j < j1; ++j) {
    const int it = j - j0;
    double2 cv[4];
    const int c0 = t0 + j * NCC + ec;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      cv[c] = (crow < n && c0 + c < n) ? A[(size_t)(c0 + c) * n + crow] : make_double2(0.0, 0.0);
    if (j + 1 < j1) {
      launch_tile(j + 1);
      issued = it + 1;
    }
    if (warp == 0) ok = mbar_wait(mbar + (it & 1), (uint32_t)((it >> 1) & 1));
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) break;
    const uint32_t base = tmem + (uint32_t)(it & 1) * ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ec;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float re[NG][2], im[NG][2];
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        tmem_ld2(base + (uint32_t)(g * NR + 2 * h), re[g]);
        tmem_ld2(base + (uint32_t)(g * NR + NCC + 2 * h), im[g]);
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float vr[NG], vi[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          vr[g] = re[g][q];
          vi[g] = im[g][q];
        }
        const int c = 2 * h + q;
        const double sc = product_scale(rexp, sCexp[(it & 3) * NCC + ec + c]);
        const double2 r = make_double2(fma(-class_sum(vr), sc, cv[c].x), fma(-class_sum(vi), sc, cv[c].y));
        if (crow < n && c0 + c < n) A[(size_t)(c0 + c) * n + crow] = r;
      }
    }
  }
  if (!ok && tid == 0) {
    atomicOr(&stat[u.stat_off], LSMS_UNIT_TIMEOUT);
    // give the tensor core a second bounded window before the accumulators are freed
    mbar_wait(mbar + (issued & 1), (uint32_t)((issued >> 1) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(TMEM_COLS));
  }
}

int gemm64_tc_chunk(const Unit* d_units, int n_units, int n_max, int k, char* fac_base, int32_t* stat,
                    cudaStream_t st) {
  LSMS_SMEM_LIMIT(k_gemm64_tc, oz::kGemmSmem);
  const int mt = n_max - k - oz::NB;
  if (mt <= 0) return LSMS_OK;
  const int rows = (mt + oz::TM - 1) / oz::TM, tiles = (mt + oz::NCC - 1) / oz::NCC;
  // few row blocks: the columns split over CTAs too, at least 4 tiles each (a CTA's staging of
  // L21 costs about as much as two tiles)
  const int want = 2 * 152 / std::max(1, rows * n_units);
  const int split = std::max(1, std::min(want, tiles / 4));
  LSMS_LAUNCH(k_gemm64_tc, dim3(rows, n_units, split), dim3(oz::NT),
              oz::kGemmSmem, st, d_units, fac_base, k, stat);
  return LSMS_OK;
}

}  // namespace lsms

// ------------------------------------------------------------------ solve
namespace lsms {

__device__ __forceinline__ double2 shfl2(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// The row interchanges of one factor panel (rows k + j <-> sp[j], j = 0..31 in
// order; sp[j] = k + j for no interchange) applied to one column by one warp.
// Lane j holds row k + j of the column in x on entry and exit; rows below the
// panel that the interchanges reach are read and written in place.  When those
// rows are all distinct (the usual case) each is read once up front and written
// once at the end and the sequence runs in registers; repeated targets take the
// sequential path through memory.
template <typename C>
__device__ __forceinline__ C panel_swaps(C x, C* col, const int* sp, int k, int lane) {
  constexpr int NB = 32;
  const int pj = sp[lane];
  const bool outj = pj >= k + NB;
  const unsigned same = __match_any_sync(0xffffffffu, outj ? pj : -1 - lane);
  const bool fast = !__any_sync(0xffffffffu, outj && __popc(same) > 1);
  if (fast) {
    C y = outj ? col[pj] : x;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int p = sp[j];
      if (p == k + j) continue;
      if (p < k + NB) {
        const int b = p - k;
        const C va = shfl2(x, j);
        const C vb = shfl2(x, b);
        if (lane == j) x = vb;
        if (lane == b) x = va;
      } else if (lane == j) {
        const C t = y;
        y = x;
        x = t;
      }
    }
    if (outj) col[pj] = y;
  } else {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int p = sp[j];
      if (p == k + j) continue;
      if (p < k + NB) {
        const int b = p - k;
        const C va = shfl2(x, j);
        const C vb = shfl2(x, b);
        if (lane == j) x = vb;
        if (lane == b) x = va;
      } else {
        if (lane == j) {
          const C t = col[p];
          col[p] = x;
          x = t;
        }
        __syncwarp();
      }
    }
  }
  return x;
}

namespace oz {

constexpr int kSolveSmem = ND * PLANE_A + STAGE_B + 3 * 4 * TM * 4 + NCC * 4 + NCC * NB * 4 + 32 +
                           NB * (NB + 1) * 16 + NB * (NCC + 1) * 16 + NB * 16 + 1024;

}  // namespace oz

// L y = P b (unit lower; each panel's row swaps applied just before its block), then
// U x = y, in place on 16 columns (slice blockIdx.y) of the unit's n x nrhs
// complex128 block X.  grid (n_units, ceil(nrhs / 16)), block 512, dynamic smem
// oz::kSolveSmem (one CTA per SM).  Per 32-row block:
//   the 32 x 32 triangle in FP64, 8 rows at a time: four warps substitute within
//   8 x 8 (4 columns x 8 rows a warp), then all threads update the block's other
//   rows; the diagonal's reciprocals are formed once per block by one warp;
//   the rows below (above, going back) take X -= L y (U x) as digit products, 128
//   rows at a time: A = the factor's rows (loaded a tile ahead, split when the
//   previous tile's products are done), B = the solved block, split once; the
//   epilogue of a tile runs under the products of the next.
// The balance takes the rows of the solved block, which spread over orders of magnitude
// (small high-l components meet large t^-1 entries), into the factor's columns.
// What bounds it: splitting the factor (each value serves 16 columns only, about
// 0.7 clocks of integer work per SM and value) and the FP64 triangle.  Measured:
// 216 matrices of n = 688, 16 columns: 3.70 ms (4.13 with eight digits) against 19.8 ms with the row updates
// on the FP64 pipe and a division per diagonal element and column; 20 matrices of
// n = 160 0.24 (0.25) against 1.00 ms.
__global__ void __launch_bounds__(oz::NT, 1) k_solve64_tc(const Unit* __restrict__ units, const char* fac_base,
                                                          char* ws, int nrhs, int32_t* stat) {
  using namespace oz;
  const Unit u = units[blockIdx.x];
  const int n = u.n;
  if (n == 0) return;  // an unused FP64 fallback slot
  const double2* A = reinterpret_cast<const double2*>(fac_base + u.fac_off);
  const int32_t* piv = reinterpret_cast<const int32_t*>(fac_base + u.piv_off);
  const int cofs = blockIdx.y * NCC, ncol = min(NCC, nrhs - cofs);
  double2* X = reinterpret_cast<double2*>(ws + u.x_off) + (size_t)cofs * n;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = sA + ND * PLANE_A;
  double2(*sT)[NB + 1] = reinterpret_cast<double2(*)[NB + 1]>(sB + STAGE_B);      // the diagonal block
  double2(*sX)[NCC + 1] = reinterpret_cast<double2(*)[NCC + 1]>(sT + NB);         // its rows of X
  double2* sD = reinterpret_cast<double2*>(sX + NB);                              // reciprocals of U's diagonal
  int* sRexp = reinterpret_cast<int*>(sD + NB);                                   // [3][4][TM], slot = tile % 3
  int* sCexp = sRexp + 3 * 4 * TM;                                                // [NCC]
  int* sKexp = sCexp + NCC;                                                       // [NCC][NB] exponents of the block
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sKexp + NCC * NB);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
  __shared__ int sp[NB];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  const int ar = tid & (TM - 1), chunk = tid >> 7;                 // A: row, chunk of 8 columns
  const int er = (warp & 3) * 32 + lane, ec = (warp >> 2) * 4;     // epilogue: TMEM lane, first column
  int issued = 0;  // products committed so far; each is waited for before the next is issued
  bool ok = true;
  int kexp = 0;    // largest exponent of the columns in row `lane` of the solved block: 2^kexp balances the factor's column
  zero_plane(sB, tid);

  // products `issued - 1` complete (bounded); CTA-uniform, also the barrier of what came before
  auto wait_products = [&]() -> bool {
    bool w = true;
    if (warp == 0 && issued > 0) w = mbar_wait(mbar, (uint32_t)((issued - 1) & 1));
    w = __syncthreads_and(w);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return w;
  };
  // X[row0 + er, ec ..] -= the products of the block's tile t
  auto epilogue = [&](int row0, int r1, int t, const double2 (&cv)[4]) {
    const int row = row0 + er;
    const int* re4 = sRexp + (t % 3) * 4 * TM + er;
    const int rexp = max(max(re4[0], re4[TM]), max(re4[2 * TM], re4[3 * TM]));
    const uint32_t base = tmem + (uint32_t)(t & 1) * ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ec;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float re[NG][2], im[NG][2];
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        tmem_ld2(base + (uint32_t)(g * NR + 2 * h), re[g]);
        tmem_ld2(base + (uint32_t)(g * NR + NCC + 2 * h), im[g]);
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float vr[NG], vi[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          vr[g] = re[g][c];
          vi[g] = im[g][c];
        }
        const int col = ec + 2 * h + c;
        const double sc = product_scale(rexp, sCexp[col]);
        const double2 x = cv[2 * h + c];
        if (row < r1 && col < ncol)
          X[(size_t)col * n + row] =
              make_double2(fma(-class_sum(vr), sc, x.x), fma(-class_sum(vi), sc, x.y));
      }
    }
  };

  const int nb = (n + NB - 1) / NB;
  for (int step = 0; step < 2 * nb && ok; ++step) {
    const bool fwd = step < nb;
    const int k = NB * (fwd ? step : 2 * nb - 1 - step);
    const int nbp = min(NB, n - k);
    const int r0 = fwd ? k + nbp : 0, r1 = fwd ? n : k;  // rows to update
    // the first tile's factor rows are requested before the triangle is solved
    double2 v[8];
    auto load_a = [&](int row0) {
      const int row = row0 + ar;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = chunk * 8 + q;
        v[q] = (row < r1 && c < nbp) ? A[(size_t)(k + c) * n + row] : make_double2(0.0, 0.0);
      }
    };
    if (r0 < r1) load_a(r0);
    for (int idx = tid; idx < NB * NB; idx += NT) {
      const int i = idx % NB, j = idx / NB;
      sT[i][j] = (i < nbp && j < nbp) ? A[(size_t)(k + j) * n + k + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
    if (tid < NB) {
      if (fwd) sp[tid] = tid < nbp ? piv[k + tid] : k + tid;
      else sD[tid] = crcp(tid < nbp ? A[(size_t)(k + tid) * n + k + tid] : make_double2(1.0, 0.0));
    }
    __syncthreads();
    {
      const bool live = warp < ncol;
      double2 x = make_double2(0.0, 0.0);
      if (live) {
        if (lane < nbp) x = X[(size_t)warp * n + k + lane];
        if (fwd) x = panel_swaps(x, X + (size_t)warp * n, sp, k, lane);
      }
      sX[lane][warp] = x;
    }
    __syncthreads();
    for (int bb = 0; bb < 4; ++bb) {
      const int b0 = 8 * (fwd ? bb : 3 - bb);
      if (warp < 4) {
        const int c = 4 * warp + (lane >> 3), r = lane & 7, i = b0 + r;
        double2 x = sX[i][c];
        if (fwd) {
#pragma unroll
          for (int j = 0; j < 7; ++j) {
            const double2 xj = shfl2(x, (lane & 24) + j);
            if (r > j) x = cfms(sT[i][b0 + j], xj, x);
          }
        } else {
#pragma unroll
          for (int j = 7; j >= 0; --j) {
            if (r == j) x = cmul(x, sD[i]);
            const double2 xj = shfl2(x, (lane & 24) + j);
            if (r < j) x = cfms(sT[i][b0 + j], xj, x);
          }
        }
        sX[i][c] = x;
      }
      __syncthreads();
      if (bb < 3) {
        const int c = tid & 15, q = tid >> 4;
        const int i = fwd ? b0 + 8 + q : q;
        if (i < (fwd ? NB : b0)) {
          double2 x = sX[i][c];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const int j = b0 + (fwd ? jj : 7 - jj);
            x = cfms(sT[i][j], sX[j][c], x);
          }
          sX[i][c] = x;
        }
        __syncthreads();
      }
    }
    {
      // the solved block: to X, and its digits into B (warp = column, lane = row; columns beyond
      // ncol are zero)
      const double2 y = sX[lane][warp];
      if (warp < ncol && lane < nbp) X[(size_t)warp * n + k + lane] = y;
      if (r0 < r1) {
        const int f = exp_field(y);
        sKexp[warp * NB + lane] = balance_exp(f);
        __syncthreads();
        kexp = 0;
#pragma unroll
        for (int c = 0; c < NCC; ++c) kexp = max(kexp, sKexp[c * NB + lane]);
        const int e = __reduce_max_sync(0xffffffffu, scale_exp(f, -kexp));
        if (lane == 0) sCexp[warp] = e;
        put_b<0>(sB, warp, lane, biased_digits(y.x, e + kexp), biased_digits(y.y, e + kexp));
      }
    }
    int t = 0;
    double2 cv[4];
    for (int row0 = r0; row0 < r1 && ok; row0 += TM, ++t) {
      int e = kNoExp;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        e = max(e, scale_exp(exp_field(v[q]), __shfl_sync(0xffffffffu, kexp, chunk * 8 + q)));
      int* rexp = sRexp + (t % 3) * 4 * TM;  // a slower warp may still read tile t - 2's
      rexp[chunk * TM + ar] = e;
      if (!(ok = wait_products())) break;  // A free, the exponents visible
      e = max(max(rexp[ar], rexp[TM + ar]), max(rexp[2 * TM + ar], rexp[3 * TM + ar]));
      {
        long long jr[8], ji[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int eq = e - __shfl_sync(0xffffffffu, kexp, chunk * 8 + q);
          jr[q] = biased_digits(v[q].x, eq);
          ji[q] = biased_digits(v[q].y, eq);
        }
        put_a<0>(sA, ar, chunk, jr, ji);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        issue_tile(tmem + (uint32_t)(t & 1) * ACC_COLS, smem_u32(sA), smem_u32(sB), smem_u32(mbar));
      }
      ++issued;
      if (row0 + TM < r1) load_a(row0 + TM);
      if (t > 0) epilogue(row0 - TM, r1, t - 1, cv);
      const int row = row0 + er;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        cv[c] = (row < r1 && ec + c < ncol) ? X[(size_t)(ec + c) * n + row] : make_double2(0.0, 0.0);
    }
    if (t > 0 && ok && (ok = wait_products())) epilogue(r0 + (t - 1) * TM, r1, t - 1, cv);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // X current for the next block, B and the accumulators free
  }
  if (!ok && tid == 0) {
    atomicOr(&stat[u.stat_off], LSMS_UNIT_TIMEOUT);
    if (issued > 0) mbar_wait(mbar, (uint32_t)((issued - 1) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

int solve64_tc_chunk(const Unit* d_units, int n_units, const char* fac_base, char* ws, int nrhs, int32_t* stat,
                     cudaStream_t st) {
  LSMS_SMEM_LIMIT(k_solve64_tc, oz::kSolveSmem);
  LSMS_LAUNCH(k_solve64_tc, dim3(n_units, (nrhs + oz::NCC - 1) / oz::NCC), dim3(oz::NT),
              oz::kSolveSmem, st, d_units,
              fac_base, ws, nrhs, stat);
  return LSMS_OK;
}

}  // namespace lsms
