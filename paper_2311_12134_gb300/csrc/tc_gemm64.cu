// Trailing update of the complex128 LU, A22 -= L21 U12, on the 5th-generation
// tensor cores (tcgen05, sm_103a): the products are formed exactly from bf16
// digits (the Ozaki scheme) and rounded to FP64 once per panel.
//
// What bounds it.  GB300's FP64 pipe retires 2 multiply-adds per SM and clock, so
// the 128 of one complex element and panel (NB = 32) cost 64 clocks; as integer
// digit products the same update needs 0.9 clocks of the tensor pipe, and what is
// left is the epilogue (one FP64 conversion and one multiply-add per real value).
//
// Digits.  Row r of L21 is scaled by its largest exponent, column c of U12 by
// its own.  A scaled value |v| < 2^E becomes the fixed-point integer
// rint(v 2^(55 - E)) and its seven balanced base-256 digits,
//   v 2^(7 - E) = sum_{s=0..6} a_s 2^(-8 s) + rest,  -128 <= a_s <= 128,
//   |rest| <= 2^-49 (2^-56 of 2^E),
// taken with integer instructions (no FP64 operation) and exact in bf16.  The 28
// digit pairs s + t <= 6 run as bf16 products with FP32 accumulation in tensor
// memory, one accumulator per class g = s + t; a class holds at most 7 pairs of
// 2^14 per real K, so the 64 real K of a panel sum exactly (below 2^23).  Left
// out are the classes g >= 7, below 2^-56 of the two scales per term: less than
// the roundings of the 128 FP64 multiply-adds that they replace.  The complex
// product is the real embedding
//   [Re C | Im C] -= [Re L | Im L] x [[Re U, Im U], [-Im U, Re U]].
// The B planes of the digits t = 0, 1, .. lie one after the other, so one
// instruction per digit s of A forms all its classes: N = 32 (7 - s) columns
// starting at class s, and A is read 7 times per 16 K instead of 28.
//
// Measured (216 matrices of n = 688, 21 panels): 14.4 ms against 165 ms for a
// register-tiled product on the FP64 pipe (0.98 of that pipe's rate); the tau
// blocks' error against a 64-bit solve is unchanged (1.4e-13).
#include <algorithm>
#include <cstdint>

#include "common.cuh"

namespace lsms {

namespace oz {

constexpr int ND = 7;                 // digits per operand, classes per accumulator
constexpr int NB = 32;                // complex panel width
constexpr int TM = 128;               // rows per CTA (TMEM lanes)
constexpr int NCC = 16;               // complex columns per tile
constexpr int NR = 2 * NCC;           // real accumulator columns per class: [Re | Im]
constexpr int NT = 512;               // threads: (row, 8-column chunk) of L21; (column, row) of a U12 tile
constexpr int PLANE_A = TM * 128;     // one digit of A: 64 real K x 2 bytes per row, 128-byte swizzle
constexpr int PLANE_B = NR * 128;
constexpr int STAGE_B = ND * PLANE_B;
constexpr int SMEM_BYTES = ND * PLANE_A + 2 * STAGE_B + 4 * TM * 4 + 4 * NCC * 4 + 64 + 1024;
constexpr uint32_t ACC_COLS = 256;    // columns between the two accumulators (ND * NR = 224 used)
constexpr uint32_t TMEM_COLS = 512;
constexpr long long kWaitLimit = 1ll << 24;  // bounded mbarrier wait (polls)
static_assert(ND * NR <= (int)ACC_COLS && NT == TM * 4 && NT == NCC * NB, "tile shape");

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// K-major operand, 128-byte swizzle, one 128-byte row per matrix row: 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// kind::f16 with bf16 A and B: D f32, both K-major, N and M.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(mbar), "r"(phase)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {  // completed by tcgen05.wait::ld
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(taddr));
}

__device__ __forceinline__ int exp_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// rint(v 2^(55 - E)) plus 128 in each of the six low bytes, E = emax - 1022 (|v| < 2^E when
// v's exponent field is at most emax): bytes 0..5 are digits 6..1 plus 128, the bits from 48
// up digit 0.  Subnormals count as zero (below 2^-1022).
__device__ __forceinline__ long long biased_digits(double v, int emax) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const long long m = e ? ((b & 0xfffffffffffffll) | 0x10000000000000ll) : 0ll;
  const int sh = e - emax + 2;  // <= 2
  const int r = min(max(-sh, 0), 62);
  const long long half = r ? 1ll << (r - 1) : 0ll;
  const long long mag = ((m << max(sh, 0)) + half) >> r;
  return (b < 0 ? -mag : mag) + 0x0000808080808080ll;
}

// Digit s of a biased value as the bits of a float (an integer of at most 8 significant
// bits: its upper 16 bits are the bf16 value, exactly).
template <int s>
__device__ __forceinline__ uint32_t digit_bits(long long j) {
  if constexpr (s == 0) {
    const uint32_t hi = (uint32_t)((unsigned long long)j >> 32) ^ 0x80000000u;
    return __float_as_uint(__uint_as_float(__byte_perm(hi, 0x4B000000u, 0x7432)) - 8421376.f);
  } else {
    const uint32_t w = s <= 2 ? (uint32_t)((unsigned long long)j >> 32) : (uint32_t)j;
    constexpr int byte = s <= 2 ? 2 - s : 6 - s;
    return __float_as_uint(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 + byte)) - 8388736.f);
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

// The class sums of one real value as a fixed-point integer in units of 2^-40 of the class-0
// weight: exact but for the last class, rounded to that unit (2^-54 of the two scales).
__device__ __forceinline__ long long class_sum(const float (&v)[ND]) {
  int i[ND];
#pragma unroll
  for (int g = 0; g < ND; ++g) i[g] = __float2int_rn(v[g]);
  const int a = i[0] * 256 + i[1];                          // below 2^29
  const int b = i[2] * 256 + i[3];                          // below 2^30
  const int c = i[4] * 256 + i[5] + ((i[6] + 128) >> 8);    // below 2^31
  return ((long long)a << 32) + (long long)b * 65536 + c;
}

}  // namespace oz

// grid (row tiles of 128, n_units, column splits), block 512, dynamic smem
// oz::SMEM_BYTES (one CTA per SM).  One CTA per 128-row block of a unit's trailing
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
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sCexp + 4 * NCC);  // [2], one per accumulator
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
  auto stage_u = [&](int j, double2 v) {
    int e = max(exp_field(v.x), exp_field(v.y));
    e = __reduce_max_sync(0xffffffffu, e);
    // (slots of 4: a slower warp may still read the exponents of tile j - 2)
    if (lane == 0) sCexp[(j & 3) * NCC + warp] = e == 0x7ff ? 1 << 14 : e;
    put_b<0>(sB + (j & 1) * STAGE_B, warp, lane, biased_digits(v.x, e), biased_digits(v.y, e));
  };
  double2 uv = load_u(j0);

  // L21: thread (row, chunk of 8 columns)
  const int ar = tid & (TM - 1), chunk = tid >> 7;
  {
    const int row = row0 + ar;
    double2 v[8];
    int e = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      v[q] = row < n ? A[(size_t)(k + chunk * 8 + q) * n + row] : make_double2(0.0, 0.0);
      e = max(e, max(exp_field(v[q].x), exp_field(v[q].y)));
    }
    sRexp[chunk * TM + ar] = e;
    __syncthreads();
    e = max(max(sRexp[ar], sRexp[TM + ar]), max(sRexp[2 * TM + ar], sRexp[3 * TM + ar]));
    long long jr[8], ji[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      jr[q] = biased_digits(v[q].x, e);
      ji[q] = biased_digits(v[q].y, e);
    }
    put_a<0>(sA, ar, chunk, jr, ji);
  }

  // epilogue: TMEM lane (warp % 4) * 32 + lane = row, complex columns 4 (warp / 4) .. + 3
  const int er = (warp & 3) * 32 + lane, ec = (warp >> 2) * 4;
  const int crow = row0 + er;
  int rexp = max(max(sRexp[er], sRexp[TM + er]), max(sRexp[2 * TM + er], sRexp[3 * TM + er]));
  if (rexp == 0x7ff) rexp = 1 << 14;

  auto issue = [&](int j, uint32_t tmem) {  // one thread: the 28 products of a tile
    const uint32_t d = tmem + (uint32_t)(j & 1) * ACC_COLS;
    const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB + (j & 1) * STAGE_B);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int s = 0; s < ND; ++s)
        mma_bf16(d + (uint32_t)(s * NR), make_desc(a0 + s * PLANE_A + ks * 32), make_desc(b0 + ks * 32),
                 make_idesc(TM, NR * (ND - s)), (ks | s) ? 1u : 0u);
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(mbar + (j & 1)))
                 : "memory");
  };
  // stage U12 of tile j (its buffer and accumulator free: tile j - 2 is done) and issue its product
  uint32_t tmem = 0;
  auto launch_tile = [&](int j) {
    stage_u(j - j0, uv);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem = *tslot;
    if (tid == 0) issue(j - j0, tmem);
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
    if (warp == 0) {
      ok = false;
      const uint32_t mb = smem_u32(mbar + (it & 1));
      for (long long q = 0; q < kWaitLimit; ++q)
        if (mbar_try_wait(mb, (uint32_t)((it >> 1) & 1))) {
          ok = true;
          break;
        }
    }
    ok = __syncthreads_and(ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) break;
    const uint32_t base = tmem + (uint32_t)(it & 1) * ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ec;
    float re[ND][4], im[ND][4];
#pragma unroll
    for (int g = 0; g < ND; ++g) {
      tmem_ld4(base + (uint32_t)(g * NR), re[g]);
      tmem_ld4(base + (uint32_t)(g * NR + NCC), im[g]);
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float vr[ND], vi[ND];
#pragma unroll
      for (int g = 0; g < ND; ++g) {
        vr[g] = re[g][c];
        vi[g] = im[g][c];
      }
      // L U = class sum x 2^(eL - 1022 + eU - 1022 - 14 - 40)
      const int ex = rexp + sCexp[(it & 3) * NCC + ec + c] - 1075;
      const double sc = __hiloint2double(ex <= 0 ? 0 : (ex >= 0x7ff ? 0x7ff80000 : ex << 20), 0);
      const double2 r = make_double2(fma(-(double)class_sum(vr), sc, cv[c].x), fma(-(double)class_sum(vi), sc, cv[c].y));
      if (crow < n && c0 + c < n) A[(size_t)(c0 + c) * n + crow] = r;
    }
  }
  if (!ok && tid == 0) {
    atomicOr(&stat[u.stat_off], LSMS_UNIT_TIMEOUT);
    // give the tensor core a second bounded window before the accumulators are freed
    const uint32_t mb = smem_u32(mbar + (issued & 1));
    for (long long q = 0; q < kWaitLimit; ++q)
      if (mbar_try_wait(mb, (uint32_t)((issued >> 1) & 1))) break;
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
  static bool attr_set = false;
  if (!attr_set) {
    LSMS_CUDA_TRY(cudaFuncSetAttribute(k_gemm64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM_BYTES));
    attr_set = true;
  }
  const int mt = n_max - k - oz::NB;
  if (mt <= 0) return LSMS_OK;
  const int rows = (mt + oz::TM - 1) / oz::TM, tiles = (mt + oz::NCC - 1) / oz::NCC;
  // few row blocks: the columns split over CTAs too, at least 4 tiles each (a CTA's staging of
  // L21 costs about as much as two tiles)
  const int want = 2 * 152 / std::max(1, rows * n_units);
  const int split = std::max(1, std::min(want, tiles / 4));
  LSMS_LAUNCH(k_gemm64_tc, dim3(rows, n_units, split), dim3(oz::NT), oz::SMEM_BYTES, st, d_units, fac_base, k, stat);
  return LSMS_OK;
}

}  // namespace lsms
