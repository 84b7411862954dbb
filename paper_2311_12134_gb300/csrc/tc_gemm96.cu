// Trailing update of large complex64 matrices, A22 -= L21 U12 with 96 complex columns
// of L at once, on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// What bounds the 32-column update (k_gemm_tc): it streams the trailing matrix once
// per 32 columns (0.84 of the memory rate; 0.61 of a 0.98 s call at n = 15,440).
// With 96 columns it is streamed a third as often; per 128 x 32 outputs and three stages
// of 32 complex K that is 2300 clocks of the tensor pipe and 3030 of memory.
// Operands as in tc_solve.cu: three bf16 parts per value, six products, one FP32
// accumulator per weight class (smallest added first); per class a value is the sum of
// 12 instructions.  The parts of the CTA's 128 x 96 block of L21 stay in shared memory
// (144 KB) for its whole walk over the columns; U12's pass through three stages of 32 K
// x 32 columns.  Warps have one role each and meet at mbarriers only (stage full / free,
// accumulator full / free): two groups of four split U12, a stage each in turn, with
// loads two of their stages ahead; one warp issues the products; two groups of four do
// the epilogues, a tile (an accumulator) each in turn.
// Measured: 108 matrices of n = 2192 18.0 ms (32-column updates 35.5), 4 of n = 15,440
// 226 ms (609).  What bounds it now is the latency of dependent products: an
// instruction takes about 115 clocks whatever its N, because the next one adds into the
// same columns (the tensor pipe is busy half of the time).  Hence the 32-column tiles (N =
// 192, 128, 64); with 16-column tiles 27 and 353 ms, with L21 in tensor memory beside
// them 29.5 and 384, with the splitting or the epilogue left out 25 and 26 instead of 27.
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "tc_bf16.cuh"

namespace lsms {

namespace tg {

using namespace tb;

constexpr int KB = kBlkK;               // complex K (columns of L per update)
constexpr int NB = 32;                  // complex K per stage
constexpr int TM = 128;                 // rows per CTA (TMEM lanes)
constexpr int NCC = 32;                 // complex columns per tile
constexpr int NR = 2 * NCC;             // real accumulator columns per class
constexpr int NW = 8;                   // splitting warps, two groups of four
constexpr int NE = 8;                   // epilogue warps, two groups of four
constexpr int NT = 32 * (NW + 1 + NE);  // and the warp that issues the products
constexpr int PLANE_B = NR * 128;       // one part of a stage: 32 complex K, 128-byte rows, 128-byte swizzle
constexpr int STAGE_B = NP * PLANE_B;
constexpr int NKC = KB / NB;            // stages per tile
constexpr int NS = 3;                   // stages in flight
constexpr int CHUNK_A = TM * 128;       // 32 complex K of one part of L21: 128-byte rows, 128-byte swizzle
constexpr int PLANE_A = NKC * CHUNK_A;
constexpr int SMEM_BYTES = NP * PLANE_A + NS * STAGE_B + (2 * NS + 4) * 8 + 64 + 1024;
constexpr uint32_t ACC_COLS = NP * NR;  // tensor memory columns of an accumulator (two of them)
constexpr uint32_t TMEM_COLS = 512;
static_assert(2 * ACC_COLS <= TMEM_COLS && SMEM_BYTES <= 227 * 1024, "tensor and shared memory");

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {  // completed by tcgen05.wait::ld
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(taddr));
}

}  // namespace tg

// grid (row tiles of 128, n_units, column splits), block 544, dynamic smem
// tg::SMEM_BYTES (one CTA per SM).  K0: first of the 96 columns of L21.
__global__ void __launch_bounds__(tg::NT, 1) k_gemm_tc96(const Unit* __restrict__ units, char* fac_base, int K0,
                                                          int32_t* stat) {
  using namespace tg;
  const Unit u = units[blockIdx.y];
  const int n = u.n;
  const int t0 = K0 + KB;
  const int row0 = t0 + blockIdx.x * TM;
  if (row0 >= n) return;
  const int tiles = (n - t0 + NCC - 1) / NCC;
  const int per = (tiles + gridDim.z - 1) / gridDim.z;
  const int j0 = blockIdx.z * per, j1 = min(tiles, j0 + per);
  if (j0 >= j1) return;
  float2* A = reinterpret_cast<float2*>(fac_base + u.fac_off);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = smem + NP * PLANE_A;
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + NS * STAGE_B);  // [NS] stage of B written
  uint64_t* freed = full + NS;                                     // [NS] its products complete
  uint64_t* acc_full = freed + NS;                                 // [2] accumulator complete
  uint64_t* acc_free = acc_full + 2;                               // [2] and read
  uint32_t* tslot = reinterpret_cast<uint32_t*>(acc_free + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == NW) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(full + i, NW / 2);
      mbar_init(freed + i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_free + i, NE / 2);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int nt = j1 - j0;
  bool ok = true;
  int issued = -1;  // last stage whose products were issued (issuing warp)

  if (warp == NW) {  // ---- the issuing warp
    for (int s = 0; s < NKC * nt; ++s) {
      const int t = s / NKC, kc = s % NKC, slot = s % NS;
      if (!(ok = mbar_wait_warp(full + slot, (uint32_t)((s / NS) & 1)))) break;
      if (kc == 0 && t >= 2 && !(ok = mbar_wait_warp(acc_free + (t & 1), (uint32_t)(((t - 2) >> 1) & 1)))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (lane == 0) {
        const uint64_t a0 = make_desc(smem_u32(sA) + kc * CHUNK_A), b0 = make_desc(smem_u32(sB + slot * STAGE_B));
        const uint32_t d = tmem + (uint32_t)(t & 1) * ACC_COLS;
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)  // the address fields of the descriptors count 16 bytes
            mma_bf16(d + (uint32_t)(p * NR), a0 + (uint64_t)((p * PLANE_A + ks * 32) >> 4), b0 + (uint64_t)((ks * 32) >> 4),
                     make_idesc(TM, NR * (NP - p)), (kc | ks | p) ? 1u : 0u);
        mma_commit(freed + slot);
        if (kc == NKC - 1) mma_commit(acc_full + (t & 1));
      }
      issued = s;
      __syncwarp();
    }
  } else if (warp < NW) {  // ---- splitting warps
    // U12: group grp takes the stages of its parity; lane = (one of two columns, pair of K rows), and the
    // columns 8, 16 and 24 further on; loads two of the group's stages ahead
    const int grp = warp >> 2, uc = 2 * (warp & 3) + (lane >> 4), kp = 2 * (lane & 15);
    const int ns = NKC * nt;
    auto load_u = [&](int s, float2 (&v)[8]) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int col = t0 + (j0 + s / NKC) * NCC + uc + 8 * h;
#pragma unroll
        for (int q = 0; q < 2; ++q)
          v[2 * h + q] =
              (s < ns && col < n) ? A[(size_t)col * n + K0 + NB * (s % NKC) + kp + q] : make_float2(0.f, 0.f);
      }
    };
    float2 u[2][8];
    load_u(grp, u[0]);
    load_u(grp + 2, u[1]);
    {  // L21: thread (row, half of the 96 columns), 16-byte units of 8 columns
      const int r = tid & (TM - 1), row = row0 + r, x = r & 7;
#pragma unroll 1
      for (int i = 0; i < 6; ++i) {
        const int unit = 6 * grp + i, kc = unit >> 2, h = unit & 3;
        uint8_t* p = sA + kc * CHUNK_A + r * 128;
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          v[q] = row < n ? A[(size_t)(K0 + 8 * unit + q) * n + row] : make_float2(0.f, 0.f);
        uint32_t re[4][NP], im[4][NP];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          split3(v[2 * q].x, v[2 * q + 1].x, re[q]);
          split3(v[2 * q].y, v[2 * q + 1].y, im[q]);
        }
#pragma unroll
        for (int s = 0; s < NP; ++s) {
          *reinterpret_cast<uint4*>(p + s * PLANE_A + ((h ^ x) << 4)) = make_uint4(re[0][s], re[1][s], re[2][s], re[3][s]);
          *reinterpret_cast<uint4*>(p + s * PLANE_A + (((4 + h) ^ x) << 4)) =
              make_uint4(im[0][s], im[1][s], im[2][s], im[3][s]);
        }
      }
    }
    // (stage 0 needs the first chunk of L21, written by the first group; later stages come after
    // an arrival of each group)
    for (int s0 = grp; s0 < ns && ok; s0 += 4) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int s = s0 + 2 * i;
        if (s >= ns) break;
        const int slot = s % NS;
        uint32_t re[4][NP], im[4][NP];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          split3(u[i][2 * h].x, u[i][2 * h + 1].x, re[h]);
          split3(u[i][2 * h].y, u[i][2 * h + 1].y, im[h]);
        }
        load_u(s + 4, u[i]);
        if (s >= NS && !(ok = mbar_wait_warp(freed + slot, (uint32_t)((s / NS - 1) & 1)))) break;
        // row uc (real output) Re at K kp, -Im at 32 + kp; row 32 + uc (imaginary) Im and Re
        const int x = uc & 7, unit = kp >> 3, off = (kp & 7) * 2;  // (uc + 8) & 7 == uc & 7
        const int o0 = ((unit ^ x) << 4) + off, o1 = (((4 + unit) ^ x) << 4) + off;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint8_t* p = sB + slot * STAGE_B + (uc + 8 * h) * 128;
          uint8_t* q = p + NCC * 128;
#pragma unroll
          for (int t = 0; t < NP; ++t) {
            *reinterpret_cast<uint32_t*>(p + t * PLANE_B + o0) = re[h][t];
            *reinterpret_cast<uint32_t*>(p + t * PLANE_B + o1) = im[h][t] ^ 0x80008000u;
            *reinterpret_cast<uint32_t*>(q + t * PLANE_B + o0) = im[h][t];
            *reinterpret_cast<uint32_t*>(q + t * PLANE_B + o1) = re[h][t];
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(full + slot);
      }
    }
  } else {  // ---- epilogue warps: TMEM lane (warp % 4) * 32 + lane = row; group eg takes tiles of its parity
    const int crow = row0 + (warp & 3) * 32 + lane;
    const int ew = warp - NW - 1, eg = ew >> 2, et = (ew & 3) * 32 + lane;
    // C tile j: 32 columns of 128 rows, 256 lines, requested into L2
    auto prefetch_c = [&](int j) {
      const int row = row0 + (et & 7) * 16;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col = t0 + j * NCC + (et >> 3) + 16 * h;
        if (j < j1 && col < n && row < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(A + (size_t)col * n + row));
      }
    };
    prefetch_c(j0 + eg);
    for (int t = eg; t < nt && ok; t += 2) {
      const int j = j0 + t;
      prefetch_c(j + 2);
      const uint32_t base = tmem + (uint32_t)eg * ACC_COLS + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
      for (int h = 0; h < NCC && ok; h += 16) {
        float2 cv[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int col = t0 + j * NCC + h + c;
          cv[c] = (crow < n && col < n) ? A[(size_t)col * n + crow] : make_float2(0.f, 0.f);
        }
        if (h == 0) {
          if (!(ok = mbar_wait_warp(acc_full + eg, (uint32_t)((t >> 1) & 1)))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
#pragma unroll
        for (int g = 0; g < 16; g += 4) {
          float re[NP][4], im[NP][4];
#pragma unroll
          for (int s = 0; s < NP; ++s) {
            tmem_ld4(base + (uint32_t)(s * NR + h + g), re[s]);
            tmem_ld4(base + (uint32_t)(s * NR + NCC + h + g), im[s]);
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int c = 0; c < 4; ++c)
            cv[g + c] = make_float2(cv[g + c].x - (re[0][c] + (re[1][c] + re[2][c])),
                                    cv[g + c].y - (im[0][c] + (im[1][c] + im[2][c])));
        }
        if (h + 16 >= NCC) {  // the accumulator is read
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_free + eg);
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int col = t0 + j * NCC + h + c;
          if (crow < n && col < n) A[(size_t)col * n + crow] = cv[c];
        }
      }
    }
  }
  if (!ok && lane == 0) {
    atomicOr(&stat[u.stat_off], LSMS_UNIT_TIMEOUT);
    // products that were issued get a second bounded window before the accumulators are freed
    if (issued >= 0) mbar_wait(freed + issued % NS, (uint32_t)((issued / NS) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == NW) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

int gemm_tc96_chunk(const Unit* d_units, int n_units, int n_max, int K0, char* fac_base, int32_t* stat,
                     cudaStream_t st) {
  LSMS_SMEM_LIMIT(k_gemm_tc96, tg::SMEM_BYTES);
  const int mt = n_max - K0 - tg::KB;
  if (mt <= 0) return LSMS_OK;
  const int rows = (mt + tg::TM - 1) / tg::TM, tiles = (mt + tg::NCC - 1) / tg::NCC;
  // about eight CTAs per SM in turn, so that the last wave is short; at least 8 tiles each (staging
  // L21 costs about as much as two)
  const int split = std::max(1, std::min(8 * 152 / std::max(1, rows * n_units), tiles / 8));
  LSMS_LAUNCH(k_gemm_tc96, dim3(rows, n_units, split), dim3(tg::NT), tg::SMEM_BYTES, st, d_units, fac_base, K0, stat);
  return LSMS_OK;
}

}  // namespace lsms
