// Complex64 triangular solves of 9 to 32 right-hand sides on the 5th-generation
// tensor cores (tcgen05, sm_103a): one chain per unit (L y = P b, then U x = y).
//
// What bounds it: one read of the factors.  128 x 32 entries are 32 KB, about 1500
// clocks of an SM's share of the memory bandwidth; the FP32 pipes need 4100 (16
// columns) or 8200 clocks for their multiply-adds.  So the rows are taken in groups
// of 128, left-looking: a group's product with everything solved before it,
//   acc = F[group, 0 .. k) y[0 .. k)        (backward: the columns right of it),
// runs on the tensor cores with the factor streamed through shared memory once for
// all columns and X read from L2 as the other operand; X is written once.  A
// right-looking form would read and write the rows of X at every block instead.
//
// Operands.  Every FP32 value is split into three bf16 parts of 8 bits (24 bits, the
// rest below 2^-25 of the value); the six products of weight 2^-16 and above run as
// bf16 tcgen05.mma with FP32 accumulation, one accumulator per weight class (the
// parts' planes of B lie one after the other, so one instruction per part of A forms
// all its classes).  Every 128 complex K the accumulators are added into FP32
// registers, smallest class first, so the tensor cores' truncating accumulation
// spans 16 instructions at most.  The complex product is the real embedding
//   [Re | Im] += [Re F | Im F] x [[Re y, Im y], [-Im y, Re y]].
// Within a group the four 32-row blocks are solved in turn in FP32 from shared memory:
// y_b = T_b^{-1} x_b with the stored inverse of the diagonal block, then the group's
// remaining rows.
//
// Measured (1,488 units of n about 850, two solves each): 16 columns 6.4 ms, 32
// columns 8.9 ms, against 11.2 and 18.4 ms (two slices of 16) for chains with the row
// updates on the FP32 pipes; the refined tau's error against 64 bits fell (n = 688:
// 2.35e-11 to 1.74e-11).  Without the L2 requests ahead 8.1 and 11.0 ms, and with loads instead of
// asynchronous copies of the group's blocks 7.2 and 9.6 ms.  What is left
// above the factor's read (2.5 ms each) is latency: two CTAs per SM, each a chain of
// split, product and wait per block and of 4 dependent blocks per group.
#include <cstdint>

#include "common.cuh"
#include "tc_bf16.cuh"

namespace lsms {

namespace ts {

using namespace tb;

constexpr int NB = 32;              // complex K per step, rows per diagonal block
constexpr int TM = 128;             // rows per group (TMEM lanes)
constexpr int NT = 256;
constexpr int kAhead = 3;           // blocks requested into L2 ahead of their loads
constexpr int WINDOW = 4;           // steps (128 complex K) between additions into registers
constexpr int PLANE_A = TM * 128;   // 64 real K x 2 bytes per row, 128-byte swizzle

template <int NCOL> constexpr int kPlaneB = 2 * NCOL * 128;
template <int NCOL> constexpr int kLdX = NCOL + 2;  // row stride of the group's X in shared memory
template <int NCOL> constexpr int kBBytes = NP * kPlaneB<NCOL> > 2 * NB * NB * 8 ? NP * kPlaneB<NCOL> : 2 * NB * NB * 8;
template <int NCOL>
constexpr int kSmem = NP * PLANE_A + kBBytes<NCOL> + TM * kLdX<NCOL> * 8 + 64 + 1024;
template <int NCOL> constexpr uint32_t kTmemCols = NP * 2 * NCOL <= 128 ? 128 : 256;
static_assert((96 + 64 + 32) * NB * 8 == NP * PLANE_A, "a group's off-diagonal blocks fill the A planes");

}  // namespace ts

// grid (n_units), block 256, dynamic smem ts::kSmem (two CTAs per SM).  In place on
// the n x nrhs complex64 block X (right-hand sides permuted by k_perm_rows before).
// Waits on the tensor core are bounded (LSMS_UNIT_TIMEOUT).
template <int NCOL>
__global__ void __launch_bounds__(ts::NT, 2) k_solve_tc(const Unit* __restrict__ units, const char* fac_base, char* ws,
                                                        int nrhs, const int32_t* done, int32_t* stat) {
  using namespace ts;
  const Unit u = units[blockIdx.x];
  if (done && done[u.stat_off]) return;
  const int n = u.n;
  const float2* __restrict__ F = reinterpret_cast<const float2*>(fac_base + u.fac_off);
  const float2* __restrict__ D = reinterpret_cast<const float2*>(fac_base + u.m64_off + diag_inv_rel_off(n));
  float2* X = reinterpret_cast<float2*>(ws + u.x32_off);
  constexpr int LDX = kLdX<NCOL>;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = smem + NP * PLANE_A;
  float2* sX = reinterpret_cast<float2*>(sB + kBBytes<NCOL>);          // the group's rows, [TM][LDX]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sX + TM * LDX);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);
  // while a group is solved the operand planes hold its off-diagonal blocks and two diagonal inverses
  float2* sL = reinterpret_cast<float2*>(sA);
  float2* sD = reinterpret_cast<float2*>(sB);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kTmemCols<NCOL>));
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

  int issued = 0;  // steps committed; each is waited for before the next is issued
  bool ok = true;
  auto wait_products = [&]() -> bool {  // bounded, CTA-uniform
    bool w = true;
    if (warp == 0 && issued > 0) w = mbar_wait(mbar, (uint32_t)((issued - 1) & 1));
    w = __syncthreads_and(w);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return w;
  };

  // A: row ar of the group, 16 columns from ac; B: column bc, RPT rows from bj; accumulators: row
  // er of the group, HC complex columns from ec
  const int ar = tid & (TM - 1), ac = (tid >> 7) * 16;
  constexpr int RPT = NCOL * NB / NT, TPC = NB / RPT, HC = NCOL / 2;
  const int bc = tid / TPC, bj = (tid % TPC) * RPT;
  const int er = (warp & 3) * 32 + lane, ec = (warp >> 2) * HC;
  const int nb = (n + NB - 1) / NB, ng = (n + TM - 1) / TM;

  for (int gi = 0; gi < 2 * ng && ok; ++gi) {
    const bool fwd = gi < ng;
    const int g0 = TM * (fwd ? gi : 2 * ng - 1 - gi);
    const int rows = min(TM, n - g0);
    const int k0 = fwd ? 0 : g0 / NB + 4, k1 = fwd ? g0 / NB : nb;  // blocks solved before this group
    float2 acc[HC];
#pragma unroll
    for (int c = 0; c < HC; ++c) acc[c] = make_float2(0.f, 0.f);
    float2 av[16], bv[RPT];
    auto load = [&](int kb) {
      const int row = g0 + ar, kc = kb * NB;
#pragma unroll
      for (int q = 0; q < 16; ++q)
        av[q] = (ar < rows && kc + ac + q < n) ? __ldg(&F[(size_t)(kc + ac + q) * n + row]) : make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < RPT; ++q)
        bv[q] = (bc < nrhs && kc + bj + q < n) ? X[(size_t)bc * n + kc + bj + q] : make_float2(0.f, 0.f);
    };
    // acc += the accumulators' classes, smallest first
    auto flush = [&]() {
      const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)ec;
#pragma unroll
      for (int h = 0; h < HC; h += 8) {
        float re[NP][8], im[NP][8];
#pragma unroll
        for (int s = 0; s < NP; ++s) {
          tmem_ld8(base + (uint32_t)(s * 2 * NCOL + h), re[s]);
          tmem_ld8(base + (uint32_t)(s * 2 * NCOL + NCOL + h), im[s]);
        }
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          acc[h + c].x += re[0][c] + (re[1][c] + re[2][c]);
          acc[h + c].y += im[0][c] + (im[1][c] + im[2][c]);
        }
      }
    };
    // The factor is requested into L2 kAhead blocks before its loads, in the order of use: the group's
    // len blocks, its four diagonal ones, then the next group's.  A block (32 columns of 128 rows) is
    // 256 lines of 128 bytes, one per thread.
    const int len = max(0, k1 - k0);
    const int g1 = fwd ? (gi + 1 < ng ? g0 + TM : g0) : g0 - TM;          // the next group
    const int n0 = gi + 1 < ng ? 0 : g1 / NB + 4, nlen = max(0, (gi + 1 < ng ? g1 / NB : nb) - n0);
    auto prefetch = [&](int t) {
      int g = g0, kb = k0 + t;
      if (t >= len) kb = g0 / NB + t - len;
      if (t >= len + 4) {
        t -= len + 4;
        g = g1;
        kb = t < nlen ? n0 + t : g1 / NB + t - nlen;
      }
      const int row = g + (tid & 7) * 16, col = kb * NB + (tid >> 3);
      if (g >= 0 && row < n && col < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(F + (size_t)col * n + row));
    };
    if (gi == 0)
      for (int t = 0; t < kAhead; ++t) prefetch(t);
    {  // the group's diagonal inverses, 64 lines each
      const int b = g0 / NB + (tid >> 6);
      if (b < nb)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(D + (size_t)b * 2 * NB * NB + (fwd ? 0 : NB * NB) + (tid & 63) * 16));
    }
    if (k0 < k1) load(k0);
    for (int kb = k0; kb < k1; ++kb) {
      prefetch(kb - k0 + kAhead);
      if (!(ok = wait_products())) break;  // the planes are free
      const int w = (kb - k0) % WINDOW;
      if (kb > k0 && w == 0) flush();
      {  // A planes: real parts of columns ac .. ac + 15 to units ac / 8 and ac / 8 + 1, imaginary parts 4 units on
        uint8_t* p = sA + ar * 128;
        const int x = ar & 7;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t re[4][NP], im[4][NP];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 v0 = av[8 * h + 2 * q], v1 = av[8 * h + 2 * q + 1];
            split3(v0.x, v1.x, re[q]);
            split3(v0.y, v1.y, im[q]);
          }
          const int unit = ac / 8 + h;
#pragma unroll
          for (int s = 0; s < NP; ++s) {
            *reinterpret_cast<uint4*>(p + s * PLANE_A + ((unit ^ x) << 4)) =
                make_uint4(re[0][s], re[1][s], re[2][s], re[3][s]);
            *reinterpret_cast<uint4*>(p + s * PLANE_A + (((4 + unit) ^ x) << 4)) =
                make_uint4(im[0][s], im[1][s], im[2][s], im[3][s]);
          }
        }
      }
      {  // B planes: row bc (real output) Re at K j, -Im at 32 + j; row NCOL + bc (imaginary) Im and Re
        const int x = bc & 7, unit = bj >> 3, off = (bj & 7) * 2;  // (NCOL + bc) & 7 == bc & 7
        uint8_t* p = sB + bc * 128;
        uint8_t* q = p + NCOL * 128;
        const int o0 = ((unit ^ x) << 4) + off, o1 = (((4 + unit) ^ x) << 4) + off;
        uint32_t re[RPT / 2][NP], im[RPT / 2][NP];
#pragma unroll
        for (int j = 0; j < RPT / 2; ++j) {
          split3(bv[2 * j].x, bv[2 * j + 1].x, re[j]);
          split3(bv[2 * j].y, bv[2 * j + 1].y, im[j]);
        }
#pragma unroll
        for (int s = 0; s < NP; ++s) {
#pragma unroll
          for (int j = 0; j < RPT / 2; ++j) {
            const int o = s * kPlaneB<NCOL> + 4 * j;
            *reinterpret_cast<uint32_t*>(p + o + o0) = re[j][s];
            *reinterpret_cast<uint32_t*>(p + o + o1) = im[j][s] ^ 0x80008000u;
            *reinterpret_cast<uint32_t*>(q + o + o0) = im[j][s];
            *reinterpret_cast<uint32_t*>(q + o + o1) = re[j][s];
          }
        }
      }
      if (kb + 1 < k1) load(kb + 1);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tid == 0) {
        const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
#pragma unroll
        for (int s = 0; s < NP; ++s)
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            mma_bf16(tmem + (uint32_t)(s * 2 * NCOL), make_desc(a0 + s * PLANE_A + ks * 32), make_desc(b0 + ks * 32),
                     make_idesc(TM, 2 * NCOL * (NP - s)), (w | ks | s) ? 1u : 0u);
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(mbar))
                     : "memory");
      }
      ++issued;
    }
    if (!ok) break;
    if (k0 < k1) {
      if (!(ok = wait_products())) break;
      flush();
    }
    // the group's off-diagonal blocks: step i (block b = i forward, 3 - i backward) updates 96 - 32 i
    // rows, forward those below block b, backward those above; and the first two diagonal inverses
    auto load_d = [&](int i) {  // into slot i & 1, completed by cp.async.wait_all
      const int b = g0 / NB + (fwd ? i : 3 - i);
      const float2* Db = D + (size_t)b * 2 * NB * NB + (fwd ? 0 : NB * NB);
      if (b < nb)
#pragma unroll
        for (int q = 0; q < NB * NB / 2 / NT; ++q) {
          const int idx = 2 * (tid + q * NT);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sD + (i & 1) * NB * NB + idx)),
                       "l"(Db + idx)
                       : "memory");
        }
    };
    // copy groups: the first two inverses and the blocks of step 0, then those of steps 1 and 2
    load_d(0);
    load_d(1);
    {
      int off = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int R = 96 - 32 * i, b = fwd ? i : 3 - i, rs = fwd ? 32 * (b + 1) : 0;
#pragma unroll 4
        for (int q = 0; q < R * NB / NT; ++q) {
          const int idx = tid + q * NT;
          const int r = rs + idx % R, c = 32 * b + idx / R;
          const bool in = r < rows && c < rows;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(sL + off + idx)),
                       "l"(F + (in ? (size_t)(g0 + c) * n + g0 + r : 0)), "r"(in ? 8 : 0)
                       : "memory");
        }
        off += R * NB;
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    }
    // x = b - acc
#pragma unroll
    for (int c = 0; c < HC; ++c) {
      float2 x = make_float2(0.f, 0.f);
      if (er < rows && ec + c < nrhs) {
        x = X[(size_t)(ec + c) * n + g0 + er];
        x = make_float2(x.x - acc[c].x, x.y - acc[c].y);
      }
      sX[er * LDX + ec + c] = x;
    }
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();
    int off = 0;
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
      const int b = fwd ? i : 3 - i, R = 96 - 32 * i, rs = fwd ? 32 * (b + 1) : 0;
      if (i == 1 || i == 2) {
        load_d(i + 1);  // its slot was last read in step i - 1
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
      prefetch(len + i + kAhead);
      if (32 * b < rows) {  // a block of the last, partial group may be missing
        // y = T^{-1} x: lane = row, warp = NCOL / 8 columns
        constexpr int CW = NCOL / 8;
        const int c0 = warp * CW;
        const float2* sDi = sD + (i & 1) * NB * NB + lane;
        float2 y0[CW], y1[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) y0[c] = y1[c] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < NB; j += 2) {
          const float2 d0 = sDi[j * NB], d1 = sDi[(j + 1) * NB];
          const float2* x0 = sX + (32 * b + j) * LDX + c0;
#pragma unroll
          for (int c = 0; c < CW; c += 2) {
            const float4 xa = *reinterpret_cast<const float4*>(x0 + c);
            const float4 xb = *reinterpret_cast<const float4*>(x0 + LDX + c);
            y0[c] = cfma(d0, make_float2(xa.x, xa.y), y0[c]);
            y0[c + 1] = cfma(d0, make_float2(xa.z, xa.w), y0[c + 1]);
            y1[c] = cfma(d1, make_float2(xb.x, xb.y), y1[c]);
            y1[c + 1] = cfma(d1, make_float2(xb.z, xb.w), y1[c + 1]);
          }
        }
        __syncwarp();  // a warp reads and writes its own columns only
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          const float2 y = make_float2(y0[c].x + y1[c].x, y0[c].y + y1[c].y);
          const int r = 32 * b + lane;
          sX[r * LDX + c0 + c] = y;
          if (r < rows && c0 + c < nrhs) X[(size_t)(c0 + c) * n + g0 + r] = y;
        }
        __syncwarp();
        // the group's remaining rows: lane = row within each of the R / 32 blocks
        if (i < 3) {
          float2 a[3][CW];
#pragma unroll
          for (int m = 0; m < 3; ++m)
            if (32 * m < R)
#pragma unroll
              for (int c = 0; c < CW; ++c) a[m][c] = sX[(rs + 32 * m + lane) * LDX + c0 + c];
#pragma unroll 4
          for (int j = 0; j < NB; ++j) {
            const float2* yj = sX + (32 * b + j) * LDX + c0;
            float4 yy[CW / 2];
#pragma unroll
            for (int c = 0; c < CW / 2; ++c) yy[c] = *reinterpret_cast<const float4*>(yj + 2 * c);
#pragma unroll
            for (int m = 0; m < 3; ++m)
              if (32 * m < R) {
                const float2 l = sL[off + j * R + 32 * m + lane];
#pragma unroll
                for (int c = 0; c < CW / 2; ++c) {
                  a[m][2 * c] = cfms(l, make_float2(yy[c].x, yy[c].y), a[m][2 * c]);
                  a[m][2 * c + 1] = cfms(l, make_float2(yy[c].z, yy[c].w), a[m][2 * c + 1]);
                }
              }
          }
#pragma unroll
          for (int m = 0; m < 3; ++m)
            if (32 * m < R)
#pragma unroll
              for (int c = 0; c < CW; ++c) sX[(rs + 32 * m + lane) * LDX + c0 + c] = a[m][c];
        }
      }
      off += R * NB;
      // step 1 needs the second group, the later steps everything issued
      if (i == 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();  // the next inverse is there, this one's slot free; after the last step X is current
    }
  }
  if (!ok && tid == 0) {
    atomicOr(&stat[u.stat_off], LSMS_UNIT_TIMEOUT);
    mbar_wait(mbar, (uint32_t)((issued - 1) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols<NCOL>));
  }
}

int solve_tc_chunk(const Unit* d_units, int n_units, const char* fac_base, char* ws, int nrhs, const int32_t* done,
                   int32_t* stat, cudaStream_t st) {
  LSMS_SMEM_LIMIT(k_solve_tc<16>, ts::kSmem<16>);
  LSMS_SMEM_LIMIT(k_solve_tc<32>, ts::kSmem<32>);
  if (nrhs < 1 || nrhs > 32) return fail(LSMS_ERR_ARG, "internal: solve_tc_chunk nrhs %d", nrhs);
  if (nrhs <= 16)
    LSMS_LAUNCH(k_solve_tc<16>, dim3(n_units), dim3(ts::NT), ts::kSmem<16>, st, d_units, fac_base, ws, nrhs, done, stat);
  else
    LSMS_LAUNCH(k_solve_tc<32>, dim3(n_units), dim3(ts::NT), ts::kSmem<32>, st, d_units, fac_base, ws, nrhs, done, stat);
  return LSMS_OK;
}

}  // namespace lsms
