// Fused degree step of the finite-element R-ChFSI filter (the loop body of Algorithm 3) on the
// tcgen05 tensor cores, in one pass over the block.
//
// The recurrence R_k = a_k A D^-1 R_{k-1} + b_k R_{k-1} + c_k R_{k-2} + a_k W Lambda_{k-1} runs on
// scaled iterates S_j = s_j R_j, with s_k = s_{k-2} / c_k chosen on the host, so that
//   S_k = S_{k-2} + alpha A D^-1 S_{k-1} + beta S_{k-1} + omega W Lambda_{k-1},
//   alpha = s_k a_k / s_{k-1},  beta = s_k b_k / s_{k-1},  omega = s_k a_k:
// the old iterate enters with coefficient 1, so the whole step is additions into the buffer that
// holds S_{k-2}.  The cell products are added with vector atomics (a dof shared by several cells
// receives one add per cell); beta S_{k-1} + omega W Lambda is added once per dof, by the cell that
// owns it (the first cell, in cell order, that contains it).  Each of S_{k-1}, S_{k-2} and W is
// then read once and S_k written once per step, the four block streams of the algorithm, plus
// the cell matrices.
//
// Per (cell, column tile): D (128 x BN, FP32 in TMEM) = T + (A_c D_c^-1) V_c, where A_c D_c^-1 is the
// cell matrix with its columns scaled by D^-1 at the cell's dofs (padded from n_c <= 128 to 128 x
// 128, packed once per operator as a K-major 128-byte-swizzled TF32 image), V_c (128 x BN) the
// cell's rows of S_{k-1}, and T the owner terms of the cell's owned rows divided by alpha, so that
// alpha D is the whole contribution of the cell.  The rows of V_c and the owned rows of W are
// gathered from the row-major blocks with 16-byte cp.async copies by 256 threads (a warp
// instruction copies whole 256-byte row segments) into a ring of 128-byte-swizzled stages, up to
// two tiles ahead of the tile being converted.  (A single loader warp issuing the copies, or TMA
// tile::gather4 copies of four 128-byte rows, moved only ~6 bytes per clock per SM.)  The same
// threads then convert: each (one cell node, half of the columns) reads its row, stores T into the
// accumulator with tcgen05.st and, after a barrier among the converters, rewrites the stage in
// place as the K-major TF32 operand of the MMA (the swizzled reads and the operand writes are both
// free of shared-memory bank conflicts).
//
// Warp roles (448 threads):
//   warp 0     cell images: one bulk copy per cell (nA buffers);
//   warp 1     MMA issuer (the whole warp walks the loop, one elected lane issues), accumulating
//              onto the owner terms in one of two TMEM accumulators of BN columns;
//   warps 2-9  gather + convert (warp w: nodes 32 (w % 4).., the TMEM lanes it may access, and
//              half of the tile's columns);
//   warps 10-13 epilogue: TMEM lanes 32 (w % 4).. (one cell node per thread); alpha scaling and
//              red.global.add.v4.f32 into the output rows.
// Every mbarrier wait is bounded; on a timeout the kernel raises the error flag, waits (bounded)
// for its copies and MMAs in flight, releases TMEM and returns.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "fe_step.cuh"
#include "prof.cuh"
#include "tc_ptx.cuh"

namespace rchfsi {
namespace {

constexpr int kNCP = 128;                       // padded cell size (MMA M and K)
constexpr int kThreads = 448;                   // 14 warps
constexpr uint32_t kABytes = kNCP * kNCP * 4;   // TF32 cell image
constexpr uint32_t kChunkBytes = kNCP * 128;    // 32 columns of V_c: 128 rows of 128 bytes
constexpr int kWRows = 80;                      // owned rows of W staged per cell (at most)
constexpr uint32_t kWChunkBytes = kWRows * 128;
constexpr int kMaxParts = 64;
constexpr int kMaxStages = 6;
constexpr int kSmemMax = 232448;                // dynamic + static shared memory per CTA

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Byte offset of element (row r, k) of a 128 x 128 K-major 128-byte-swizzled FP32 image.
__device__ __forceinline__ uint32_t sw_off4(int r, int k) {
  const int kb = k >> 5, byte = (k & 31) * 4;
  const int chunk = (byte >> 4) ^ (r & 7);
  return (uint32_t)kb * kNCP * 128 + (uint32_t)r * 128 + (chunk << 4) + (byte & 15);
}

// (A_c D_c^-1) images: column k of cell c scaled by dinv[dofs(c, k)], rounded to TF32.
__global__ void pack_scaled_kernel(int64_t n_cells, int nc, const double* __restrict__ A, const int* __restrict__ dofs,
                                   const double* __restrict__ dinv, uint8_t* __restrict__ img) {
  const int64_t per_cell = (int64_t)kNCP * kNCP;
  const int64_t total = n_cells * per_cell;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = e / per_cell;
    const int r = (int)((e % per_cell) / kNCP), k = (int)(e % kNCP);
    const double v = (r < nc && k < nc) ? A[(c * nc + r) * nc + k] * dinv[dofs[c * nc + k]] : 0.0;
    *reinterpret_cast<float*>(img + c * per_cell * 4 + sw_off4(r, k)) = tf32_rna((float)v);
  }
}

struct StepPartDev {
  const int* dofs;
  const int8_t* own_pos;  // per cell 128 entries: >= 0 when the cell owns its node k
  const uint8_t* img;
  const float* V;
  const float* W;
  float* U;
  const float* lam;
  const double* coef;
  int64_t n_cells, cell_off;
  float alpha, beta, omega, sign;
  int nc, n, ntiles, owner;  // owner = 0: no owner terms in this part
  const float* V2;  // V and U of the odd steps of a loop
  float* U2;
};

struct StepBatch {
  StepPartDev part[kMaxParts];
  int64_t total_cells;
  int nparts, nA, nslots;
  uint32_t tmem_cols;
  int* err;
  // a loop of degree steps (fe_step_t_kernel only, nsteps > 1): alpha, beta, omega per step in `coefs` in place of the
  // parts' own, lam advances by n per step, and the CTAs meet between steps at the counter *sync
  int nsteps;
  int* sync;
  float coefs[3 * kTableSteps];
};

__device__ __forceinline__ int part_of(const StepBatch& p, int64_t g) {
  int q = 0;
  while (q + 1 < p.nparts && g >= p.part[q + 1].cell_off) ++q;
  return q;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc::smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(tc::smem_u32(bar))
               : "memory");
}

// 16-byte asynchronous copy global -> shared (L2 only); `in` = false writes 16 zero bytes instead.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in) {
  // no memory clobber: the copy is ordered by the mbarrier that completes with it, and loads that
  // feed later copies may be scheduled ahead of it
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(in ? 16 : 0));
}

// Arrive on `bar` once every cp.async this thread issued before has completed (the barrier's count
// includes this arrival).
__device__ __forceinline__ void cp_async_arrive_noinc(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Byte offset of element (row r, k) of a K-major 128-byte-swizzled FP32 operand with `rows` rows
// per 32-element K block.
__device__ __forceinline__ uint32_t img_off(int r, int k, int rows) {
  const int kb = k >> 5, byte = (k & 31) * 4;
  return (uint32_t)kb * rows * 128 + (uint32_t)r * 128 + ((((byte >> 4) ^ (r & 7))) << 4) + (byte & 15);
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1) fe_step_kernel(const __grid_constant__ StepBatch p) {
  constexpr int NCH = BN / 32;
  constexpr int CPR = BN / 4;                     // 16-byte chunks per row of a tile
  constexpr int HB = BN / 2;                      // columns of one converter thread per tile
  constexpr uint32_t kHalf = NCH * kChunkBytes;   // 128 rows of BN FP32 values
  constexpr uint32_t kSlotBytes = kHalf + NCH * kWChunkBytes;  // V rows (then the operand), owned W rows
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t afull[2], aempty[2], bfull[kMaxStages], bempty[kMaxStages], ifull[kMaxStages],
      accfull[2], accempty[2], cvt_read, mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + (size_t)p.nA * kABytes;
  float* sL = reinterpret_cast<float*>(sB + (size_t)p.nslots * kSlotBytes);  // Lambda of each stage's columns

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&afull[i], 1);
      tc::mbar_init(&aempty[i], 1);
      tc::mbar_init(&accfull[i], 1);
      tc::mbar_init(&accempty[i], 128);
    }
    for (int i = 0; i < kMaxStages; ++i) {
      tc::mbar_init(&bfull[i], 256);  // every gathering thread, once its copies have landed
      tc::mbar_init(&bempty[i], 1);
      tc::mbar_init(&ifull[i], 256);
    }
    tc::mbar_init(&cvt_read, 256);
    tc::mbar_init(&mma_done, 1);
    tc::fence_barrier_init();
    abort_flag = 0;
  }
  if (warp == 1) {
    tc::tmem_alloc(&tmem_slot, p.tmem_cols);
    tc::tmem_relinquish();
    tc::tc_fence_before();
  }
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  volatile int* vabort = &abort_flag;
  auto fail = [&]() {
    *vabort = 1;
    atomicExch(p.err, 1);
  };
  const int64_t G = gridDim.x;
  const int nA = p.nA, nS = p.nslots;

  if (warp == 0) {
    // ---------------- cell images: one bulk copy per cell into nA buffers
    if (lane == 0) {
      int64_t cl = 0;
      for (int64_t g = blockIdx.x; g < p.total_cells; g += G, ++cl) {
        const int ab = (int)(cl % nA);
        if (*vabort || !tc::mbar_wait(&aempty[ab], (uint32_t)((cl / nA) & 1) ^ 1u)) {
          fail();
          break;
        }
        const StepPartDev& P = p.part[part_of(p, g)];
        tc::mbar_arrive_expect_tx(&afull[ab], kABytes);
        bulk_g2s(sA + (size_t)ab * kABytes, P.img + (g - P.cell_off) * (int64_t)kABytes, kABytes, &afull[ab]);
      }
      if (*vabort)  // let the copies already issued land before the shared memory is released (bounded)
        for (int64_t c2 = (cl > nA ? cl - nA : 0); c2 < cl; ++c2) tc::mbar_wait(&afull[c2 % nA], (uint32_t)((c2 / nA) & 1));
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: accumulates onto the owner terms the converters stored
    const bool leader = tc::elect_one();
    constexpr uint32_t idesc = tc::instr_desc(2u, kNCP, BN);  // TF32, both operands K-major
    int64_t j = 0, cl = 0;
    bool stop = false;
    for (int64_t g = blockIdx.x; g < p.total_cells && !stop; g += G, ++cl) {
      const StepPartDev& P = p.part[part_of(p, g)];
      const int ab = (int)(cl % nA);
      for (int t = 0; t < P.ntiles; ++t, ++j) {
        const int s = (int)(j % nS), xb = (int)(j & 1);
        bool ok = !*vabort;
        if (ok && t == 0) ok = tc::mbar_wait(&afull[ab], (uint32_t)((cl / nA) & 1));
        if (ok) ok = tc::mbar_wait(&ifull[s], (uint32_t)((j / nS) & 1));
        if (!__all_sync(0xffffffffu, ok)) {
          if (leader) fail();
          stop = true;
          break;
        }
        tc::tc_fence_after();
        const uint64_t a0 = tc::sw128_desc(tc::smem_u32(sA + (size_t)ab * kABytes));
        const uint64_t b0 = tc::sw128_desc(tc::smem_u32(sB + (size_t)s * kSlotBytes));
        const uint32_t d = tmem + (uint32_t)(xb * BN);
#pragma unroll
        for (int kk = 0; kk < kNCP / 8; ++kk) {
          const int kel = kk * 8;
          const uint32_t aoff = (uint32_t)(kel >> 5) * kNCP * 128 + (uint32_t)((kel & 31) * 4);
          const uint32_t boff = (uint32_t)(kel >> 5) * BN * 128 + (uint32_t)((kel & 31) * 4);
          if (leader) tc::mma_tf32(d, tc::desc_add(a0, aoff), tc::desc_add(b0, boff), idesc, 1u);
        }
        __syncwarp();
        if (leader) {
          tc::mma_commit(&bempty[s]);
          tc::mma_commit(&accfull[xb]);
          if (t == P.ntiles - 1) tc::mma_commit(&aempty[ab]);
        }
        __syncwarp();
      }
    }
    // every MMA issued has completed before TMEM is released
    if (leader) {
      tc::mma_commit(&mma_done);
      tc::mbar_wait(&mma_done, 0u);
    }
    __syncwarp();
  } else if (warp < 10) {
    // ---------------- gather + convert (256 threads)
    // Gather (all 256 threads, coalesced: a warp instruction copies whole 256-byte row segments):
    // the tile's rows of V and owned rows of W as 16-byte cp.async copies into the 128-byte-swizzled
    // stage, and the tile's Lambda values; each thread arrives on the stage's barrier once its copies
    // have landed.  Tiles are gathered `ahead` tiles ahead of the one being converted.
    // Convert (thread (k, h): cell node k = TMEM lane k, half h of the columns): the owner terms
    // into the accumulator (tcgen05.st), then, once all threads have read the stage, the stage
    // rewritten in place as the K-major TF32 operand.
    const int gt = threadIdx.x - 64;         // 0..255
    const int k = (warp & 3) * 32 + lane;
    const int h = (warp - 2) >> 2;
    const int ahead = nS - 1;  // tiles gathered ahead: tile j + ahead reuses the stage of tile j - 1
    // gather cursor (the tile `ahead` tiles ahead of the one converted): this thread copies the rows
    // kr = (it * 256 + gt) / CPR of every tile, the same for all tiles of a cell, so their offsets
    // and owner flags are loaded once per cell
    constexpr int kIt = kNCP * CPR / 256;
    int64_t gg = blockIdx.x, jg = 0;
    int tg = 0;
    int64_t rowoff[kIt];
    int ownpos[kIt];
    auto gather = [&]() -> bool {
      if (gg >= p.total_cells) return true;
      const StepPartDev& P = p.part[part_of(p, gg)];
      const int s = (int)(jg % nS);
      const int64_t cell = gg - P.cell_off;
      if (tg == 0) {
#pragma unroll
        for (int it = 0; it < kIt; ++it) {
          const int kr = (it * 256 + gt) / CPR;
          rowoff[it] = (int64_t)__ldg(P.dofs + cell * P.nc + min(kr, P.nc - 1)) * P.n;  // padding rows repeat
          ownpos[it] = (P.owner && kr < P.nc) ? (int)__ldg(P.own_pos + cell * kNCP + kr) : -1;
        }
      }
      if (!tc::mbar_wait(&bempty[s], (uint32_t)((jg / nS) & 1) ^ 1u)) return false;
      const int c0 = tg * BN;
      uint8_t* slot = sB + (size_t)s * kSlotBytes;
#pragma unroll
      for (int it = 0; it < kIt; ++it) {
        const int e = it * 256 + gt;
        const int kr = e / CPR, ch = e % CPR, col = c0 + 4 * ch;
        const bool in = col < P.n;
        const uint32_t off = (uint32_t)(ch >> 3) * kChunkBytes + (uint32_t)kr * 128 + (uint32_t)(((ch & 7) ^ (kr & 7)) << 4);
        cp_async16(slot + off, P.V + rowoff[it] + (in ? col : 0), in);
        if (ownpos[it] >= 0) {  // owned row: W row into position ownpos of the compact W area
          const int o = ownpos[it];
          const uint32_t woff = (uint32_t)(ch >> 3) * kWChunkBytes + (uint32_t)o * 128 + (uint32_t)(((ch & 7) ^ (o & 7)) << 4);
          cp_async16(slot + kHalf + woff, P.W + rowoff[it] + (in ? col : 0), in);
        }
      }
      for (int e = gt; e < BN / 4; e += 256) {
        const int col = c0 + 4 * e;
        const bool in = col < P.n;
        cp_async16(sL + (size_t)s * BN + 4 * e, P.lam + (in ? col : 0), in);
      }
      cp_async_arrive_noinc(&bfull[s]);
      ++jg;
      if (++tg == P.ntiles) {
        tg = 0;
        gg += G;
      }
      return true;
    };
    bool stop = false;
    for (int a = 0; a < ahead && !stop; ++a)
      if (!gather()) {
        fail();
        stop = true;
      }
    int64_t j = 0;
    for (int64_t g = blockIdx.x; g < p.total_cells && !stop; g += G) {
      const StepPartDev& P = p.part[part_of(p, g)];
      const int64_t cell = g - P.cell_off;
      const bool real = k < P.nc;
      const int o = (real && P.owner) ? (int)__ldg(P.own_pos + cell * kNCP + k) : -1;  // compact W row
      const bool own = o >= 0;
      float al = P.alpha, be = P.beta, om = P.omega;
      if (P.coef) {
        al = (float)__ldg(P.coef);
        be = (float)__ldg(P.coef + 1);
        om = (float)__ldg(P.coef + 2);
      }
      al *= P.sign;
      const float rbe = be / al, rom = om / al;  // owner terms divided by alpha
      for (int t = 0; t < P.ntiles; ++t, ++j) {
        const int s = (int)(j % nS), xb = (int)(j & 1);
        bool ok = !*vabort && tc::mbar_wait(&bfull[s], (uint32_t)((j / nS) & 1));
        if (ok) ok = tc::mbar_wait(&accempty[xb], (uint32_t)((j >> 1) & 1) ^ 1u);
        if (!ok) fail();
        if (!__all_sync(0xffffffffu, ok && !*vabort)) {
          stop = true;
          break;
        }
        tc::tc_fence_after();
        uint8_t* slot = sB + (size_t)s * kSlotBytes;
        const uint8_t* vrow = slot + (size_t)k * 128;
        const uint8_t* wrow = slot + kHalf + (size_t)(own ? o : 0) * 128;
        const float* lam = sL + (size_t)s * BN;
        const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(xb * BN + h * HB);
        float4 v[HB / 4];
#pragma unroll
        for (int c16 = 0; c16 < HB / 16; ++c16) {
          float tv[16];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int col = h * HB + c16 * 16 + 4 * u;      // column within the tile
            const int c = col >> 5, qd = (col & 31) >> 2;  // 32-column chunk, 16-byte chunk in the row
            // 16-byte chunk qd of staged row k sits at chunk qd ^ (k % 8) (the 128-byte swizzle)
            const uint32_t off = (uint32_t)c * kChunkBytes + (uint32_t)((qd ^ (k & 7)) << 4);
            float4 x = *reinterpret_cast<const float4*>(vrow + off);
            const uint32_t woff = (uint32_t)c * kWChunkBytes + (uint32_t)((qd ^ (o & 7)) << 4);
            if (!real) x = make_float4(0.f, 0.f, 0.f, 0.f);
            v[c16 * 4 + u] = x;
            float4 tq = make_float4(0.f, 0.f, 0.f, 0.f);
            if (own) {
              // (FP32 Lambda: a conversion from FP64 would hold the SM's FP64 pipe ~16 clocks per warp)
              const float4 wv = *reinterpret_cast<const float4*>(wrow + woff);
              const float4 lv = *reinterpret_cast<const float4*>(lam + col);
              tq.x = rbe * x.x + rom * lv.x * wv.x;
              tq.y = rbe * x.y + rom * lv.y * wv.y;
              tq.z = rbe * x.z + rom * lv.z * wv.z;
              tq.w = rbe * x.w + rom * lv.w * wv.w;
            }
            tv[4 * u] = tq.x;
            tv[4 * u + 1] = tq.y;
            tv[4 * u + 2] = tq.z;
            tv[4 * u + 3] = tq.w;
          }
          tc::tmem_st16(taddr + c16 * 16, tv);
        }
        tc::tmem_wait_st();
        // once every converter has read its part of the stage (a bounded wait on a barrier that
        // completes one phase per tile), rewrite the stage as the K-major operand
        tc::mbar_arrive(&cvt_read);
        ok = tc::mbar_wait(&cvt_read, (uint32_t)(j & 1));
        if (!ok) fail();
        if (!__all_sync(0xffffffffu, ok && !*vabort)) {
          stop = true;
          break;
        }
#pragma unroll
        for (int u = 0; u < HB / 4; ++u) {
          const int col = h * HB + 4 * u;
          const float4 x = v[u];
          *reinterpret_cast<float*>(slot + img_off(col, k, BN)) = tf32_rna(x.x);
          *reinterpret_cast<float*>(slot + img_off(col + 1, k, BN)) = tf32_rna(x.y);
          *reinterpret_cast<float*>(slot + img_off(col + 2, k, BN)) = tf32_rna(x.z);
          *reinterpret_cast<float*>(slot + img_off(col + 3, k, BN)) = tf32_rna(x.w);
        }
        fence_proxy_async();  // the generic-proxy writes, before the MMA reads them
        tc::tc_fence_before();
        tc::mbar_arrive(&ifull[s]);
        // the tile `ahead` further on, into the stage of tile j - 1 (free once its MMA is done)
        if (!gather()) {
          fail();
          stop = true;
        }
      }
    }
    // copies still in flight land before the shared memory is released
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ---------------- epilogue
    const int q = warp & 3;              // TMEM lane quarter this warp may access
    const int i = q * 32 + lane;         // cell-local node of this thread's accumulator row
    int64_t j = 0;
    bool stop = false;
    for (int64_t g = blockIdx.x; g < p.total_cells && !stop; g += G) {
      const StepPartDev& P = p.part[part_of(p, g)];
      const int64_t cell = g - P.cell_off;
      float al = P.coef ? (float)__ldg(P.coef) : P.alpha;
      al *= P.sign;
      const int64_t row = (i < P.nc) ? (int64_t)__ldg(P.dofs + cell * P.nc + i) * P.n : -1;
      for (int t = 0; t < P.ntiles; ++t, ++j) {
        const int xb = (int)(j & 1);
        const int c0 = t * BN;
        bool ok = !*vabort && tc::mbar_wait(&accfull[xb], (uint32_t)((j >> 1) & 1));
        if (!ok) fail();
        if (!__all_sync(0xffffffffu, ok && !*vabort)) {
          stop = true;
          break;
        }
        tc::tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(xb * BN);
#pragma unroll
        for (int cc = 0; cc < BN; cc += 16) {
          float v[16];
          tc::tmem_ld16(taddr + cc, v);
          if (row >= 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int col = c0 + cc + 4 * u;
              if (col < P.n)
                red_add_v4(P.U + row + col, al * v[4 * u], al * v[4 * u + 1], al * v[4 * u + 2], al * v[4 * u + 3]);
            }
          }
        }
        tc::tc_fence_before();
        tc::mbar_arrive(&accempty[xb]);
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, p.tmem_cols);
  }
}

// ---------------------------------------------------------------- the transposed step
// The same step with the block's columns as the rows of the MMA: D^T (128 columns x 128 nodes) = T^T + V_c^T
// (A_c D_c^-1)^T.  V_c^T is the A operand and lives in TMEM (lane = column), so a converter thread reads its
// column of the staged rows (a warp reads 128 consecutive bytes per row) and writes it with tcgen05.st: no
// rewriting of the stage into a K-major image, no barrier among the converters, and the stage is free as soon
// as it has been read.  The cell image is the B operand as it stands (K-major).  In the epilogue a warp holds
// 32 consecutive columns of one node, so every red is a whole 128-byte line.
//   warp 0      cell images in four 32-wide K blocks, each refilled as soon as the last tile's MMAs on it are done
//   warp 1      MMA issuer (M = 128 columns, N = 128 nodes)
//   warps 2-9   convert: TMEM quarter w % 4 = 32 columns, half of the nodes each
//   warps 10-17 epilogue: the same quarters, half of the nodes each
//   warps 18-21 gather: half tiles of 64 columns into a ring of stages
// At 16^3 cells x 600 columns the step above took 857 us, and 610 us without any of its gathers and reds: its
// chain of conversion, barrier and rewriting was the bound, not memory (0.41 ms at the copy rate).  This one takes
// 498 us there; below about 64 columns, where half of its 128 lanes are idle, a launch of the other is faster (6^3 x 48: 11.0
// against 13 us; 10.3 us a step when one launch does them all), so both stand: fe_step_tile picks for a single
// filter, fe_step_tune by time for the graphs of the batched filters.
constexpr int kTThreads = 704;
constexpr int kTGather = 128;
constexpr int kTStages = 3;
constexpr uint32_t kTV = kNCP * 256;                    // 128 rows x 64 FP32
constexpr uint32_t kTStage = kTV + (kWRows + 1) * 256;  // the owned rows of W and a row of zeros
constexpr uint32_t kABlock = kABytes / 4;               // 32 K values of the cell image
constexpr int kTab = 4;                                 // cells whose tables are held

struct CellTab {
  int dof[kNCP];
  int orow[kWRows];   // dofs of the owned rows, in compact order
  uint8_t pos[kNCP];  // row of W in the stage: compact position of an owned node, else the row of zeros
};
constexpr size_t kTSmem = kABytes + kTStages * ((size_t)kTStage + 64 * 4) + kTab * sizeof(CellTab) + 1024;

// (predicated inside: a branch around each add made an add wait for the address of the one before, 130 clocks)
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d, bool on) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %5, 0;\n@p red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n}" ::"l"(p),
               "f"(a), "f"(b), "f"(c), "f"(d), "r"((uint32_t)on)
               : "memory");
}

// v[i] of lane 4 q + j (i, j < 4) goes to v[j] of lane 4 q + i.
__device__ __forceinline__ void quad_transpose(float* v, int lane) {
  const bool b0 = lane & 1, b1 = lane & 2;
  const float s0 = __shfl_xor_sync(0xffffffffu, b0 ? v[0] : v[1], 1);
  const float s1 = __shfl_xor_sync(0xffffffffu, b0 ? v[2] : v[3], 1);
  const float x0 = b0 ? s0 : v[0], x1 = b0 ? v[1] : s0, x2 = b0 ? s1 : v[2], x3 = b0 ? v[3] : s1;
  const float t0 = __shfl_xor_sync(0xffffffffu, b1 ? x0 : x2, 2);
  const float t1 = __shfl_xor_sync(0xffffffffu, b1 ? x1 : x3, 2);
  v[0] = b1 ? t0 : x0;
  v[1] = b1 ? t1 : x1;
  v[2] = b1 ? x2 : t0;
  v[3] = b1 ? x3 : t1;
}

// D[tmem] += A[tmem] * B[smem]^T, TF32.
__device__ __forceinline__ void mma_tf32_ts(uint32_t d, uint32_t a, uint64_t b_desc, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, 1, 0;\n"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b_desc), "r"(idesc)
      : "memory");
}

// The CTA's cells, step by step.
struct StepCell {
  int64_t g;
  int st;
  __device__ __forceinline__ bool first() const { return g == (int64_t)blockIdx.x; }
  __device__ __forceinline__ bool last(const StepBatch& p) const { return g + gridDim.x >= p.total_cells; }
  __device__ __forceinline__ void next(const StepBatch& p) {
    g += gridDim.x;
    if (g >= p.total_cells) {
      g = blockIdx.x;
      ++st;
    }
  }
};

// *p >= want (acquire), with the limit of the other waits; false also once another CTA has failed.
__device__ __forceinline__ bool wait_steps(const int* p, int want, const int* err) {
  const long long t0 = clock64();
  for (int spin = 0;; ++spin) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (v >= want) return true;
    if (clock64() - t0 > tc::kWaitCycles) return false;
    if ((spin & 255) == 255 && *(volatile const int*)err) return false;
  }
}

__global__ void __launch_bounds__(kTThreads, 1) fe_step_t_kernel(const __grid_constant__ StepBatch p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t afull[4], aempty[4], bfull[kTStages], bempty[kTStages], ifull[2], accfull[2],
      accempty[2], tfree[kTab], mma_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + kABytes;
  float* sL = reinterpret_cast<float*>(sB + (size_t)kTStages * kTStage);  // Lambda of each stage's columns
  CellTab* tabs = reinterpret_cast<CellTab*>(sL + kTStages * 64);
  for (int i = threadIdx.x; i < kTStages * 64; i += kTThreads)  // the rows of zeros
    reinterpret_cast<float*>(sB + (size_t)(i / 64) * kTStage + kTV + kWRows * 256)[i % 64] = 0.f;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) {
      tc::mbar_init(&afull[i], 1);
      tc::mbar_init(&aempty[i], 1);
    }
    for (int i = 0; i < kTStages; ++i) {
      tc::mbar_init(&bfull[i], kTGather + 1);  // every gathering thread's copies, and the cell's table
      tc::mbar_init(&bempty[i], 128);          // the converters of the stage's 64 columns
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&ifull[i], 256);
      tc::mbar_init(&accfull[i], 1);
      tc::mbar_init(&accempty[i], 256);
    }
    for (int i = 0; i < kTab; ++i) tc::mbar_init(&tfree[i], 8);
    tc::mbar_init(&mma_done, 1);
    tc::fence_barrier_init();
    abort_flag = 0;
  }
  if (warp == 1) {
    tc::tmem_alloc(&tmem_slot, 512);
    tc::tmem_relinquish();
    tc::tc_fence_before();
  }
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;  // D of tile parity x at 128 x, the V operand at 256 + 128 x
  volatile int* vabort = &abort_flag;
  auto fail = [&]() {
    *vabort = 1;
    atomicExch(p.err, 1);
  };

  if (warp == 0) {
    // ---------------- cell images
    if (lane == 0) {
      int64_t cl = 0;
      int issued = 0;
      for (StepCell it{blockIdx.x, 0}; it.st < p.nsteps && !*vabort; it.next(p), ++cl) {
        const int64_t g = it.g;
        const StepPartDev& P = p.part[part_of(p, g)];
        const uint8_t* src = P.img + (g - P.cell_off) * (int64_t)kABytes;
        for (issued = 0; issued < 4; ++issued) {
          if (*vabort || !tc::mbar_wait(&aempty[issued], (uint32_t)(cl & 1) ^ 1u)) {
            fail();
            break;
          }
          tc::mbar_arrive_expect_tx(&afull[issued], kABlock);
          bulk_g2s(sA + (size_t)issued * kABlock, src + (size_t)issued * kABlock, kABlock, &afull[issued]);
        }
      }
      if (*vabort) {  // copies already issued land before the shared memory is released (bounded)
        // the last cell begun is cl - 1: blocks from `issued` on still hold the one before
        for (int b = 0; b < 4; ++b) {
          const int64_t c = b < issued ? cl - 1 : cl - 2;
          if (c >= 0) tc::mbar_wait(&afull[b], (uint32_t)(c & 1));
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: accumulates onto the owner terms the converters stored
    const bool leader = tc::elect_one();
    constexpr uint32_t idesc = tc::instr_desc(2u, 128, kNCP);  // TF32, B K-major
    const uint64_t b0 = tc::sw128_desc(tc::smem_u32(sA));
    uint32_t j = 0, cl = 0;
    bool stop = false;
    for (StepCell it{blockIdx.x, 0}; it.st < p.nsteps && !stop; it.next(p), ++cl) {
      const int64_t g = it.g;
      const StepPartDev& P = p.part[part_of(p, g)];
      const int ntiles = P.ntiles;
      for (int t = 0; t < ntiles && !stop; ++t, ++j) {
        const uint32_t xb = (uint32_t)(j & 1);
        bool ok = !*vabort && tc::mbar_wait(&ifull[xb], (uint32_t)((j >> 1) & 1));
        const uint32_t d = tmem + xb * 128u, a = tmem + 256u + xb * 128u;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
          if (ok && t == 0) ok = tc::mbar_wait(&afull[kb], (uint32_t)(cl & 1));
          if (kb == 0 || t == 0) {
            if (!__all_sync(0xffffffffu, ok)) {
              if (leader) fail();
              stop = true;
              break;
            }
            tc::tc_fence_after();
          }
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            if (leader) mma_tf32_ts(d, a + (uint32_t)(kb * 32 + kk * 8), tc::desc_add(b0, kb * kABlock + kk * 32), idesc);
          __syncwarp();
          if (leader && t == ntiles - 1) tc::mma_commit(&aempty[kb]);
          __syncwarp();
        }
        if (leader && !stop) tc::mma_commit(&accfull[xb]);
        __syncwarp();
      }
    }
    // every MMA issued has completed before TMEM is released
    if (leader) {
      tc::mma_commit(&mma_done);
      tc::mbar_wait(&mma_done, 0u);
    }
    __syncwarp();
  } else if (warp < 10) {
    // ---------------- convert: this thread's column c of the tile, nodes k0 .. k0 + 63
    const int q = warp & 3, k0 = 64 * ((warp - 2) >> 2), hp = q >> 1;
    const int cs = (q & 1) * 32 + lane;  // column within the half tile
    // (j: tiles so far, 32 bits and its low ones only; s0, ph0: stage and phase of the tile's first half)
    uint32_t j = 0, cl = 0, ph0 = 0;
    int s0 = 0;
    bool stop = false;
    for (StepCell it{blockIdx.x, 0}; it.st < p.nsteps && !stop; it.next(p), ++cl) {
      const int64_t g = it.g;
      const StepPartDev& P = p.part[part_of(p, g)];
      const CellTab& tab = tabs[cl % kTab];
      const int n = P.n, ntiles = P.ntiles;
      float al = P.alpha, be = P.beta, om = P.omega;
      if (p.nsteps > 1) {
        al = p.coefs[3 * it.st];
        be = p.coefs[3 * it.st + 1];
        om = p.coefs[3 * it.st + 2];
      } else if (P.coef) {
        al = (float)__ldg(P.coef);
        be = (float)__ldg(P.coef + 1);
        om = (float)__ldg(P.coef + 2);
      }
      al *= P.sign;
      const float rbe = be / al, rom = om / al;  // owner terms divided by alpha
      for (int t = 0; t < ntiles; ++t, ++j) {
        const int nh = n - 128 * t > 64 ? 2 : 1;  // half tiles
        const uint32_t xb = (uint32_t)(j & 1);
        bool ok = !*vabort && tc::mbar_wait(&accempty[xb], (uint32_t)((j >> 1) & 1) ^ 1u);
        const bool wrap = s0 + hp >= kTStages;
        const int s = wrap ? s0 + hp - kTStages : s0 + hp;
        if (ok && hp < nh) ok = tc::mbar_wait(&bfull[s], ph0 ^ (wrap ? 1u : 0u));
        if (!ok) fail();
        if (!__all_sync(0xffffffffu, ok)) {
          stop = true;
          break;
        }
        tc::tc_fence_after();
        if (hp < nh) {
          const float* V = reinterpret_cast<const float*>(sB + (size_t)s * kTStage) + cs;
          const uint8_t* W = reinterpret_cast<const uint8_t*>(V) + kTV;
          const float rl = rom * sL[s * 64 + cs];
          const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16) + xb * 128u + (uint32_t)k0;
#pragma unroll
          for (int kb = 0; kb < 64; kb += 16) {
            float x[16], d[16];
            const uint4 pk = *reinterpret_cast<const uint4*>(tab.pos + k0 + kb);
            const uint32_t pw[4] = {pk.x, pk.y, pk.z, pk.w};
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              x[u] = V[(k0 + kb + u) * 64];
              // byte u of the positions, times the 256 bytes of a row
              d[u] = *reinterpret_cast<const float*>(W + __byte_perm(pw[u >> 2], 0, 0x4404u | (uint32_t)((u & 3) << 4)));
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const bool own = ((pw[u >> 2] >> (8 * (u & 3))) & 0xffu) != (uint32_t)kWRows;
              d[u] = fmaf(rl, d[u], own ? rbe * x[u] : 0.f);
              x[u] = tf32_rna(x[u]);
            }
            tc::tmem_st16(lane_addr + (uint32_t)kb, d);
            tc::tmem_st16(lane_addr + 256u + (uint32_t)kb, x);
          }
          tc::mbar_arrive(&bempty[s]);
          tc::tmem_wait_st();
          tc::tc_fence_before();
        }
        tc::mbar_arrive(&ifull[xb]);
        s0 += nh;
        if (s0 >= kTStages) {
          s0 -= kTStages;
          ph0 ^= 1u;
        }
      }
    }
  } else if (warp < 18) {
    // ---------------- epilogue
    const int q = warp & 3, k0 = 64 * ((warp - 10) >> 2);
    uint32_t j = 0, cl = 0;
    bool stop = false;
    for (StepCell it{blockIdx.x, 0}; it.st < p.nsteps && !stop; it.next(p), ++cl) {
      const int64_t g = it.g;
      const StepPartDev& P = p.part[part_of(p, g)];
      const CellTab& tab = tabs[cl % kTab];
      const int nc = P.nc, n = P.n, ntiles = P.ntiles;
      float al = p.nsteps > 1 ? p.coefs[3 * it.st] : P.coef ? (float)__ldg(P.coef) : P.alpha;
      al *= P.sign;
      float* Ub = (it.st & 1) ? P.U2 : P.U;
      for (int t = 0; t < ntiles; ++t, ++j) {
        const uint32_t xb = (uint32_t)(j & 1);
        const int col4 = 128 * t + q * 32 + (lane & ~3);
        // (ifull: the acquire that makes the cell's table visible here)
        bool ok = !*vabort && tc::mbar_wait(&ifull[xb], (uint32_t)((j >> 1) & 1)) &&
                  tc::mbar_wait(&accfull[xb], (uint32_t)((j >> 1) & 1));
        if (!ok) fail();
        if (!__all_sync(0xffffffffu, ok)) {
          stop = true;
          break;
        }
        tc::tc_fence_after();
        if (128 * t + q * 32 < n) {
          const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + xb * 128u + (uint32_t)k0;
          float* U = Ub + col4;
#pragma unroll
          for (int kb = 0; kb < 64; kb += 16) {
            float v[16];
            tc::tmem_ld16(taddr + (uint32_t)kb, v);
            // four lanes exchange four nodes, so that each holds four columns of one: a quarter of the adds
#pragma unroll
            for (int g4 = 0; g4 < 16; g4 += 4) {
              quad_transpose(v + g4, lane);
              const int i = k0 + kb + g4 + (lane & 3);
              red_add_v4(U + (int64_t)tab.dof[i] * n, al * v[g4], al * v[g4 + 1], al * v[g4 + 2], al * v[g4 + 3],
                         col4 < n && i < nc);
            }
          }
        }
        tc::tc_fence_before();
        tc::mbar_arrive(&accempty[xb]);
      }
      const bool meet = it.last(p) && it.st + 1 < p.nsteps;
      if (meet) __threadfence();  // this step's adds, before the other CTAs read the rows
      __syncwarp();
      if (lane == 0 && !stop) {
        tc::mbar_arrive(&tfree[cl % kTab]);
        if (meet) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.sync) : "memory");
      }
    }
  } else {
    // ---------------- gather: 16 lanes copy one 256-byte row segment
    const int gt = threadIdx.x - 576;
    const int ch = gt & 15, r0 = gt >> 4;
    uint32_t cl = 0, ph = 1;  // ph: phase parity that frees stage s
    int s = 0;
    bool stop = false;
    for (StepCell it{blockIdx.x, 0}; it.st < p.nsteps; it.next(p), ++cl) {
      const int64_t g = it.g;
      const StepPartDev& P = p.part[part_of(p, g)];
      const int64_t cell = g - P.cell_off;
      CellTab& tab = tabs[cl % kTab];
      const int nc = P.nc, n = P.n;
      // the cell's tables, once its predecessor in the same place is done with
      bool ok = !stop && !*vabort && tc::mbar_wait(&tfree[cl % kTab], (uint32_t)((cl / kTab) & 1) ^ 1u);
      // a step reads what the one before has added: once all its adds (eight epilogue warps per CTA) are in
      if (ok && it.st > 0 && it.first() && gt == 0) ok = wait_steps(p.sync, it.st * 8 * (int)gridDim.x, p.err);
      const float* Vb = (it.st & 1) ? P.V2 : P.V;
      int o = -1;
      if (ok) {
        const int d = __ldg(P.dofs + cell * nc + min(gt, nc - 1));  // padding rows repeat
        if (P.owner && gt < nc) o = (int)__ldg(P.own_pos + cell * kNCP + gt);
        tab.dof[gt] = d;
        tab.pos[gt] = (uint8_t)(o >= 0 ? o : kWRows);
        if (o >= 0) tab.orow[o] = d;
      }
      // barriers of the gather warps: owned rows of the cell, and whether any thread gave up
      uint32_t nown, bad;
      asm volatile("{\n.reg .pred q;\nsetp.ge.s32 q, %1, 0;\nbarrier.cta.red.popc.u32 %0, 2, 128, q;\n}"
                   : "=r"(nown)
                   : "r"(o)
                   : "memory");
      asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %1, 0;\nbarrier.cta.red.popc.u32 %0, 2, 128, q;\n}"
                   : "=r"(bad)
                   : "r"((int)!ok)
                   : "memory");
      if (bad) {
        fail();
        break;
      }
      int rows[kNCP / 8];
#pragma unroll
      for (int i = 0; i < kNCP / 8; ++i) rows[i] = tab.dof[r0 + 8 * i];
      for (int hs = 0; hs * 64 < n; ++hs) {
        if (*vabort || !tc::mbar_wait(&bempty[s], ph)) {
          fail();
          stop = true;  // (the gather warps leave together, at the vote of the next cell)
          break;
        }
        const int col = hs * 64 + 4 * ch;
        const bool in = col < n;
        const float* Vc = Vb + (in ? col : 0);
        const float* Wc = P.W + (in ? col : 0);
        uint8_t* dst = sB + (size_t)s * kTStage + r0 * 256 + ch * 16;
#pragma unroll
        for (int i = 0; i < kNCP / 8; ++i)  // (rows of padding nodes: zeros)
          cp_async16(dst + i * 2048, Vc + (int64_t)rows[i] * n, in && r0 + 8 * i < nc);
        for (int r = r0; r < (int)nown; r += 8)
          cp_async16(dst + kTV + (r - r0) * 256, Wc + (int64_t)tab.orow[r] * n, in);
        if (gt < 16) cp_async16(sL + s * 64 + 4 * gt, P.lam + (int64_t)it.st * n + (in ? col : 0), in);
        cp_async_arrive_noinc(&bfull[s]);
        if (gt == 0) tc::mbar_arrive(&bfull[s]);
        if (++s == kTStages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    // copies still in flight land before the shared memory is released
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// Shared-memory plan of a tile width: cell-image buffers and stages (V rows, owned W rows) that fit.
struct Plan {
  int nA, nslots;
  size_t smem;
};

Plan make_plan(int BN) {
  // the deepest ring of stages that fits beside one cell image (the gathers run nslots - 1 tiles
  // ahead); a second image buffer only when it leaves at least three stages
  const size_t stage = (size_t)(BN / 32) * (kChunkBytes + kWChunkBytes) + (size_t)BN * 4;
  const size_t cap = kSmemMax - 1024 - 512;  // alignment slack and the kernel's static shared memory
  for (int nA : {1, 2}) {
    for (int ns = kMaxStages; ns >= (nA == 2 ? 3 : 2); --ns) {
      const size_t need = (size_t)nA * kABytes + (size_t)ns * stage;
      if (need <= cap) return Plan{nA, ns, need + 1024};
    }
  }
  return Plan{0, 0, 0};
}

const uint8_t* scaled_images(cudaStream_t s, FeOp& op, const double* dinv) {
  if (!op.imgADtf.p || !op.imgAD_packed) {
    op.imgADtf.ensure((size_t)kABytes * op.n_cells);
    const int64_t total = op.n_cells * (int64_t)kNCP * kNCP;
    const unsigned blocks = (unsigned)std::min<int64_t>((total + 255) / 256, 152 * 32);
    pack_scaled_kernel<<<blocks, 256, 0, s>>>(op.n_cells, op.nc, op.A64.p, op.dofs.p, dinv, op.imgADtf.p);
    op.imgAD_packed = true;
    RC_LAUNCH();
  }
  return op.imgADtf.p;
}

template <int BN>
void launch(cudaStream_t s, const StepBatch& b, const Plan& pl, unsigned grid) {
  set_smem_limit(reinterpret_cast<const void*>(fe_step_kernel<BN>), kSmemMax - 512);
  fe_step_kernel<BN><<<grid, kThreads, pl.smem, s>>>(b);
  RC_LAUNCH();
}

std::mutex g_tune_mu;
std::map<std::tuple<int, int64_t, int, int>, int> g_tune;

}  // namespace

bool fe_step_supported(const FeOp& op, int n, int precision) {
  return precision == RCHFSI_TF32 && n % 4 == 0 && n >= 4 && op.nc <= kNCP && op.own_pos.p != nullptr &&
         op.own_max <= kWRows;
}

// Up to 32 columns fill a quarter of the 128 lanes of the transposed step, whose time per cell does not depend on the
// width below 64; the other form's tile of 32 columns takes less, and loses a launch per step.  So it is taken where
// there are at least four cell products per SM, or where the steps do not fit one launch anyway.  Whole calls in
// us, 128 in one launch / 32 per step, degree 20: 16 columns 6^3 cells 302 / 325, 7^3 365 / 363, 8^3 442 / 410,
// 9^3 538 / 459, 10^3 689 / 583, 14^3 1592 / 1354; 32 columns 8^3 443 / 452, 9^3 537 / 500, 10^3 700 / 630, 14^3
// 1603 / 1440; 36 columns (two tiles) 8^3 440 / 570, 14^3 1607 / 1966; complex 32 columns 4^3 365 / 362, 6^3 669 / 637,
// 8^3 1325 / 1158.  Degree 110, one launch per step either way, 32 columns: 6^3 1514 / 1297, 10^3 3555 / 2885.
int fe_step_tile(const FeOp& op, int n, int num_sms, bool loop) {
  const int64_t items = op.n_cells * (op.cplx ? 4 : 1);
  return n <= 32 && (!loop || items >= 4 * (int64_t)num_sms) ? 32 : 128;
}

void fe_step_prepare(cudaStream_t s, FeOp& op) {
  scaled_images(s, op, op.Dinv.p);
  if (op.cplx) scaled_images(s, *op.imag, op.Dinv.p);
}

int fe_step_parts(FeOp& op, const float* V, const float* W, float* U, const float* lam, int n, float alpha,
                  float beta, float omega, const double* coef, FeStepPart* out) {
  if (!op.cplx) {
    out[0] = FeStepPart{&op, V, W, U, lam, coef, op.m, n, alpha, beta, omega, 1.f, true};
    return 1;
  }
  // complex operator on the real embedding: rows [0, mc) real parts, [mc, 2 mc) imaginary parts
  //   U_r += alpha (Ar V_r - Ai V_i),   U_i += alpha (Ai V_r + Ar V_i)
  // and the owner terms of each half once (with the Ar part of that half)
  const int64_t mc = op.mc, off = mc * (int64_t)n;
  FeOp& im = *op.imag;
  out[0] = FeStepPart{&op, V, W, U, lam, coef, mc, n, alpha, beta, omega, 1.f, true};
  out[1] = FeStepPart{&im, V + off, W, U, lam, coef, mc, n, alpha, beta, omega, -1.f, false};
  out[2] = FeStepPart{&im, V, W, U + off, lam, coef, mc, n, alpha, beta, omega, 1.f, false};
  out[3] = FeStepPart{&op, V + off, W + off, U + off, lam, coef, mc, n, alpha, beta, omega, 1.f, true};
  return 4;
}

void fe_step_batch(cudaStream_t s, const FeStepPart* parts, int nparts, int BN, int num_sms, const FeStepLoop* loop) {
  RC_CHECK(nparts >= 1 && nparts <= kMaxParts, RCHFSI_ERR_INVALID_ARG, "fused FE step: 1..64 parts per launch");
  RC_CHECK(BN == 32 || BN == 64 || BN == 96 || BN == 128, RCHFSI_ERR_INVALID_ARG,
           "fused FE step: column tile of 32, 64, 96 or 128");
  const Plan pl = BN == 128 ? Plan{1, kTStages, kTSmem} : make_plan(BN);
  RC_CHECK(pl.nA > 0, RCHFSI_ERR_INVALID_ARG, "fused FE step: no shared-memory plan for this tile");
  const int nsteps = loop ? loop->steps : 1;
  RC_CHECK(nsteps == 1 || (BN == 128 && nsteps >= 1 && nsteps <= kTableSteps && loop->sync), RCHFSI_ERR_INVALID_ARG,
           "fused FE loop: tiles of 128 columns, at most kTableSteps steps and a counter");
  StepBatch b{};
  b.nparts = nparts;
  b.nsteps = nsteps;
  if (nsteps > 1) {
    b.sync = loop->sync;
    std::copy(loop->coefs, loop->coefs + 3 * nsteps, b.coefs);
  }
  b.nA = pl.nA;
  b.nslots = pl.nslots;
  int64_t off = 0;
  double flops = 0.0, bytes = 0.0;
  for (int q = 0; q < nparts; ++q) {
    const FeStepPart& t = parts[q];
    FeOp& op = *t.op;
    RC_CHECK(op.nc <= kNCP && t.n % 4 == 0 && op.own_pos.p && op.own_max <= kWRows, RCHFSI_ERR_INVALID_ARG,
             "fused FE step: n_c <= 128, n a multiple of 4, owner positions and at most 80 owned dofs per cell");
    StepPartDev& P = b.part[q];
    RC_CHECK(((uintptr_t)t.V & 15) == 0 && ((uintptr_t)t.W & 15) == 0 && ((uintptr_t)t.U & 15) == 0,
             RCHFSI_ERR_INVALID_ARG, "fused FE step: blocks must start on 16-byte boundaries");
    P.dofs = op.dofs.p;
    P.own_pos = op.own_pos.p;
    P.owner = t.owner ? 1 : 0;
    // the scaled images use the D^-1 of the rows the part reads (both halves share it)
    P.img = scaled_images(s, op, op.Dinv.p);
    P.V = t.V;
    P.W = t.W;
    P.U = t.U;
    if (nsteps > 1) {  // the two blocks change places
      P.V2 = loop->U + (t.V - loop->V);
      P.U2 = loop->V + (t.U - loop->U);
    }
    P.lam = t.lam;
    P.coef = t.coef;
    P.n_cells = op.n_cells;
    P.cell_off = off;
    P.alpha = t.alpha;
    P.beta = t.beta;
    P.omega = t.omega;
    P.sign = t.sign;
    P.nc = op.nc;
    P.n = t.n;
    P.ntiles = (t.n + BN - 1) / BN;
    off += op.n_cells;
    const double nc = op.nc, C = (double)op.n_cells;
    flops += 2.0 * nc * nc * C * t.n;
    // algorithmic bytes: the cell images, and for the owner part of each row half the four block
    // streams (V read, U read and written, W read); a complex operator's cross parts re-read V
    bytes += 4.0 * nc * nc * C + (t.owner ? 16.0 * (double)t.rows * t.n : 0.0);
  }
  b.total_cells = off;
  b.err = parts[0].op->err;
  uint32_t cols = 32;
  while (cols < (uint32_t)(2 * BN)) cols <<= 1;
  b.tmem_cols = cols;
  const unsigned grid = (unsigned)std::min<int64_t>(b.total_cells, (int64_t)num_sms);
  prof::Scope ps(s, RCHFSI_KERNEL_FE_CELL, flops * nsteps, bytes * nsteps);
  switch (BN) {
    case 32: launch<32>(s, b, pl, grid); break;
    case 64: launch<64>(s, b, pl, grid); break;
    case 128:
      set_smem_limit(reinterpret_cast<const void*>(fe_step_t_kernel), kSmemMax - 512);
      if (nsteps > 1) {
        void* args[] = {(void*)&b};
        RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(fe_step_t_kernel), dim3(grid), dim3(kTThreads),
                                            args, kTSmem, s));
      } else {
        fe_step_t_kernel<<<grid, kTThreads, kTSmem, s>>>(b);
      }
      RC_LAUNCH();
      break;
    default: launch<96>(s, b, pl, grid); break;
  }
}

int fe_step_tune(cudaStream_t s, int num_sms, FeOp& op, int n, const float* V, const float* W, const float* lam) {
  const auto key = std::make_tuple(op.nc, (int64_t)op.n_cells, n, op.cplx ? 1 : 0);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) return it->second;
  }
  std::vector<int> cand;
  for (int bn : {32, 64, 96})
    if (bn <= std::max(32, (n + 31) / 32 * 32) && make_plan(bn).nA > 0) cand.push_back(bn);
  cand.push_back(128);
  DevBuf<float> scratch;
  float* out = scratch.ensure((size_t)op.m * n);
  cudaEvent_t e0, e1;
  RC_CUDA(cudaEventCreate(&e0));
  RC_CUDA(cudaEventCreate(&e1));
  int best = cand[0];
  float best_ms = 1e30f;
  for (int bn : cand) {
    FeStepPart parts[4];
    const int np = fe_step_parts(op, V, W, out, lam, n, 1.f, 0.5f, 0.25f, nullptr, parts);
    fe_step_batch(s, parts, np, bn, num_sms);  // warm-up
    RC_CUDA(cudaEventRecord(e0, s));
    for (int r = 0; r < 2; ++r) fe_step_batch(s, parts, np, bn, num_sms);
    RC_CUDA(cudaEventRecord(e1, s));
    RC_CUDA(cudaEventSynchronize(e1));
    float ms = 0.f;
    RC_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    if (ms < best_ms) {
      best_ms = ms;
      best = bn;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[key] = best;
  return best;
}

}  // namespace rchfsi
