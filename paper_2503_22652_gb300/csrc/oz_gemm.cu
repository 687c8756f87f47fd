// FP64-accurate products from BF16 tensor-core slices (see oz_gemm.cuh for the scheme).
//
// oz_gemm_kernel: persistent CTAs (one per SM) walking (128 x 64 output tile, K range) items.
// Warp 0 (one lane) streams, per 64-wide K chunk, the 7 A and the 7 B slices of the tile (16 KB and
// 8 KB each, whole 128-byte rows, 128-byte swizzle) with TMA, every slice into a slot of its own ring;
// warp 1 (the whole warp, one elected lane issuing) runs, for each A slice s, the products with B
// slices t <= 6 - s (4 x tcgen05.mma kind::f16, K = 16) into the TMEM accumulator of level s + t,
// GROUP chunks (128 K terms) per exact accumulation group.  Pass s is the last to read A slice s and
// B slice 6 - s, so each pass ends with one commit that frees both and the next chunk's slices arrive
// while this one is multiplied.  TMEM holds 8 level blocks of 64 columns,
// 7 for the group and one spare, rotated so that the next group's first writes go to blocks in the
// order they are freed; warps 2-17 (four per TMEM lane quarter, 16 columns each) fold level L of a
// group as soon as the group's pass L is done: tcgen05.ld and one 64-bit multiply-add into exact integer
// accumulators.  The final value, two conversions scaled by exponent arithmetic and one FP64 add, is stored
// (or, with split-K, written as a partial and summed by a second kernel) while the next item's MMAs run.
// The host splits K only as far as the items fill the CTAs.
// Bound: issue of the 128 x 64 x 16 MMAs by one warp beside 16 busy epilogue warps.  A pass runs its A tile (16 K
// values) against all its B slices before the next, with the tile kept in the collector: 35 clocks per MMA alone
// instead of 48 (shared-memory reads of A).  Measured per MMA in the kernel: 86 clocks with stages of whole 32-wide
// chunks, 87 with a ring and an arrival barrier per slice, 68 with the arrivals merged into five per chunk (a wait
// that finds its data there still costs about 130 clocks), 57 with the levels folded in integers.  262144 x 600 x 600:
// 6.79 -> 4.6 ms, the Gram matrix of 600 columns of 262144 4.03 -> 2.75 ms.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "oz_gemm.cuh"
#include "oz_digits.cuh"
#include "prof.cuh"
#include "tc_ptx.cuh"

namespace rchfsi {
namespace {

constexpr int S = kOzSlices;
constexpr int BM = 128;
constexpr int KC = 64;            // K tile of the slicing kernel (K is padded to a multiple of it)
constexpr int KCH = 64;           // K chunk of the products: one 128-byte row of BF16 per slice
// Chunks accumulated in TMEM before a drain: 2 x 64 = 128 K terms per exact FP32 sum (bounds of the sums: oz_gemm.cuh).
constexpr int GROUP = 2;
constexpr int kMaxSplitChunks = 1 << 14;  // 2^20 K terms: what the epilogue's integers hold exactly
constexpr int kARing = 8;         // A slices in flight (a power of two)
constexpr int kBRing = 8;         // B slices 6 .. 1 in flight (a power of two); slice 0 alternates between two slots
constexpr int kPassRing = 16;     // barriers of finished passes: more than the passes the producer runs ahead
constexpr int BN = 64;            // output tile columns
constexpr int kThreads = 576;     // 18 warps: TMA producer, MMA issuer, 16 epilogue warps
constexpr int kEpiThreads = 512;
constexpr uint32_t kASlice = BM * 128;       // 16 KB per A slice of a chunk
constexpr uint32_t kBSlice = BN * 128;       // 8 KB per B slice of a chunk
constexpr uint32_t kSmemBytes = kARing * kASlice + (kBRing + 2) * kBSlice;  // 208 KB
constexpr uint32_t kTmemCols = 512;          // 8 level blocks x 64 columns

// ---------------------------------------------------------------- slicing
// Row exponents, K-contiguous rows: one warp per (row, K slice), the K range split over
// blockIdx.y so that a few hundred rows still fill the GPU; slices meet in ex by atomicMax (ex
// preset to INT_MIN), slice_kernel maps rows without a nonzero element to 0.
__global__ void rowexp_kcontig(int64_t R, int64_t K, const double* __restrict__ X, int64_t rs, int* ex) {
  const int64_t r = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (r >= R) return;
  const int64_t kb = (K + gridDim.y - 1) / gridDim.y, k0 = (int64_t)blockIdx.y * kb;
  const int64_t k1 = k0 + kb < K ? k0 + kb : K;
  const double* x = X + r * rs;
  unsigned long long top = 0;  // the largest magnitude, as bits: one exponent for all
  for (int64_t k = k0 + lane; k < k1; k += 256) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = k + 32 * u < k1 ? x[k + 32 * u] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      top = max(top, (unsigned long long)__double_as_longlong(v[u]) & 0x7fffffffffffffffULL);
  }
  int e = exp_of(__longlong_as_double((long long)top));
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  if (lane == 0) atomicMax(ex + r, e);
}

// Row exponents, rows contiguous across threads (element (r, k) at X[r + k * ks]): 32 rows per
// block (coalesced), the K range split over the block's 8 warps and over blockIdx.y.  Partial maxima
// meet in ex by atomicMax (ex preset to INT_MIN); slice_kernel maps rows without a nonzero
// element to 0.
__global__ void __launch_bounds__(256) rowexp_rcontig(int64_t R, int64_t K, const double* __restrict__ X, int64_t ks,
                                                      int* ex) {
  __shared__ int red[8][32];
  const int64_t r = (int64_t)blockIdx.x * 32 + threadIdx.x;
  int e = -100000;
  if (r < R)
    for (int64_t k = threadIdx.y + 8 * (int64_t)blockIdx.y; k < K; k += 8 * (int64_t)gridDim.y)
      e = max(e, exp_of(X[r + k * ks]));
  red[threadIdx.y][threadIdx.x] = e;
  __syncthreads();
  if (threadIdx.y == 0 && r < R) {
#pragma unroll
    for (int y = 1; y < 8; ++y) e = max(e, red[y][threadIdx.x]);
    atomicMax(ex + r, e);
  }
}

// Slices of a 32-row x 64-k tile, 256 threads: four neighbouring k per thread, stored as 8 bytes per slice.
// K-contiguous rows come straight into registers, both rows of a thread and their exponents in flight together
// (VEC: 16-byte loads, where rows start on 16 bytes); others through shared memory.
// Bound by HBM: 600 rows of 262144 took 743 us with two k per thread, all rows through shared memory and an
// exponent loaded per row after the barrier; 498 us now (6.9 TB/s).
__device__ __forceinline__ void slice4(const double* x, int e, uint32_t* o, int64_t plane) {
  float t[4][S];
#pragma unroll
  for (int u = 0; u < 4; ++u) digits7(fixed56(x[u], e), t[u]);
#pragma unroll
  for (int s = 0; s < S; ++s)
    *reinterpret_cast<uint2*>(o + s * plane) = make_uint2(bf16_pair(t[0][s], t[1][s]), bf16_pair(t[2][s], t[3][s]));
}

template <bool KCONTIG, bool VEC>
__global__ void __launch_bounds__(256) slice_kernel(int64_t R, int64_t Rp, int64_t K, int64_t Kp,
                                                    const double* __restrict__ X, int64_t rs, int64_t ks, int* ex,
                                                    __nv_bfloat16* __restrict__ out) {
  __shared__ double tile[KCONTIG ? 1 : 32][KC + 1];
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.y * 32, k0 = (int64_t)blockIdx.x * KC;
  const int kq = (tid & 15) * 4, ra = tid >> 4;  // this thread's k and first row (the other 16 further on)
  double x[2][4];
  int e[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t r = r0 + ra + 16 * h;
    e[h] = r < R ? ex[r] : 0;
    if (KCONTIG) {
      const double* p = X + (r < R ? r : 0) * rs + k0 + kq;
      const int64_t left = r < R ? K - k0 - kq : 0;  // elements of the row from here on
#pragma unroll
      for (int u = 0; u < 4; u += 2) {
        double2 v = make_double2(0.0, 0.0);
        if (VEC && left > u + 1) v = *reinterpret_cast<const double2*>(p + u);
        if (!VEC && left > u + 1) v.y = p[u + 1];
        if (left == u + 1 || (!VEC && left > u)) v.x = p[u];
        x[h][u] = v.x;
        x[h][u + 1] = v.y;
      }
    }
  }
  if (!KCONTIG) {
    for (int kk = tid >> 5; kk < KC; kk += 8) {
      const int64_t r = r0 + (tid & 31), k = k0 + kk;
      tile[tid & 31][kk] = (r < R && k < K) ? X[r * rs + k * ks] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int u = 0; u < 4; ++u) x[h][u] = tile[ra + 16 * h][kq + u];
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t r = r0 + ra + 16 * h;
    if (r >= R) continue;
    // a row without a nonzero element has the exponent 0 (the blocks of the row agree on it; the one
    // at k0 = 0 stores it, and another block reads either value)
    if (e[h] <= -100000) {
      e[h] = 0;
      if (k0 == 0 && kq == 0) ex[r] = 0;
    }
    // digits t_s of x 2^(-e) = sum_s t_s 2^(-8(s+1)): |t_0| <= 256, |t_s| <= 128, each exact in BF16
    slice4(x[h], e[h], reinterpret_cast<uint32_t*>(out + r * Kp + k0 + kq), Rp * Kp / 2);
  }
}

// Exponents and slices of RB rows in one pass, the rows held in shared memory between the two: one
// read of X instead of two and one launch instead of four (preset, exponents, fix, slices).  Rows
// R .. Rp - 1 are written as zeros.  256 threads.
template <bool KCONTIG>
__global__ void __launch_bounds__(256) slice_rows_kernel(int RB, int64_t R, int64_t Rp, int64_t K, int64_t Kp,
                                                         const double* __restrict__ X, int64_t rs, int64_t ks, int* ex,
                                                         __nv_bfloat16* __restrict__ out) {
  extern __shared__ double tile[];  // RB x (K + 1)
  __shared__ int rex[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t r0 = (int64_t)blockIdx.x * RB, ld = K + 1;
  if (tid < RB) rex[tid] = -100000;
  __syncthreads();
  if (KCONTIG) {
    // a warp per run of 128 elements of a row, four loads in flight per lane
    const int runs = (int)((K + 127) / 128);
    for (int t = warp; t < RB * runs; t += 8) {
      const int rr = t / runs;
      const int64_t k0 = (int64_t)(t - rr * runs) * 128 + lane, r = r0 + rr;
      if (r >= R) continue;
      double v[4];
      int e = -100000;
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = k0 + 32 * u < K ? X[r * rs + k0 + 32 * u] : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k0 + 32 * u < K) tile[rr * ld + k0 + 32 * u] = v[u];
        e = max(e, exp_of(v[u]));
      }
      e = __reduce_max_sync(0xffffffffu, e);
      if (lane == 0) atomicMax(&rex[rr], e);
    }
  } else {
    // RB consecutive rows (a power of two) by 256 / RB k per step
    const int rr = tid & (RB - 1);
    const int kst = 256 / RB;
    const int64_t r = r0 + rr;
    int e = -100000;
    for (int64_t k0 = tid / RB; k0 < K; k0 += 4 * kst) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = r < R && k0 + u * kst < K ? X[r + (k0 + u * kst) * ks] : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k0 + u * kst < K) tile[rr * ld + k0 + u * kst] = v[u];
        e = max(e, exp_of(v[u]));
      }
    }
    atomicMax(&rex[rr], e);
  }
  __syncthreads();
  if (tid < RB && r0 + tid < R) ex[r0 + tid] = rex[tid] == -100000 ? 0 : rex[tid];
  const int segs = (int)(Kp / KC);
  for (int t = warp; t < RB * segs; t += 8) {
    const int rr = t / segs, k = (t - rr * segs) * KC + 2 * lane;
    const int64_t r = r0 + rr;
    if (r >= Rp) break;
    uint32_t* o2 = reinterpret_cast<uint32_t*>(out + r * Kp + k);
    const int e = rex[rr] == -100000 ? 0 : rex[rr];
    float t0[S], t1[S];
    digits7(r < R && k < K ? fixed56(tile[rr * ld + k], e) : 0, t0);
    digits7(r < R && k + 1 < K ? fixed56(tile[rr * ld + k + 1], e) : 0, t1);
#pragma unroll
    for (int s = 0; s < S; ++s) o2[(int64_t)s * Rp * Kp / 2] = bf16_pair(t0[s], t1[s]);
  }
}

// ---------------------------------------------------------------- the product
struct OzArgs {
  int M, N;
  int MP, NP;      // rows per slice in the A and B slice tensors
  int chunks_per_split, nchunks;
  int n_tiles;     // column tiles
  int m_fast;      // > 0: that many row tiles, walked fastest (fewer than column tiles)
  int kept;        // output tiles computed (all, or those reaching the upper triangle)
  int64_t items;   // kept x splits
  const int* ea;
  const int* eb;
  double* C;       // final output (nsplit == 1) or partials [split][N][M]
  int64_t ldc;
  int partial;
  int upper;       // only tiles that reach the upper triangle (i <= j) are computed
  int* err;
};

// Level blocks in TMEM: 8 blocks of 64 columns, 7 holding the levels of the current accumulation
// group and one spare.  perm packs, per level L = 0..6, its block (4 bits each; bits 28-31: the
// spare).  The next group puts level 0 in the spare and levels 6, 5, .., 1 in the blocks of levels
// 0, 1, .., 5, the order in which the epilogue frees them, so its MMAs start before this group is
// fully drained.
__device__ __forceinline__ uint32_t perm_block(uint32_t perm, int L) { return (perm >> (4 * L)) & 7u; }
__device__ __forceinline__ uint32_t perm_next(uint32_t perm) {
  uint32_t n = perm_block(perm, 7);
  for (int L = 1; L < S; ++L) n |= perm_block(perm, S - 1 - L) << (4 * L);
  return n | (perm_block(perm, 6) << 28);
}
constexpr uint32_t kPerm0 = 0x76543210u;

// Work item -> (row tile, column tile, K split).  Items run split-major, the side with fewer tiles fastest, so
// CTAs working at the same time share the slices of the longer operand and the split's K range in L2.  With
// `upper`, row tile tm keeps only the column tiles tn >= tm BM / BN (those reaching i <= j).
struct OzItem {
  int tm, tn, split;
};
__device__ __forceinline__ OzItem oz_item(const OzArgs& p, int64_t it) {
  OzItem r;
  r.split = (int)(it / p.kept);
  int t = (int)(it - (int64_t)r.split * p.kept);
  if (!p.upper) {
    if (p.m_fast > 0) {
      r.tn = t / p.m_fast;
      r.tm = t - r.tn * p.m_fast;
    } else {
      r.tm = t / p.n_tiles;
      r.tn = t - r.tm * p.n_tiles;
    }
    return r;
  }
  int tm = 0;
  for (;; ++tm) {
    const int row = p.n_tiles - (tm * BM) / BN;
    if (t < row) break;
    t -= row;
  }
  r.tm = tm;
  r.tn = (tm * BM) / BN + t;
  return r;
}

__global__ void __launch_bounds__(kThreads, 1)
    oz_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, OzArgs p) {
  extern __shared__ uint8_t smem_raw[];
  // lev[g & 1][L]: level L of accumulation group g has all its products (two sets, so that the next
  // group's levels never complete a phase that the epilogue is still waiting for)
  // arrivals by chunk parity: A slices 0 | 1, 2 | 3, 4 | 5, 6 and all B slices (a wait of the issuer costs about
  // 130 clocks, four MMAs, even when it finds its data there)
  __shared__ __align__(8) uint64_t afull[2][4], bfull[2], pass_done[kPassRing], lev[2][S], bfree[8], mdone;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sB = smem + kARing * kASlice;   // ring of B slices 6 .. 1
  uint8_t* sB0 = sB + kBRing * kBSlice;    // two slots of B slice 0

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      for (int g = 0; g < 4; ++g) tc::mbar_init(&afull[i][g], 1);
      tc::mbar_init(&bfull[i], 1);
    }
    for (int i = 0; i < kPassRing; ++i) tc::mbar_init(&pass_done[i], 1);
    for (int L = 0; L < S; ++L) {
      tc::mbar_init(&lev[0][L], 1);
      tc::mbar_init(&lev[1][L], 1);
    }
    for (int b = 0; b < 8; ++b) tc::mbar_init(&bfree[b], kEpiThreads);
    tc::mbar_init(&mdone, 1);
    tc::fence_barrier_init();
    abort_flag = 0;
    tc::prefetch_tmap(&mapA);
    tc::prefetch_tmap(&mapB);
  }
  if (warp == 1) {
    tc::tmem_alloc(&tmem_slot, kTmemCols);
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
  auto chunks_of = [&](int split) {
    const int c0 = split * p.chunks_per_split;
    return min(p.nchunks, c0 + p.chunks_per_split) - c0;
  };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer.  Counted over the whole launch: chunk cg, pass 7 cg + s (it reads A
      // slice s), B ring entry 6 cg + (6 - t) for slice t >= 1.  Order of the loads = order of first use.
      int64_t cg = 0;
      int64_t seen = -1;  // passes up to this one are known to be done
      int armed = 0;      // arrivals of chunk cg armed so far: A group 0, B, A groups 1 .. 3
      bool ok = true;
      auto pass_is_done = [&](int64_t pass) -> bool {
        if (pass <= seen) return true;
        if (*vabort || !tc::mbar_wait(&pass_done[pass & (kPassRing - 1)], (uint32_t)(pass / kPassRing) & 1u)) return false;
        seen = pass;
        return true;
      };
      for (int64_t it = blockIdx.x; it < p.items && ok; it += G) {
        const OzItem w = oz_item(p, it);
        const int nch = chunks_of(w.split), c_begin = w.split * p.chunks_per_split;
        for (int ci = 0; ci < nch; ++ci) {
          const int k0 = (c_begin + ci) * KCH, z = (int)(cg & 1);
          armed = 0;
          auto load_a = [&](int s) {
            const int64_t pass = S * cg + s;  // the slot's previous slice was read by pass - kARing
            if (!pass_is_done(pass - kARing)) return false;
            const int slot = (int)(pass & (kARing - 1)), g = (s + 1) / 2;
            if (s == 0 || (s & 1)) {
              tc::mbar_arrive_expect_tx(&afull[z][g], s == 0 ? kASlice : 2 * kASlice);
              ++armed;
            }
            tc::tma_load_2d(smem + (size_t)slot * kASlice, &mapA, &afull[z][g], k0, s * p.MP + w.tm * BM);
            return true;
          };
          ok = load_a(0) && pass_is_done(S * (cg - 2) + S - 1);
          if (!ok) break;
          tc::mbar_arrive_expect_tx(&bfull[z], S * kBSlice);
          ++armed;
          tc::tma_load_2d(sB0 + (size_t)z * kBSlice, &mapB, &bfull[z], k0, w.tn * BN);
          for (int t = S - 1; t >= 1 && ok; --t) {
            const int64_t q = (S - 1) * cg + (S - 1 - t), o = q - kBRing;  // o: the slot's previous entry
            ok = o < 0 || pass_is_done(S * (o / (S - 1)) + o % (S - 1));
            if (ok)
              tc::tma_load_2d(sB + (size_t)(q & (kBRing - 1)) * kBSlice, &mapB, &bfull[z], k0, t * p.NP + w.tn * BN);
          }
          for (int s = 1; s < S && ok; ++s) ok = load_a(s);
          if (!ok) break;
          ++cg;
        }
      }
      if (!ok) {
        fail();
        // wait for copies that may still be landing in this CTA's shared memory: whole chunks by their barriers,
        // the copies of the unfinished one (its arrivals may never complete) for a time far above a copy's
        for (int64_t c = (cg > 2 ? cg - 2 : 0); c < cg; ++c) {
          const int z = (int)(c & 1);
          if (c == cg - 2 && armed) continue;  // (its barriers are in use by chunk cg, and its copies were all read)
          for (int g = 0; g < 4; ++g) tc::mbar_wait(&afull[z][g], (uint32_t)(c >> 1) & 1u);
          tc::mbar_wait(&bfull[z], (uint32_t)(c >> 1) & 1u);
        }
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000LL) {}
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the whole warp walks the unrolled (s, t, k) sequence with
    // warp-uniform values, one elected lane issues
    const bool leader = tc::elect_one();
    const uint32_t idesc = tc::instr_desc(1u, BM, BN);  // BF16 x BF16 -> FP32, M = 128
    uint32_t perm = kPerm0, use_par = 0;  // use_par bit b: parity of the uses of level block b so far
    int64_t cg = 0, gidx = 0;
    bool ok = true;
    const uint64_t a_base = tc::sw128_desc(tc::smem_u32(smem)), b_base = tc::sw128_desc(tc::smem_u32(sB)),
                   b0_base = tc::sw128_desc(tc::smem_u32(sB0));
    for (int64_t it = blockIdx.x; it < p.items && ok; it += G) {
      const OzItem wi = oz_item(p, it);
      const int nch = chunks_of(wi.split);
      for (int ci = 0; ci < nch && ok; ++ci, ++cg) {
        const bool first = (ci % GROUP) == 0, last = (ci % GROUP) == GROUP - 1 || ci == nch - 1;
        uint32_t dcol[S];  // TMEM columns of the levels
        uint64_t bd[S];    // descriptors of the chunk's B slices
#pragma unroll
        for (int L = 0; L < S; ++L) dcol[L] = tmem + perm_block(perm, L) * (uint32_t)BN;
        const uint32_t z = (uint32_t)cg & 1u, par = (uint32_t)(cg >> 1) & 1u;
        bd[0] = tc::desc_add(b0_base, z * kBSlice);
#pragma unroll
        for (int t = 1; t < S; ++t)
          bd[t] = tc::desc_add(b_base, ((uint32_t)((S - 1) * cg + (S - 1 - t)) & (kBRing - 1)) * kBSlice);
        // a wait that runs out is looked at once per chunk: the products in between then run on whatever the
        // slots hold, and the launch fails
        bool w = !*vabort;
        w &= tc::mbar_wait(&bfull[z], par);
        w &= tc::mbar_wait(&afull[z][0], par);
        auto wait_blocks = [&](int t) {  // the epilogue releases blocks in the order 6, 5, .., 1 of the next group
          const uint32_t blk = perm_block(perm, t);
          w &= tc::mbar_wait(&bfree[blk], ((use_par >> blk) & 1u) ^ 1u);
        };
        if (first) wait_blocks(5);
        tc::tc_fence_after();
        // one A tile (16 K values) against B slices t0, t0 + 1, .., kept in the collector between them
        auto run = [&](int s, int n, auto slice) {
          const uint64_t a0 = tc::desc_add(a_base, ((uint32_t)(S * cg + s) & (kARing - 1)) * kASlice);
#pragma unroll
          for (int kk = 0; kk < KCH / 16; ++kk)
#pragma unroll
            for (int u = 0; u < n; ++u) {
              const int t = slice(u);
              tc::mma_f16_run(leader, u, n, dcol[s + t], tc::desc_add(a0, kk * 32), tc::desc_add(bd[t], kk * 32), idesc,
                              first && s == 0 && kk == 0 ? 0u : 1u);
            }
        };
        auto pass_end = [&](int s) {
          __syncwarp();
          if (leader) {
            tc::mma_commit(&pass_done[(S * cg + s) & (kPassRing - 1)]);  // A slice s and B slice 6 - s are free
            if (last) tc::mma_commit(&lev[gidx & 1][s]);                 // level s of the group has all its products
          }
          __syncwarp();
        };
        // pass 0 in two runs, the first into the blocks that are released early (0: the spare, 6, 5)
        run(0, 3, [](int u) { return u == 0 ? 0 : S - u; });
        if (first) {
          wait_blocks(1);
          use_par ^= 0xffu & ~(1u << perm_block(perm, 7));  // the seven blocks of this group
        }
        w &= tc::mbar_wait(&afull[z][1], par);
        tc::tc_fence_after();
        run(0, 4, [](int u) { return 4 - u; });
        pass_end(0);
        run(1, 6, [](int u) { return u; });
        pass_end(1);
        w &= tc::mbar_wait(&afull[z][2], par);
        tc::tc_fence_after();
        run(2, 5, [](int u) { return u; });
        pass_end(2);
        run(3, 4, [](int u) { return u; });
        pass_end(3);
        w &= tc::mbar_wait(&afull[z][3], par);
        tc::tc_fence_after();
        run(4, 3, [](int u) { return u; });
        pass_end(4);
        run(5, 2, [](int u) { return u; });
        pass_end(5);
        run(6, 1, [](int u) { return u; });
        pass_end(6);
        ok = __all_sync(0xffffffffu, w);
        if (!ok) break;
        if (last) {
          perm = perm_next(perm);
          ++gidx;
        }
      }
    }
    if (!ok && leader) fail();
    // every issued MMA completes (bounded wait) before the TMEM is released
    __syncwarp();
    if (leader) tc::mma_commit(&mdone);
    __syncwarp();
    tc::mbar_wait(&mdone, 0);
  } else {
    // ---------------- epilogue: 16 warps, lane quarter q, 16 columns each.  Level L of a group is
    // folded into the integer accumulators as soon as
    // the group's pass L is done, and its block released; the final value of an item is stored while
    // the next item's MMAs run.  (Every instruction here delays the issuing warp: with a scaling and a TwoSum in
    // FP32 per level, seven instructions per value, an MMA took 68 clocks.)
    const int q = warp & 3, hq = (warp - 2) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hq * 16);
    uint32_t perm = kPerm0;
    int64_t gidx = 0;  // accumulation groups drained so far
    bool ok = true;
    for (int64_t it = blockIdx.x; it < p.items && ok; it += G) {
      const OzItem wi = oz_item(p, it);
      const int ngroups = (chunks_of(wi.split) + GROUP - 1) / GROUP;
      // sum_L D_L 2^(48 - 8 L) = top 2^32 + low over all groups (at most kMaxSplitChunks / GROUP), exact in 64-bit
      // integers: a conversion and one wide multiply-add per level and column
      long long top[16], low[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) top[u] = low[u] = 0;
      for (int g = 0; g < ngroups && ok; ++g, ++gidx) {
        uint64_t* lv = lev[gidx & 1];
        const uint32_t par = (uint32_t)((gidx >> 1) & 1);
#pragma unroll
        for (int L = 0; L < S; ++L) {
          const bool w = !*vabort && tc::mbar_wait(&lv[L], par);
          ok = __all_sync(0xffffffffu, w);
          if (!ok) break;
          tc::tc_fence_after();
          const uint32_t blk = perm_block(perm, L);
          float v[16];
          tc::tmem_ld16(lane_base + blk * (uint32_t)BN, v);
          tc::tc_fence_before();
          tc::mbar_arrive(&bfree[blk]);
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int d = __float2int_rn(v[u]);
            if (L < 3) top[u] += (long long)d * (1 << (16 - 8 * (L < 3 ? L : 2)));
            else low[u] += (long long)d * (1 << (24 - 8 * (L < 3 ? 3 : L - 3)));
          }
        }
        perm = perm_next(perm);
      }
      if (!ok) {
        fail();
        break;
      }
      const int64_t i = (int64_t)wi.tm * BM + q * 32 + lane;
      if (i < p.M) {
        const int ei = p.ea[i];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int64_t jcol = (int64_t)wi.tn * BN + hq * 16 + u;
          if (jcol < p.N) {
            // (top 2^32 + low) 2^(e_i + f_j - 64): `top` is exact in FP64, `low` 2^-32 of its scale
            const int pw = ei + p.eb[jcol] - 64;
            const double v = fixed_to_f64(top[u], pw + 32) + fixed_to_f64(low[u], pw);
            if (p.partial) p.C[((int64_t)wi.split * p.N + jcol) * p.M + i] = v;
            else p.C[jcol * p.ldc + i] = v;
          }
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
}

// Sum of the split-K partials; `mirror`: of the upper triangle, written to both.
__global__ void oz_sum_kernel(int64_t M, int64_t N, int nsplit, const double* __restrict__ part, double* C,
                              int64_t ldc, int mirror) {
  const int64_t total = M * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / M, i = e - j * M;
    if (mirror && i > j) continue;
    double acc = 0.0;
    for (int s = 0; s < nsplit; ++s) acc += part[(int64_t)s * total + e];
    C[j * ldc + i] = acc;
    if (mirror && i < j) C[i * ldc + j] = acc;
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::mutex mu;
  std::lock_guard<std::mutex> lk(mu);
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    RC_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q));
    RC_CHECK(q == cudaDriverEntryPointSuccess && ptr, RCHFSI_ERR_CUDA, "cuTensorMapEncodeTiled not available");
    fn = (PFN_cuTensorMapEncodeTiled_v12000)ptr;
  }
  return fn;
}

// All slices of an operand as one 2D BF16 tensor: S*R rows of Kp elements.
CUtensorMap slice_map(const OzOperand& op, int box_rows) {
  CUtensorMap m;
  RC_CHECK(((uintptr_t)op.sl.p & 15) == 0 && (op.Kp * 2) % 16 == 0, RCHFSI_ERR_INVALID_ARG, "slice alignment");
  cuuint64_t dims[2] = {(cuuint64_t)op.Kp, (cuuint64_t)(S * op.Rp)};
  cuuint64_t strides[1] = {(cuuint64_t)(op.Kp * 2)};
  cuuint32_t box[2] = {(cuuint32_t)KCH, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)op.sl.p, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  RC_CHECK(r == CUDA_SUCCESS, RCHFSI_ERR_CUDA, "cuTensorMapEncodeTiled failed for a slice tensor");
  return m;
}

}  // namespace

namespace {
int sm_count() {
  static const int n = [] {
    int d = 0, c = 152;
    if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, d) != cudaSuccess)
      c = 152;
    return c;
  }();
  return n;
}
}  // namespace

void oz_slice(cudaStream_t s, int64_t R, int64_t K, const double* X, int64_t rs, int64_t ks, OzOperand& op) {
  RC_CHECK(R > 0 && K > 0, RCHFSI_ERR_INVALID_ARG, "oz_slice: empty operand");
  RC_CHECK(ks == 1 || rs == 1, RCHFSI_ERR_INVALID_ARG, "oz_slice: one of the strides must be 1");
  op.R = R;
  op.Rp = std::max<int64_t>(R, 32);  // the 128-row TMA box must fit in the S * Rp rows of the tensor
  op.K = K;
  op.Kp = (K + KC - 1) / KC * KC;
  op.sl.ensure((size_t)S * op.Rp * op.Kp);
  op.ex.ensure((size_t)R);
  prof::Scope ps(s, RCHFSI_KERNEL_RR_AUX, 0.0, 8.0 * R * K + 2.0 * S * op.Rp * op.Kp);
  // One pass with the rows in shared memory, when RB rows of K fit (64 KB: three CTAs per SM) and
  // there are CTAs for most of the SMs; RB is 8 (16) rows where rows are contiguous across threads, so
  // that a load covers whole 64-byte runs, and down to 1 for few K-contiguous rows.  Measured against
  // the separate passes (us, exponents + fix + slices -> one pass, without the launches in between):
  // 60 x 60 18 -> 4.2, 240 x 240 19 -> 8, 4000 x 240 by rows 23 -> 11.6, 262144 x 600 by rows 1120 -> 943.
  int rb = 0;
  const size_t row = ((size_t)K + 1) * sizeof(double);
  if (ks == 1) {
    for (int c : {8, 4, 2, 1})
      if (rb == 0 && c * row <= 66 * 1024 && (c == 1 || (int64_t)cdiv(R, c) >= sm_count() / 2)) rb = c;
    if ((int64_t)R * 4 < sm_count()) rb = K <= 1024 ? rb : 0;  // few long rows: split along K instead
  } else if (8 * row <= 66 * 1024) {
    rb = 8;
  }
  if (rb > 0) {
    const unsigned g = cdiv(op.Rp, rb);
    const size_t smem = rb * row;
    if (ks == 1) {
      set_smem_limit(reinterpret_cast<const void*>(slice_rows_kernel<true>), 68 * 1024);
      slice_rows_kernel<true><<<g, 256, smem, s>>>(rb, R, op.Rp, K, op.Kp, X, rs, ks, op.ex.p, op.sl.p);
    } else {
      set_smem_limit(reinterpret_cast<const void*>(slice_rows_kernel<false>), 68 * 1024);
      slice_rows_kernel<false><<<g, 256, smem, s>>>(rb, R, op.Rp, K, op.Kp, X, rs, ks, op.ex.p, op.sl.p);
    }
    RC_LAUNCH();
    return;
  }
  if (op.Rp > R) RC_CUDA(cudaMemsetAsync(op.sl.p, 0, sizeof(__nv_bfloat16) * S * op.Rp * op.Kp, s));
  RC_CUDA(cudaMemsetAsync(op.ex.p, 0x80, sizeof(int) * R, s));  // 0x80808080: below every exponent
  if (ks == 1) {
    // K slices of >= 256 elements, enough (row, slice) warps for ~16 per SM
    const unsigned rw = cdiv(R, 8);
    const unsigned kb = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>(cdiv(K, 256), (int64_t)(sm_count() * 16 * 8) / std::max<int64_t>(R, 1)));
    rowexp_kcontig<<<dim3(rw, kb), 256, 0, s>>>(R, K, X, rs, op.ex.p);
  } else {
    // enough blocks to fill the GPU a few times over, each warp walking at least 8 k
    const unsigned rw = cdiv(R, 32);
    const unsigned kb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(cdiv(K, 64), (int64_t)(sm_count() * 16) / rw));
    rowexp_rcontig<<<dim3(rw, kb), dim3(32, 8), 0, s>>>(R, K, X, ks, op.ex.p);
  }
  RC_LAUNCH();
  RC_CHECK(cdiv(R, 32) <= 65535u, RCHFSI_ERR_INVALID_ARG, "oz_slice: too many rows");
  dim3 grid((unsigned)(op.Kp / KC), cdiv(R, 32));
  const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && rs % 2 == 0;
  if (ks != 1) slice_kernel<false, false><<<grid, 256, 0, s>>>(R, op.Rp, K, op.Kp, X, rs, ks, op.ex.p, op.sl.p);
  else if (vec) slice_kernel<true, true><<<grid, 256, 0, s>>>(R, op.Rp, K, op.Kp, X, rs, ks, op.ex.p, op.sl.p);
  else slice_kernel<true, false><<<grid, 256, 0, s>>>(R, op.Rp, K, op.Kp, X, rs, ks, op.ex.p, op.sl.p);
  RC_LAUNCH();
}

namespace {

// Split-K count: the smallest with which the (tile, split) items fill whole rounds of one item per
// persistent CTA to >= 90% (else the best found); a few output tiles (N x N products) go down to one
// chunk per split, since a chunk is 3.3 us of MMAs in a CTA.
int choose_split(int tiles, int nchunks, int num_sms, double* eff_out) {
  const int max_split = std::max(1, std::min(64, nchunks));
  double best = -1.0;
  int nsplit = 1;
  for (int ns = 1; ns <= max_split; ++ns) {
    const int64_t ctas = (int64_t)tiles * ns;
    const int64_t waves = (ctas + num_sms - 1) / num_sms;
    const double eff = (double)ctas / (double)(waves * num_sms);
    if (eff > best + 1e-9) {
      best = eff;
      nsplit = ns;
    }
    if (eff >= 0.9) break;
  }
  *eff_out = best;
  return nsplit;
}

// C(i, j) = C(j, i) for i > j (column-major n x n)
__global__ void mirror_upper_kernel(int n, double* C, int64_t ldc) {
  const int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(t / n), i = (int)(t - (int64_t)j * n);
    if (i > j) C[(int64_t)j * ldc + i] = C[(int64_t)i * ldc + j];
  }
}

// Output tiles of a product that reach the upper triangle (all of them unless `upper`).
int kept_tiles(int m_tiles, int n_tiles, bool upper) {
  if (!upper) return m_tiles * n_tiles;
  int t = 0;
  for (int bm = 0; bm < m_tiles; ++bm) t += std::max(0, n_tiles - (bm * BM) / BN);
  return t;
}

}  // namespace

void oz_gemm(cudaStream_t s, int num_sms, const OzOperand& A, const OzOperand& B, double* C, int64_t ldc,
             DevBuf<double>& ws, int* err, bool symmetric) {
  RC_CHECK(A.K == B.K && A.Kp == B.Kp, RCHFSI_ERR_INVALID_ARG, "oz_gemm: K mismatch");
  const int64_t M = A.R, N = B.R;
  RC_CHECK(!symmetric || M == N, RCHFSI_ERR_INVALID_ARG, "oz_gemm: a symmetric product is square");
  RC_CHECK(M < (1LL << 31) && N < (1LL << 31), RCHFSI_ERR_INVALID_ARG, "oz_gemm: too large");
  const int m_tiles = (int)((M + BM - 1) / BM), n_tiles = (int)((N + BN - 1) / BN);
  const int nchunks = (int)(A.Kp / KCH);
  const int kept = kept_tiles(m_tiles, n_tiles, symmetric);
  // persistent CTAs over (tile, K split) items: split K only as far as the items then fill the CTAs
  double eff = 0.0;
  int nsplit = choose_split(kept, nchunks, num_sms, &eff);
  nsplit = std::max(nsplit, (nchunks + kMaxSplitChunks - 1) / kMaxSplitChunks);
  const int per = (nchunks + nsplit - 1) / nsplit;
  nsplit = (nchunks + per - 1) / per;
  const CUtensorMap ma = slice_map(A, BM);
  const CUtensorMap mb = slice_map(B, BN);
  constexpr size_t smem = (size_t)kSmemBytes + 1024;
  set_smem_limit(reinterpret_cast<const void*>(oz_gemm_kernel), (int)smem);
  OzArgs p;
  p.M = (int)M;
  p.N = (int)N;
  p.MP = (int)A.Rp;
  p.NP = (int)B.Rp;
  p.chunks_per_split = per;
  p.nchunks = nchunks;
  p.n_tiles = n_tiles;
  p.m_fast = m_tiles < n_tiles ? m_tiles : 0;
  p.kept = kept;
  p.items = (int64_t)kept * nsplit;
  p.ea = A.ex.p;
  p.eb = B.ex.p;
  p.err = err;
  p.partial = nsplit > 1;
  p.upper = symmetric ? 1 : 0;
  if (nsplit > 1) {
    p.C = ws.ensure((size_t)nsplit * M * N);
    p.ldc = M;
  } else {
    p.C = C;
    p.ldc = ldc;
  }
  const unsigned grid = (unsigned)std::min<int64_t>(p.items, num_sms);
  {
    // tensor-core flops of the 28 slice products; bytes: the slices once and the FP64 output
    // (a symmetric product computes the kept tiles only: the flops of those tiles)
    const double frac = (double)kept / ((double)m_tiles * n_tiles);
    prof::Scope ps(s, RCHFSI_KERNEL_GEMM_F64_EMU, 2.0 * M * N * A.Kp * (S * (S + 1) / 2) * frac,
                   2.0 * S * (double)(M + N) * A.Kp + 8.0 * M * N);
    oz_gemm_kernel<<<grid, kThreads, smem, s>>>(ma, mb, p);
    RC_LAUNCH();
  }
  if (nsplit > 1) {
    const int64_t total = M * N;
    const unsigned blocks = (unsigned)std::min<int64_t>((total + 255) / 256, (int64_t)num_sms * 8);
    oz_sum_kernel<<<blocks, 256, 0, s>>>(M, N, nsplit, p.C, C, ldc, symmetric ? 1 : 0);
    RC_LAUNCH();
  }
  if (symmetric && nsplit == 1) {
    const unsigned blocks = (unsigned)std::min<int64_t>((M * N + 255) / 256, (int64_t)num_sms * 4);
    mirror_upper_kernel<<<blocks, 256, 0, s>>>((int)M, C, ldc);
    RC_LAUNCH();
  }
}

}  // namespace rchfsi
