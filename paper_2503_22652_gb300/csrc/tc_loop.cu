// The degree loop of the dense filter in one persistent launch on the tcgen05 tensor cores.
//
// One launch per degree step and split-K sum (tc_gemm.cu) spends more on launches, on draining the
// pipeline and on the sum than on the products: at m = 4000, N = 240 a step took 20.8 us for the product,
// 7.2 us for the sum and ~7 us of gaps, against 8 us of TF32 MMAs; at m = 1000, N = 60 the four parts
// are all latency.  Here every CTA keeps one (128-row tile, K split) of the product for all steps:
//   warp 0     TMA producer: the A chunks of the next step are requested while this step is still
//              being summed (they do not depend on it); the R chunks follow, each as soon as the row
//              tile it comes from is marked ready;
//   warp 1     tcgen05.mma issuer (whole warp, one elected lane) into one of two TMEM accumulators;
//   warps 2-9  write the CTA's partial tile to a workspace (L2), count it in, and when all splits of
//              the row tile are in, sum the CTA's own share (N / nsplit columns) in split order, apply
//              the recurrence and store the new R.  R_k, R_{k-1} and W of the share stay in registers
//              for the whole loop.
// (Clusters of 2 or 4 row tiles that load R once and multicast it were no faster: 673 and 702 us against 663
// at m = 4000, N = 240, where a step loads 1.5 MB per CTA; L2 is not the bound.)
//
// Ordering without a grid barrier.  ready[t] counts the shares of row tile t stored for each step, parts[t]
// the partial tiles.  A CTA starts step k + 1 on chunk i when ready[tile of i] shows step k.  Because a row
// tile is only finished with the partial tiles of all its splits, which together read all of R, every
// buffer may be reused two steps later: R (two buffers), the partial tiles (two sets), the two
// accumulators.  All CTAs are resident (cooperative launch) and every wait is bounded; after a failed
// wait the kernel raises the error flag, waits for copies in flight and returns.
#include <cudaTypedefs.h>

#include <algorithm>
#include <type_traits>

#include "prof.cuh"
#include "tc_loop.cuh"
#include "tc_ptx.cuh"

namespace rchfsi {
namespace {

constexpr int kBM = 128;
constexpr int kRowBytes = 128;
constexpr int kMaxStages = 8;
constexpr int kThreads = 320;
constexpr int kSmemCap = 232448 - 2048;  // dynamic shared memory: the limit less the static part
constexpr int kCntStride = 32;  // ints between two counters: one 128-byte line each

struct LoopArgs {
  int M, N, ld, BN, m_tiles, nsplit, kb_per_split, stages, steps;
  uint32_t acc_cols;
  float* ws;
  void* R0;
  void* R1;
  const void* W;
  const float* coef;
  const float* lam;
  int* cnt;  // parts[m_tiles], then ready[m_tiles]
  int* err;
};

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void from_f(float& d, float v) { d = v; }
__device__ __forceinline__ void from_f(__nv_bfloat16& d, float v) { d = __float2bfloat16_rn(v); }

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(int* p) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// *p >= want, waiting at most as long as the mbarrier waits do; false also once another CTA has failed.
__device__ __forceinline__ bool wait_count(const int* p, int want, const int* err) {
  if (ld_acquire(p) >= want) return true;
  const long long t0 = clock64();
  for (int spin = 0; ld_acquire(p) < want; ++spin) {
    if (clock64() - t0 > tc::kWaitCycles) return false;
    if ((spin & 255) == 255 && *(volatile const int*)err) return false;
  }
  return true;
}

// Barrier of the epilogue threads that also tells each of them whether any passed `bad`.
__device__ __forceinline__ bool epi_any(bool bad) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, 256, p;\nselp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)bad)
      : "memory");
  return r != 0;
}

// EC: columns of the share per epilogue thread (at most).
template <typename T, int EC>
__global__ void __launch_bounds__(kThreads, 1)
    tc_loop_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapR0,
                   const __grid_constant__ CUtensorMap mapR1, const LoopArgs p) {
  constexpr bool kBF16 = std::is_same<T, __nv_bfloat16>::value;
  constexpr int BK = kRowBytes / (int)sizeof(T);
  constexpr int KMMA = kBF16 ? 16 : 8;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float s_lam[2 * EC];  // Lambda of the share's columns in the current step

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = blockIdx.x, split = blockIdx.y;
  const int nkb_total = (p.M + BK - 1) / BK;
  const int kb_begin = split * p.kb_per_split;
  const int nkb = min(nkb_total, kb_begin + p.kb_per_split) - kb_begin;
  const int nS = p.stages;
  int* parts = p.cnt;
  int* ready = p.cnt + (size_t)p.m_tiles * kCntStride;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t a_bytes = kBM * kRowBytes;
  const uint32_t b_bytes = (uint32_t)p.BN * kRowBytes;
  const uint32_t stage_bytes = a_bytes + b_bytes;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      tc::mbar_init(&full_bar[s], 1);
      tc::mbar_init(&empty_bar[s], 1);
    }
    tc::mbar_init(&acc_bar[0], 1);
    tc::mbar_init(&acc_bar[1], 1);
    tc::fence_barrier_init();
    abort_flag = 0;
    tc::prefetch_tmap(&mapA);
    tc::prefetch_tmap(&mapR0);
    tc::prefetch_tmap(&mapR1);
  }
  if (warp == 1) {
    tc::tmem_alloc(&tmem_slot, 2 * p.acc_cols);
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

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer
      // (slots and phases are counted up: a 64-bit remainder per use made this loop, at 1290 clocks a chunk, the
      // bound of large operators)
      const int pre = min(nS, nkb);  // A chunks of a step requested before its R is known to be ready
      int sa = 0, sr = 0;     // slots of the next A and the next R chunk
      uint32_t ph = 1;        // phase parity that frees slot sa
      bool ok = true;
      for (int k = 0; k < p.steps && ok; ++k) {
        const CUtensorMap* mapR = (k & 1) ? &mapR1 : &mapR0;
        int seen = -1;  // last row tile found ready
        auto put_a = [&](int i) -> bool {
          if (*vabort || !tc::mbar_wait(&empty_bar[sa], ph)) return false;
          tc::mbar_arrive_expect_tx(&full_bar[sa], stage_bytes);
          tc::tma_load_2d(smem + (size_t)sa * stage_bytes, &mapA, &full_bar[sa], (kb_begin + i) * BK, mt * kBM);
          if (++sa == nS) {
            sa = 0;
            ph ^= 1u;
          }
          return true;
        };
        auto put_r = [&](int i) -> bool {
          const int k0 = (kb_begin + i) * BK, tile = k0 / kBM;
          if (k > 0 && tile != seen) {
            if (*vabort || !wait_count(ready + (size_t)tile * kCntStride, k * p.nsplit, p.err)) return false;
            fence_proxy_async_global();  // the rows were stored through the generic proxy
            seen = tile;
          }
          tc::tma_load_2d(smem + (size_t)sr * stage_bytes + a_bytes, mapR, &full_bar[sr], k0, 0);
          if (++sr == nS) sr = 0;
          return true;
        };
        for (int i = 0; i < pre && ok; ++i) ok = put_a(i);
        for (int i = 0; i < nkb && ok; ++i) {
          if (i >= pre) ok = put_a(i);
          if (ok) ok = put_r(i);
        }
      }
      if (!ok) fail();
      // every slot has been released by all its readers: nothing of this CTA's ring is still in flight
      // (slots the ring never reached are in their first phase, which their waits of parity 1 pass)
      for (int i = 0; i < nS && ok; ++i) {
        ok = tc::mbar_wait(&empty_bar[sa], ph);
        if (++sa == nS) {
          sa = 0;
          ph ^= 1u;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer
    const bool leader = tc::elect_one();
    const uint32_t idesc = tc::instr_desc(kBF16 ? 1u : 2u, kBM, p.BN);
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int k = 0; k < p.steps && ok; ++k) {
      const uint32_t acc = tmem + (uint32_t)(k & 1) * p.acc_cols;
      for (int i = 0; i < nkb; ++i) {
        const bool w = !*vabort && tc::mbar_wait(&full_bar[s], ph);
        ok = __all_sync(0xffffffffu, w);
        if (!ok) {
          if (leader) fail();
          break;
        }
        tc::tc_fence_after();
        const uint32_t a_base = tc::smem_u32(smem + (size_t)s * stage_bytes);
        const uint64_t a0 = tc::sw128_desc(a_base), b0 = tc::sw128_desc(a_base + a_bytes);
#pragma unroll
        for (int kk = 0; kk < BK / KMMA; ++kk) {
          if (leader) {
            const uint64_t ad = tc::desc_add(a0, kk * 32), bd = tc::desc_add(b0, kk * 32);
            const uint32_t accumulate = (i > 0 || kk > 0) ? 1u : 0u;
            if (kBF16) tc::mma_f16(acc, ad, bd, idesc, accumulate);
            else tc::mma_tf32(acc, ad, bd, idesc, accumulate);
          }
        }
        __syncwarp();
        if (leader) tc::mma_commit(&empty_bar[s]);
        __syncwarp();
        if (++s == nS) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (ok && leader) tc::mma_commit(&acc_bar[k & 1]);
      __syncwarp();
    }
  } else {
    // ---------------- partial tile, sum of the own share, recurrence
    const int q = warp & 3, h = (warp - 2) >> 2;
    const int et = threadIdx.x - 64;
    const int64_t row = (int64_t)mt * kBM + q * 32 + lane;
    const bool in = row < p.M;
    const int cw = (p.N + p.nsplit - 1) / p.nsplit;        // columns of a share
    const int c0 = split * cw, c1 = min(p.N, c0 + cw);     // this CTA's share; this thread: c0 + h + 2 j
    const size_t tile_floats = (size_t)p.BN * kBM;
    const size_t set_floats = (size_t)p.m_tiles * p.nsplit * tile_floats;
    const T* W = static_cast<const T*>(p.W);
    // W of the share in shared memory (each thread its own values), R_k and R_{k-1} in registers
    float* sW = reinterpret_cast<float*>(smem + (size_t)nS * stage_bytes) + h * kBM + q * 32 + lane;
    float cur[EC], prev[EC];
#pragma unroll
    for (int j = 0; j < EC; ++j) {
      const int col = c0 + h + 2 * j;
      const bool mine = in && col < c1;
      const int64_t o = (int64_t)col * p.ld + row;
      cur[j] = mine ? to_f(static_cast<const T*>(p.R0)[o]) : 0.f;
      sW[2 * j * kBM] = mine && W ? to_f(W[o]) : 0.f;
      prev[j] = 0.f;
    }
    for (int k = 0; k < p.steps; ++k) {
      const float ca = __ldg(p.coef + 3 * k), cb = __ldg(p.coef + 3 * k + 1), cc = __ldg(p.coef + 3 * k + 2);
      if (W && et < c1 - c0) s_lam[et] = __ldg(p.lam + (size_t)k * p.N + c0 + et);
      float* set = p.ws + (size_t)(k & 1) * set_floats + (size_t)mt * p.nsplit * tile_floats;
      bool bad = *vabort || !tc::mbar_wait(&acc_bar[k & 1], (uint32_t)((k >> 1) & 1));
      if (!__any_sync(0xffffffffu, bad)) {
        tc::tc_fence_after();
        float* out = set + (size_t)split * tile_floats + q * 32 + lane;
        const uint32_t base = tmem + (uint32_t)(k & 1) * p.acc_cols + ((uint32_t)(q * 32) << 16);
        for (int g = 16 * h; g < p.BN; g += 32) {
          float v[16];
          tc::tmem_ld16(base + g, v);
#pragma unroll
          for (int t = 0; t < 16; ++t)
            if (g + t < p.N) __stcg(out + (size_t)(g + t) * kBM, v[t]);
        }
        tc::tc_fence_before();
      }
      if (epi_any(bad)) {
        fail();
        break;
      }
      bad = false;
      if (et == 0) {
        red_release(parts + (size_t)mt * kCntStride);
        bad = !wait_count(parts + (size_t)mt * kCntStride, (k + 1) * p.nsplit, p.err);
      }
      if (epi_any(bad)) {
        fail();
        break;
      }
      // (columns past the share are read and not used, instead of a branch around each load: with the branches
      // every load waited for the one before it, 24k of the 80k clocks of a step at m = 4000, N = 240)
      float sum[EC];
#pragma unroll
      for (int j = 0; j < EC; ++j) sum[j] = 0.f;
      const float* src = set + (size_t)(c0 + h) * kBM + q * 32 + lane;
      if (c0 < c1) {
#pragma unroll(32 / EC)
        for (int s = 0; s < p.nsplit; ++s) {
          float v[EC];
#pragma unroll
          for (int j = 0; j < EC; ++j) v[j] = __ldcg(src + (size_t)s * tile_floats + 2 * j * kBM);
#pragma unroll
          for (int j = 0; j < EC; ++j) sum[j] += v[j];
        }
      }
      T* dst = static_cast<T*>((k & 1) ? p.R0 : p.R1) + (int64_t)(c0 + h) * p.ld + row;
      int64_t ld2 = 2 * (int64_t)p.ld;
      asm volatile("" : "+l"(ld2));  // the column offsets are formed here, not kept in registers between steps
#pragma unroll
      for (int j = 0; j < EC; ++j) {
        const int col = c0 + h + 2 * j;
        float v = ca * sum[j] + cb * cur[j];
        v += cc * prev[j];
        if (W) v += sW[2 * j * kBM] * (ca * s_lam[h + 2 * j]);
        T o;
        from_f(o, v);
        prev[j] = cur[j];
        cur[j] = to_f(o);
        if (in && col < c1) *dst = o;
        dst += ld2;
      }
      fence_proxy_async_global();  // the next step reads these rows by TMA
      epi_any(false);
      if (et == 0) red_release(ready + (size_t)mt * kCntStride);
    }
  }
  __syncthreads();
  if (*vabort) {
    // copies that were in flight land before the shared memory is released: far below 1 ms
    const long long t0 = clock64();
    while (clock64() - t0 < 4000000LL) {}
  }
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 2 * p.acc_cols);
  }
}

CUtensorMap make_map(const void* base, bool bf16, int64_t inner, int64_t outer, int64_t ld, int box_rows) {
  CUtensorMap m;
  const size_t es = bf16 ? 2 : 4;
  RC_CHECK(((uintptr_t)base & 15) == 0 && (ld * es) % 16 == 0, RCHFSI_ERR_INVALID_ARG,
           "filter loop: blocks start and rows advance by multiples of 16 bytes");
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * es)};
  cuuint32_t box[2] = {(cuuint32_t)(kRowBytes / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  const auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
  const CUresult r = fn(&m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                        const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  RC_CHECK(r == CUDA_SUCCESS, RCHFSI_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return m;
}

using Kernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, LoopArgs);

constexpr int elems_of(int e) { return e <= 2 ? 2 : e <= 8 ? 8 : 32; }
template <typename T>
Kernel pick(int elems) {
  const int ec = elems_of(elems);
  return ec == 2 ? tc_loop_kernel<T, 2> : ec == 8 ? tc_loop_kernel<T, 8> : tc_loop_kernel<T, 32>;
}

}  // namespace

// One CTA per (row tile, K split), all resident: at least four splits, so that a share of up to 64 columns fits
// the epilogue's registers, and N in one tile.  Against the per-step launches (whole filter calls, degree 20 to
// 30): m = 1000, N = 60 330 -> 180 us; m = 1537, N = 99 BF16 470 -> 263 us; m = 4000, N = 240 1117 -> 810 us.
TcLoopPlan tc_loop_plan(int num_sms, int64_t M, int64_t N, bool bf16) {
  TcLoopPlan p;
  p.M = M;
  p.N = N;
  p.bf16 = bf16;
  const int BK = kRowBytes / (bf16 ? 2 : 4);
  if (N > 256 || M > 32 * 1024) return p;
  p.m_tiles = (int)((M + kBM - 1) / kBM);
  const int nkb = (int)((M + BK - 1) / BK);
  const int ns = std::min(num_sms / p.m_tiles, nkb);
  if (ns < 4) return p;
  p.BN = (int)((N + 15) / 16 * 16);
  p.kb_per_split = (nkb + ns - 1) / ns;
  p.nsplit = (nkb + p.kb_per_split - 1) / p.kb_per_split;
  p.elems = (int)(((N + p.nsplit - 1) / p.nsplit + 1) / 2);
  if (p.elems > 32) return p;
  p.acc_cols = 16;
  while (p.acc_cols < (uint32_t)p.BN) p.acc_cols <<= 1;
  const size_t stage = (size_t)(kBM + p.BN) * kRowBytes;
  const size_t wbytes = (size_t)2 * elems_of(p.elems) * kBM * sizeof(float);  // W of the share
  p.stages = (int)std::min<size_t>(kMaxStages, (kSmemCap - 1024 - wbytes) / stage);
  p.smem = p.stages * stage + wbytes + 1024;
  p.ws_floats = 2 * (size_t)p.m_tiles * p.nsplit * p.BN * kBM + 2 * 32 * kBM;  // (a share is read past its end)
  p.counters = 2 * (size_t)p.m_tiles * kCntStride;
  p.ok = true;
  return p;
}

void tc_loop(cudaStream_t s, const TcLoopPlan& p, int64_t M, int64_t N, bool bf16, const void* A, int64_t ld, void* R0,
             void* R1, const void* W, const float* coef, const float* lam, int steps, float* ws, int* counters,
             int* err) {
  CUtensorMap ma = make_map(A, bf16, M, M, ld, kBM);
  CUtensorMap m0 = make_map(R0, bf16, M, N, ld, p.BN);
  CUtensorMap m1 = make_map(R1, bf16, M, N, ld, p.BN);
  LoopArgs a;
  a.M = (int)M;
  a.N = (int)N;
  a.ld = (int)ld;
  a.BN = p.BN;
  a.m_tiles = p.m_tiles;
  a.nsplit = p.nsplit;
  a.kb_per_split = p.kb_per_split;
  a.stages = p.stages;
  a.steps = steps;
  a.acc_cols = p.acc_cols;
  a.ws = ws;
  a.R0 = R0;
  a.R1 = R1;
  a.W = W;
  a.coef = coef;
  a.lam = lam;
  a.cnt = counters;
  a.err = err;
  const Kernel kf = bf16 ? pick<__nv_bfloat16>(p.elems) : pick<float>(p.elems);
  set_smem_limit(reinterpret_cast<const void*>(kf), kSmemCap);
  const double es = bf16 ? 2 : 4;
  // per step: A and R once, and the new R (the operator stays in L2 between steps where it fits)
  prof::Scope ps(s, RCHFSI_KERNEL_FILTER_TC, 2.0 * M * M * N * steps,
                 steps * (es * ((double)M * M + 2.0 * M * N)) + (W ? es * M * N : 0.0));
  void* args[] = {&ma, &m0, &m1, &a};
  RC_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kf), dim3(p.m_tiles, p.nsplit), dim3(kThreads),
                                      args, p.smem, s));
  RC_LAUNCH();
}

}  // namespace rchfsi
