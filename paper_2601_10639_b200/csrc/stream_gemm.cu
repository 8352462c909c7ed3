// bf16 contraction for batches of few rows (decode steps): the weight matrix streams through the tensor
// cores once and the whole batch is the narrow operand.
//
//   C[t, f] = sum_k X(t, k) W(f, k)         X [T, K], W [F, K] row-major bf16, T <= 256
//
// The roles of the operands are swapped against the general kernel: 128 rows of W (256 for a CTA pair)
// are the MMA's M, the batch padded to a multiple of 16 is its N.  A 256 x 256 tile of the general
// kernel computes and stages 128 rows of batch per CTA whether they exist or not, and one row of such
// tiles leaves most SMs without work.  Here the contraction is cut along k over the CTAs (pairs) of a
// cluster until every SM streams an equal share of W; the CTAs leave their fp32 sums in shared memory,
// and each adds one share of the batch over the cluster in ascending k and runs the epilogue on it,
// four neighbouring features per thread, so that table rows, G, H and y move in whole 128-byte lines.
//
// Bound: streaming W, on top of a chain of launch, first loads, last MMA, exchange and epilogue of some 5 us per
// kernel.  33.5 MB of cold weights take 9.6 us, 3.5 TB/s over the kernel: 4.6 us of streaming at the memory's 7.3
// TB/s and that chain.  (One SM draws at most 70 - 98 GB/s.)
// Measured, a forward pass (two of these kernels against two general ones) replayed from a graph, weights in L2 / not:
//   d_model 2048, d_ff 8192   16 rows 30.8 -> 14.9 / 32.5 -> 19.2 us     128 rows 29.8 -> 23.6 / 31.3 -> 28.0 us
//   d_model 1024, d_ff 2816   16 rows 22.0 ->  9.3 / 23.0 -> 10.8 us     128 rows 22.9 -> 14.9 / 23.8 -> 16.5 us
// Loading W before the kernel that writes X has finished gained nothing: the two then share the memory's
// bandwidth (23.7 us against 21.2 with it left out, 16 rows, weights not in L2).
#include <cuda.h>

#include "ptx_sm100.cuh"
#include "stem_internal.h"

namespace stem {
namespace {

constexpr int BM = 128;                 // rows of W per CTA
constexpr int BK = 64;
constexpr int kMaxT = 256;
constexpr int kMaxStages = 12;
constexpr int kEpiThreads = 256;
constexpr int kThreads = 64 + kEpiThreads;
constexpr long long kWaitLimitCycles = 2000000000ll;  // ~1 s at boost clock
constexpr int kWBytes = BM * BK * 2;

// bars: full[kMaxStages], empty[kMaxStages], done, drain; then tensor-memory address, abort flag, ids
constexpr int kNumBars = 2 * kMaxStages + 2;
constexpr int kTailBytes = kNumBars * 8 + 16 + kMaxT * 4;

__device__ __forceinline__ float fast_sigmoid(float g) {   // as in the general kernel
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * g));
  return fmaf(t, 0.5f, 0.5f);
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int V> struct Int { static constexpr int value = V; };

template <int KIND, int CTAS>
__global__ void __launch_bounds__(kThreads)
stream_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, int T, int F, int K,
                   int n_pad, int stages, int ksplit, int tmem_cols, EpiParams ep) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t x_bytes = static_cast<uint32_t>(n_pad / CTAS) * (BK * 2);
  const uint32_t stage_bytes = kWBytes + x_bytes;
  const uint32_t tail = max(stages * stage_bytes, static_cast<uint32_t>(n_pad) * BM * 4u);
  const uint32_t bars = base + tail;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (kMaxStages + s); };
  const uint32_t done_bar = bars + 8u * (2 * kMaxStages), drain_bar = done_bar + 8u;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + tail + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + tail + kNumBars * 8 + 4);
  int* s_ids = reinterpret_cast<int*>(base_ptr + tail + kNumBars * 8 + 16);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool clustered = CTAS * ksplit > 1;
  const uint32_t crank = clustered ? ptx::cluster_ctarank() : 0u;
  const uint32_t rank = CTAS == 2 ? crank & 1u : 0u, leader = crank - rank;
  const int slice = static_cast<int>(crank) / CTAS;
  const int f0 = (static_cast<int>(blockIdx.x) / (CTAS * ksplit) * CTAS + static_cast<int>(rank)) * BM;
  const int k_blocks = (K + BK - 1) / BK;
  const int kb0 = k_blocks * slice / ksplit, kb1 = k_blocks * (slice + 1) / ksplit;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { ptx::mbar_init(full_bar(s), 1); ptx::mbar_init(empty_bar(s), 1); }
    ptx::mbar_init(done_bar, 1);
    ptx::mbar_init(drain_bar, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tensormap(&tmW);
    ptx::prefetch_tensormap(&tmX);
  }
  if (warp == 1) {
    if (CTAS == 2) {
      ptx::tmem_alloc_pair(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), tmem_cols);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(ptx::smem_u32(const_cast<uint32_t*>(tmem_slot)), tmem_cols);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  // a pair signals each other's barriers from here on; single CTAs meet only at the exchange of sums
  if (CTAS == 2) ptx::cluster_sync(); else __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  int issued = 0;   // producer: k blocks handed to TMA so far
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      auto load = [&](uint32_t dst, const CUtensorMap* map, int s, int k0, int row) {
        if (CTAS == 2) ptx::tma_load_2d_pair(dst, map, ptx::mapa(full_bar(s), leader), k0, row);
        else ptx::tma_load_2d(dst, map, full_bar(s), k0, row);
      };
      ptx::grid_dependency_wait();
      ptx::grid_launch_dependents();
      int s = 0; uint32_t ph = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!ptx::mbar_wait_bounded(empty_bar(s), ph ^ 1u, abort_flag, kWaitLimitCycles)) {
          report_error(ep.status, STEM_ERR_TIMEOUT, 1);
          *abort_flag = 1; break;
        }
        if (rank == 0) ptx::mbar_arrive_expect_tx(full_bar(s), CTAS * stage_bytes);
        load(base + s * stage_bytes, &tmW, s, kb * BK, f0);
        load(base + s * stage_bytes + kWBytes, &tmX, s, kb * BK, rank * (n_pad / CTAS));
        ++issued;
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      const uint32_t idesc = ptx::make_idesc_bf16(BM * CTAS, n_pad, false, false);
      const uint16_t pair_mask = static_cast<uint16_t>(3u << leader);
      ptx::grid_dependency_wait();   // nothing is read here, but the limit of the waits below must not run before
      int s = 0; uint32_t ph = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!ptx::mbar_wait_bounded(full_bar(s), ph, abort_flag, kWaitLimitCycles)) {
          report_error(ep.status, STEM_ERR_TIMEOUT, 2);
          *abort_flag = 1; ok = false; break;
        }
        ptx::tc_fence_after();
        const uint32_t w_src = base + s * stage_bytes, x_src = w_src + kWBytes;
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          const uint64_t ad = ptx::make_smem_desc(w_src + kk * 32, 16, 1024), bd = ptx::make_smem_desc(x_src + kk * 32, 16, 1024);
          if (CTAS == 2) ptx::mma_bf16_ss_pair(tmem_base, ad, bd, idesc, (kb > kb0 || kk > 0) ? 1u : 0u);
          else ptx::mma_bf16_ss(tmem_base, ad, bd, idesc, (kb > kb0 || kk > 0) ? 1u : 0u);
        }
        if (CTAS == 2) ptx::mma_commit_pair(empty_bar(s), pair_mask); else ptx::mma_commit(empty_bar(s));
        if (++s == stages) { s = 0; ph ^= 1u; }
      }
      if (ok) {
        if (CTAS == 2) ptx::mma_commit_pair(done_bar, pair_mask); else ptx::mma_commit(done_bar);
      } else {
        // let MMAs already issued finish before TMEM is freed
        if (CTAS == 2) ptx::mma_commit_pair(drain_bar, static_cast<uint16_t>(1u << leader)); else ptx::mma_commit(drain_bar);
        int zero = 0;
        ptx::mbar_wait_bounded(drain_bar, 0, &zero, kWaitLimitCycles);
      }
    }
  } else {
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int et = threadIdx.x - 64;
    // final stage: features f .. f + 3 of the tokens first, first + step, ... of this CTA's share
    const int f = f0 + (et & 31) * 4, first = slice + ksplit * (et >> 5), step = ksplit * (kEpiThreads / 32);
    const bool f_ok = f < F;
    // Eight 16-byte reads of the CTAs' sums are in flight per thread: those of 4 tokens from 2 CTAs, or of 2
    // tokens from 4 CTAs at a time.
    const int batch = ksplit <= 2 ? 4 : 2;
    uint2 e[4];
    auto request = [&](int t0) {      // table-row pieces of the next tokens
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = t0 + i * step;
        if (KIND == kEpiGate && f_ok && i < batch && t < T)
          e[i] = __ldg(reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(ep.E) + static_cast<size_t>(s_ids[t]) * F + f));
      }
    };
    if (KIND == kEpiGate) {
      if (et < T) {
        int id = ep.ids != nullptr ? ep.ids[et] : et;
        if (id < 0 || id >= ep.V) {
          report_error(ep.status, STEM_ERR_ID_RANGE, et);
          id = id < 0 ? 0 : ep.V - 1;
        }
        s_ids[et] = id;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
      request(first);
    }
    bool mine = ptx::mbar_wait_bounded(done_bar, 0, abort_flag, kWaitLimitCycles);
    mine = __all_sync(0xffffffffu, mine);
    if (!mine) {
      if (lane == 0) { report_error(ep.status, STEM_ERR_TIMEOUT, 4); *abort_flag = 1; }
      ok = false;
    } else {
      // Every copy of this CTA has landed and every MMA on it is complete: the operand ring is free for
      // the sums, token by token (128 features of a token side by side).
      ptx::tc_fence_after();
      const int q = warp & 3, half = (warp - 2) >> 2;
      float* part = reinterpret_cast<float*>(base_ptr) + q * 32 + lane;
      for (int c = half * 16; c < n_pad; c += 32) {
        uint32_t v[16];
        ptx::tmem_ld_32x16(tmem_base + c + (static_cast<uint32_t>(q * 32) << 16), v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) part[(c + i) * BM] = __uint_as_float(v[i]);
      }
      ptx::tc_fence_before();
    }
    __syncwarp();
    // Every epilogue thread of the cluster meets here, also after a timeout (the other warps: below).
    if (clustered) ptx::cluster_sync(); else asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
    if (ok && f_ok) {
      const uint32_t sums = base + 16u * (et & 31);
      // (Rolled up on purpose: this runs once, and a body unrolled over the tokens took 8300 cycles to fetch.)
      auto finish = [&](auto tokens, auto ctas) {
        constexpr int TB = decltype(tokens)::value, KB = decltype(ctas)::value;
#pragma unroll 1
        for (int t0 = first; t0 < T; t0 += TB * step) {
          uint2 cur[TB];
          float a[TB][4];
#pragma unroll
          for (int i = 0; i < TB; ++i) { cur[i] = e[i]; a[i][0] = a[i][1] = a[i][2] = a[i][3] = 0.0f; }
          if (t0 + TB * step < T) request(t0 + TB * step);
#pragma unroll 1
          for (int k0 = 0; k0 < ksplit; k0 += KB) {
            float p[KB][TB][4];
#pragma unroll
            for (int k = 0; k < KB; ++k) {
              const uint32_t src = sums + 4u * BM * t0;
              const uint32_t at = clustered ? ptx::mapa(src, min(k0 + k, ksplit - 1) * CTAS + rank) : src;
#pragma unroll
              for (int i = 0; i < TB; ++i) {
                p[k][i][0] = p[k][i][1] = p[k][i][2] = p[k][i][3] = 0.0f;
                if (k0 + k < ksplit && t0 + i * step < T) ptx::ld_shared_cluster_f32x4(at + 4u * BM * i * step, p[k][i]);
              }
            }
#pragma unroll
            for (int k = 0; k < KB; ++k)
#pragma unroll
              for (int i = 0; i < TB; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) a[i][j] += p[k][i][j];
          }
#pragma unroll
          for (int i = 0; i < TB; ++i) {
            const int t = t0 + i * step;
            if (t < T) {
              const size_t o = static_cast<size_t>(t) * F + f;
              const uint2 acc = make_uint2(pack_bf16(a[i][0], a[i][1]), pack_bf16(a[i][2], a[i][3]));
              if (KIND == kEpiGate) {
                const float u[4] = {__uint_as_float(cur[i].x << 16), __uint_as_float(cur[i].x & 0xFFFF0000u),
                                    __uint_as_float(cur[i].y << 16), __uint_as_float(cur[i].y & 0xFFFF0000u)};
                float h[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) h[j] = a[i][j] * fast_sigmoid(a[i][j]) * u[j];
                *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(ep.H) + o) =
                    make_uint2(pack_bf16(h[0], h[1]), pack_bf16(h[2], h[3]));
                if (ep.G) *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(ep.G) + o) = acc;
              } else {
                *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(ep.out) + o) = acc;
              }
            }
          }
        }
      };
      if (batch == 4) finish(Int<4>{}, Int<2>{}); else finish(Int<2>{}, Int<4>{});
    }
    __syncwarp();
  }

  if (clustered && warp < 2) { __syncwarp(); ptx::cluster_sync(); }   // (the epilogue warps': above)
  __syncthreads();
  if (*abort_flag != 0 && threadIdx.x == 0) {
    // wait (bounded) for copies still in flight; the second CTA of a pair cannot poll the barriers
    // its bytes are counted on and waits out a fixed interval (far longer than a copy takes)
    int zero = 0;
    if (rank == 0) {
      for (int j = issued > stages ? issued - stages : 0; j < issued; ++j)
        ptx::mbar_wait_bounded(full_bar(j % stages), (j / stages) & 1, &zero, kWaitLimitCycles / 16);
    } else {
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000ll) { }
    }
  }
  // No CTA of a cluster leaves (or frees TMEM) while another can still signal its barriers, read its
  // shared memory or write its accumulators.
  if (clustered) ptx::cluster_sync(); else __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    if (CTAS == 2) ptx::tmem_dealloc_pair(tmem_base, tmem_cols); else ptx::tmem_dealloc(tmem_base, tmem_cols);
  }
}

// Row-major bf16 [rows, cols]; box = 64 columns x box_rows rows, 128-byte swizzle.
bool encode_operand(CUtensorMap* map, const void* ptr, int rows, int cols, int box_rows) {
  const auto fn = reinterpret_cast<CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                                CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                                CUtensorMapFloatOOBfill)>(tensor_map_encode_fn());
  if (!fn) return false;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(cols) * 2};
  const cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shared memory of a CTA: batches of up to 128 rows leave room for a second CTA on the SM.  (With all of it
// a forward pass of 128 rows took 38.8 us against 33.3: two rounds of clusters of 8.)
constexpr int kMaxSmem = 232448;
int smem_budget(int n_pad) { return n_pad <= 128 ? 113 * 1024 : kMaxSmem; }

// Single CTAs or pairs, and CTAs along k.  What a CTA must load sets the pace: its k range times 128 rows
// of W and its rows of X (half of the batch in a pair), times the rounds its clusters take.  Narrow
// batches get no more CTAs than there are SMs, though two fit one: the second place is a cluster's that
// finds its GPC full (twice the CTAs at half the k range measured the same at 16 rows and 10 % slower at 128).
// (The MMA's N is a multiple of 16, in a pair of 32.)
struct Plan { int ctas, ksplit, n_pad; long long rows; };
Plan make_plan(int T, int F, int K) {
  const int k_blocks = (K + BK - 1) / BK, slots = device_sm_count();
  Plan best{1, 1, 0, 0};
  for (int ctas = 1; ctas <= 2; ++ctas) {
    const int tiles = (F + BM * ctas - 1) / (BM * ctas), n_pad = (T + 16 * ctas - 1) / (16 * ctas) * (16 * ctas);
    for (int sp = 1; sp * ctas <= 8; ++sp) {
      if (sp > 1 && (k_blocks < 2 * sp || static_cast<long long>(tiles) * ctas * sp > slots)) break;
      const int at_once = n_pad <= 128 ? slots / (ctas * sp) : clusters_at_once(ctas * sp);
      const long long rounds = (tiles + at_once - 1) / at_once;
      const long long rows = rounds * ((k_blocks + sp - 1) / sp) * (BM + n_pad / ctas);
      if (best.rows == 0 || rows < best.rows) best = {ctas, sp, n_pad, rows};
    }
  }
  return best;
}

template <int KIND, int CTAS>
cudaError_t launch_inst(const void* X, const void* W, int T, int F, int K, const Plan& pl, const EpiParams& ep,
                        cudaStream_t stream) {
  const int n_pad = pl.n_pad, ksplit = pl.ksplit;
  auto kern = stream_gemm_kernel<KIND, CTAS>;
  static PerDeviceOnce configured;
  if (cudaError_t ce = configured.run([&] {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
      }))
    return ce;
  CUtensorMap tmW, tmX;
  if (!encode_operand(&tmW, W, F, K, BM) || !encode_operand(&tmX, X, T, K, n_pad / CTAS)) return cudaErrorNotSupported;
  const int k_blocks = (K + BK - 1) / BK, my_blocks = (k_blocks + ksplit - 1) / ksplit;
  const int stage_bytes = kWBytes + n_pad / CTAS * BK * 2;
  const int budget = smem_budget(n_pad) - kTailBytes - 1024;
  int stages = budget / stage_bytes;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages > my_blocks) stages = my_blocks;
  int ring = stages * stage_bytes;
  if (ring < n_pad * BM * 4) ring = n_pad * BM * 4;    // the sums take the ring's place
  int tmem_cols = 32;
  while (tmem_cols < n_pad) tmem_cols *= 2;
  const int tiles = (F + BM * CTAS - 1) / (BM * CTAS);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles * CTAS * ksplit));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = ring + kTailBytes + 1024;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(CTAS * ksplit);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CTAS * ksplit > 1 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tmW, tmX, T, F, K, n_pad, stages, ksplit, tmem_cols, ep);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Clusters of `size` CTAs that run at once with one CTA per SM (an SM left over in a GPC is no help to a
// cluster that needs more of them: 15 clusters of 8, not 18).  Asked once per device and size.
int clusters_at_once(int size) {
  static int cached[64][9] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return device_sm_count() / size;
  if (cached[dev][size] == 0) {
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(device_sm_count() / size * size));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kMaxSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(size);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto kern = stream_gemm_kernel<kEpiStore, 1>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = device_sm_count() / size;
    }
    cached[dev][size] = n;
  }
  return cached[dev][size];
}

cudaError_t launch_stream_gemm(int T, int F, int K, const void* X, const void* W, EpiKind kind, const EpiParams& ep,
                               cudaStream_t stream) {
  if (T <= 0 || F <= 0) return cudaSuccess;
  if (T > kMaxT || K <= 0 || (F % 8) || (K % 8) || (kind != kEpiGate && kind != kEpiStore) ||
      (kind == kEpiStore && (ep.out_fp32 || ep.accumulate)))
    return cudaErrorNotSupported;
  const Plan pl = make_plan(T, F, K);
  if (kind == kEpiGate) {
    if (pl.ctas == 2) return launch_inst<kEpiGate, 2>(X, W, T, F, K, pl, ep, stream);
    return launch_inst<kEpiGate, 1>(X, W, T, F, K, pl, ep, stream);
  }
  if (pl.ctas == 2) return launch_inst<kEpiStore, 2>(X, W, T, F, K, pl, ep, stream);
  return launch_inst<kEpiStore, 1>(X, W, T, F, K, pl, ep, stream);
}

// Above 128 rows a CTA has no room for a second one beside it and the exchange (fp32 sums of the whole batch)
// grows, so the lines depend on how much W there is to stream.  Measured, a forward pass with both kernels general /
// with both so / with only the second so, weights in L2, replayed from a graph, us at 144, 192, 256 rows:
//   2048 x 8192   29.9 / 23.7 / 25.9   31.2 / 25.2 / 26.9   32.1 / 31.0 / 31.7
//   1800 x 6000   27.8 / 22.2 / 24.4   28.6 / 24.2 / 25.8   30.0 / 27.8 / 28.1
//   1536 x 5000   25.4 / 20.0 / 22.3   25.6 / 22.2 / 23.9   26.8 / 25.8 / 26.3
//   1280 x 4096   29.1 / 17.1 / 18.6   29.2 / 18.9 / 19.7   30.1 / 21.8 / 21.5
//   2048 x 2048   24.2 / 16.5 / 20.2   24.5 / 17.2 / 20.4   25.1 / 19.8 / 22.4
//   1024 x 4096   27.9 / 16.6 / 17.3   28.1 / 18.0 / 18.4   28.7 / 20.6 / 20.0
//   1024 x 2816   23.1 / 19.1 / 16.7   23.3 / 17.3 / 17.6   23.9 / 19.6 / 19.2
//    768 x 2048   19.1 / 15.0 / 15.1   19.2 / 19.8 / 16.1   19.9 / 19.5 / 17.5
// The first kernel goes general where this form of it loses (K up to 1280 at 256 rows, 2.9 M weights at 144); between
// 193 and 256 rows the line at 10 M weights also leaves it general where this form would be up to 2.6 us faster (K of
// 1536 and 2048 with fewer weights).  The second one (a plain store) takes this form for a short k range per CTA too: up
// to 3000 rows of operands, 6 blocks x 384 at 1024 x 2816.
bool stream_gemm_pays(int T, int F, int K, EpiKind kind) {
  const long long weights = static_cast<long long>(F) * K;
  if (T <= 128 || (T <= 192 && weights >= 4000000) || (T <= kMaxT && weights >= 10000000)) return true;
  return kind == kEpiStore && T <= kMaxT && make_plan(T, F, K).rows <= 3000;
}

}  // namespace stem
