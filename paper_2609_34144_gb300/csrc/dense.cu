// Dense projections of the residual sites beyond the attention output (App. B.1, B.4): the
// output projection W_O of the anchor rows and the two GEMMs of the anchor FFN, as one
// persistent tcgen05 kernel per GEMM over the rows of every anchor.
//
//   C[anchor i, row r, :] = act(A[a_frame[i], r, :] W^T + bias),  r < S,
//
// bf16 A and W (K contiguous), f32 accumulation in TMEM, bias (+ GELU, tanh form) in the
// epilogue, C in bf16 or f32.
//
// Two SMs work on one tile of 256 rows x BN columns (BN = 256 or 128): CTA pairs
// (cta_group::2), persistent, one CTA per SM.  Each CTA loads its own 128 rows of A and half of
// the tile's rows of W, and the pair's UMMAs (M = 256) read both halves: 32 KB per 64-wide k-step
// and SM at BN = 256, where a CTA on its own needs 48 KB for the same work.  A 128 x 256 tile per
// CTA was bound by that stream: 48 KB took ~1,000 cycles of an SM against 544 of UMMAs.
// The two 128-row halves of a tile are independent row tiles (any anchor each), so that nothing
// is padded to 256 rows; where the rows of all anchors lie one after another (activations in the
// workspace) they are tiled as one run of rows.  Rows past the end read as zero through the
// tensor map [frame][row][k] and are not written.
// Warp roles (384 threads, one CTA per SM):
//   warp 0      TMA producer: A (128 x 64) and W (BN / 2 x 64) k-slices into a 6-stage ring; both
//               CTAs' copies complete on the leader's barrier
//   warp 1      TMEM owner; in the leader also the UMMA issuer (converged, one elected lane),
//               accumulating each tile in one of two 256-column TMEM buffers
//   warps 4..11 epilogue: one output row per thread and half of the tile's columns per warp
//               (warps 4-7 the first half, warps 8-11 the second), tcgen05.ld of 32 columns at a
//               time, bias (vector loads issued before the TMEM load), GELU, conversion and
//               vector stores; the buffer is handed back to the issuer, so the next tile's
//               mainloop overlaps this tile's epilogue.
// Every wait is bounded; on a timeout a CTA records an error word and leaves its loops; the
// cluster barrier at the end keeps both CTAs' shared memory until nothing is in flight.
#include <cuda_bf16.h>

#include "dense_plan.h"
#include "internal.h"
#include "ptx.cuh"

namespace cast {
namespace {

__device__ unsigned int g_dense_error;

constexpr int GBM = 128, GBK = 64, kGStages = 6, kMaxBN = 256;
constexpr int kGThreads = 384;
constexpr int kEpiWarps = 8;
constexpr int kABytes = GBM * GBK * 2;                                // own rows of A
constexpr int kStageBytes = kABytes + (kMaxBN / 2) * GBK * 2;         // ... and half the tile's rows of W
constexpr int kEpiStage = 32 * 128;                                   // 128 bytes of 32 rows per epilogue warp
constexpr int kGBarOff = kGStages * kStageBytes + kEpiWarps * kEpiStage;
constexpr int kGSmem = kGBarOff + 256 + 1024;                         // + barriers + alignment slack

struct GemmKArgs {
  int S, N, n_k, bn;      // rows per anchor, output columns, k-steps, columns per tile
  int seg_rows, seg_tiles, n_half;   // rows and 128-row tiles of one run of A rows; tiles in all
  int n_col, n_items;     // column tiles; pairs of row tiles x column tiles
  const void* bias;
  void* c;
  int64_t ldc;
  int c_f32, bias_f32, gelu;
  unsigned long long wait_ns;
  int a_frame[CAST_MAX_ANCHORS];   // frame of A of each run
  int c_frame[CAST_MAX_ANCHORS];   // frame of C of each anchor
};

struct GBars {
  uint64_t full[kGStages], empty[kGStages];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t fin;
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ bool g_aborted(const GBars* b) {
  return *reinterpret_cast<const volatile int*>(&b->abort) != 0;
}
__device__ __forceinline__ void g_set_abort(GBars* b) {
  atomicExch(&b->abort, 1);
  atomicExch(&g_dense_error, 1u);
}
// GELU in its tanh form, 0.5 x (1 + tanh(sqrt(2/pi) (x + 0.044715 x^3))), with the hardware
// tanh approximation
__device__ __forceinline__ float gelu_tanh(float x) {
  const float u = 0.7978845608028654f * fmaf(0.044715f * x, x * x, x);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  return 0.5f * x * (1.f + t);
}

// Item t -> row tile q of this CTA (2 rp + rank) as (run, first row), and column tile; column
// tiles innermost.  A row tile past the last starts past the run's rows: it reads zeros and
// writes nothing.
struct GTile {
  int seg, row0, n0;
};
__device__ __forceinline__ GTile tile_of(const GemmKArgs& a, int t, int rank) {
  GTile g;
  const int rp = t / a.n_col;
  g.n0 = (t - rp * a.n_col) * a.bn;
  const int q = 2 * rp + rank;
  g.seg = q < a.n_half ? q / a.seg_tiles : 0;
  g.row0 = q < a.n_half ? (q - g.seg * a.seg_tiles) * GBM : a.seg_tiles * GBM;
  return g;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGThreads, 1)
    k_gemm(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w,
           const __grid_constant__ GemmKArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  GBars* bars = reinterpret_cast<GBars*>(smem + kGBarOff);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t lim = a.wait_ns;
  const int rank = (int)cluster_ctarank();
  const int first = blockIdx.x >> 1, stride = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kGStages; ++s) {
      mbar_init(&bars->full[s], 1);    // the leader's: its expected bytes cover both CTAs' copies
      mbar_init(&bars->empty[s], 1);   // released by the UMMA issuer in both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->acc_full[b], 1);
      mbar_init(&bars->acc_empty[b], 2 * kEpiWarps);   // the leader's: both CTAs' epilogue warps
    }
    mbar_init(&bars->fin, 1);
    bars->abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&bars->tmem_base, 512);
    tmem_relinquish_pair();
    tc_fence_before();
  }
  __syncthreads();
  cluster_barrier();   // the peer's barriers exist before anything signals them
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  // A comes from the kernel before when this one is its programmatic dependent (a no-op for an
  // ordinary launch); this kernel's own dependent may take SMs as they become free
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------------------------------------ TMA producer
      tma_prefetch_desc(&tm_a);
      tma_prefetch_desc(&tm_w);
      const int half_n = a.bn / 2;
      const uint32_t pair_bytes = 2u * (uint32_t)(kABytes + half_n * GBK * 2);
      int it = 0;
      bool ok = true;
      for (int t = first; ok && t < a.n_items; t += stride) {
        const GTile g = tile_of(a, t, rank);
        const int frame = a.a_frame[g.seg];
        for (int ks = 0; ks < a.n_k; ++ks, ++it) {
          const int s = it % kGStages;
          // the UMMAs that read this stage (in both CTAs) have completed
          if (g_aborted(bars) || !mbar_wait(&bars->empty[s], ((uint32_t)(it / kGStages) & 1u) ^ 1u, lim)) {
            g_set_abort(bars);
            ok = false;
            break;
          }
          uint8_t* st = smem + s * kStageBytes;
          if (rank == 0) mbar_arrive_expect_tx(&bars->full[s], pair_bytes);
          const uint32_t bar = cluster_addr(&bars->full[s], 0);
          tma_load_3d_pair(st, &tm_a, bar, ks * GBK, g.row0, frame);
          tma_load_2d_pair(st + kABytes, &tm_w, bar, ks * GBK, g.n0 + rank * half_n);
        }
      }
      if (rank == 0)   // (whatever ended the loop) the last copies have landed before shared memory is released
        for (int l = it > kGStages ? it - kGStages : 0; l < it; ++l)
          mbar_wait(&bars->full[l % kGStages], (uint32_t)(l / kGStages) & 1u, lim);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------------------ UMMA issuer
      // (converged warp and uniform operands: see the attention kernel)
      const uint32_t idesc = idesc_bf16_f32(2 * GBM, a.bn, false, false);
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      const uint32_t base = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
      const uint64_t d0 = sdesc_sw128(base, 16, 1024);
      const bool lead = elect_one();
      auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity, lim));
      };
      int s = 0, lt = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = first; ok && t < a.n_items; t += stride, ++lt) {
        const int buf = lt & 1;
        if (g_aborted(bars) || !wait(&bars->acc_empty[buf], ((uint32_t)(lt >> 1) & 1u) ^ 1u)) {
          ok = false;
          break;
        }
        tc_fence_after();
        for (int ks = 0; ks < a.n_k; ++ks) {
          if (!wait(&bars->full[s], ph)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (lead) {
            const uint64_t da = d0 + (uint64_t)(s * (kStageBytes >> 4));
#pragma unroll
            for (int kk = 0; kk < GBK / 16; ++kk)
              umma_bf16_ss_pair(tm + buf * kMaxBN, da + (uint64_t)(kk * 2), da + (uint64_t)((kABytes >> 4) + kk * 2),
                                idesc, (ks > 0 || kk > 0) ? 1u : 0u);
            umma_commit_pair(&bars->empty[s]);   // the stage is free once these UMMAs have read it
          }
          __syncwarp();
          if (++s == kGStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        if (lead) umma_commit_pair(&bars->acc_full[buf]);
        __syncwarp();
      }
      if (!ok && lane == 0) g_set_abort(bars);
      // every issued UMMA has completed before TMEM and the peer's shared memory are released
      if (lead) umma_commit_pair(&bars->fin);
      __syncwarp();
    }
    // (the peer waits as well: after this no commit can still signal its barriers)
    mbar_wait(&bars->fin, 0, lim);
    __syncwarp();
  } else if (warp >= 4) {
    // ------------------------------------------------------------ epilogue
    const int q4 = warp & 3, half = (warp - 4) >> 2;
    const int row = q4 * 32 + lane;
    uint8_t* stage = smem + kGStages * kStageBytes + (warp - 4) * kEpiStage;
    int lt = 0;
    for (int t = first; t < a.n_items; t += stride, ++lt) {
      const int buf = lt & 1;
      const bool w = !g_aborted(bars) && mbar_wait(&bars->acc_full[buf], (uint32_t)(lt >> 1) & 1u, lim);
      if (!__all_sync(0xffffffffu, w)) {
        g_set_abort(bars);
        break;
      }
      tc_fence_after();
      const GTile g = tile_of(a, t, rank);
      const bool live = g.row0 + row < a.seg_rows;
      // row of all anchors -> (anchor, row of its frame)
      const int R = g.seg * a.seg_rows + g.row0 + row;
      const int anchor = live ? R / a.S : 0;
      const uint32_t tl = tmem + buf * kMaxBN + ((uint32_t)(q4 * 32) << 16);
      const int64_t crow = live ? ((int64_t)a.c_frame[anchor] * a.S + (R - anchor * a.S)) * a.ldc : -1;
      // 128 bytes of every row at a time (64 bf16 or 32 f32 columns): formed row by row, staged in
      // shared memory and stored by eight lanes per row, so that a store writes whole lines (row
      // by row, a 16-byte store of the warp touched 32 lines: the first GEMM of the
      // Matrix-Game-shaped FFN took 93 us with that, 77 us with whole lines)
      const int step = a.c_f32 ? 32 : 64, n_steps = a.bn / 2 / step;
#pragma unroll 1
      for (int cs = 0; cs < n_steps; ++cs) {
        const int col = half * (a.bn / 2) + cs * step;   // first column within the tile
#pragma unroll
        for (int sub = 0; sub < 2; ++sub) {
          if (sub * 32 >= step) break;
          const int n0 = g.n0 + col + sub * 32;
          // bias of the 32 columns (the same for every row): vector loads in flight before the
          // TMEM load
          float bv[32];
          if (a.bias && n0 + 32 <= a.N) {
            if (a.bias_f32) {
              const float4* bp = reinterpret_cast<const float4*>(static_cast<const float*>(a.bias) + n0);
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const float4 v4 = __ldg(bp + q);
                bv[4 * q] = v4.x; bv[4 * q + 1] = v4.y; bv[4 * q + 2] = v4.z; bv[4 * q + 3] = v4.w;
              }
            } else {
              const uint4* bp = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(a.bias) + n0);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint4 u4 = __ldg(bp + q);
                const uint32_t wds[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  bv[8 * q + 2 * e] = __uint_as_float(wds[e] << 16);
                  bv[8 * q + 2 * e + 1] = __uint_as_float(wds[e] & 0xFFFF0000u);
                }
              }
            }
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c) {
              const int n = n0 + c;
              bv[c] = 0.f;
              if (a.bias && n < a.N)
                bv[c] = a.bias_f32 ? __ldg(static_cast<const float*>(a.bias) + n)
                                   : __bfloat162float(__ldg(static_cast<const __nv_bfloat16*>(a.bias) + n));
            }
          }
          uint32_t v[32];
          tmem_ld_x32(tl + col + sub * 32, v);   // warp-collective: every lane loads
          if (cs == n_steps - 1 && (sub + 1) * 32 >= step) {
            // the accumulator buffer is free for the tile after next
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(&bars->acc_empty[buf], 0));
          }
          float y[32];
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const float x = __uint_as_float(v[c]) + bv[c];
            y[c] = a.gelu ? gelu_tanh(x) : x;
          }
          // 16-byte piece p of the row at slot p ^ (row & 7): conflict-free both ways
          if (a.c_f32) {
#pragma unroll
            for (int p = 0; p < 8; ++p)
              *reinterpret_cast<float4*>(stage + lane * 128 + ((p ^ (lane & 7)) << 4)) =
                  make_float4(y[4 * p], y[4 * p + 1], y[4 * p + 2], y[4 * p + 3]);
          } else {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              uint32_t pk[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                __nv_bfloat162 b2 = __floats2bfloat162_rn(y[8 * p + 2 * e], y[8 * p + 2 * e + 1]);
                pk[e] = *reinterpret_cast<uint32_t*>(&b2);
              }
              *reinterpret_cast<uint4*>(stage + lane * 128 + (((sub * 4 + p) ^ (lane & 7)) << 4)) =
                  make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
        }
        __syncwarp();
        const int piece = lane & 7, elts = a.c_f32 ? 4 : 8;   // this lane's 16 bytes of each row
        const int n = g.n0 + col + piece * elts;
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += 4) {
          const int r = r0 + (lane >> 3);
          const uint4 w4 = *reinterpret_cast<const uint4*>(stage + r * 128 + ((piece ^ (r & 7)) << 4));
          const int64_t at = __shfl_sync(0xffffffffu, crow, r);
          // N is a multiple of 8, so a 16-byte piece lies inside the row or past its end
          if (at >= 0 && n < a.N)
            *reinterpret_cast<uint4*>(static_cast<char*>(a.c) + (at + n) * (a.c_f32 ? 4 : 2)) = w4;
        }
        __syncwarp();
      }
    }
  }
  // the last UMMA has completed (fin), every epilogue thread of both CTAs has read its TMEM and
  // no signal to the other CTA is outstanding
  tc_fence_before();
  cluster_barrier();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
  cluster_barrier();
}

// bf16 [depth][rows][inner] (rank 2 when depth == 0), box 64 x box_rows (x 1), 128-B swizzle
bool make_gemm_map(CUtensorMap* m, const void* base, uint64_t inner, uint64_t rows,
                   uint64_t row_stride_bytes, uint64_t depth, uint64_t depth_stride_bytes,
                   uint32_t box_rows) {
  EncodeTiledFn fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[3] = {inner, rows, depth};
  cuuint64_t strides[2] = {row_stride_bytes, depth_stride_bytes};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, depth ? 3 : 2, const_cast<void*>(base), dims, strides,
            box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cast_status gemm_anchor_rows(const AnchorGemm& g, cudaStream_t st) {
  if (g.n_anchors < 1 || g.S < 1 || g.N < 1 || g.K < 1) return CAST_OK;
  const int nsm = sm_count();
  const int pairs = nsm > 1 ? nsm / 2 : 1;
  GemmKArgs k{};
  k.S = g.S;
  k.N = g.N;
  k.n_k = (g.K + GBK - 1) / GBK;
  // rows of every anchor one after another: one run of rows
  bool run = g.a_frame_stride == (int64_t)g.S * g.lda;
  for (int j = 1; j < g.n_anchors; ++j) run = run && g.a_frame[j] == g.a_frame[j - 1] + 1;
  const int n_seg = run ? 1 : g.n_anchors;
  k.seg_rows = run ? g.n_anchors * g.S : g.S;
  k.seg_tiles = (k.seg_rows + GBM - 1) / GBM;
  k.n_half = n_seg * k.seg_tiles;
  const int row_pairs = (k.n_half + 1) / 2;
  k.bn = tile_columns(row_pairs, g.N, k.n_k, pairs);
  k.n_col = (g.N + k.bn - 1) / k.bn;
  k.n_items = row_pairs * k.n_col;
  CUtensorMap ma, mw;
  const char* abase = static_cast<const char*>(g.a) + (run ? (int64_t)g.a_frame[0] * g.a_frame_stride * 2 : 0);
  if (!make_gemm_map(&ma, abase, (uint64_t)g.K, (uint64_t)k.seg_rows, (uint64_t)g.lda * 2,
                     run ? 1 : (uint64_t)g.a_frames, (uint64_t)(run ? k.seg_rows * g.lda : g.a_frame_stride) * 2, GBM) ||
      !make_gemm_map(&mw, g.w, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.ldw * 2, 0, 0, (uint32_t)k.bn / 2))
    return fail(CAST_ERR_CUDA, "dense: cuTensorMapEncodeTiled failed");
  k.bias = g.bias;
  k.c = g.c;
  k.ldc = g.ldc;
  k.c_f32 = g.c_dtype == CAST_F32;
  k.bias_f32 = g.bias_dtype == CAST_F32;
  k.gelu = g.gelu ? 1 : 0;
  k.wait_ns = 2000000000ull;
  for (int j = 0; j < g.n_anchors; ++j) {
    k.a_frame[j] = run ? 0 : g.a_frame[j];
    k.c_frame[j] = g.c_frame[j];
  }
  static std::atomic<uint64_t> attr_done{0};
  if (!once_per_device(attr_done, [] {
        return cudaFuncSetAttribute(k_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem) ==
               cudaSuccess;
      }))
    return check_launch("dense GEMM smem attribute");
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * (k.n_items < pairs ? k.n_items : pairs), 1, 1);
  cfg.blockDim = dim3(kGThreads, 1, 1);
  cfg.dynamicSmemBytes = kGSmem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g.dependent ? 1 : 0;
  if (cudaLaunchKernelEx(&cfg, k_gemm, ma, mw, k) != cudaSuccess) return check_launch("dense GEMM kernel");
  return check_launch("dense GEMM kernel");
}

unsigned int dense_error_word(cudaStream_t st, bool clear) {
  unsigned int v = 0;
  cudaMemcpyFromSymbolAsync(&v, g_dense_error, sizeof(v), 0, cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  if (clear && v) {
    const unsigned int z = 0;
    cudaMemcpyToSymbolAsync(g_dense_error, &z, sizeof(z), 0, cudaMemcpyHostToDevice, st);
    cudaStreamSynchronize(st);
  }
  return v;
}

}  // namespace cast
