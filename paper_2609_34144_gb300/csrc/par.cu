// Phase-Aware Reconstruction of skipped frames (Section 4.3, Eqs. cross, confidence, gate,
// fcpasm; App. A.2).  On every tile: the anchors' spectra, the channel-pooled
//   Z = sum_c w_c F_b conj(F_a),  W = sum_c w_c |F_b||F_a|
// of each anchor pair, from them reliability, phases theta, confidence and gate g (the transport),
// and R_t = IRFFT2((1-alpha) F_a e^{i g alpha theta} + alpha F_b e^{-i g (1-alpha) theta}).
//
// bf16 residuals: two launches over every tile, on the tensor cores.
//   K_stats_tc (tile, pair, chunk range): the transforms as one GEMM with the tile's DFT matrix per
//       128-channel chunk, Z and W summed over channels into one record in the workspace.
//   K_blend_tc (tile, targets of a pair, chunk range): the transport from the records, then the
//       blend: on one tile, Eq. (fcpasm) is exactly two circular convolutions,
//         R_t = h_a (*) R_a + h_b (*) R_b,  h = IDFT2 of the Hermitian-extended phasors
//         phi_a = (1-alpha) e^{i g alpha theta}, phi_b = alpha e^{-i g (1-alpha) theta},
//       so one UMMA chain per pair of targets computes [H_t1 ; H_t2] [X_a ; X_b] for 128 channels.
//   Measured (GB300, 16 frames of 44x80 x 3072, 5 anchors): 160 -> 107 us against three launches
//   per tile kind (register transforms, a transport that wrote the matrices, a blend that loaded
//   them for every tile and chunk; edge tiles on a second stream).
//
// f32 residuals: three passes per tile kind (full 8x8 tiles / truncated edge tiles).
//   K_stats (tile, channel chunk): one thread per channel streams the anchors of the tile in
//       time order through a TMA 4-D map ([frame][row][col][channel], out-of-range rows/cols/
//       channels arrive as zeros), forms each tile spectrum in registers (the previous anchor's
//       spectrum stays in shared memory) and, for every anchor pair with targets, reduces Z and W
//       over the chunk's channels (warp transpose reductions) into one record in the workspace.
//   K_transport (tile, pair): sums the records of the tile's channel chunks in chunk order
//       (deterministic) and writes theta and g.
//   K_blend (tile, channel chunk): streams the anchors again (an L2 hit at these sizes), forms
//       their spectra and writes every target straight from registers.
// The passes are chained as programmatic dependents (the transport releases the blend at its
// end), the full-tile chain on the caller's stream and the edge-tile chain on a side stream.
//
// The CTAs of a pass never wait on each other, so the passes fill the GPU whatever the number
// of anchor pairs.  Global traffic beyond the algorithmic bytes: a second read of the anchors
// (bf16: of each anchor once per pair and pass, from L2) and the records.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "dft.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace cast {
namespace {

constexpr int kCC = 128;           // channels per CTA (one thread each)
constexpr int kNB = 40;            // stored bins of an 8-wide tile: 8 x 5
constexpr int kNV = 3 * kNB;       // (Re Z, Im Z, W) per bin, record index = 3 * bin + component
constexpr int kRec = kNV;          // record slots per chunk (96 + 1 used for 8x8 tiles)
constexpr int kCoefBatch = 4;

__device__ unsigned int g_par_error;   // 1: a wait gave up

// Non-redundant (bin, component) values of an 8x8 tile's Z / W record, encoded bin * 4 +
// component (0: Re Z, 1: Im Z, 2: W): mirrors (ky > 4 in the kx = 0 and kx = 4 columns) are
// conjugates of their representatives, the self-conjugate bins have Im Z = 0, and DC needs
// only W (reduced separately).  96 values = three 32-value transpose groups.
__host__ __device__ __forceinline__ constexpr int fast_value(int n) {
  return
      n == 0 ? 4 :
      n == 1 ? 5 :
      n == 2 ? 6 :
      n == 3 ? 8 :
      n == 4 ? 9 :
      n == 5 ? 10 :
      n == 6 ? 12 :
      n == 7 ? 13 :
      n == 8 ? 14 :
      n == 9 ? 16 :
      n == 10 ? 18 :
      n == 11 ? 20 :
      n == 12 ? 21 :
      n == 13 ? 22 :
      n == 14 ? 24 :
      n == 15 ? 25 :
      n == 16 ? 26 :
      n == 17 ? 28 :
      n == 18 ? 29 :
      n == 19 ? 30 :
      n == 20 ? 32 :
      n == 21 ? 33 :
      n == 22 ? 34 :
      n == 23 ? 36 :
      n == 24 ? 37 :
      n == 25 ? 38 :
      n == 26 ? 40 :
      n == 27 ? 41 :
      n == 28 ? 42 :
      n == 29 ? 44 :
      n == 30 ? 45 :
      n == 31 ? 46 :
      n == 32 ? 48 :
      n == 33 ? 49 :
      n == 34 ? 50 :
      n == 35 ? 52 :
      n == 36 ? 53 :
      n == 37 ? 54 :
      n == 38 ? 56 :
      n == 39 ? 57 :
      n == 40 ? 58 :
      n == 41 ? 60 :
      n == 42 ? 61 :
      n == 43 ? 62 :
      n == 44 ? 64 :
      n == 45 ? 65 :
      n == 46 ? 66 :
      n == 47 ? 68 :
      n == 48 ? 69 :
      n == 49 ? 70 :
      n == 50 ? 72 :
      n == 51 ? 73 :
      n == 52 ? 74 :
      n == 53 ? 76 :
      n == 54 ? 77 :
      n == 55 ? 78 :
      n == 56 ? 80 :
      n == 57 ? 82 :
      n == 58 ? 84 :
      n == 59 ? 85 :
      n == 60 ? 86 :
      n == 61 ? 88 :
      n == 62 ? 89 :
      n == 63 ? 90 :
      n == 64 ? 92 :
      n == 65 ? 93 :
      n == 66 ? 94 :
      n == 67 ? 96 :
      n == 68 ? 98 :
      n == 69 ? 104 :
      n == 70 ? 105 :
      n == 71 ? 106 :
      n == 72 ? 108 :
      n == 73 ? 109 :
      n == 74 ? 110 :
      n == 75 ? 112 :
      n == 76 ? 113 :
      n == 77 ? 114 :
      n == 78 ? 124 :
      n == 79 ? 125 :
      n == 80 ? 126 :
      n == 81 ? 128 :
      n == 82 ? 129 :
      n == 83 ? 130 :
      n == 84 ? 132 :
      n == 85 ? 133 :
      n == 86 ? 134 :
      n == 87 ? 144 :
      n == 88 ? 145 :
      n == 89 ? 146 :
      n == 90 ? 148 :
      n == 91 ? 149 :
      n == 92 ? 150 :
      n == 93 ? 152 :
      n == 94 ? 153 :
      n == 95 ? 154 :
      0;
}

// A unit of the bf16 kernels: a tile, a range of its channel chunks and an item (a pair, or a group of
// targets), items innermost, so that a tile's anchors are read from L2 by the CTAs of neighbouring units.
struct Unit {
  int tile, part, item;
};

struct ParKArgs {
  char* r;
  const float* wch;
  float* rec;     // workspace [tile][pair j][chunk][kRec]: each chunk's Z / W record
  float* trans;   // workspace [tile][pair j][2][kNB]: theta and g per bin (f32)
  int F, Hg, Wg, C, n_chunk;             // n_chunk: channel chunks of kCC channels
  int tile_base;                         // global index of tile 0 of this launch's kind
  int th, tw, tiles_x, tiles_y, n_tile, n_tseg;
  int n_anchor;
  int anchor_frame[CAST_MAX_ANCHORS];
  int pair_tbeg[CAST_MAX_ANCHORS + 1];   // targets of pair j (anchors j-1, j) in [tbeg[j], tbeg[j+1])
  int target_frame[CAST_MAX_FRAMES];
  float target_alpha[CAST_MAX_FRAMES];
  // bf16 path (tensor cores)
  int whole_y, whole_x;                  // complete tiles in a column, in a row
  int after_own;                         // the launch before on the stream is one of this library's kernels
  int n_act, n_grp;                      // pairs with targets; groups of up to two targets of a pair
  int st_parts, st_cpp, bl_parts, bl_cpp;   // K_stats_tc / K_blend_tc: channel-chunk ranges and chunks in each
  Unit st_step, bl_step;                 // ... and the CTAs' stride over the units
  // per tile shape (bit 0: last column of tiles, truncated; bit 1: last row): where the stored bin
  // b's sums stand in a record (BinSlot), and the bin of each slot (255: none)
  unsigned char bin_slot[4][40], slot_bin[4][34];
  unsigned char act_pair[CAST_MAX_ANCHORS];
  unsigned char grp_pair[CAST_MAX_FRAMES], grp_nt[CAST_MAX_FRAMES];
  short grp_t0[CAST_MAX_FRAMES];
  int seg_pair0[CAST_MAX_ANCHORS];       // time segment s covers pairs seg_pair0[s] .. seg_pair1[s]
  int seg_pair1[CAST_MAX_ANCHORS];
  float tau_low, tau_high, q, T, eps, eta_rel, eta_abs, band;
  int gate_mode;
  unsigned long long wait_ns;
  // 8x8 tiles: record entry t (3 * bin + component) = sign * reduced value |fast_src[t]| - 1,
  // 0 = not needed (Z at DC) or identically zero (Im Z at self-conjugate bins)
  signed char fast_src[kNV];
};


struct TileGeom {
  int y0, x0, h, w;
};

// Tile i of one kind.  With 8x8 tiles: full tiles (row-major over the full-tile grid) or edge
// tiles (the truncated last column of every tile row, then the truncated last row).  Other
// tile sides: every tile, row-major, in the edge kind.
__device__ __forceinline__ TileGeom tile_geom(const ParKArgs& a, int i, bool full) {
  TileGeom g;
  if (a.th != 8 || a.tw != 8) {
    const int ty = i / a.tiles_x, tx = i - (i / a.tiles_x) * a.tiles_x;
    g.y0 = ty * a.th;
    g.x0 = tx * a.tw;
    g.h = min(a.th, a.Hg - g.y0);
    g.w = min(a.tw, a.Wg - g.x0);
    return g;
  }
  const int fy = a.Hg / 8, fx = a.Wg / 8;   // full tiles per column / row
  int ty, tx;
  if (full) {
    ty = i / fx;
    tx = i - ty * fx;
  } else if (a.Wg % 8 != 0 && i < a.tiles_y) {
    ty = i;
    tx = fx;
  } else {
    ty = fy;
    tx = i - (a.Wg % 8 != 0 ? a.tiles_y : 0);
  }
  g.y0 = ty * 8;
  g.x0 = tx * 8;
  g.h = min(8, a.Hg - g.y0);
  g.w = min(8, a.Wg - g.x0);
  return g;
}

// Warp transpose-reduction of 32 values: lane l returns the warp sum of v[l].
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int off = 16, n = 16; off > 0; off >>= 1, n >>= 1) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i < n) {
        const float send = hi ? v[i] : v[i + n];
        const float keep = hi ? v[i + n] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    }
  }
  return v[0];
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// sin and cos of x = 2 pi k + r with |r| <= pi (Cody-Waite split of 2 pi into two parts),
// then the hardware approximations on the reduced argument.
__device__ __forceinline__ void sincos_reduced(float x, float* s, float* c) {
  const float k = rintf(x * 0.159154943091895336f);
  float r = fmaf(-k, 6.28318548202514648f, x);
  r = fmaf(-k, -1.74845553e-07f, r);
  __sincosf(r, s, c);
}

// Geometry of the stored bins of one tile shape (App. A.2), computed once per CTA: per bin
// b = ky * 5 + kx the representative (mirrors point at their conjugate), the pooling weight
// kappa (0: not stored, DC, or outside the tile), the flags, the gate threshold tau(nu) and
// whether the band cut forces g = 0.
struct BinInfo {
  float tau[kNB], kap[kNB];
  unsigned char rep[kNB], valid[kNB], selfc[kNB], mirror[kNB], cut[kNB];
};

__device__ void bin_info(const ParKArgs& a, const TileGeom& g, BinInfo& bi, int tid) {
  if (tid >= kNB) return;
  const int b = tid, ky = b / 5, kx = b % 5, hw2 = g.w / 2;
  const bool valid = ky < g.h && kx <= hw2;
  const bool edge = kx == 0 || ((g.w % 2 == 0) && kx == hw2);
  const bool selfc = edge && (ky == 0 || ((g.h % 2 == 0) && 2 * ky == g.h));
  const bool mirror = edge && !selfc && 2 * ky > g.h;
  bi.valid[b] = valid;
  bi.selfc[b] = selfc;
  bi.mirror[b] = mirror;
  bi.rep[b] = (unsigned char)(mirror ? (g.h - ky) * 5 + kx : b);
  bi.kap[b] = (valid && b != 0) ? (edge ? 1.f : 2.f) : 0.f;
  const int kys = ky <= (g.h - 1) / 2 ? ky : ky - g.h;
  const float hh = (float)(g.h / 2) / (float)g.h, ww = (float)hw2 / (float)g.w;
  const float rmax = sqrtf(hh * hh + ww * ww);
  const float fy = (float)kys / (float)g.h, fx = (float)kx / (float)g.w;
  const float nu = rmax > 0.f ? sqrtf(fy * fy + fx * fx) / rmax : 0.f;
  bi.tau[b] = a.tau_low + (a.tau_high - a.tau_low) * powf(nu, a.q);
  bool cut = false;
  if (a.band >= 0.f) {
    const float ry = (float)kys * 8.f / (float)g.h, rx = (float)kx * 8.f / (float)g.w;
    cut = sqrtf(ry * ry + rx * rx) > a.band;
  }
  bi.cut[b] = cut;
}

// Per-tile transport of one anchor pair (one warp): theta and g of the stored bins lane and
// lane + 32 from the pooled Z, W record (App. A.2).
__device__ void tile_transport(const ParKArgs& a, const TileGeom& g, const BinInfo& bi,
                               const float* zw, float (&th)[2], float (&gate)[2], float* own_th,
                               int* own_rel, int lane) {
  const float inv_hw = 1.f / (float)(g.h * g.w);
  float Zr[2], Zi[2], Wv[2], Za[2], t[2];
  float wmax = 0.f;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int b = lane + 32 * s;
    const bool v = b < kNB && bi.valid[b];
    Zr[s] = v ? zw[3 * b] * inv_hw : 0.f;
    Zi[s] = v ? zw[3 * b + 1] * inv_hw : 0.f;
    Wv[s] = v ? zw[3 * b + 2] * inv_hw : 0.f;
    Za[s] = sqrt_approx(Zr[s] * Zr[s] + Zi[s] * Zi[s]);
    t[s] = atan2f(Zi[s], Zr[s]);
    if (t[s] <= -3.14159265358979f) t[s] = 3.14159265358979f;   // principal branch (-pi, pi]
    if (v) wmax = fmaxf(wmax, Wv[s]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
  const float eta = a.eta_rel * wmax + a.eta_abs;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int b = lane + 32 * s;
    if (b < kNB) {
      own_th[b] = t[s];
      own_rel[b] = bi.valid[b] && Wv[s] > eta && Za[s] > eta;
    }
  }
  __syncwarp();
  float num = 0.f, den = 0.f;
  int any = 0;
  float thv[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int b = lane + 32 * s;
    thv[s] = 0.f;
    if (b < kNB) {
      const int rep = bi.rep[b] < kNB ? bi.rep[b] : 0;
      const bool rel = bi.valid[b] && own_rel[rep];
      float tv = own_th[rep];
      if (bi.mirror[b]) tv = -tv;
      thv[s] = (!rel || bi.selfc[b]) ? 0.f : tv;
      if (rel && bi.kap[b] > 0.f) {
        num += bi.kap[b] * Za[s];
        den += bi.kap[b] * Wv[s];
        any = 1;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
    any |= __shfl_xor_sync(0xffffffffu, any, o);
  }
  const float c = any ? __fdividef(num, den + a.eps) : 0.f;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int b = lane + 32 * s;
    th[s] = gate[s] = 0.f;
    if (b >= kNB) continue;
    const float tau = bi.tau[b];
    float gv = rcp_approx(1.f + __expf((tau - c) * rcp_approx(a.T)));
    if (a.gate_mode == CAST_GATE_ZERO) gv = 0.f;
    if (a.gate_mode == CAST_GATE_ONE) gv = 1.f;
    if (bi.cut[b]) gv = 0.f;   // outside the band
    th[s] = any ? thv[s] : 0.f;
    gate[s] = gv;
  }
}

__device__ __forceinline__ void grid_dependency_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Dynamic shared memory of a streaming f32 CTA with cc channels: the TMA stage (one anchor tile,
// 128-byte aligned; one, so that three CTAs fit an SM) and the previous anchor's spectrum
// [value][thread].
__host__ __device__ constexpr size_t stage_bytes(int cc) { return (size_t)64 * cc * sizeof(float); }
__host__ __device__ constexpr size_t spec_bytes(int cc) { return (size_t)2 * kNB * cc * sizeof(float); }
__host__ __device__ constexpr size_t par_dyn_smem(int cc) { return stage_bytes(cc) + spec_bytes(cc) + 128; }

// K_stats (STATS) and K_blend (!STATS): grid (n_chunk, n_tiles_of_kind * n_tseg), CC threads,
// one channel each.  A time segment covers the anchor pairs seg_pair0 .. seg_pair1 (it starts
// one anchor earlier).  FULL: every tile of the launch is 8x8 (the specialised fast path).
template <int CC, bool FULL, bool STATS>
__global__ void __launch_bounds__(CC, 3)
    k_par(const __grid_constant__ CUtensorMap tm, const __grid_constant__ ParKArgs a) {
  extern __shared__ uint8_t dsm_raw[];
  const uint32_t raw = smem_u32(dsm_raw);
  uint8_t* dsm = dsm_raw + (((raw + 127u) & ~127u) - raw);   // TMA boxes without swizzle: 128 B
  constexpr int cc = CC;
  constexpr int nwarp = CC / 32;
  float* stage = reinterpret_cast<float*>(dsm);                      // [y][x][channel] of one anchor tile
  float* s_fprev = reinterpret_cast<float*>(dsm + stage_bytes(cc));   // [value][thread]
  __shared__ float s_red[STATS ? nwarp : 1][128];
  __shared__ float4 s_coef[STATS ? 1 : kCoefBatch][kNB];
  __shared__ __align__(8) uint64_t s_full;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunk = blockIdx.x;
  const int tile = blockIdx.y / a.n_tseg, seg = blockIdx.y - tile * a.n_tseg;
  const int tg = a.tile_base + tile;                  // tile index in the workspace
  const int j0 = a.seg_pair0[seg] - 1, j1 = a.seg_pair1[seg];   // anchors of this segment
  const TileGeom g = tile_geom(a, tile, FULL);
  const int c = chunk * cc + tid;
  const bool active = c < a.C;
  const float wc = active ? (a.wch ? __ldg(a.wch + c) : 1.f) : 0.f;
  // bytes one TMA box delivers: cc channels x tile_w x tile_h (must match the tensor map)
  const uint32_t box_bytes = (uint32_t)(cc * a.tw * a.th * sizeof(float));
  if (tid == 0) {
    mbar_init(&s_full, 1);
    fence_barrier_init();
    tma_prefetch_desc(&tm);
    mbar_arrive_expect_tx(&s_full, box_bytes);
    tma_load_4d(stage, &tm, &s_full, chunk * cc, g.x0, g.y0, a.anchor_frame[j0]);
  }
  launch_dependents();
  __syncthreads();
  // K_blend reads theta and g, written by the preceding K_transport
  if (!STATS) grid_dependency_wait();
  bool ok = true;          // CTA-uniform; after a failed wait no more TMA is issued
  const int64_t frame_elems = (int64_t)a.Hg * a.Wg * a.C;
  float* out = reinterpret_cast<float*>(a.r);

  for (int j = j0; j <= j1; ++j) {
    float re[8][5], im[8][5];
    {
      const bool got = ok && mbar_wait(&s_full, (uint32_t)(j - j0) & 1u, a.wait_ns);
      float x[8][8];
      if (FULL) {
#pragma unroll
        for (int y = 0; y < 8; ++y)
#pragma unroll
          for (int xx = 0; xx < 8; ++xx) x[y][xx] = stage[(y * 8 + xx) * cc + tid];
      } else {
#pragma unroll
        for (int y = 0; y < 8; ++y)
#pragma unroll
          for (int xx = 0; xx < 8; ++xx)
            x[y][xx] = (y < g.h && xx < g.w) ? stage[(y * a.tw + xx) * cc + tid] : 0.f;
      }
      // the stage is free: the next anchor goes into it while this one is transformed
      if (__syncthreads_or(ok && !got)) {
        if (tid == 0) atomicExch(&g_par_error, 1u);
        ok = false;
      }
      if (ok && tid == 0 && j < j1) {
        mbar_arrive_expect_tx(&s_full, box_bytes);
        tma_load_4d(stage, &tm, &s_full, chunk * cc, g.x0, g.y0, a.anchor_frame[j + 1]);
      }
      if (FULL) dft::fwd2d(x, 8, 8, re, im);
      else dft::fwd2d(x, g.h, g.w, re, im);
    }
    const bool has_targets = j > j0 && a.pair_tbeg[j + 1] > a.pair_tbeg[j];
    const float* fa = s_fprev;   // spectrum of anchor j-1 (this thread's column)
    if (STATS && has_targets) {
      // this chunk's Z = sum w F_b conj(F_a), W = sum w |F_b||F_a| (Eq. cross)
      if (FULL) {
        // the 96 non-redundant values in three transpose groups, W at DC by a warp sum
#pragma unroll
        for (int grp = 0; grp < 3; ++grp) {
          float v[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const int code = fast_value(grp * 32 + e);
            const int b = code >> 2, comp = code & 3;
            const float ar = fa[(2 * b) * cc + tid], ai = fa[(2 * b + 1) * cc + tid];
            const float br = re[b / 5][b % 5], bi = im[b / 5][b % 5];
            v[e] = comp == 0 ? wc * (br * ar + bi * ai)
                 : comp == 1 ? wc * (bi * ar - br * ai)
                             : wc * sqrt_approx((ar * ar + ai * ai) * (br * br + bi * bi));
          }
          s_red[warp][grp * 32 + lane] = warp_transpose_sum(v, lane);
        }
        float wdc = wc * fabsf(re[0][0]) * fabsf(fa[tid]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wdc += __shfl_xor_sync(0xffffffffu, wdc, o);
        if (lane == 0) s_red[warp][96] = wdc;
      } else {
#pragma unroll
        for (int grp = 0; grp < 4; ++grp) {
          float v[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const int vi = grp * 32 + e;
            if (vi < kNV) {
              const int b = vi / 3, comp = vi % 3;
              const float ar = fa[(2 * b) * cc + tid], ai = fa[(2 * b + 1) * cc + tid];
              const float br = re[b / 5][b % 5], bi = im[b / 5][b % 5];
              v[e] = comp == 0 ? wc * (br * ar + bi * ai)
                   : comp == 1 ? wc * (bi * ar - br * ai)
                               : wc * sqrt_approx((ar * ar + ai * ai) * (br * br + bi * bi));
            } else {
              v[e] = 0.f;
            }
          }
          s_red[warp][grp * 32 + lane] = warp_transpose_sum(v, lane);
        }
      }
      __syncthreads();
      constexpr int nrec = FULL ? 97 : kNV;
      if (tid < nrec) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < nwarp; ++w) sum += s_red[w][tid];
        a.rec[(((int64_t)tg * a.n_anchor + j) * a.n_chunk + chunk) * kRec + tid] = sum;
      }
      // s_red is rewritten only after the next anchor's stage barrier
    }
    if (!STATS && has_targets) {
      // every target of the pair (Eq. fcpasm), ortho scale folded into the coefficients
      const float* th = a.trans + ((int64_t)tg * a.n_anchor + j) * 2 * kNB;
      const float* gg = th + kNB;
      const float inv_hw = 1.f / (float)(g.h * g.w);
      for (int t0 = a.pair_tbeg[j]; t0 < a.pair_tbeg[j + 1]; t0 += kCoefBatch) {
        const int nt = min(kCoefBatch, a.pair_tbeg[j + 1] - t0);
        for (int e = tid; e < nt * kNB; e += cc) {
          const int k = e / kNB, b = e % kNB;
          const float al = a.target_alpha[t0 + k];
          const float tb = __ldcg(th + b), gb = __ldcg(gg + b);
          float sa, ca, sb, cb;
          sincos_reduced(gb * al * tb, &sa, &ca);
          sincos_reduced(-gb * (1.f - al) * tb, &sb, &cb);
          const float fa_ = (1.f - al) * inv_hw, fb_ = al * inv_hw;
          s_coef[k][b] = make_float4(fa_ * ca, fa_ * sa, fb_ * cb, fb_ * sb);
        }
        __syncthreads();
        for (int k = 0; k < nt; ++k) {
          float hr[8][5], hi[8][5];
#pragma unroll
          for (int b = 0; b < kNB; ++b) {
            const int ky = b / 5, kx = b % 5;
            const float4 cf = s_coef[k][b];
            const float ar = fa[(2 * b) * cc + tid], ai = fa[(2 * b + 1) * cc + tid];
            const float br = re[ky][kx], bi = im[ky][kx];
            hr[ky][kx] = cf.x * ar - cf.y * ai + cf.z * br - cf.w * bi;
            hi[ky][kx] = cf.x * ai + cf.y * ar + cf.z * bi + cf.w * br;
          }
          float* dst = out + (int64_t)a.target_frame[t0 + k] * frame_elems +
                   ((int64_t)g.y0 * a.Wg + g.x0) * a.C + c;
          const int64_t row_step = (int64_t)a.Wg * a.C;
          const int w = FULL ? 8 : g.w, C = a.C;
          // keeps the compiler from hoisting the stores over the blend (register pressure)
          asm volatile("" ::: "memory");
          auto emit = [&](int yy, const float* row) {
            if (!active) return;
            float* d = dst + yy * row_step;
#pragma unroll
            for (int xx = 0; xx < 8; ++xx)
              if (xx < w) d[(int64_t)xx * C] = row[xx];
          };
          if (FULL) dft::inv2d_emit(hr, hi, 8, 8, emit);
          else dft::inv2d_emit(hr, hi, g.h, g.w, emit);
        }
        __syncthreads();   // s_coef is rewritten by the next batch
      }
    }
    // this anchor's spectrum becomes the previous one (thread-private column)
    if (j < j1) {
#pragma unroll
      for (int b = 0; b < kNB; ++b) {
        s_fprev[(2 * b) * cc + tid] = re[b / 5][b % 5];
        s_fprev[(2 * b + 1) * cc + tid] = im[b / 5][b % 5];
      }
    }
  }
}

// ------------------------------------------------------------------ K_stats_tc (bf16)
// Z and W of every anchor pair with targets on the tensor cores.  A unit is one (tile, pair) with
// a range of 128-channel chunks.  Per chunk the two anchors' tiles arrive by TMA ([8 x 8 tokens]
// [channels], 128-byte swizzle) and one UMMA chain each transforms them: D[channel][column] =
// X^T F with the tile's DFT as a 112-column operand in shared memory, M = 128 channels, K = 64
// tokens, D in TMEM.  A thread then owns one channel and a quarter of the bins (26 of the 98 sums: Re Z,
// Im Z, W of 30 complex bins, Z and W of 4 real ones): it reads its columns of both spectra from TMEM
// and adds its products in registers, which are reduced over the channels once per unit.
// The 8x8 transform is exact: every twiddle is an integer plus an integer times sqrt(1/2), so the
// columns hold the two integer parts (0, +-1) of each value and the thread forms A + sqrt(1/2) B
// in f32.  Other tile shapes hold the twiddles in three bf16 pieces (24 bits), accumulated into
// the A columns.
// Bound by issue slots: 16 warps of ~250 instructions per chunk (130 of them FMAs of the 8 bins of
// a warpgroup), ~1,100 cycles a chunk.  The register transform it replaces spent 1,400
// instructions per channel and anchor, half of them on transposing every chunk's sums between
// lanes: 45 us for the 50 full tiles and 22 us beside it for the 10 edge tiles of the
// HY-World-shaped call; this kernel takes 42 us for both.
constexpr int kStSumWarps = 16, kStSumThreads = 32 * kStSumWarps;
constexpr int kStThreads = 128 + kStSumThreads, kStStages = 4;
constexpr int kNCpx = 30, kNOdd = 24, kNReal = 4;       // complex bins (the first 24 with sqrt(1/2) parts), real bins
constexpr int kStN = 112;                               // columns: four warpgroups of 28
constexpr int kStTile = 64 * 128 * 2;                   // one anchor tile, 16 KB
constexpr int kStPiece = kStN * 128;                    // one operand piece [112][64] bf16, 14 KB
constexpr int kStSums = 3 * kNCpx + 2 * kNReal;         // 98
constexpr int kQOdd = kNOdd / 4, kQCpx = kQOdd + 2;     // complex bins of a warpgroup: six odd ones and a pair of even
constexpr int kQCols = kStN / 4;                        // its columns: A and B (re, im) of the odd bins, then the pair or the reals
constexpr int kStSmem = kStStages * 2 * kStTile + 3 * kStPiece + 2 * kStSumWarps * 32 * 4 + 1024;
static_assert(kStSums <= kRec, "record slots");

// Record slots of the stored bins of an h x w tile: complex representatives in bin order (8x8:
// those with an odd frequency first), self-conjugate (real) bins 0..3 apart; mirrors point at
// their representative.  255: not stored.
constexpr int kSlotMirror = 64, kSlotReal = 128;
void make_slots(int h, int w, unsigned char* bin_slot, unsigned char* slot_bin) {
  const bool full = h == 8 && w == 8;
  for (int q = 0; q < kNCpx + kNReal; ++q) slot_bin[q] = 255;
  int n_cpx = 0, n_even = kNOdd, n_real = 0;
  for (int pass = 0; pass < 2; ++pass)   // representatives, then mirrors
    for (int b = 0; b < kNB; ++b) {
      const int ky = b / 5, kx = b % 5;
      const bool edge = kx == 0 || (w % 2 == 0 && kx == w / 2);
      const bool real = edge && (ky == 0 || (h % 2 == 0 && 2 * ky == h));
      const bool mirror = edge && !real && 2 * ky > h;
      if (ky >= h || kx > w / 2) {
        bin_slot[b] = 255;
      } else if (mirror) {
        if (pass == 1) bin_slot[b] = bin_slot[(h - ky) * 5 + kx] | kSlotMirror;
      } else if (pass == 0) {
        const int slot = real ? n_real++ : full && ((ky | kx) & 1) == 0 ? n_even++ : n_cpx++;
        bin_slot[b] = (unsigned char)(slot | (real ? kSlotReal : 0));
        slot_bin[real ? kNCpx + slot : slot] = (unsigned char)b;
      }
    }
}

__device__ __forceinline__ int tile_shape(const ParKArgs& a, const TileGeom& g) {
  return (g.h < a.th ? 2 : 0) + (g.w < a.tw ? 1 : 0);
}

__device__ __forceinline__ void stats_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kStSumThreads) : "memory"); }

// A tile's transform as the swizzled K-major operand [112 columns][64 tokens] (one piece for
// 8x8, three for other shapes).  Runs once or twice per CTA, when its instructions are not yet
// cached, so the code is kept short (unrolled, it took 6 us of the kernel).
__device__ void build_dft_operand(const ParKArgs& a, const TileGeom& g, uint8_t* img, int tid) {
  // rows 0-2: bf16 pieces of cos and -sin of m / turn of a turn; 8x8: row 0 the integers, row 1
  // the factors of sqrt(1/2)
  __shared__ unsigned short s_tab[3][2][64];
  __shared__ unsigned char bins[kNCpx + kNReal];
  const int h = g.h, w = g.w;
  const bool full = h == 8 && w == 8;
  const int turn = full ? 8 : h * w;
  if (tid < 2 * 64 && (tid & 63) < turn) {
    const int im = tid >> 6, m = tid & 63;
    float sv, cv;
    sincospif(2.f * (float)m / (float)turn, &sv, &cv);
    float v = im ? -sv : cv;
    const bool odd = full && (m & 1);
    if (full) v = odd ? copysignf(1.f, v) : rintf(v);
#pragma unroll 1
    for (int p = 0; p < 3; ++p) {
      const __nv_bfloat16 b = __float2bfloat16_rn(full ? (p == (odd ? 1 : 0) ? v : 0.f) : v);
      s_tab[p][im][m] = __bfloat16_as_ushort(b);
      if (!full) v -= __bfloat162float(b);
    }
  } else if (tid >= 128 && tid < 128 + kNCpx + kNReal) {
    bins[tid - 128] = a.slot_bin[tile_shape(a, g)][tid - 128];
  }
  stats_sync();
#pragma unroll 1
  for (int e = tid; e < kStN * 8; e += kStSumThreads) {
    const int col = e >> 3, y = e & 7;
    const int wg = col / kQCols, r = col - wg * kQCols;
    const bool bpart = r >= 2 * kQOdd && r < 4 * kQOdd;
    int slot = wg * kQOdd + (r % (2 * kQOdd)) / 2, im = r & 1;
    if (r >= 4 * kQOdd && wg < 3) slot = kNOdd + 2 * wg + (r - 4 * kQOdd) / 2;
    else if (r >= 4 * kQOdd) slot = kNCpx + r - 4 * kQOdd, im = 0;
    const int b = bins[slot], ky = b / 5, kx = b % 5;
    const bool live = b != 255 && y < h && (full || !bpart);
    uint8_t* dst = img + col * 128 + ((y ^ (col & 7)) << 4);
#pragma unroll 1
    for (int p = 0; p < (full ? 1 : 3); ++p) {
      // e^{-2 pi i (ky y / h + kx x / w)}: angle m in units of 1 / turn, stepping with x
      const unsigned short* t = s_tab[full ? (int)bpart : p][im];
      const int dm = full ? kx : (kx * h) % turn;
      int m = (full ? ky * y : ky * y * w) % turn;
#pragma unroll 1
      for (int x = 0; x < 8; ++x) {
        *reinterpret_cast<unsigned short*>(dst + p * kStPiece + 2 * x) = live && x < w ? t[m] : (unsigned short)0;
        m += dm;
        if (m >= turn) m -= turn;
      }
    }
  }
}

// One anchor's tile of 128 channels into [64-channel half][8 y + x] of shared memory, one box per
// half: tiles of eight columns come from the map [frame][row][column], narrower ones from a map
// [frame][row][tile][column of the tile] with a box of eight columns, whose columns past the tile's
// side are out of range and arrive as zeros (no token of a neighbouring tile is read).  The last,
// truncated column of narrower tiles is loaded row by row.  Rows past the tile's side, and here the
// columns, are not written: they are zero (zero_stages, once per CTA) and stay so.  Row by row for
// every tile, one thread issued up to 32 copies a chunk: HY-World-shaped PAR took 335 us with 8x4
// tiles, 242 us with 8x6 and 267 us with 7x5, with boxes 234, 199 and 198 us.
struct TileMaps {
  const CUtensorMap *box, *row;   // a tile; one row of it
};
__device__ __forceinline__ bool whole_tiles(const ParKArgs& a) { return a.th == 8 && a.tw == 8; }
__device__ __forceinline__ bool boxed(const ParKArgs& a, const TileGeom& g) { return a.tw == 8 || g.w == a.tw; }
__device__ __forceinline__ uint32_t anchor_tile_bytes(const ParKArgs& a, const TileGeom& g) {
  return (uint32_t)(2 * a.th * (boxed(a, g) ? 8 : a.tw) * 128);
}
__device__ __forceinline__ void load_anchor_tile(const ParKArgs& a, const TileMaps& tm, uint8_t* dst, uint64_t* bar,
                                                 int ch, const TileGeom& g, int frame) {
  for (int b = 0; b < 2; ++b) {
    if (a.tw == 8) {
      tma_load_4d(dst + b * 8192, tm.box, bar, ch + b * 64, g.x0, g.y0, frame);
    } else if (g.w == a.tw) {
      tma_load_5d(dst + b * 8192, tm.box, bar, ch + b * 64, 0, g.x0 / a.tw, g.y0, frame);
    } else {
      for (int y = 0; y < a.th; ++y)
        tma_load_4d(dst + b * 8192 + y * 1024, tm.row, bar, ch + b * 64, g.x0, g.y0 + y, frame);
    }
  }
}
__device__ __forceinline__ void zero_stages(const ParKArgs& a, uint8_t* p, int bytes) {
  if (whole_tiles(a)) return;
  for (int e = threadIdx.x * 16; e < bytes; e += blockDim.x * 16) *reinterpret_cast<uint4*>(p + e) = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
}

// Tile i of the bf16 kernels: the complete tiles (row-major), then the truncated last column of every
// tile row, then the truncated last row, so that tiles of one shape follow one another (a CTA that
// comes to another shape builds its operand and twiddles anew: row-major over all tiles, the
// Matrix-Game-shaped PAR took 70 us with 7x5 tiles, 57 us in this order).
__device__ __forceinline__ TileGeom any_tile(const ParKArgs& a, int i) {
  const int n = a.whole_y * a.whole_x;
  int ty, tx;
  if (i < n) {
    ty = i / a.whole_x;
    tx = i - ty * a.whole_x;
  } else if (a.whole_x < a.tiles_x && i - n < a.tiles_y) {
    ty = i - n;
    tx = a.whole_x;
  } else {
    ty = a.whole_y;
    tx = i - n - (a.whole_x < a.tiles_x ? a.tiles_y : 0);
  }
  TileGeom g;
  g.y0 = ty * a.th;
  g.x0 = tx * a.tw;
  g.h = min(a.th, a.Hg - g.y0);
  g.w = min(a.tw, a.Wg - g.x0);
  return g;
}

// The units of a CTA: blockIdx.x, then every gridDim.x-th.  Stepping in (tile, part, item) costs no
// division: the divisions took ~1,000 cycles of every role and unit, and a unit of one channel chunk has
// ~1,100 cycles of work in the statistics (16 frames of 44x80 x 64 channels: 6x6 tiles 42 -> 40 us, 4x4
// tiles 59 -> 54 us).
__device__ __forceinline__ Unit first_unit(int n_part, int n_item) {
  Unit u;
  const int q = blockIdx.x / n_item;
  u.item = blockIdx.x - q * n_item;
  u.tile = q / n_part;
  u.part = q - u.tile * n_part;
  return u;
}
__device__ __forceinline__ void next_unit(Unit& u, const Unit& step, int n_part, int n_item) {
  u.item += step.item;
  u.part += step.part;
  u.tile += step.tile;
  if (u.item >= n_item) u.item -= n_item, ++u.part;
  if (u.part >= n_part) u.part -= n_part, ++u.tile;
}

template <bool WEIGHTED>
__global__ void __launch_bounds__(kStThreads, 1)
    k_par_stats_tc(const __grid_constant__ CUtensorMap tm_box, const __grid_constant__ CUtensorMap tm_row,
                   const __grid_constant__ ParKArgs a) {
  extern __shared__ uint8_t dsm_raw[];
  const uint32_t raw_addr = smem_u32(dsm_raw);
  uint8_t* dsm = dsm_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint8_t* s_x = dsm;
  uint8_t* s_img = dsm + kStStages * 2 * kStTile;
  float* s_red = reinterpret_cast<float*>(s_img + 3 * kStPiece);   // [2][16 warps][32]
  __shared__ __align__(8) uint64_t b_full[kStStages], b_empty[kStStages], b_dfull[2], b_dempty[2], b_img,
      b_seen;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t lim = a.wait_ns;
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    if (s_abort) return false;
    if (mbar_wait(bar, parity, lim)) return true;
    s_abort = 1;
    atomicExch(&g_par_error, 1u);
    return false;
  };
  // Behind a kernel of someone else this CTA takes no TMEM until that one has ended: it may let its
  // dependents start before its own CTAs have allocated theirs, and would then wait for the columns
  // of a CTA that waits for its end.  (The attention and the GEMM leave no room for another CTA on
  // their SM.)
  if (!a.after_own) grid_dependency_wait();
  if (tid == 0) {
    for (int s = 0; s < kStStages; ++s) {
      mbar_init(&b_full[s], 1);
      mbar_init(&b_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&b_dfull[b], 1);
      mbar_init(&b_dempty[b], kStSumWarps);
    }
    mbar_init(&b_img, 1);
    mbar_init(&b_seen, 2);   // both issuers
    fence_barrier_init();
    s_abort = 0;
  }
  if (warp == 1) {
    tmem_alloc(&s_tmem, 512);
    tmem_relinquish();
    tc_fence_before();
  }
  zero_stages(a, s_x, kStStages * 2 * kStTile);
  launch_dependents();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int nck = a.n_chunk, n_part = a.st_parts, n_item = a.n_act;   // an item: a pair with targets
  const auto c0_of = [&](const Unit& u) { return u.part * a.st_cpp; };
  const auto c1_of = [&](const Unit& u) { return min(nck, (u.part + 1) * a.st_cpp); };

  if (warp < 4) {
    if (warp == 0 && lane == 0) {
      // -------------------------------------------------------------- anchor producer
      const TileMaps tm{&tm_box, &tm_row};
      tma_prefetch_desc(&tm_box);
      grid_dependency_wait();   // the anchors (what the sums need besides comes after them)
      int n = 0;
      bool ok = true;
      for (Unit x = first_unit(n_part, n_item); ok && x.tile < a.n_tile; next_unit(x, a.st_step, n_part, n_item)) {
        const TileGeom g = any_tile(a, x.tile);
        for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
          const int s = n % kStStages;
          if (n >= kStStages && !wait(&b_empty[s], (uint32_t)((n / kStStages) - 1) & 1u)) { ok = false; break; }
          mbar_arrive_expect_tx(&b_full[s], 2 * anchor_tile_bytes(a, g));
          for (int q = 0; q < 2; ++q)
            load_anchor_tile(a, tm, s_x + (2 * s + q) * kStTile, &b_full[s], c * 128, g, a.anchor_frame[a.act_pair[x.item] - 1 + q]);
        }
      }
      // (whatever ended the loop) the last copies have landed before shared memory is released
      for (int l = n > kStStages ? n - kStStages : 0; l < n; ++l)
        mbar_wait(&b_full[l % kStStages], (uint32_t)(l / kStStages) & 1u, lim);
    } else if (warp & 1) {
      // -------------------------------------------------------------- UMMA issuers (converged)
      // warps 1 and 3 take alternate chunks and accumulators: the ~500 cycles that an issuer
      // spends on waits and commits per chunk pass while the other one's UMMAs run
      constexpr uint32_t idesc = idesc_bf16_f32(128, kStN, true, false);
      const int buf = warp >> 1;
      const uint32_t tmu = __shfl_sync(0xffffffffu, tmem, 0) + (uint32_t)(buf * 256);
      const uint32_t xb = __shfl_sync(0xffffffffu, smem_u32(s_x), 0), ib = __shfl_sync(0xffffffffu, smem_u32(s_img), 0);
      const uint64_t dx = sdesc_sw128(xb, 8192, 1024), di = sdesc_sw128(ib, 16, 1024);
      const bool lead = elect_one();
      int n = 0, last = -1, shape = -1, builds = 0;
      bool ok = true;
      for (Unit x = first_unit(n_part, n_item); ok && x.tile < a.n_tile; next_unit(x, a.st_step, n_part, n_item)) {
        const TileGeom g = any_tile(a, x.tile);
        if (g.h * 16 + g.w != shape) {
          shape = g.h * 16 + g.w;
          if (!(ok = __all_sync(0xffffffffu, wait(&b_img, (uint32_t)builds++ & 1u)))) break;
          if (lane == 0) mbar_arrive(&b_seen);
        }
        const bool pieces = !(g.h == 8 && g.w == 8);
        for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
          if ((n & 1) != buf) continue;
          const int s = n % kStStages;
          // half of the warp waits for the anchors, half for the accumulator
          const bool w = lane < 16 ? wait(&b_full[s], (uint32_t)(n / kStStages) & 1u)
                                   : n < 2 || wait(&b_dempty[buf], (uint32_t)((n >> 1) - 1) & 1u);
          if (!(ok = __all_sync(0xffffffffu, w))) break;
          __syncwarp();   // (a vote orders no memory) what the other half waited for, the lead sees after this
          tc_fence_after();
          if (lead) {
            const uint64_t da = dx + (uint64_t)(2 * s * (kStTile >> 4));
            auto chain = [&](int q, int p) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                umma_bf16_ss(tmu + (uint32_t)(q * 128), da + (uint64_t)(q * (kStTile >> 4) + kk * (2048 >> 4)),
                             di + (uint64_t)(p * (kStPiece >> 4) + kk * 2), idesc, (p | kk) ? 1u : 0u);
            };
            chain(0, 0);
            if (pieces) chain(0, 1), chain(0, 2);
            chain(1, 0);
            if (pieces) chain(1, 1), chain(1, 2);
            umma_commit(&b_empty[s]);
            umma_commit(&b_dfull[buf]);
          }
          __syncwarp();
          last = n;
        }
      }
      // the UMMAs issued so far have completed before shared memory and TMEM are released
      if (last >= 0) mbar_wait(&b_dfull[buf], (uint32_t)(last >> 1) & 1u, lim);
      __syncwarp();
    }
  } else {
    // ---------------------------------------------------------------- sums
    // One channel per thread (and per TMEM lane) in each of four warpgroups, a quarter of the bins
    // in each: four warps per scheduler cover the latency of the TMEM reads and square roots
    // (two warpgroups with half of the bins took 1,160 cycles a chunk).  Warpgroup w has the
    // complex bins 6 w .. 6 w + 5 and 24 + 2 w, 25 + 2 w, the last one the real bins instead.
    const int wg = (warp >> 2) - 1, q4 = warp & 3, ctid = tid - 128;
    const uint32_t td0 = tmem + ((uint32_t)(q4 * 32) << 16);
    constexpr float kR = 0.70710678118654752f;
    int n = 0, shape = 0, flip = 0;   // shape: operands built so far << 8 | sides of the last one
    bool ok = true;
    for (Unit x = first_unit(n_part, n_item); x.tile < a.n_tile; next_unit(x, a.st_step, n_part, n_item), flip ^= 1) {
      const TileGeom g = any_tile(a, x.tile);
      if (g.h * 16 + g.w != (shape & 255)) {
        // every UMMA that read the operand has completed: its chunk has been waited for
        const int builds = shape >> 8;
        shape = (builds + 1) << 8 | (g.h * 16 + g.w);
        build_dft_operand(a, g, s_img, ctid);
        fence_proxy_async_smem();
        stats_sync();
        // an issuer without a chunk since then may not have seen the operand before this one: its
        // barrier must not run a second phase ahead of it
        if (ctid == 0 && (builds == 0 || wait(&b_seen, (uint32_t)(builds - 1) & 1u))) mbar_arrive(&b_img);
      }
      // Re Z, Im Z, W of the complex bins; of the last warpgroup, Z of the real bins in zr[6],
      // zr[7], zi[6], zi[7] and W in wv[6], wv[7], ex[0], ex[1]
      float zr[kQCpx], zi[kQCpx], wv[kQCpx], ex[2] = {0.f, 0.f};
#pragma unroll
      for (int c = 0; c < kQCpx; ++c) zr[c] = zi[c] = wv[c] = 0.f;
      // one complex bin; the weight comes last, so that no square of it is formed (w^2 leaves the range
      // of a float long before w |F_a| |F_b| does)
      float wc = 1.f;
      auto add = [&](int s, float ra, float ia, float rb, float ib) {
        const float aw = sqrt_approx(fmaf(ra, ra, ia * ia) * fmaf(rb, rb, ib * ib));
        if (WEIGHTED) {
          zr[s] = fmaf(wc, fmaf(rb, ra, ib * ia), zr[s]);
          zi[s] = fmaf(wc, fmaf(ib, ra, -rb * ia), zi[s]);
          wv[s] = fmaf(wc, aw, wv[s]);
        } else {
          zr[s] = fmaf(rb, ra, fmaf(ib, ia, zr[s]));
          zi[s] = fmaf(ib, ra, fmaf(-rb, ia, zi[s]));
          wv[s] += aw;
        }
      };
      for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
        const int buf = n & 1, ch = c * 128 + q4 * 32 + lane;
        if (!(ok = __all_sync(0xffffffffu, wait(&b_dfull[buf], (uint32_t)(n >> 1) & 1u)))) break;
        tc_fence_after();
        if (WEIGHTED) wc = ch < a.C ? __ldcg(a.wch + ch) : 1.f;
        // the warpgroup's columns of anchors a and b, then the buffer goes back to its issuer
        uint32_t va[64];
        tmem_ld_x32_async(td0 + (uint32_t)(buf * 256 + wg * kQCols), va);
        tmem_ld_x32_async(td0 + (uint32_t)(buf * 256 + 128 + wg * kQCols), va + 32);
        tmem_wait_ld_x64(va);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&b_dempty[buf]);
        const float *fa = reinterpret_cast<const float*>(va), *fb = fa + 32;
#pragma unroll
        for (int e = 0; e < 2 * kQOdd; e += 2)   // A + sqrt(1/2) B
          add(e / 2, fmaf(kR, fa[2 * kQOdd + e], fa[e]), fmaf(kR, fa[2 * kQOdd + e + 1], fa[e + 1]),
              fmaf(kR, fb[2 * kQOdd + e], fb[e]), fmaf(kR, fb[2 * kQOdd + e + 1], fb[e + 1]));
        fa += 4 * kQOdd;
        fb += 4 * kQOdd;
        if (wg < 3) {
          add(kQOdd, fa[0], fa[1], fb[0], fb[1]);
          add(kQOdd + 1, fa[2], fa[3], fb[2], fb[3]);
        } else {
          const float z0 = wc * (fa[0] * fb[0]), z1 = wc * (fa[1] * fb[1]), z2 = wc * (fa[2] * fb[2]), z3 = wc * (fa[3] * fb[3]);
          zr[kQOdd] += z0;
          zr[kQOdd + 1] += z1;
          zi[kQOdd] += z2;
          zi[kQOdd + 1] += z3;
          wv[kQOdd] += fabsf(z0);
          wv[kQOdd + 1] += fabsf(z1);
          ex[0] += fabsf(z2);
          ex[1] += fabsf(z3);
        }
      }
      // sums over the channels by a warp transpose (8 Re Z | 8 Im Z | 8 W | 2 more), then over the
      // warpgroup's four warps in order
      {
        float t[32];
#pragma unroll
        for (int e = 0; e < 32; ++e)
          t[e] = e < kQCpx ? zr[e < kQCpx ? e : 0]
               : e < 2 * kQCpx ? zi[e < 2 * kQCpx ? e - kQCpx : 0]
               : e < 3 * kQCpx ? wv[e < 3 * kQCpx ? e - 2 * kQCpx : 0]
               : e < 3 * kQCpx + 2 ? ex[e < 3 * kQCpx + 2 ? e - 3 * kQCpx : 0] : 0.f;
        s_red[(flip * kStSumWarps + warp - 4) * 32 + lane] = warp_transpose_sum(t, lane);
      }
      // (the warps leave together: a thread left behind would wait in this barrier)
      if (bar_sync_or(2, kStSumThreads, !ok || s_abort)) break;
      if (ctid < kStSums) {
        // record slot (30 Re Z | 30 Im Z | 30 W | 4 Z | 4 W) -> warpgroup and place in its sums
        const int part = ctid / kNCpx, slot = ctid - part * kNCpx;
        int of = 3, at;
        if (part < 3) {
          of = slot < kNOdd ? slot / kQOdd : (slot - kNOdd) >> 1;
          at = part * kQCpx + (slot < kNOdd ? slot - of * kQOdd : kQOdd + ((slot - kNOdd) & 1));
        } else {
          const int r = slot & 3;   // Z: zr, zr, zi, zi; W: wv, wv, ex, ex
          at = (slot < kNReal ? (r >> 1) : 2 + (r >> 1)) * kQCpx + (slot >= kNReal && r >= 2 ? 0 : kQOdd) + (r & 1);
        }
        float sum = 0.f;
#pragma unroll
        for (int w4 = 0; w4 < 4; ++w4) sum += s_red[(flip * kStSumWarps + of * 4 + w4) * 32 + at];
        a.rec[(((int64_t)x.tile * a.n_anchor + a.act_pair[x.item]) * a.n_chunk + x.part) * kRec + ctid] = sum;
      }
      // the other half of s_red is written next, this one only after the next unit's barrier
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// Sum of `n` record entries kRec apart, in order, twelve loads in flight per round.
__device__ __forceinline__ float record_sum(const float* r, int n) {
  float sum = 0.f;
  for (int q0 = 0; q0 < n; q0 += 12) {
    float v[12];
#pragma unroll
    for (int u = 0; u < 12; ++u) v[u] = q0 + u < n ? __ldcg(r + (int64_t)(q0 + u) * kRec) : 0.f;
#pragma unroll
    for (int u = 0; u < 12; ++u) sum += v[u];
  }
  return sum;
}

// ------------------------------------------------------------------ K_transport (f32)
// grid (n_tiles_of_kind, n_anchor - 1), 128 threads; block y = pair j - 1.
template <bool FULL>
__global__ void __launch_bounds__(128) k_par_transport(const __grid_constant__ ParKArgs a) {
  __shared__ float s_zw[kNV];
  __shared__ float s_own_th[kNB];
  __shared__ int s_own_rel[kNB];
  __shared__ BinInfo s_bins;
  const int tid = threadIdx.x;
  const int tile = blockIdx.x, j = blockIdx.y + 1, tg = a.tile_base + tile;
  if (!(a.pair_tbeg[j + 1] > a.pair_tbeg[j])) {   // no target: no record
    launch_dependents();
    return;
  }
  const TileGeom g = tile_geom(a, tile, FULL);
  bin_info(a, g, s_bins, tid);
  grid_dependency_wait();   // the records come from the preceding K_stats
  if (tid < kNV) {
    int k = tid, sign = 1;
    if (FULL) {
      const int src = a.fast_src[tid];
      k = (src > 0 ? src : -src) - 1;
      sign = src < 0 ? -1 : 1;
    }
    const float sum =
        k >= 0 ? record_sum(a.rec + ((int64_t)tg * a.n_anchor + j) * a.n_chunk * kRec + k, a.n_chunk) : 0.f;
    s_zw[tid] = sign < 0 ? -sum : sum;
  }
  __syncthreads();
  if (tid < 32) {
    float th[2], gate[2];
    tile_transport(a, g, s_bins, s_zw, th, gate, s_own_th, s_own_rel, tid);
    float* tr = a.trans + ((int64_t)tg * a.n_anchor + j) * 2 * kNB;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int b = tid + 32 * s;
      if (b < kNB) {
        tr[b] = th[s];
        tr[kNB + b] = gate[s];
      }
    }
  }
  launch_dependents();
}

// ------------------------------------------------------------------ K_blend_tc (bf16)
// Persistent, one CTA per SM, 512 threads.  A unit is one (tile, group of up to two targets of a
// pair) with a range of 128-channel chunks: its blend matrices (two targets stacked into the
// M = 128 operand, rows 0-63 and 64-127; two bf16 pieces) stay in TMEM while the chunks stream
// past, [H_t1 ; H_t2] [X_a ; X_b] per chunk (2 pieces x 8 K-steps, N = 128):
//   warp 0       X_a and X_b of each chunk (TMA, [8 x 8 tokens][channels], the MN-major operand),
//                four stages of 32 KB
//   warps 2, 3   the transport of each unit (records -> theta, g), alternate units, up to two ahead
//   warps 12..15 the matrices: the convolution kernels h of the unit's targets, a table of their
//                128 distinct 16-byte rows each, and from it one operand row per thread into TMEM
//                (two pieces of 64 columns, two units' worth), one unit ahead of the UMMAs
//   warp 1       UMMA issuer (converged), A from TMEM, D in one of two 128-column TMEM buffers
//   warps 4..11  epilogue: two sets of four warps take alternate chunks; a warp converts 32 output
//                tokens x 64 channels at a time into one of its two 4 KB staging tiles, which it
//                stores with TMA by itself (no barrier between warps).
// Bound by the tensor pipe (1,088 cycles a chunk) and the output stream.  A kernel of its own for
// the transport, which wrote 32 KB of matrices per (tile, target), and a blend that loaded them
// for every (tile, chunk) - 64 KB per 32 KB of output through the ~50 bytes per clock that an SM
// takes from L2, one staging tile for all warps - took 11 and 68 us for the full tiles of the
// HY-World-shaped call, 9.5 and 19 us beside them for the edge tiles.  A unit's transport is one chain
// of ~5,500 cycles, its matrices take ~3,500: with one transport warp (and a second issuer in place of
// the other) a unit could not take less than six chunks (HY-World-shaped call 109 -> 107 us, with 4x4
// tiles 388 -> 339 us).  With the matrices in shared
// memory the UMMAs read both operands from there (128 bytes per clock, as much as an SM has).
constexpr int kTbStages = 4;
constexpr int kTbPlane = 64 * 128 * 2;          // one anchor tile of a chunk, 16 KB
constexpr int kTbStage = 2 * kTbPlane;          // X_a and X_b
constexpr int kTbOut = 32 * 128;                // a warp's 32 tokens x 64 channels
constexpr int kTbThreads = 512;
constexpr int kTbMat = 128, kTbD = 256;         // TMEM columns: matrices of unit k at (k & 1) * 128, D buffers at 256

// The transport of one unit, by one warp.
struct TransportShared {
  BinInfo bins;
  float zw[kNV], own_th[kNB];
  int own_rel[kNB];
  unsigned char slot[kNB];
};
constexpr int kZwPer = (kNV + 31) / 32;   // entries of zw per lane: lane, lane + 32, ...
__device__ void transport_shape(const ParKArgs& a, const TileGeom& g, TransportShared& m, int (&at)[kZwPer], int lane) {
#pragma unroll 1
  for (int b = lane; b < kNB; b += 32) {
    bin_info(a, g, m.bins, b);
    m.slot[b] = a.bin_slot[tile_shape(a, g)][b];
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < kZwPer; ++i) {
    const int e = lane + 32 * i, b = min(e / 3, kNB - 1), comp = e - 3 * (e / 3), code = m.slot[b], slot = code & 63;
    // Re Z, Im Z, W of complex slot s stand at s, 30 + s, 60 + s, Z and W of real slot s at 90 + s, 94 + s
    at[i] = comp * kNCpx + slot;
    if (code & kSlotReal) at[i] = comp == 1 ? -1 : 3 * kNCpx + (comp == 2 ? kNReal : 0) + slot;
    if (code == 255 || e >= kNV) at[i] = -1;
  }
}
__device__ void unit_transport(const ParKArgs& a, const TileGeom& g, int tile, int j, TransportShared& m,
                               const int (&at)[kZwPer], float (&th)[2], float (&gate)[2], int lane) {
  const float* rec = a.rec + ((int64_t)tile * a.n_anchor + j) * a.n_chunk * kRec;
  // this lane's entries, summed over the parts in order, sixteen loads in flight
  float sum[kZwPer];
#pragma unroll
  for (int i = 0; i < kZwPer; ++i) sum[i] = 0.f;
  for (int q0 = 0; q0 < a.st_parts; q0 += 4) {
    float v[kZwPer][4];
#pragma unroll
    for (int i = 0; i < kZwPer; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        v[i][q] = at[i] >= 0 && q0 + q < a.st_parts ? __ldcg(rec + (int64_t)(q0 + q) * kRec + at[i]) : 0.f;
#pragma unroll
    for (int i = 0; i < kZwPer; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) sum[i] += v[i][q];
  }
#pragma unroll
  for (int i = 0; i < kZwPer; ++i) {
    const int e = lane + 32 * i;
    if (e < kNV) m.zw[e] = (e % 3) == 1 && (m.slot[e / 3] & kSlotMirror) && at[i] >= 0 ? -sum[i] : sum[i];
  }
  __syncwarp();
  tile_transport(a, g, m.bins, m.zw, th, gate, m.own_th, m.own_rel, lane);
  __syncwarp();
}

// The matrices of one unit, by 128 threads (barrier 3): thread = (side, dy, xo).
// Row m = output token 8 yo + xo, column 64 side + 8 yi + xi = input token of anchor a (side 0)
// or b (side 1); entry h_side((yo - yi) mod h, (xo - xi) mod w) with
// h_side(d) = (1 / (h w)) sum over stored bins of kappa' Re(phi_side e^{2 pi i (ky dy / h + kx dx / w)}),
// kappa' = 1 on the kx = 0 and Nyquist columns (every ky stored), 2 elsewhere;
// phi_a = (1 - alpha) e^{i g alpha theta}, phi_b = alpha e^{-i g (1 - alpha) theta}.  The sum runs
// over kx first (one complex value per (ky, dx)), then over ky.
struct MatrixShared {
  uint4 row[2][2][2][64];   // [target][piece][side][8 dy + xo]: entries (xo - xi) mod w, xi = 0..7, of row dy
  float4 phi[2][kNB];
  float2 col[2][2][64];     // [target][side][8 ky + dx]
  float h[2][2][64];        // [target][side][8 dy + dx]
};
constexpr int kTbSmem = kTbStages * kTbStage + 16 * kTbOut + (int)sizeof(MatrixShared) + 1024;

__device__ __forceinline__ void matrix_sync() { asm volatile("bar.sync 3, 128;" ::: "memory"); }

__global__ void __launch_bounds__(kTbThreads, 1)
    k_par_blend_tc(const __grid_constant__ CUtensorMap tm_box, const __grid_constant__ CUtensorMap tm_row,
                   const __grid_constant__ CUtensorMap tm_out, const __grid_constant__ ParKArgs a) {
  extern __shared__ uint8_t dsm_raw[];
  const uint32_t raw_addr = smem_u32(dsm_raw);
  uint8_t* dsm = dsm_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);   // 128-byte swizzle atoms
  uint8_t* s_x = dsm;
  uint8_t* s_out = dsm + kTbStages * kTbStage;
  MatrixShared& m = *reinterpret_cast<MatrixShared*>(s_out + 16 * kTbOut);
  __shared__ __align__(8) uint64_t b_xfull[kTbStages], b_xempty[kTbStages], b_mfull[2], b_mempty[2], b_dfull[2],
      b_dempty[2], b_tready[2], b_tfree[2];
  __shared__ float s_th[2][kNB], s_gate[2][kNB];   // of the units whose matrices are next
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t lim = a.wait_ns;
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    if (s_abort) return false;
    if (mbar_wait(bar, parity, lim)) return true;
    s_abort = 1;
    atomicExch(&g_par_error, 1u);
    return false;
  };
  if (tid == 0) {
    for (int s = 0; s < kTbStages; ++s) {
      mbar_init(&b_xfull[s], 1);
      mbar_init(&b_xempty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&b_mfull[b], 128);
      mbar_init(&b_mempty[b], 1);
      mbar_init(&b_tready[b], 1);
      mbar_init(&b_tfree[b], 1);
      mbar_init(&b_dfull[b], 1);
      mbar_init(&b_dempty[b], 4);
    }
    fence_barrier_init();
    s_abort = 0;
  }
  if (warp == 1) {
    tmem_alloc(&s_tmem, 512);
    tmem_relinquish();
    tc_fence_before();
  }
  zero_stages(a, s_x, kTbStages * kTbStage);
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  // (the warps that read what earlier launches wrote, 0, 2 and 3, wait for the grid before)
  const int n_part = a.bl_parts, n_item = a.n_grp;   // an item: up to two targets of a pair
  const auto c0_of = [&](const Unit& u) { return u.part * a.bl_cpp; };
  const auto c1_of = [&](const Unit& u) { return min(a.n_chunk, (u.part + 1) * a.bl_cpp); };

  if (warp == 0) {
    if (lane == 0) {
      // -------------------------------------------------------------- anchor producer
      const TileMaps tm{&tm_box, &tm_row};
      tma_prefetch_desc(&tm_box);
      // the anchors may come from the launch before the statistics, whose grid waited for it
      grid_dependency_wait();
      int n = 0;
      bool ok = true;
      for (Unit x = first_unit(n_part, n_item); ok && x.tile < a.n_tile; next_unit(x, a.bl_step, n_part, n_item)) {
        const TileGeom g = any_tile(a, x.tile);
        const int j = a.grp_pair[x.item];
        for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
          const int s = n % kTbStages;
          if (n >= kTbStages && !wait(&b_xempty[s], (uint32_t)((n / kTbStages) - 1) & 1u)) { ok = false; break; }
          mbar_arrive_expect_tx(&b_xfull[s], 2 * anchor_tile_bytes(a, g));
          for (int q = 0; q < 2; ++q)
            load_anchor_tile(a, tm, s_x + s * kTbStage + q * kTbPlane, &b_xfull[s], c * 128, g, a.anchor_frame[j - 1 + q]);
        }
      }
      for (int l = n > kTbStages ? n - kTbStages : 0; l < n; ++l)
        mbar_wait(&b_xfull[l % kTbStages], (uint32_t)(l / kTbStages) & 1u, lim);
    }
  } else if (warp >= 12) {
    // ---------------------------------------------------------------- matrices
    const int mt = tid - 384, side = mt >> 6, dy = (mt >> 3) & 7, dx = mt & 7;   // dy also ky, dx also xo
    // this thread's operand row (TMEM lane): target slot and output token
    const int rts = mt >> 6, ryo = (mt >> 3) & 7, rxo = mt & 7;
    const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    int k = 0, shape = -1;
    float2 twx[5], twy[8];   // e^{2 pi i kx dx / w}, e^{2 pi i ky dy / h}; 0 past the stored bins
    for (Unit x = first_unit(n_part, n_item); x.tile < a.n_tile; next_unit(x, a.bl_step, n_part, n_item), ++k) {
      const TileGeom g = any_tile(a, x.tile);
      const int h = g.h, w = g.w, t0 = a.grp_t0[x.item], nt = a.grp_nt[x.item];
      if (h * 16 + w != shape) {
        shape = h * 16 + w;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          float sv, cv;
          sincospif(2.f * (float)(q * dx % w) / (float)w, &sv, &cv);
          twx[q] = q <= w / 2 ? make_float2(cv, sv) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float sv, cv;
          sincospif(2.f * (float)(q * dy % h) / (float)h, &sv, &cv);
          twy[q] = q < h ? make_float2(cv, sv) : make_float2(0.f, 0.f);
        }
      }
      // (the four warps leave together)
      if (bar_sync_or(3, 128, !wait(&b_tready[k & 1], (uint32_t)(k >> 1) & 1u))) break;
      if (mt < 2 * kNB) {
        const int ts = mt / kNB, b = mt - ts * kNB, ky = b / 5, kx = b % 5;
        float4 ph = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ts < nt && ky < h && kx <= w / 2) {
          const float al = a.target_alpha[t0 + ts];
          const bool edge = kx == 0 || ((w % 2 == 0) && kx == w / 2);
          const float kap = (edge ? 1.f : 2.f) / (float)(h * w);
          float sa, ca, sb, cb;
          const float gt = s_gate[k & 1][b] * s_th[k & 1][b];
          sincosf(gt * al, &sa, &ca);
          sincosf(-gt * (1.f - al), &sb, &cb);
          ph = make_float4(kap * (1.f - al) * ca, kap * (1.f - al) * sa, kap * al * cb, kap * al * sb);
        }
        m.phi[ts][b] = ph;
      }
      matrix_sync();
      if (mt == 0) mbar_arrive(&b_tfree[k & 1]);   // theta and g have been read
#pragma unroll
      for (int ts = 0; ts < 2; ++ts) {
        float cr = 0.f, ci = 0.f;
#pragma unroll
        for (int kx = 0; kx < 5; ++kx) {
          const float4 ph = m.phi[ts][dy * 5 + kx];
          const float pr = side ? ph.z : ph.x, pi = side ? ph.w : ph.y;
          cr = fmaf(pr, twx[kx].x, fmaf(-pi, twx[kx].y, cr));
          ci = fmaf(pr, twx[kx].y, fmaf(pi, twx[kx].x, ci));
        }
        m.col[ts][side][dy * 8 + dx] = make_float2(cr, ci);
      }
      matrix_sync();
#pragma unroll
      for (int ts = 0; ts < 2; ++ts) {
        float acc = 0.f;
#pragma unroll
        for (int ky = 0; ky < 8; ++ky) {
          const float2 c = m.col[ts][side][ky * 8 + dx];
          acc = fmaf(c.x, twy[ky].x, fmaf(-c.y, twy[ky].y, acc));
        }
        m.h[ts][side][dy * 8 + dx] = acc;
      }
      matrix_sync();
      // the distinct rows of 8 input columns in two bf16 pieces
#pragma unroll
      for (int ts = 0; ts < 2; ++ts) {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int xi = 0; xi < 8; xi += 2) {
          float v[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int d = dx - xi - q + (dx < xi + q ? w : 0);
            v[q] = dy < h && dx < w && xi + q < w ? m.h[ts][side][dy * 8 + d] : 0.f;
          }
          const __nv_bfloat162 b1 = __floats2bfloat162_rn(v[0], v[1]);
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[0] - __low2float(b1), v[1] - __high2float(b1));
          hi[xi / 2] = *reinterpret_cast<const uint32_t*>(&b1);
          lo[xi / 2] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        m.row[ts][0][side][dy * 8 + dx] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        m.row[ts][1][side][dy * 8 + dx] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      }
      // the UMMAs of the unit before the last have read their matrices
      const int mb = k & 1;
      if (bar_sync_or(3, 128, k >= 2 && !wait(&b_mempty[mb], (uint32_t)((k >> 1) - 1) & 1u))) break;
      tc_fence_after();
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
          uint32_t v[32];
#pragma unroll
          for (int yi = 0; yi < 8; ++yi) {
            const int d = ryo - yi + (ryo < yi ? h : 0);
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (yi < h && ryo < h) q = m.row[rts][p][sd][d * 8 + rxo];
            v[4 * yi] = q.x;
            v[4 * yi + 1] = q.y;
            v[4 * yi + 2] = q.z;
            v[4 * yi + 3] = q.w;
          }
          tmem_st_x32_async(tm + (uint32_t)(mb * kTbMat + p * 64 + sd * 32), v);
        }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&b_mfull[mb]);
    }
  } else if (warp == 2 || warp == 3) {
    // ---------------------------------------------------------------- transport
    // warps 2 and 3 take alternate units
    __shared__ TransportShared both[2];
    const int me = warp & 1;
    TransportShared& ms = both[me];
    int k = 0, shape = -1, at[kZwPer];
    for (Unit x = first_unit(n_part, n_item); x.tile < a.n_tile; next_unit(x, a.bl_step, n_part, n_item), ++k) {
      if ((k & 1) != me) continue;
      const TileGeom g = any_tile(a, x.tile);
      const bool fresh = g.h * 16 + g.w != shape;
      shape = g.h * 16 + g.w;
      if (fresh) transport_shape(a, g, ms, at, lane);
      if (k == me) grid_dependency_wait();   // the records of K_stats_tc
      float th[2], gate[2];
      unit_transport(a, g, x.tile, a.grp_pair[x.item], ms, at, th, gate, lane);
      // only the hand-over waits for the matrix warps to have read the unit before the last
      if (!__all_sync(0xffffffffu, k < 2 || wait(&b_tfree[me], (uint32_t)((k >> 1) - 1) & 1u))) break;
#pragma unroll
      for (int s = 0; s < 2; ++s)
        if (lane + 32 * s < kNB) {
          s_th[me][lane + 32 * s] = th[s];
          s_gate[me][lane + 32 * s] = gate[s];
        }
      __syncwarp();
      if (lane == 0) mbar_arrive(&b_tready[me]);
    }
  } else if (warp < 4) {
    // ---------------------------------------------------------------- UMMA issuer (converged)
    constexpr uint32_t idesc = idesc_bf16_f32(128, 128, false, true);
    const uint32_t tmu = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t xb = __shfl_sync(0xffffffffu, smem_u32(s_x), 0);
    const uint64_t dx = sdesc_sw128(xb, 8192, 1024);
    const bool lead = elect_one();
    int n = 0, k = 0, last = -1;
    bool ok = true;
    for (Unit x = first_unit(n_part, n_item); ok && x.tile < a.n_tile; next_unit(x, a.bl_step, n_part, n_item), ++k) {
      const int mb = k & 1;
      if (!(ok = __all_sync(0xffffffffu, wait(&b_mfull[mb], (uint32_t)(k >> 1) & 1u)))) break;
      tc_fence_after();
      for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
        const int s = n % kTbStages, buf = n & 1;
        // half of the warp waits for the anchors, half for the accumulator
        const bool w = lane < 16 ? wait(&b_xfull[s], (uint32_t)(n / kTbStages) & 1u)
                                 : n < 2 || wait(&b_dempty[buf], (uint32_t)((n >> 1) - 1) & 1u);
        if (!(ok = __all_sync(0xffffffffu, w))) break;
        __syncwarp();   // (a vote orders no memory) what the other half waited for, the lead sees after this
        tc_fence_after();
        if (lead) {
          const uint64_t db = dx + (uint64_t)(s * (kTbStage >> 4));
#pragma unroll
          for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              umma_bf16_ts(tmu + (uint32_t)(kTbD + buf * 128), tmu + (uint32_t)(mb * kTbMat + p * 64 + kk * 8),
                           db + (uint64_t)(((kk >> 2) * kTbPlane + (kk & 3) * 2048) >> 4), idesc, (p | kk) ? 1u : 0u);
          umma_commit(&b_xempty[s]);
          umma_commit(&b_dfull[buf]);
        }
        __syncwarp();
        last = n;
      }
      // the last reads of the unit's matrices
      if (ok && lead) umma_commit(&b_mempty[mb]);
      __syncwarp();
    }
    // the UMMAs issued so far have completed before shared memory and TMEM are released
    if (last >= 0) mbar_wait(&b_dfull[last & 1], (uint32_t)(last >> 1) & 1u, lim);
    __syncwarp();
  } else if (warp >= 4) {   // 4..11
    // ---------------------------------------------------------------- epilogue
    const int set = (warp - 4) >> 2, q = warp & 3;   // TMEM lanes 32 q .. 32 q + 31
    const int ts = q >> 1;                           // target slot of this warp
    const int o = 32 * (q & 1) + lane, yo = o >> 3, xo = o & 7;   // output token 8 y + x
    const bool valid = yo < a.th && xo < a.tw, four = a.th >= 4 * (q & 1) + 4;   // four rows of the tile are this warp's
    uint8_t* out0 = s_out + (warp - 4) * 2 * kTbOut;   // two tiles, row yo & 3 at 1 KB each
    const int doff = (yo & 3) * 1024 + xo * 128;
    int n = 0;
    bool ok = true;
    for (Unit x = first_unit(n_part, n_item); ok && x.tile < a.n_tile; next_unit(x, a.bl_step, n_part, n_item)) {
      const TileGeom g = any_tile(a, x.tile);
      const bool mine = ts < a.grp_nt[x.item];
      const int frame = mine ? a.target_frame[a.grp_t0[x.item] + ts] : 0, y0 = g.y0 + 4 * (q & 1);
      for (int c = c0_of(x), c1 = c1_of(x); c < c1; ++c, ++n) {
        if ((n & 1) != set) continue;
        if (!__all_sync(0xffffffffu, wait(&b_dfull[set], (uint32_t)(n >> 1) & 1u))) { ok = false; break; }
        tc_fence_after();
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(kTbD + set * 128);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          // 64 channels (one 128-byte box) at a time
          uint32_t r[64];
          tmem_ld_x64(ta + 64 * half, r);
          if (half == 1) {   // the whole buffer is in registers: it goes back to the issuer
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&b_dempty[set]);
          }
          uint32_t pk[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1]));
            pk[e] = *reinterpret_cast<const uint32_t*>(&b2);
          }
          uint8_t* out = out0 + half * kTbOut;
          if (lane == 0) bulk_wait_read_1();   // the store before the last has read this tile
          __syncwarp();
          if (mine && valid)
#pragma unroll
            for (int c8 = 0; c8 < 8; ++c8)
              *reinterpret_cast<uint4*>(out + doff + ((c8 ^ xo) << 4)) =
                  make_uint4(pk[4 * c8], pk[4 * c8 + 1], pk[4 * c8 + 2], pk[4 * c8 + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          const int ch = c * 128 + 64 * half;
          if (lane == 0) {
            if (mine && ch < a.C && four && boxed(a, g)) {   // four rows at once
              if (y0 < a.Hg && a.tw == 8) tma_store_4d(&tm_out, out, ch, g.x0, y0, frame);
              else if (y0 < a.Hg) tma_store_5d(&tm_out, out, ch, 0, g.x0 / a.tw, y0, frame);
            } else if (mine && ch < a.C) {   // the last rows of a tile, or a truncated column: one row at a time
              for (int yy = 4 * (q & 1); yy < min(a.th, 4 * (q & 1) + 4) && g.y0 + yy < a.Hg; ++yy)
                tma_store_4d(&tm_row, out + (yy & 3) * 1024, ch, g.x0, g.y0 + yy, frame);
            }
            bulk_commit();   // one group per half, also where nothing is stored
          }
        }
      }
    }
    if (lane == 0) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// 4-D map [F][Hg][Wg][C] with a 128-byte-swizzled box (64 bf16 channels, bw, bh, 1)
bool make_r_map_sw(CUtensorMap* m, const cast_par_args& a, int bw, int bh) {
  EncodeTiledFn fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.Wg, (cuuint64_t)a.Hg, (cuuint64_t)a.F};
  cuuint64_t strides[3] = {a.C * 2ull, (cuuint64_t)a.Wg * a.C * 2, (cuuint64_t)a.Hg * a.Wg * a.C * 2};
  cuuint32_t box[4] = {64, (cuuint32_t)bw, (cuuint32_t)bh, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, a.r, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 5-D map [F][Hg][complete tiles of a row][column of a tile][C] with a 128-byte-swizzled box (64 bf16
// channels, 8 columns, 1, bh, 1)
bool make_tile_map_sw(CUtensorMap* m, const cast_par_args& a, int bh) {
  EncodeTiledFn fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t tw = (cuuint64_t)a.params.tile_w, token = a.C * 2ull;
  cuuint64_t dims[5] = {(cuuint64_t)a.C, tw, (cuuint64_t)a.Wg / tw, (cuuint64_t)a.Hg, (cuuint64_t)a.F};
  cuuint64_t strides[4] = {token, tw * token, a.Wg * token, (cuuint64_t)a.Hg * a.Wg * token};
  cuuint32_t box[5] = {64, 8, 1, (cuuint32_t)bh, 1};
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, a.r, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// f32 4-D map [F][Hg][Wg][C], box (cc channels, tw, th, 1), zero fill out of range
bool make_r_map(CUtensorMap* m, const cast_par_args& a, int cc) {
  EncodeTiledFn fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t elt = 4;
  cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.Wg, (cuuint64_t)a.Hg, (cuuint64_t)a.F};
  cuuint64_t strides[3] = {a.C * elt, (cuuint64_t)a.Wg * a.C * elt, (cuuint64_t)a.Hg * a.Wg * a.C * elt};
  cuuint32_t box[4] = {(cuuint32_t)cc, (cuuint32_t)a.params.tile_w, (cuuint32_t)a.params.tile_h, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.r, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16: two launches over every tile, each a programmatic dependent of the launch before it on the
// stream (behind one of this library's, the statistics kernel sets itself up and builds its operand
// while that one ends).
cast_status launch_tc(const CUtensorMap& tm_box, const CUtensorMap& tm_row, const CUtensorMap& tm_out, ParKArgs& k,
                      cudaStream_t st) {
  static std::atomic<uint64_t> attr_done{0};
  if (!once_per_device(attr_done, [] {
        return cudaFuncSetAttribute(k_par_stats_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStSmem) ==
                   cudaSuccess &&
               cudaFuncSetAttribute(k_par_stats_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStSmem) ==
                   cudaSuccess &&
               cudaFuncSetAttribute(k_par_blend_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTbSmem) ==
                   cudaSuccess;
      }))
    return check_launch("PAR kernel attributes");
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  const auto grid_of = [&](int n_part, int n_item, Unit& step) {   // CTAs, and their stride over the units
    const int n = (int)std::min<int64_t>((int64_t)k.n_tile * n_part * n_item, sm_count());
    step.item = n % n_item;
    step.part = n / n_item % n_part;
    step.tile = n / n_item / n_part;
    return dim3(n, 1, 1);
  };
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid_of(k.st_parts, k.n_act, k.st_step);
  cfg.blockDim = dim3(kStThreads, 1, 1);
  cfg.dynamicSmemBytes = kStSmem;
  cfg.stream = st;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k.wch ? k_par_stats_tc<true> : k_par_stats_tc<false>, tm_box, tm_row, k) != cudaSuccess)
    return check_launch("PAR statistics kernel");
  cudaLaunchConfig_t bc{};
  bc.gridDim = grid_of(k.bl_parts, k.n_grp, k.bl_step);
  bc.blockDim = dim3(kTbThreads, 1, 1);
  bc.dynamicSmemBytes = kTbSmem;
  bc.stream = st;
  bc.attrs = pdl;
  bc.numAttrs = 1;
  if (cudaLaunchKernelEx(&bc, k_par_blend_tc, tm_box, tm_row, tm_out, k) != cudaSuccess)
    return check_launch("PAR tensor-core blend kernel");
  return check_launch("PAR kernels");
}

// f32, one tile kind on one stream: K_stats, then K_transport and K_blend as programmatic dependents.
template <bool FULL>
cast_status launch_kind(const CUtensorMap& tm, const ParKArgs& k, int n_tiles, cudaStream_t st) {
  const size_t smem = par_dyn_smem(kCC);
  static std::atomic<uint64_t> attr_done{0};
  if (!once_per_device(attr_done, [smem] {
        return cudaFuncSetAttribute(k_par<kCC, FULL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem) == cudaSuccess &&
               cudaFuncSetAttribute(k_par<kCC, FULL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem) == cudaSuccess;
      }))
    return check_launch("PAR kernel attributes");
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(k.n_chunk, n_tiles * k.n_tseg, 1);
  cfg.blockDim = dim3(kCC, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (cudaLaunchKernelEx(&cfg, k_par<kCC, FULL, true>, tm, k) != cudaSuccess)
    return check_launch("PAR statistics kernel");
  cudaLaunchConfig_t tc{};
  tc.gridDim = dim3(n_tiles, k.n_anchor - 1, 1);
  tc.blockDim = dim3(128, 1, 1);
  tc.stream = st;
  tc.attrs = pdl;
  tc.numAttrs = 1;
  if (cudaLaunchKernelEx(&tc, k_par_transport<FULL>, k) != cudaSuccess)
    return check_launch("PAR transport kernel");
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_par<kCC, FULL, false>, tm, k) != cudaSuccess)
    return check_launch("PAR blend kernel");
  return check_launch("PAR kernels");
}

// Side streams for the edge-tile launches, each with the events that fork it from and join it back
// into a caller's stream.  A call takes one for itself until it has joined it (another caller's record
// between this call's record and wait would make the edge tiles wait for the wrong stream) and passes
// over those that a capture still holds, except its own capture's.  At most kMaxForks per device are
// made, on demand, and kept; a call that finds none runs both kinds on its own stream.
// (Both kinds in one launch need no second stream, but the 8x8 tiles run slower beside the other path's
// code: PAR sweep 205 -> 224 us, one tile of 128 channels 15 -> 21 us.)
constexpr int kMaxForks = 16;
struct ForkStream {
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};
struct ForkPool {
  std::mutex mu;
  ForkStream idle[kMaxForks];
  int n_idle = 0, n_made = 0;
};
class ForkLease {
 public:
  explicit ForkLease(cudaStream_t st) {
    static ForkPool pools[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    unsigned long long cid = 0;
    if (!capture_of(st, cs, cid)) return;
    ForkPool& p = pools[dev];
    std::lock_guard<std::mutex> lock(p.mu);
    for (int i = p.n_idle - 1; i >= 0; --i) {
      cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
      unsigned long long id = 0;
      if (!capture_of(p.idle[i].side, s, id)) continue;
      if (s != cudaStreamCaptureStatusNone && !(s == cs && id == cid)) continue;
      f_ = p.idle[i];
      p.idle[i] = p.idle[--p.n_idle];
      pool_ = &p;
      return;
    }
    if (p.n_made == kMaxForks) return;
    // (creating a stream takes no part in a capture that is open)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (cudaStreamCreateWithFlags(&f_.side, cudaStreamNonBlocking) == cudaSuccess &&
        cudaEventCreateWithFlags(&f_.fork, cudaEventDisableTiming) == cudaSuccess &&
        cudaEventCreateWithFlags(&f_.join, cudaEventDisableTiming) == cudaSuccess) {
      ++p.n_made;
      pool_ = &p;
    } else {
      if (f_.fork) cudaEventDestroy(f_.fork);
      if (f_.side) cudaStreamDestroy(f_.side);
      cudaGetLastError();   // (the call goes on without a side stream)
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
  ~ForkLease() {
    if (!pool_) return;
    std::lock_guard<std::mutex> lock(pool_->mu);
    pool_->idle[pool_->n_idle++] = f_;
  }
  ForkLease(const ForkLease&) = delete;
  ForkLease& operator=(const ForkLease&) = delete;
  explicit operator bool() const { return pool_ != nullptr; }
  const ForkStream& operator*() const { return f_; }

 private:
  static bool capture_of(cudaStream_t st, cudaStreamCaptureStatus& status, unsigned long long& id) {
    if (cudaStreamGetCaptureInfo(st, &status, &id) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  ForkPool* pool_ = nullptr;
  ForkStream f_;
};

// Time segments of consecutive anchor pairs (pairs 1 .. n_anchor-1), as even as possible.
ParKArgs with_segments(const ParKArgs& k0, int nseg) {
  ParKArgs k = k0;
  const int npair = k.n_anchor - 1;
  k.n_tseg = nseg;
  int pair = 1;
  for (int sg = 0; sg < nseg; ++sg) {
    const int left = npair - (pair - 1), segs_left = nseg - sg;
    const int take = (left + segs_left - 1) / segs_left;
    k.seg_pair0[sg] = pair;
    k.seg_pair1[sg] = pair + take - 1;
    pair += take;
  }
  return k;
}

cast_status launch_f32(const CUtensorMap& tm, const ParKArgs& k0, const ParPlan& p, cudaStream_t st) {
  ParKArgs kf = with_segments(k0, p.n_tseg_full), ke = with_segments(k0, p.n_tseg_edge);
  kf.tile_base = 0;
  ke.tile_base = p.n_full;
  if (p.n_edge == 0) return launch_kind<true>(tm, kf, p.n_full, st);
  if (p.n_full == 0) return launch_kind<false>(tm, ke, p.n_edge, st);
  ForkLease fork(st);
  if (!fork) {
    const cast_status s = launch_kind<false>(tm, ke, p.n_edge, st);
    return s != CAST_OK ? s : launch_kind<true>(tm, kf, p.n_full, st);
  }
  // full tiles on the caller's stream, edge tiles concurrently on the side stream
  const ForkStream& f = *fork;
  if (cudaEventRecord(f.fork, st) != cudaSuccess || cudaStreamWaitEvent(f.side, f.fork, 0) != cudaSuccess)
    return check_launch("PAR fork");
  const cast_status se = launch_kind<false>(tm, ke, p.n_edge, f.side);
  const cast_status sf = se != CAST_OK ? se : launch_kind<true>(tm, kf, p.n_full, st);
  // (also after a failed launch: what is already on the side stream belongs to the caller's)
  if (cudaEventRecord(f.join, f.side) != cudaSuccess || cudaStreamWaitEvent(st, f.join, 0) != cudaSuccess)
    return sf != CAST_OK ? sf : check_launch("PAR join");
  return sf;
}

}  // namespace

ParPlan par_plan(const cast_par_args& a) {
  ParPlan p{};
  int na = 0;
  for (int f = 0; f < a.F; ++f) na += a.anchor_mask[f] ? 1 : 0;
  p.n_anchor = na;
  p.n_pair = na > 0 ? na - 1 : 0;
  p.n_target = a.F - na;
  const int th = a.params.tile_h, tw = a.params.tile_w;
  p.tiles_y = (a.Hg + th - 1) / th;
  p.tiles_x = (a.Wg + tw - 1) / tw;
  p.n_tile = p.tiles_y * p.tiles_x;
  // 8x8 tiles take the specialised kernel; with smaller tile sides every tile is an edge tile
  if (th == 8 && tw == 8) {
    p.n_full = (a.Hg / 8) * (a.Wg / 8);
    p.n_edge = p.n_tile - p.n_full;
  } else {
    p.n_full = 0;
    p.n_edge = p.n_tile;
  }
  // channel chunks of kCC channels, one CTA each
  p.chunk = kCC;
  p.n_chunk = (a.C + kCC - 1) / kCC;
  // time segments: split the anchor pairs so that the CTAs of a kind cover the SMs about
  // two deep for full tiles and four deep for the (fewer, longer-running) edge tiles, which
  // run concurrently on the side stream; each segment re-reads its first anchor.  Measured at
  // the Matrix-Game size (3 pairs: full tiles 2 segments, 0.049 ms against 0.053 ms with 3)
  // and the PAR sweep (edge tiles 3 segments, 2 % faster than 2).
  const int nsm = sm_count();
  auto segs = [&](int n_tiles, int depth) {
    const int want_ctas = depth * nsm;
    const int per_seg = n_tiles * p.n_chunk;
    int nseg = per_seg > 0 ? (want_ctas + per_seg - 1) / per_seg : 1;
    if (nseg > p.n_pair) nseg = p.n_pair;
    return nseg < 1 ? 1 : nseg;
  };
  p.n_tseg_full = segs(p.n_full, 2);
  p.n_tseg_edge = segs(p.n_edge, 4);
  // workspace: the chunk records [tile][pair][chunk][kRec] and, f32, theta and g [tile][pair][2][kNB]
  p.rec_bytes = align_up((size_t)p.n_tile * (na > 0 ? na : 1) * p.n_chunk * kRec * sizeof(float));
  p.trans_bytes = a.dtype == CAST_F32 ? align_up((size_t)p.n_tile * (na > 0 ? na : 1) * 2 * kNB * sizeof(float)) : 0;
  p.total_bytes = p.n_target > 0 ? p.rec_bytes + p.trans_bytes : 0;
  return p;
}

namespace {
struct FastSrc {
  signed char v[kNV];
};
FastSrc make_fast_src() {
  FastSrc f{};
  // record entry t = 3 * bin + comp of an 8x8 tile from the 96 reduced values (+ W at DC = 96)
  int pos[40 * 4];
  for (int q = 0; q < 160; ++q) pos[q] = -1;
  for (int n = 0; n < 96; ++n) pos[fast_value(n)] = n;
  for (int t = 0; t < kNV; ++t) {
    const int b = t / 3, comp = t % 3, ky = b / 5, kx = b % 5;
    const bool edge = kx == 0 || kx == 4;
    const bool selfc = edge && (ky == 0 || ky == 4);
    const bool mirror = edge && !selfc && ky > 4;
    const int r = mirror ? (8 - ky) * 5 + kx : b;
    int src = 0;
    if (r == 0) src = comp == 2 ? 96 + 1 : 0;                 // DC: only W
    else if (comp == 1 && selfc) src = 0;                     // Im Z of a real bin
    else src = (pos[r * 4 + comp] + 1) * ((mirror && comp == 1) ? -1 : 1);
    f.v[t] = (signed char)src;
  }
  return f;
}
}  // namespace

cast_status launch_par(const cast_par_args& a, void* ws, cudaStream_t st, bool after_own) {
  const ParPlan p = par_plan(a);
  if (p.n_target == 0) return CAST_OK;   // every frame is an anchor: reconstruction bypassed
  ParKArgs k{};
  k.r = static_cast<char*>(a.r);
  k.wch = a.channel_weight;
  k.F = a.F;
  k.Hg = a.Hg;
  k.Wg = a.Wg;
  k.C = a.C;
  k.th = a.params.tile_h;
  k.tw = a.params.tile_w;
  k.tiles_x = p.tiles_x;
  k.tiles_y = p.tiles_y;
  k.n_tile = p.n_tile;
  k.n_chunk = p.n_chunk;
  k.rec = static_cast<float*>(ws);
  k.trans = reinterpret_cast<float*>(static_cast<char*>(ws) + p.rec_bytes);
  int anchors[CAST_MAX_FRAMES];
  int na = 0;
  for (int f = 0; f < a.F; ++f)
    if (a.anchor_mask[f]) anchors[na++] = f;
  k.n_anchor = na;
  for (int j = 0; j < na; ++j) k.anchor_frame[j] = anchors[j];
  // targets grouped by pair j (anchors j-1, j), j = 1..na-1 (Eq. block)
  int nt = 0;
  for (int j = 0; j <= na; ++j) k.pair_tbeg[j] = 0;
  for (int j = 1; j < na; ++j) {
    k.pair_tbeg[j] = nt;
    const int a0 = anchors[j - 1], a1 = anchors[j];
    auto add = [&](int t) {
      k.target_frame[nt] = t;
      k.target_alpha[nt] = (float)((double)(t - a0) / (double)(a1 - a0));
      ++nt;
    };
    if (j == 1)
      for (int t = 0; t < a0; ++t) add(t);
    for (int t = a0 + 1; t < a1; ++t) add(t);
    if (j == na - 1)
      for (int t = a1 + 1; t < a.F; ++t) add(t);
  }
  k.pair_tbeg[na] = nt;
  const cast_par_params& pp = a.params;
  k.tau_low = pp.tau_low;
  k.tau_high = pp.tau_high;
  k.q = pp.q;
  k.T = pp.T;
  k.eps = pp.eps;
  k.eta_rel = pp.eta_rel;
  k.eta_abs = pp.eta_abs;
  k.band = pp.band_radius;
  k.gate_mode = pp.gate_mode;
  k.wait_ns = 2000000000ull;
  static const FastSrc fast_src = make_fast_src();
  std::copy(fast_src.v, fast_src.v + kNV, k.fast_src);

  if (a.dtype == CAST_BF16) {
    k.whole_y = a.Hg / k.th;
    k.whole_x = a.Wg / k.tw;
    for (int q = 0; q < 4; ++q) {
      const int h = (q & 2) ? a.Hg % k.th : k.th, w = (q & 1) ? a.Wg % k.tw : k.tw;
      if (h > 0 && w > 0) make_slots(h, w, k.bin_slot[q], k.slot_bin[q]);
    }
    k.after_own = after_own ? 1 : 0;
    for (int j = 1; j < na; ++j) {
      if (k.pair_tbeg[j + 1] > k.pair_tbeg[j]) k.act_pair[k.n_act++] = (unsigned char)j;
      for (int t = k.pair_tbeg[j]; t < k.pair_tbeg[j + 1]; t += 2, ++k.n_grp) {
        k.grp_pair[k.n_grp] = (unsigned char)j;
        k.grp_t0[k.n_grp] = (short)t;
        k.grp_nt[k.n_grp] = (unsigned char)std::min(2, k.pair_tbeg[j + 1] - t);
      }
    }
    // The range of chunks a unit takes.  CTAs stride the units (contiguous ranges of units per CTA
    // lose the anchors' reuse in L2: HY-World-shaped 109 -> 123 us); a unit takes its chunks
    // and what does not overlap with the neighbours' work, and the first one `start` more (all in
    // chunks): the statistics' reduction takes about one chunk (1,100 cycles) and their start four
    // (6,000 cycles until the first products: the DFT operand); a unit of the blend counts as at least
    // six (3, 4 or 5 give the HY-World-shaped call 124 / 107 / 108 us and one with 8 anchors 141 / 142 /
    // 140, six 107 and 132) and the first one eight.
    const int nsm = sm_count();
    auto split = [&](int64_t units, int extra, int least, int start, int& parts, int& cpp) {
      int64_t best = -1;
      for (int q = 1; q <= p.n_chunk; ++q) {
        const int c = (p.n_chunk + q - 1) / q;
        if ((p.n_chunk + c - 1) / c != q) continue;   // the same ranges as with fewer parts
        const int64_t n = (units * q + nsm - 1) / nsm;
        const int64_t cost = start + (n - 1) * std::max(c + extra, least) + c + extra;
        if (best < 0 || cost < best) {
          best = cost;
          parts = q;
          cpp = c;
        }
      }
    };
    split((int64_t)p.n_tile * k.n_act, 1, 0, 4, k.st_parts, k.st_cpp);
    split((int64_t)p.n_tile * k.n_grp, 0, 6, 8, k.bl_parts, k.bl_cpp);
    CUtensorMap tm_box, tm_row, tm_out;
    bool ok = make_r_map_sw(&tm_row, a, k.tw, 1);
    if (k.tw == 8) {
      ok = ok && make_r_map_sw(&tm_box, a, 8, k.th) && make_r_map_sw(&tm_out, a, 8, 4);
    } else if (a.Wg >= k.tw) {
      ok = ok && make_tile_map_sw(&tm_box, a, k.th) && make_tile_map_sw(&tm_out, a, 4);
    } else {   // no complete tile in a row: everything row by row
      tm_box = tm_out = tm_row;
    }
    if (!ok) return fail(CAST_ERR_CUDA, "PAR: cuTensorMapEncodeTiled failed");
    return launch_tc(tm_box, tm_row, tm_out, k, st);
  }
  CUtensorMap tm;
  if (!make_r_map(&tm, a, p.chunk)) return fail(CAST_ERR_CUDA, "PAR: cuTensorMapEncodeTiled failed");
  return launch_f32(tm, k, p, st);
}

unsigned int par_error_word(cudaStream_t st, bool clear) {
  unsigned int v = 0;
  cudaMemcpyFromSymbolAsync(&v, g_par_error, sizeof(v), 0, cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  if (clear && v) {
    const unsigned int z = 0;
    cudaMemcpyToSymbolAsync(g_par_error, &z, sizeof(z), 0, cudaMemcpyHostToDevice, st);
    cudaStreamSynchronize(st);
  }
  return v;
}

}  // namespace cast
