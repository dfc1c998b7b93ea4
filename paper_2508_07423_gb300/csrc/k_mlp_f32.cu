// FP32 SIMT kernels of the embedding MLP and the interaction network.
//
// Row-tiled register products: a lane keeps rows x columns of a layer's output
// in registers, the input rows of its tile are staged in shared memory, and the
// inputs of an output element are added in increasing k order, two columns per
// packed FMA. The interaction-network kernels work per warp (WarpTile), the
// embedding per block of 256 threads.
//
//  k_embed_f32     embedding MLP (Sec. "Hit Embedding and Rough Graph
//                  Construction") on (r/s0, phi/s1, z/s2), ReLU between layers
//  k_gnn_f32<MODE> node encoder on (x/s3, y/s4, z/s5); edge encoder on
//                  [h_src, h_dst]; node step: m = [sum_out e, sum_in e]
//                  (Eq. of m^k_l), h <- h + N_k([h, m]); edge step:
//                  e <- e + E_k([e, h_src, h_dst]) with the updated h, and at
//                  the last step the classifier and the cut (Sec. "Graph Neural
//                  Network and Classifiers"). Sub-networks are
//                  Linear -> LayerNorm -> ReLU -> Linear.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "internal.cuh"
#include "msg.cuh"
#include "tc_ptx.cuh"

namespace gnntrk {

int device_sms();

namespace {

constexpr int kThreads = 256;                      // embedding kernel
constexpr int kRowGroups = 32;                     // lanes of a warp
constexpr int kColGroups = kThreads / kRowGroups;  // warps of the embedding block

// Interaction network: every warp owns whole rows. Lane (rg = lane / 8,
// cg = lane % 8) holds RM rows (rg + 4 i) x CW columns (32 c + 4 cg + u) of a
// layer's output in registers; a warp covers WR = 4 RM rows and all H columns,
// so a row's LayerNorm is a reduction over the 8 lanes of its row group and no
// block-wide barrier is needed. A lane's part of a reduction is summed in
// column order and the 8 parts pairwise (0+1, 2+3, ... first), so the result
// does not depend on RM: every tile height gives the same bits. Inputs are
// staged row-major in the warp's own shared-memory slice with a row stride of
// H + 4 floats: the four rows a warp reads at one k fall in distinct bank
// quads, and the eight lanes of a row group read the same address (broadcast).
template <int H_, int RM_>
struct WarpTile {
  static constexpr int H = H_, RM = RM_;
  static constexpr int CW = H / 8;   // columns per lane
  static constexpr int RG = 4;       // row groups
  static constexpr int WR = RG * RM; // rows per warp
  static constexpr int NJ = H / 32;  // float4 column chunks per lane
  static constexpr int LDH = H + 4;  // row stride of staged rows (floats)
};

// Variant chosen per (hidden index, kernel family: 0 encoders, 1 node step,
// 2 edge step and classifier); set by the autotuner, process wide.
std::atomic<int> g_f32_variant[3][3] = {};

enum GMode : int { G_NODE_ENC = 0, G_EDGE_ENC = 1, G_NODE_UPD = 2, G_EDGE_UPD = 3,
                   G_EDGE_UPD_CLS = 4, G_CLS = 5, G_TRIP = 6 };

__device__ __forceinline__ bool input_bad(const Ws& w) {
  return (*(volatile int32_t*)&w.counters[C_STATUS] & ST_INPUT) != 0;
}

// first column of a lane's chunk c
__device__ __forceinline__ int col_of(int c, int cg) { return 32 * c + 4 * cg; }

// acc[i][4c+u] (+)= sum_{k < KV} A[rg + RG i][k] * W[k * ldo + col_of(c) + u], k ascending;
// A row-major with stride LDA (K a multiple of 4, KV <= K valid); the weights
// in global memory, or (SW) in shared memory
template <class T, int K, int KV, int LDA, bool SW>
__device__ __forceinline__ void warp_product(const float* A, const float* W, int ldo, int rg, int cg,
                                             float (&acc)[T::RM][T::CW]) {
  constexpr int RM = T::RM, NC = T::NJ;
  const float* wp = W + 4 * cg;
#pragma unroll 2
  for (int k0 = 0; k0 < K; k0 += 4) {
    float4 a[RM];
#pragma unroll
    for (int i = 0; i < RM; ++i)
      a[i] = *reinterpret_cast<const float4*>(A + (rg + T::RG * i) * LDA + k0);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (KV < K && k0 + t >= KV) break;
      float4 q[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float* wc = wp + (k0 + t) * ldo + 32 * c;
        q[c] = SW ? *reinterpret_cast<const float4*>(wc) : __ldg(reinterpret_cast<const float4*>(wc));
      }
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const float av = t == 0 ? a[i].x : (t == 1 ? a[i].y : (t == 2 ? a[i].z : a[i].w));
        const float2 a2 = make_float2(av, av);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          // two columns per packed FMA (each lane rounds like fmaf)
          float2 c01 = __ffma2_rn(a2, make_float2(q[c].x, q[c].y),
                                  make_float2(acc[i][4 * c], acc[i][4 * c + 1]));
          float2 c23 = __ffma2_rn(a2, make_float2(q[c].z, q[c].w),
                                  make_float2(acc[i][4 * c + 2], acc[i][4 * c + 3]));
          acc[i][4 * c] = c01.x;
          acc[i][4 * c + 1] = c01.y;
          acc[i][4 * c + 2] = c23.x;
          acc[i][4 * c + 3] = c23.y;
        }
      }
    }
  }
}

template <class T>
__device__ __forceinline__ void acc_bias(const float* b, int cg, float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int c = 0; c < T::NJ; ++c) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(b + col_of(c, cg)));
#pragma unroll
    for (int i = 0; i < T::RM; ++i) {
      acc[i][4 * c] = v.x;
      acc[i][4 * c + 1] = v.y;
      acc[i][4 * c + 2] = v.z;
      acc[i][4 * c + 3] = v.w;
    }
  }
}

// acc += S[rg + RG i][col] (each lane reads only its own elements)
template <class T>
__device__ __forceinline__ void acc_add_smem(const float* S, int rg, int cg,
                                             float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int i = 0; i < T::RM; ++i)
#pragma unroll
    for (int c = 0; c < T::NJ; ++c) {
      const float4 v =
          *reinterpret_cast<const float4*>(S + (rg + T::RG * i) * T::LDH + col_of(c, cg));
      acc[i][4 * c] += v.x;
      acc[i][4 * c + 1] += v.y;
      acc[i][4 * c + 2] += v.z;
      acc[i][4 * c + 3] += v.w;
    }
}

// acc += X[rows[r]][offx + col] (TWO: + Y[rows2[r]][offy + col], the two added
// first), straight from global memory (missing rows read row 0; their result
// is dropped)
template <class T, bool TWO>
__device__ __forceinline__ void acc_add_rows(const int* rows, const float* X, int64_t ldx,
                                             const int* rows2, const float* Y, int64_t ldy,
                                             int rg, int cg, float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int i = 0; i < T::RM; ++i) {
    const int r = rg + T::RG * i;
    const float* x = X + size_t(max(rows[r], 0)) * ldx;
    const float* y = TWO ? Y + size_t(max(rows2[r], 0)) * ldy : nullptr;
#pragma unroll
    for (int c = 0; c < T::NJ; ++c) {
      float4 v = __ldcg(reinterpret_cast<const float4*>(x + col_of(c, cg)));
      if constexpr (TWO) {
        const float4 u = __ldcg(reinterpret_cast<const float4*>(y + col_of(c, cg)));
        v.x += u.x;
        v.y += u.y;
        v.z += u.z;
        v.w += u.w;
      }
      acc[i][4 * c] += v.x;
      acc[i][4 * c + 1] += v.y;
      acc[i][4 * c + 2] += v.z;
      acc[i][4 * c + 3] += v.w;
    }
  }
}

template <class T>
__device__ __forceinline__ void acc_store_smem(float* S, int rg, int cg,
                                               const float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int i = 0; i < T::RM; ++i)
#pragma unroll
    for (int c = 0; c < T::NJ; ++c)
      *reinterpret_cast<float4*>(S + (rg + T::RG * i) * T::LDH + col_of(c, cg)) =
          make_float4(acc[i][4 * c], acc[i][4 * c + 1], acc[i][4 * c + 2], acc[i][4 * c + 3]);
}

// rows of the warp to global: dst[rows[r] * ld + off + col] (rows < 0 skipped)
template <class T>
__device__ __forceinline__ void acc_store_rows(float* dst, int64_t ld, int off, const int* rows,
                                               int rg, int cg, const float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int i = 0; i < T::RM; ++i) {
    const int row = rows[rg + T::RG * i];
    if (row < 0) continue;
    float* d = dst + size_t(row) * ld + off;
#pragma unroll
    for (int c = 0; c < T::NJ; ++c)
      *reinterpret_cast<float4*>(d + col_of(c, cg)) =
          make_float4(acc[i][4 * c], acc[i][4 * c + 1], acc[i][4 * c + 2], acc[i][4 * c + 3]);
  }
}

// Sums over the 8 lanes of a row group for every row: part[i] is this lane's
// part of row i; pairwise, by a butterfly that hands half of the remaining rows
// to the other lane of each pair, so that the work after the sum (a division, a
// square root) runs once per row and not in all 8 lanes: with 8 rows per lane
// LayerNorm takes 2.7 k cycles per tile instead of 6.2 k (hidden 64). tot[j] is
// the sum of row row_of<T>(j, cg) (with fewer rows than lanes several lanes
// hold the same row).
template <class T>
struct RowSums {
  static constexpr int M = T::RM < 8 ? T::RM : 8;  // lanes that hold distinct rows
  static constexpr int N = T::RM / M;              // rows per lane
  static_assert(T::RM % M == 0 && (M & (M - 1)) == 0, "whole butterflies");
};

template <class T>
__device__ __forceinline__ int row_of(int j, int cg) {
  return j * RowSums<T>::M + (cg & (RowSums<T>::M - 1));
}

template <class T>
__device__ __forceinline__ void row_sums(const float (&part)[T::RM], int cg,
                                         float (&tot)[RowSums<T>::N]) {
  float v[T::RM];
#pragma unroll
  for (int i = 0; i < T::RM; ++i) v[i] = part[i];
  int n = T::RM;
#pragma unroll
  for (int o = 1; o < 8; o *= 2) {
    if (n > RowSums<T>::N) {
      const bool up = (cg & o) != 0;
#pragma unroll
      for (int j = 0; j < T::RM / 2; ++j) {
        if (2 * j >= n) break;
        const float keep = up ? v[2 * j + 1] : v[2 * j], send = up ? v[2 * j] : v[2 * j + 1];
        v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
      n /= 2;
    } else {
#pragma unroll
      for (int j = 0; j < RowSums<T>::N; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
    }
  }
#pragma unroll
  for (int j = 0; j < RowSums<T>::N; ++j) tot[j] = v[j];
}

// the value that row_sums' owner of row i holds, in every lane of the row group
template <class T>
__device__ __forceinline__ float row_value(const float (&own)[RowSums<T>::N], int i, int lane) {
  constexpr int M = RowSums<T>::M;
  return __shfl_sync(0xffffffffu, own[i / M], (lane & ~(M - 1)) | (i % M));
}

// per row: ReLU((v - mean) / sqrt(var + eps)) over the H columns
template <class T>
__device__ __forceinline__ void acc_ln_relu(float (&acc)[T::RM][T::CW], int lane) {
  constexpr int CW = T::CW, RM = T::RM, H = T::H, N = RowSums<T>::N;
  const int cg = lane & 7;
  float part[RM], mean[N], inv[N];
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    part[i] = 0.f;
#pragma unroll
    for (int c = 0; c < CW; ++c) part[i] += acc[i][c];
  }
  row_sums<T>(part, cg, mean);
#pragma unroll
  for (int j = 0; j < N; ++j) mean[j] /= float(H);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const float m = row_value<T>(mean, i, lane);
    part[i] = 0.f;
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      acc[i][c] -= m;
      part[i] = fmaf(acc[i][c], acc[i][c], part[i]);
    }
  }
  row_sums<T>(part, cg, inv);
#pragma unroll
  for (int j = 0; j < N; ++j) inv[j] = 1.0f / sqrtf(inv[j] / float(H) + kLnEps);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const float r = row_value<T>(inv, i, lane);
#pragma unroll
    for (int c = 0; c < CW; ++c) acc[i][c] = fmaxf(acc[i][c] * r, 0.f);
  }
}

// bias + dot product of every row (after LayerNorm and ReLU) with the 1-unit
// layer L: out[j] is row row_of<T>(j, cg)'s
template <class T>
__device__ __forceinline__ void row_dots(const float (&acc)[T::RM][T::CW], const LayerF32& L, int cg,
                                         float (&out)[RowSums<T>::N]) {
  float part[T::RM];
#pragma unroll
  for (int i = 0; i < T::RM; ++i) part[i] = 0.f;
#pragma unroll
  for (int c = 0; c < T::NJ; ++c)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float wv = __ldg(L.WT + size_t(col_of(c, cg) + u) * L.ldo);
#pragma unroll
      for (int i = 0; i < T::RM; ++i) part[i] = fmaf(acc[i][4 * c + u], wv, part[i]);
    }
  row_sums<T>(part, cg, out);
#pragma unroll
  for (int j = 0; j < RowSums<T>::N; ++j) out[j] = L.b[0] + out[j];
}

// S[r][col] = X[rows[r]][offx + col] (+ Y[rows2[r]][offy + col]), zero for rows < 0;
// 8 lanes per row, one float4 column chunk each, four rows per instruction.
// Loads are unconditional (row 0 stands in for a missing row, its value is
// then dropped) so that a lane's loads (up to 16 at a time) are in flight
// together.
template <class T, bool TWO>
__device__ __forceinline__ void stage_rows(float* S, const int* rows, const float* X, int64_t ldx,
                                           int offx, const int* rows2, const float* Y,
                                           int64_t ldy, int offy, int lane) {
  constexpr int NR = T::WR / 4, NJ = T::NJ, LD = T::LDH;
  constexpr int G = NR * NJ <= 16 ? NR : 16 / NJ;  // rows per lane and batch of loads
  static_assert(NR % G == 0, "whole batches");
  const int gr = lane >> 3, q = lane & 7;
#pragma unroll 1
  for (int i0 = 0; i0 < NR; i0 += G) {
    float4 v[G][NJ];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const int row = rows[gr + 4 * (i0 + i)];
      const int rx = max(row, 0);
      const int ry = TWO ? (row >= 0 ? rows2[gr + 4 * (i0 + i)] : 0) : 0;
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        v[i][j] = __ldcg(reinterpret_cast<const float4*>(X + size_t(rx) * ldx + offx + 32 * j + 4 * q));
        if (TWO) {
          const float4 y =
              __ldcg(reinterpret_cast<const float4*>(Y + size_t(ry) * ldy + offy + 32 * j + 4 * q));
          v[i][j].x += y.x;
          v[i][j].y += y.y;
          v[i][j].z += y.z;
          v[i][j].w += y.w;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const int r = gr + 4 * (i0 + i);
      const bool ok = rows[r] >= 0;
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        *reinterpret_cast<float4*>(S + r * LD + 32 * j + 4 * q) =
            ok ? v[i][j] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}

// ---------------------------------------------------------------------------
// interaction network, one kernel per mode
// ---------------------------------------------------------------------------
struct GnnArgs {
  Batch b;
  Ws w;
  EdgeProj proj;  // node kernels: projections for the next edge layer
  Mlp2F32 m;    // the sub-network of this kernel
  Mlp2F32 cls;  // classifier (G_EDGE_UPD_CLS, G_CLS)
  float fs[6];
  float cut;
  int rescore_only;
  float band_lo, band_hi;
  Sel sel;
  // G_TRIP: one triplet list (its two edges, count on the device) and outputs
  const int32_t* t1;
  const int32_t* t2;
  const int32_t* tn;
  float* tlogit;
  uint8_t* tkeep;
  int short_rounds;  // see k_gnn_f32
};

__host__ __device__ constexpr bool g_edge_rows(int mode) {
  return mode != G_NODE_ENC && mode != G_NODE_UPD;
}

// matrix m (H rows, row stride ldo = H) of a tile's layer sequence
template <int MODE>
__device__ __forceinline__ const float* layer_mat(const GnnArgs& p, int m) {
  if constexpr (MODE == G_NODE_ENC) return m == 0 ? p.m.l2.WT : m == 1 ? p.proj.src.WT : p.proj.dst.WT;
  if constexpr (MODE == G_NODE_UPD)
    return m < 3 ? p.m.l1.WT + size_t(m) * p.m.l2.in * p.m.l1.ldo
                 : m == 3 ? p.m.l2.WT : m == 4 ? p.proj.src.WT : p.proj.dst.WT;
  if constexpr (MODE == G_EDGE_ENC) return p.m.l2.WT;
  if constexpr (MODE == G_CLS) return p.cls.l1.WT;
  if constexpr (MODE == G_TRIP) return p.m.l1.WT + size_t(m) * p.m.l1.out * p.m.l1.ldo;
  return m == 0 ? p.m.l1.WT : m == 1 ? p.m.l2.WT : p.cls.l1.WT;
}

// Where a kernel reads its layer weights: copies of the whole matrices in shared
// memory (hidden 32 and 64), or a ring of chunks in shared memory that bulk
// copies refill as the block's warps walk through the layers (hidden 128, whose
// matrices do not fit).
enum Weights : int { W_BLOCK = 1, W_RING = 2 };

// The H x H matrices of a kernel (MATS of them, in the order its layers use
// them) and the shared memory their source takes.
template <int H, int MATS_, int WEIGHTS>
struct WeightSource {
  static constexpr int MATS = MATS_;
  static constexpr bool COPIES = WEIGHTS == W_BLOCK, RING = WEIGHTS == W_RING;
  // ring: KC rows of a matrix per chunk, NST chunks
  static constexpr int KC = 16, NST = 4;
  // copies with their barrier, or chunks with their barriers and counts
  static constexpr int FLOATS = COPIES ? MATS * H * H + 4 : NST * KC * H + 4 * NST;
};

// Shape of one kernel: a tall and a short warp tile, warps per block (one block
// per SM: fewer, larger blocks measured faster at the same number of warps,
// the layer weights being there once) and the source of the weights.
//
// A warp's row buffer holds one tall tile: its input segments pass through the
// buffer in turn, the residual row is read again and the projected rows are
// added straight from global memory, which leaves room for 12-20 warps of tall
// tiles. Short tiles are for calls of few rows: more warps share the rows, and
// every input segment has a buffer of its own, so that all gathers are in
// flight at once. Every output element is the same sum in the same order in
// both.
template <int H_, int RM_, int RM_SHORT_, int MODE_, int NW_, int WEIGHTS_>
struct GnnShape {
  using Args = GnnArgs;
  using Tall = WarpTile<H_, RM_>;
  using Short = WarpTile<H_, RM_SHORT_>;
  static constexpr int H = H_, MODE = MODE_, NW = NW_;
  // input segments with a buffer of their own in a short tile
  static constexpr int SEGS = MODE == G_NODE_UPD ? 3 : MODE == G_NODE_ENC || MODE == G_CLS ? 1 : 2;
  static constexpr int ROWS = Tall::WR > SEGS * Short::WR ? Tall::WR : SEGS * Short::WR;
  // row buffers, features of the node encoder (8 floats per row), row ids
  static constexpr int FEATS = MODE == G_NODE_ENC ? 8 * Tall::WR : 0;
  static constexpr int IDS = Tall::WR * (g_edge_rows(MODE) ? 3 : 1);
  static constexpr int WARP_FLOATS = ROWS * Tall::LDH + FEATS + IDS;
  // H x H matrices a tile's layers use, in this order (layer_mat)
  static constexpr int MATS = MODE == G_NODE_ENC ? 3
                              : MODE == G_NODE_UPD ? 6
                              : MODE == G_EDGE_UPD || MODE == G_TRIP ? 2
                              : MODE == G_EDGE_UPD_CLS ? 3 : 1;
  using W = WeightSource<H, MATS, WEIGHTS_>;
  static constexpr size_t SMEM = (size_t(NW) * WARP_FLOATS + W::FLOATS) * 4;
  static __device__ __forceinline__ const float* mat(const Args& p, int m) {
    return layer_mat<MODE>(p, m);
  }
};

// The ring of weight chunks of one block: chunk g (g = 0, 1, ...) is rows
// [(g % CPL) KC, + KC) of matrix (g / CPL) % MATS and lies in stage g % NST;
// a stage's barrier completes when its bytes have landed, and the last of the
// `users` warps that have a tile to finish a chunk refills the stage with chunk
// g + NST. A wait that runs out (of chunk `late`) latches ST_TIMEOUT; the warp then
// waits no more and no longer counts as done with a chunk, so that no stage whose
// copy may still be in flight is refilled: of the chunks that it has not seen land,
// only late .. late + NST - 1 can have been asked for.
constexpr long long kRingWaitCycles = 4000000000LL;  // about 2 s

template <class X>
struct WeightRing {
  using W = typename X::W;
  static constexpr int STAGE = W::KC * X::H;  // floats per chunk
  static constexpr int CPL = X::H / W::KC;    // chunks per matrix
  float* buf;
  uint64_t* full;
  int* done;
  int g = 0, total = 0, users = 0;
  int late = -1;

  __device__ __forceinline__ void load(const typename X::Args& p, int c) {
    const int m = (c / CPL) % W::MATS, k = (c % CPL) * W::KC;
    uint64_t* f = full + c % W::NST;
    tc::mbar_expect_tx(f, STAGE * 4);
    tc::bulk_g2s(buf + (c % W::NST) * STAGE, X::mat(p, m) + size_t(k) * X::H, STAGE * 4, f);
  }
  __device__ __forceinline__ void init(float* smem) {  // (a block barrier follows)
    buf = smem;
    full = reinterpret_cast<uint64_t*>(smem + W::NST * STAGE);
    done = reinterpret_cast<int*>(full + W::NST);
    if (threadIdx.x == 0) {
      for (int s = 0; s < W::NST; ++s) {
        tc::mbar_init(full + s, 1);
        done[s] = 0;
      }
      tc::fence_mbar_init();
    }
  }
  // the block walks `tiles` tiles
  __device__ __forceinline__ void start(const typename X::Args& p, int tiles) {
    total = tiles * W::MATS * CPL;
    if (threadIdx.x == 0)
      for (int c = 0; c < W::NST && c < total; ++c) load(p, c);
  }
  // the next matrix of the sequence times the staged rows A
  template <class T>
  __device__ __forceinline__ void product(const typename X::Args& p, const float* A, int rg, int cg,
                                          float (&acc)[T::RM][T::CW]) {
#pragma unroll 1
    for (int c = 0; c < CPL; ++c) {
      const int st = g % W::NST;
      if (late < 0 && !tc::mbar_wait_bounded(full + st, (g / W::NST) & 1, kRingWaitCycles)) {
        late = g;
        set_status(p.w.counters, ST_TIMEOUT);
      }
      warp_product<T, W::KC, W::KC, T::LDH, true>(A + c * W::KC, buf + st * STAGE, X::H, rg, cg,
                                                  acc);
      __syncwarp();  // every lane is done with the chunk
      if ((threadIdx.x & 31) == 0 && late < 0 && g + W::NST < total) {
        __threadfence_block();
        if (atomicAdd(done + st, 1) == users - 1) {
          done[st] = 0;
          __threadfence_block();
          load(p, g + W::NST);
        }
      }
      ++g;
    }
  }
  // before the warp ends, after a wait that ran out: the copies that may be in flight
  __device__ __forceinline__ void drain() {
    if (late < 0 || (threadIdx.x & 31) != 0) return;
    for (int c = late; c < late + W::NST && c < total; ++c)
      tc::mbar_wait_bounded(full + c % W::NST, (c / W::NST) & 1, kRingWaitCycles / W::NST);
  }
};

// The weights a kernel multiplies by: matrix m of its layer sequence from the
// copies in shared memory, or from the ring (which serves the matrices of every
// tile in their order). One thread asks for the copies in bulk, and they land while
// the block waits for the kernel before it: copied by the block's threads they took
// longer than that wait in kernels of a few microseconds, which hold an SM each (one
// run-3 event, 18 such kernels: 417 -> 403 us per call alone, 253 -> 218 with eight
// handles on eight streams).
template <class X>
struct LayerWeights {
  using W = typename X::W;
  const typename X::Args& p;
  WeightRing<X> ring;
  const float* copies = nullptr;
  uint64_t* bar = nullptr;  // of the copies

  // block-wide, before pdl_wait (the weights are constant); smem: W::FLOATS floats
  __device__ __forceinline__ LayerWeights(const typename X::Args& a, float* smem) : p(a) {
    if constexpr (W::RING) ring.init(smem);
    if constexpr (W::COPIES) {
      constexpr int N = X::H * X::H;
      copies = smem;
      bar = reinterpret_cast<uint64_t*>(smem + W::MATS * N);
      if (threadIdx.x == 0) {
        tc::mbar_init(bar, 1);
        tc::fence_mbar_init();
        tc::mbar_expect_tx(bar, W::MATS * N * 4);
        for (int m = 0; m < W::MATS; ++m) tc::bulk_g2s(smem + m * N, X::mat(p, m), N * 4, bar);
      }
    }
    __syncthreads();
  }
  // block-wide, before the first use of the copies and before any return (no copy may
  // land after the block is gone); false: the wait ran out
  __device__ __forceinline__ bool landed() {
    if constexpr (W::COPIES) {
      if (__syncthreads_or(!tc::mbar_wait_bounded(bar, 0, kRingWaitCycles))) {
        if (threadIdx.x == 0) {
          set_status(p.w.counters, ST_TIMEOUT);
          tc::mbar_wait_bounded(bar, 0, kRingWaitCycles);
        }
        return false;
      }
    }
    return true;
  }
  // the block walks tiles of `step` rows (per block) from block0 on
  __device__ __forceinline__ void start(int block0, int step, int hi) {
    if constexpr (W::RING) ring.start(p, (hi - block0 + step - 1) / step);
  }
  // the block's round of tiles that begins at `first` (its warp 0's tile; the
  // warps' tiles are `stride` rows apart)
  __device__ __forceinline__ void round(int first, int stride, int hi) {
    if constexpr (W::RING) ring.users = min(X::NW, (hi - first + stride - 1) / stride);
  }
  // acc += A (staged rows) x matrix m
  template <class T>
  __device__ __forceinline__ void product(const float* A, int m, int rg, int cg,
                                          float (&acc)[T::RM][T::CW]) {
    constexpr int H = X::H;
    if constexpr (W::RING)
      ring.template product<T>(p, A, rg, cg, acc);
    else
      warp_product<T, H, H, T::LDH, true>(A, copies + m * H * H, H, rg, cg, acc);
  }
  // before a block ends (after a timeout: no copy may land after it is gone)
  __device__ __forceinline__ void finish() {
    if constexpr (W::RING) ring.drain();
  }
};

// The block's tiles of T::WR rows of positions [lo, hi): tile t goes to block
// t % gridDim.x, warp (t / gridDim.x) % NW, so that few tiles spread over all
// blocks.
template <class X, class T>
__device__ __forceinline__ void gnn_rows(const GnnArgs& p, LayerWeights<X>& weights, float* sm,
                                         int lo, int hi) {
  constexpr int MODE = X::MODE, NW = X::NW, H = X::H;
  constexpr bool MULTI = T::RM == X::Short::RM;  // a row buffer per input segment
  constexpr int RM = T::RM, CW = T::CW, WR = T::WR, LD = T::LDH;
  constexpr bool EDGE_ROWS = g_edge_rows(MODE);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* B0 = sm + warp * X::WARP_FLOATS;  // [WR][H + 4]
  float* B1 = MULTI && X::SEGS > 1 ? B0 + WR * LD : B0;
  float* B2 = MULTI && X::SEGS > 2 ? B0 + 2 * WR * LD : B0;
  float* F = B0 + X::ROWS * LD;  // node encoder: [WR][8] features
  int* rows = reinterpret_cast<int*>(F + X::FEATS);
  int* srcs = EDGE_ROWS ? rows + WR : nullptr;
  int* dsts = EDGE_ROWS ? srcs + WR : nullptr;
  (void)B1;
  (void)B2;
  const Ws& w = p.w;
  const int rg = lane >> 3, cg = lane & 7;
  const int tstride = gridDim.x * NW * WR;
  const int block0 = lo + blockIdx.x * WR;
  if (block0 >= hi) return;  // no rows for this block
  weights.start(block0, tstride, hi);

  // Edge rows: the index chain (row id from the list, then its source and
  // target) is loaded ahead in registers, lane r holding row r (and r + 32) of
  // a tile: the row ids two tiles ahead and the source / target one tile
  // ahead are loaded during a tile and first used in the next one, so a tile's
  // row gathers start without waiting for its indices.
  constexpr bool AHEAD = EDGE_ROWS && MODE != G_TRIP;
  constexpr int NI = (WR + 31) / 32;
  const int base0 = block0 + warp * gridDim.x * WR;
  auto row_at = [&](int b, int i) {
    const int r = lane + 32 * i, pos = b + r;
    return (r < WR && pos < hi) ? sel_row(p.sel, pos) : -1;
  };
  int r_cur[NI], s_cur[NI], d_cur[NI], r_next[NI];
  if constexpr (AHEAD) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      r_cur[i] = row_at(base0, i);
      s_cur[i] = r_cur[i] >= 0 ? w.src[r_cur[i]] : 0;
      d_cur[i] = r_cur[i] >= 0 ? w.col[r_cur[i]] : 0;
      r_next[i] = row_at(base0 + tstride, i);
    }
  }
  for (int base = base0; base < hi; base += tstride) {
    weights.round(base - base0 + block0, int(gridDim.x) * WR, hi);
    // ---- rows of this warp -----------------------------------------------
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int r = lane + 32 * i;
      if constexpr (AHEAD) {
        if (r < WR) {
          rows[r] = r_cur[i];
          srcs[r] = s_cur[i];
          dsts[r] = d_cur[i];
        }
        s_cur[i] = r_next[i] >= 0 ? w.src[r_next[i]] : 0;
        d_cur[i] = r_next[i] >= 0 ? w.col[r_next[i]] : 0;
        r_cur[i] = r_next[i];
        r_next[i] = row_at(base + 2 * tstride, i);
      } else if (r < WR) {
        const int pos = base + r;
        const bool in = pos < hi;
        rows[r] = in ? (MODE == G_TRIP ? pos : sel_row(p.sel, pos)) : -1;
        if constexpr (MODE == G_TRIP) {
          srcs[r] = in ? p.t1[pos] : 0;
          dsts[r] = in ? p.t2[pos] : 0;
        }
      }
    }
    __syncwarp();
    float acc[RM][CW];

    if constexpr (MODE == G_NODE_ENC || MODE == G_NODE_UPD) {
      if constexpr (MODE == G_NODE_ENC) {
        // features (x/s3, y/s4, z/s5) of each hit, column 3 zero
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int r = lane + 32 * i;
          if (r >= WR) break;
          const int row = rows[r];
          float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
          if (row >= 0) {
            const float4 q = w.pos[row];
            f = make_float4(q.x / p.fs[3], q.y / p.fs[4], q.z / p.fs[5], 0.f);
          }
          *reinterpret_cast<float4*>(F + r * 8) = f;
        }
        __syncwarp();
        acc_bias<T>(p.m.l1.b, cg, acc);
        warp_product<T, 4, 3, 8, false>(F, p.m.l1.WT, p.m.l1.ldo, rg, cg, acc);
        acc_ln_relu<T>(acc, lane);
        acc_store_smem<T>(B0, rg, cg, acc);
        __syncwarp();
        acc_bias<T>(p.m.l2.b, cg, acc);
        weights.template product<T>(B0, 0, rg, cg, acc);
        __syncwarp();  // all lanes are done reading B0
      } else {
        // [h, sum_out e, sum_in e] (the two sums written into the node's
        // projection row by k_msg_f32)
        stage_rows<T, false>(B0, rows, w.hstate, H, 0, nullptr, nullptr, 0, 0, lane);
        if constexpr (MULTI) {
          stage_rows<T, false>(B1, rows, w.pstate, 2 * H, 0, nullptr, nullptr, 0, 0, lane);
          stage_rows<T, false>(B2, rows, w.pstate, 2 * H, H, nullptr, nullptr, 0, 0, lane);
        }
        __syncwarp();
        acc_bias<T>(p.m.l1.b, cg, acc);
        weights.template product<T>(B0, 0, rg, cg, acc);
        if constexpr (!MULTI) {
          __syncwarp();
          stage_rows<T, false>(B0, rows, w.pstate, 2 * H, 0, nullptr, nullptr, 0, 0, lane);
          __syncwarp();
        }
        weights.template product<T>(B1, 1, rg, cg, acc);
        if constexpr (!MULTI) {
          __syncwarp();
          stage_rows<T, false>(B0, rows, w.pstate, 2 * H, H, nullptr, nullptr, 0, 0, lane);
          __syncwarp();
        }
        weights.template product<T>(B2, 2, rg, cg, acc);
        acc_ln_relu<T>(acc, lane);
        __syncwarp();  // all lanes are done reading B1 (which is B0 without MULTI)
        acc_store_smem<T>(B1, rg, cg, acc);
        __syncwarp();
        acc_bias<T>(p.m.l2.b, cg, acc);
        weights.template product<T>(B1, 3, rg, cg, acc);
        if constexpr (MULTI) {
          acc_add_smem<T>(B0, rg, cg, acc);  // residual h
        } else {
          acc_add_rows<T, false>(rows, w.hstate, H, nullptr, nullptr, 0, rg, cg, acc);
          __syncwarp();  // all lanes are done reading B0
        }
      }
      acc_store_rows<T>(w.hstate, H, 0, rows, rg, cg, acc);
      // ---- projections of the new node state for the next edge layer -------
      acc_store_smem<T>(B0, rg, cg, acc);
      __syncwarp();
      acc_bias<T>(p.proj.src.b, cg, acc);
      weights.template product<T>(B0, X::MATS - 2, rg, cg, acc);
      acc_store_rows<T>(w.pstate, 2 * H, 0, rows, rg, cg, acc);
      acc_bias<T>(p.proj.dst.b, cg, acc);
      weights.template product<T>(B0, X::MATS - 1, rg, cg, acc);
      acc_store_rows<T>(w.pstate, 2 * H, H, rows, rg, cg, acc);
    } else if constexpr (MODE == G_TRIP) {
      // ---- triplet classifier: [e^K(first), e^K(second)] -> Linear ->
      //      LayerNorm -> ReLU -> dot, then the triplet cut -----------------
      stage_rows<T, false>(B0, srcs, w.estate, H, 0, nullptr, nullptr, 0, 0, lane);
      if constexpr (MULTI)
        stage_rows<T, false>(B1, dsts, w.estate, H, 0, nullptr, nullptr, 0, 0, lane);
      __syncwarp();
      acc_bias<T>(p.m.l1.b, cg, acc);
      weights.template product<T>(B0, 0, rg, cg, acc);
      if constexpr (!MULTI) {
        __syncwarp();
        stage_rows<T, false>(B0, dsts, w.estate, H, 0, nullptr, nullptr, 0, 0, lane);
        __syncwarp();
      }
      weights.template product<T>(B1, 1, rg, cg, acc);
      acc_ln_relu<T>(acc, lane);
      float lg[RowSums<T>::N];
      row_dots<T>(acc, p.m.l2, cg, lg);
#pragma unroll
      for (int j = 0; j < RowSums<T>::N; ++j) {
        const int row = rows[rg + T::RG * row_of<T>(j, cg)];
        if (cg < RowSums<T>::M && row >= 0) {
          p.tlogit[row] = lg[j];
          p.tkeep[row] = lg[j] >= p.cut ? 1 : 0;
        }
      }
    } else {
      if constexpr (MODE != G_CLS) {
        // ---- layer 1: b + W_e e + (W_src h_src + W_dst h_dst, projected) ----
        if constexpr (MULTI)
          stage_rows<T, true>(B1, srcs, w.pstate, 2 * H, 0, dsts, w.pstate, 2 * H, H, lane);
        if constexpr (MODE != G_EDGE_ENC)
          stage_rows<T, false>(B0, rows, w.estate, H, 0, nullptr, nullptr, 0, 0, lane);
        __syncwarp();
        acc_bias<T>(p.m.l1.b, cg, acc);
        if constexpr (MODE != G_EDGE_ENC) weights.template product<T>(B0, 0, rg, cg, acc);
        if constexpr (MULTI) {
          acc_add_smem<T>(B1, rg, cg, acc);
        } else {
          acc_add_rows<T, true>(srcs, w.pstate, 2 * H, dsts, w.pstate + H, 2 * H, rg, cg, acc);
        }
        acc_ln_relu<T>(acc, lane);
        if constexpr (!MULTI) __syncwarp();  // all lanes are done reading B0 (= B1)
        acc_store_smem<T>(B1, rg, cg, acc);
        __syncwarp();
        // ---- layer 2 (+ residual e) -----------------------------------------
        acc_bias<T>(p.m.l2.b, cg, acc);
        weights.template product<T>(B1, MODE == G_EDGE_ENC ? 0 : 1, rg, cg, acc);
        if constexpr (MODE != G_EDGE_ENC) {
          if constexpr (MULTI)
            acc_add_smem<T>(B0, rg, cg, acc);
          else
            acc_add_rows<T, false>(rows, w.estate, H, nullptr, nullptr, 0, rg, cg, acc);
        }
        if constexpr (MODE != G_EDGE_UPD_CLS) acc_store_rows<T>(w.estate, H, 0, rows, rg, cg, acc);
        if constexpr (MODE == G_EDGE_UPD_CLS) {
          if constexpr (!MULTI) __syncwarp();  // all lanes are done reading B0
          acc_store_smem<T>(B0, rg, cg, acc);
        }
      } else {
        stage_rows<T, false>(B0, rows, w.estate, H, 0, nullptr, nullptr, 0, 0, lane);
      }
      if constexpr (MODE == G_EDGE_UPD_CLS || MODE == G_CLS) {
        // ---- classifier: Linear -> LayerNorm -> ReLU -> dot, then the cut ----
        __syncwarp();
        acc_bias<T>(p.cls.l1.b, cg, acc);
        weights.template product<T>(B0, X::MATS - 1, rg, cg, acc);
        acc_ln_relu<T>(acc, lane);
        float lg[RowSums<T>::N];
        row_dots<T>(acc, p.cls.l2, cg, lg);
#pragma unroll
        for (int j = 0; j < RowSums<T>::N; ++j) {
          const int row = rows[rg + T::RG * row_of<T>(j, cg)];
          if (cg < RowSums<T>::M && row >= 0) {
            bool write = true;
            if (p.rescore_only) {
              const float old = w.logit[row];
              write = old > p.band_lo && old < p.band_hi;
            }
            if (write) {
              w.logit[row] = lg[j];
              w.keep[row] = lg[j] >= p.cut ? 1 : 0;
            }
          }
        }
      }
    }
    __syncwarp();  // the next tile overwrites this warp's shared memory
  }
  weights.finish();
}

template <class X>
__global__ void __launch_bounds__(X::NW * 32, 1) k_gnn_f32(const GnnArgs p) {
  extern __shared__ __align__(16) float sm[];
  const Ws& w = p.w;
  LayerWeights<X> weights(p, sm + X::NW * X::WARP_FLOATS);
  pdl_begin();
  if (!weights.landed() || input_bad(w)) return;
  int lo, hi;
  if constexpr (X::MODE == G_TRIP) {
    if (*(volatile int32_t*)&w.counters[C_STATUS] & ST_CAPACITY) return;
    lo = 0;
    hi = min(*p.tn, int(w.t_cap));
    if (hi <= 0) return;
  } else {
    if (!sel_rows(p.b, w, p.sel, g_edge_rows(X::MODE), lo, hi)) return;
  }
  // short tiles while they fill at most `short_rounds` rounds of the grid's
  // warps (launch_shape; the number of rows of an edge kernel or of a row list
  // is known only here)
  const int64_t short_rows = int64_t(gridDim.x) * X::NW * X::Short::WR;
  if (hi - lo <= p.short_rounds * short_rows)
    gnn_rows<X, typename X::Short>(p, weights, sm, lo, hi);
  else
    gnn_rows<X, typename X::Tall>(p, weights, sm, lo, hi);
}

// ---------------------------------------------------------------------------
// messages of the node step (msg.cuh) from the FP32 edge rows, written to the
// node's projection row P[v] = [m_out | m_in] (the node step reads it there and
// then overwrites the row with the new projections)
// ---------------------------------------------------------------------------
template <int H>
struct MsgF32 {
  static constexpr int LANES = H / 4;
  using Chunk = float4;
  struct Acc {
    float2 a = make_float2(0.f, 0.f), b = a;
    __device__ __forceinline__ void add(const float4& v) {
      a = __fadd2_rn(a, make_float2(v.x, v.y));
      b = __fadd2_rn(b, make_float2(v.z, v.w));
    }
    __device__ __forceinline__ void finish() {}
  };
  static __device__ __forceinline__ float4 load(const Ws& w, int e, int q) {
    return __ldg(reinterpret_cast<const float4*>(w.estate + size_t(e) * H) + q);
  }
  static __device__ __forceinline__ void store(const Ws& w, int row, int side, int q, const Acc& s) {
    *(reinterpret_cast<float4*>(w.pstate + size_t(row) * 2 * H + side * H) + q) =
        make_float4(s.a.x, s.a.y, s.b.x, s.b.y);
  }
};

// (5 blocks per SM: row lists of the re-score, random in the batch, want warps)
template <int H>
__global__ void __launch_bounds__(256, 5) k_msg_f32(Batch b, Ws w, Sel sel) {
  pdl_begin();
  if (input_bad(w)) return;
  int lo, hi;
  if (!sel_rows(b, w, sel, false, lo, hi)) return;
  message_sums<MsgF32<H>>(w, sel, lo, hi);
}

// ---- transposed register tiles of the embedding MLP -------------------------
// acc[i][j] = b[c0 + j] + sum_k A[k][r0 + i] * W[k][c0 + j]
// A: shared [K][TM]; W: global [K][ldo] (transposed weights)
template <int RM, int CW, int TM>
__device__ __forceinline__ void tile_layer(const float* As, int K, const LayerF32& L, int r0,
                                           int c0, float (&acc)[RM][CW]) {
  static_assert(CW % 4 == 0 && (RM == 2 || RM == 4), "tile shape");
#pragma unroll
  for (int j = 0; j < CW; j += 4) {
    const float4 bb = __ldg(reinterpret_cast<const float4*>(L.b + c0 + j));
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      acc[i][j] = bb.x;
      acc[i][j + 1] = bb.y;
      acc[i][j + 2] = bb.z;
      acc[i][j + 3] = bb.w;
    }
  }
  const float* wp = L.WT + c0;
#pragma unroll 2
  for (int k = 0; k < K; ++k) {
    float a[RM];
    if constexpr (RM == 4) {
      const float4 v = *reinterpret_cast<const float4*>(As + k * TM + r0);
      a[0] = v.x;
      a[1] = v.y;
      a[2] = v.z;
      a[3] = v.w;
    } else {
      const float2 v = *reinterpret_cast<const float2*>(As + k * TM + r0);
      a[0] = v.x;
      a[1] = v.y;
    }
    const float4* w4 = reinterpret_cast<const float4*>(wp + size_t(k) * L.ldo);
#pragma unroll
    for (int j = 0; j < CW; j += 4) {
      const float4 q = __ldg(w4 + j / 4);
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        // two columns per packed FMA (each lane rounds like fmaf)
        const float2 a2 = make_float2(a[i], a[i]);
        const float2 c01 = __ffma2_rn(a2, make_float2(q.x, q.y), make_float2(acc[i][j], acc[i][j + 1]));
        const float2 c23 = __ffma2_rn(a2, make_float2(q.z, q.w), make_float2(acc[i][j + 2], acc[i][j + 3]));
        acc[i][j] = c01.x;
        acc[i][j + 1] = c01.y;
        acc[i][j + 2] = c23.x;
        acc[i][j + 3] = c23.y;
      }
    }
  }
}

// store acc transposed into S[c][row] (one vector store per column)
template <int RM, int CW, int TM>
__device__ __forceinline__ void tile_store_t(float* S, int r0, int c0, const float (&acc)[RM][CW],
                                             bool relu) {
#pragma unroll
  for (int j = 0; j < CW; ++j) {
    float v[RM];
#pragma unroll
    for (int i = 0; i < RM; ++i) v[i] = relu ? fmaxf(acc[i][j], 0.f) : acc[i][j];
    if constexpr (RM == 4)
      *reinterpret_cast<float4*>(S + (c0 + j) * TM + r0) = make_float4(v[0], v[1], v[2], v[3]);
    else
      *reinterpret_cast<float2*>(S + (c0 + j) * TM + r0) = make_float2(v[0], v[1]);
  }
}

// ---------------------------------------------------------------------------
// embedding MLP
// ---------------------------------------------------------------------------
struct EmbedLayers {
  LayerF32 l[kMaxEmbedLayers];
};

constexpr int kEmbedTM = 128;

template <int CW>
__device__ __forceinline__ void embed_layer_tiled(const float* X, float* Y, const LayerF32& L,
                                                  int tid, bool relu) {
  float acc[4][CW];
  const int r0 = (tid % kRowGroups) * 4, c0 = (tid / kRowGroups) * CW;
  tile_layer<4, CW, kEmbedTM>(X, L.in, L, r0, c0, acc);
  tile_store_t<4, CW, kEmbedTM>(Y, r0, c0, acc, relu);
}

__global__ void __launch_bounds__(kThreads, 3) k_embed_f32(Batch b, Ws w, EmbedLayers em,
                                                        int n_embed, int D, GraphParams g,
                                                        int maxw) {
  extern __shared__ __align__(16) float sm[];
  pdl_begin();
  if (input_bad(w)) return;
  const int tid = threadIdx.x;
  for (int base = blockIdx.x * kEmbedTM; base < b.n_hits; base += gridDim.x * kEmbedTM) {
    float* X = sm;
    float* Y = sm + maxw * kEmbedTM;
    for (int r = tid; r < kEmbedTM; r += kThreads) {
      const int v = base + r;
      float f0 = 0.f, f1 = 0.f, f2 = 0.f;
      if (v < b.n_hits) {
        const float4 p = w.pos[v];
        f0 = sqrtf(p.x * p.x + p.y * p.y) / g.fs[0];
        f1 = atan2f(p.y, p.x) / g.fs[1];
        f2 = p.z / g.fs[2];
      }
      X[r] = f0;
      X[kEmbedTM + r] = f1;
      X[2 * kEmbedTM + r] = f2;
    }
    __syncthreads();
    for (int l = 0; l < n_embed; ++l) {
      const LayerF32& L = em.l[l];
      const bool relu = l + 1 < n_embed;
      const int cw = L.ldo / kColGroups;
      if (L.ldo % 32 == 0 && (cw == 4 || cw == 8 || cw == 16)) {
        // register-tiled: 32 row groups x 8 column groups of ldo/8 columns
        if (cw == 4)
          embed_layer_tiled<4>(X, Y, L, tid, relu);
        else if (cw == 8)
          embed_layer_tiled<8>(X, Y, L, tid, relu);
        else
          embed_layer_tiled<16>(X, Y, L, tid, relu);
      } else {
        // any other width (the D-wide output): one thread per (row, output)
        for (int t = tid; t < kEmbedTM * L.out; t += kThreads) {
          const int r = t % kEmbedTM, o = t / kEmbedTM;
          float a = L.b[o];
          for (int k = 0; k < L.in; ++k) a = fmaf(X[k * kEmbedTM + r], L.WT[k * L.ldo + o], a);
          Y[o * kEmbedTM + r] = relu ? fmaxf(a, 0.f) : a;
        }
      }
      __syncthreads();
      float* t = X;
      X = Y;
      Y = t;
    }
    for (int t = tid; t < kEmbedTM * D; t += kThreads) {
      const int r = t / D, d = t % D, v = base + r;
      if (v < b.n_hits) w.emb[size_t(v) * D + d] = X[d * kEmbedTM + r];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// embedding MLP, 3 -> W -> ... -> W -> D with NH layers W -> W in the middle: the
// warp tiles and weight sources of the interaction-network kernels. A lane of
// the last layer takes one row and four outputs.
// ---------------------------------------------------------------------------
struct EmbedArgs {
  Batch b;
  Ws w;
  EmbedLayers em;
  int D;
  float fs[3];
};

template <int W_, int RM_, int NH_, int NW_, int WEIGHTS_>
struct EmbedShape {
  using Args = EmbedArgs;
  using Tall = WarpTile<W_, RM_>;
  using Short = WarpTile<W_, W_ == 128 ? 2 : 1>;
  static constexpr int H = W_, NH = NH_, NW = NW_;
  static constexpr int WARP_FLOATS = Tall::WR * (Tall::LDH + 8);  // rows, features
  using W = WeightSource<W_, NH_, WEIGHTS_>;
  static constexpr int LAST = W_ * 16;  // last layer, D <= 16
  static constexpr size_t SMEM = (size_t(NW) * WARP_FLOATS + W::FLOATS + LAST) * 4;
  static __device__ __forceinline__ const float* mat(const Args& p, int m) { return p.em.l[1 + m].WT; }
};

template <class T>
__device__ __forceinline__ void acc_relu(float (&acc)[T::RM][T::CW]) {
#pragma unroll
  for (int i = 0; i < T::RM; ++i)
#pragma unroll
    for (int c = 0; c < T::CW; ++c) acc[i][c] = fmaxf(acc[i][c], 0.f);
}

template <class X, class T>
__device__ __forceinline__ void embed_rows(const EmbedArgs& p, LayerWeights<X>& weights, float* sm) {
  constexpr int NW = X::NW, H = X::H, WR = T::WR, LD = T::LDH;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rg = lane >> 3, cg = lane & 7;
  const int n = p.b.n_hits;
  float* A = sm + warp * X::WARP_FLOATS;  // [WR][H + 4]
  float* F = A + WR * LD;                 // [WR][8] features
  const float* last = sm + NW * X::WARP_FLOATS + X::W::FLOATS;
  const int tstride = gridDim.x * NW * WR;
  const int block0 = blockIdx.x * WR;
  if (block0 >= n) return;  // no rows for this block
  const LayerF32& lo = p.em.l[X::NH + 1];  // W -> D
  weights.start(block0, tstride, n);
  const int base0 = block0 + warp * gridDim.x * WR;
  for (int base = base0; base < n; base += tstride) {
    weights.round(base - base0 + block0, int(gridDim.x) * WR, n);
    if (lane < WR) {
      const int v = base + lane;
      float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
      if (v < n) {
        const float4 q = p.w.pos[v];
        f.x = sqrtf(q.x * q.x + q.y * q.y) / p.fs[0];
        f.y = atan2f(q.y, q.x) / p.fs[1];
        f.z = q.z / p.fs[2];
      }
      *reinterpret_cast<float4*>(F + lane * 8) = f;
    }
    __syncwarp();
    float acc[T::RM][T::CW];
    acc_bias<T>(p.em.l[0].b, cg, acc);
    warp_product<T, 4, 3, 8, false>(F, p.em.l[0].WT, p.em.l[0].ldo, rg, cg, acc);
    acc_relu<T>(acc);
    acc_store_smem<T>(A, rg, cg, acc);
    __syncwarp();
#pragma unroll 1
    for (int l = 0; l < X::NH; ++l) {
      acc_bias<T>(p.em.l[1 + l].b, cg, acc);
      weights.template product<T>(A, l, rg, cg, acc);
      acc_relu<T>(acc);
      __syncwarp();  // all lanes are done reading A
      acc_store_smem<T>(A, rg, cg, acc);
      __syncwarp();
    }
    for (int t = lane; t < WR * (lo.ldo / 4); t += 32) {
      const int r = t % WR, o = 4 * (t / WR), v = base + r;
      if (v >= n) continue;
      float4 y = __ldg(reinterpret_cast<const float4*>(lo.b + o));
      const float* a = A + r * LD;
#pragma unroll 4
      for (int k = 0; k < H; k += 4) {
        const float4 x = *reinterpret_cast<const float4*>(a + k);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float xv = u == 0 ? x.x : (u == 1 ? x.y : (u == 2 ? x.z : x.w));
          const float4 q = *reinterpret_cast<const float4*>(last + (k + u) * lo.ldo + o);
          y.x = fmaf(xv, q.x, y.x);
          y.y = fmaf(xv, q.y, y.y);
          y.z = fmaf(xv, q.z, y.z);
          y.w = fmaf(xv, q.w, y.w);
        }
      }
      float* e = p.w.emb + size_t(v) * p.D + o;
      if (p.D % 4 == 0) {
        *reinterpret_cast<float4*>(e) = y;
      } else {
        e[0] = y.x;
        if (o + 1 < p.D) e[1] = y.y;
        if (o + 2 < p.D) e[2] = y.z;
        if (o + 3 < p.D) e[3] = y.w;
      }
    }
    __syncwarp();  // the next tile overwrites A and F
  }
  weights.finish();
}

template <class X>
__global__ void __launch_bounds__(X::NW * 32, 1) k_embed_tiles(const EmbedArgs p) {
  extern __shared__ __align__(16) float sm[];
  const LayerF32& lo = p.em.l[X::NH + 1];
  for (int i = threadIdx.x; i < X::H * lo.ldo; i += X::NW * 32)
    sm[X::NW * X::WARP_FLOATS + X::W::FLOATS + i] = lo.WT[i];
  LayerWeights<X> weights(p, sm + X::NW * X::WARP_FLOATS);  // (ends with a block barrier)
  pdl_begin();
  if (!weights.landed() || input_bad(p.w)) return;
  // short tiles while they fill at most one round of the grid's warps, as the
  // interaction-network kernels
  if (p.b.n_hits <= int64_t(gridDim.x) * X::NW * X::Short::WR)
    embed_rows<X, typename X::Short>(p, weights, sm);
  else
    embed_rows<X, typename X::Tall>(p, weights, sm);
}

// occupancy of (kernel, block size, shared memory), queried once and cached
int blocks_per_sm(const void* fn, int threads, size_t smem) {
  struct Entry {
    const void* fn;
    int threads;
    size_t smem;
    int n;
  };
  static Entry cache[64];
  static int used = 0;
  static std::mutex mu;  // handles may launch from several host threads
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < used; ++i)
    if (cache[i].fn == fn && cache[i].threads == threads && cache[i].smem == smem) return cache[i].n;
  int n = 0;
  // the attribute is an upper bound: set it once to the device maximum, so a
  // later configuration with less shared memory never lowers it
  bool seen = false;
  for (int i = 0; i < used; ++i) seen = seen || cache[i].fn == fn;
  if (!seen) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem);
  n = n > 0 ? n : 1;
  if (used < 64) cache[used++] = Entry{fn, threads, smem, n};
  return n;
}

constexpr int f32_family(int mode) {
  return (mode == G_NODE_ENC || mode == G_EDGE_ENC) ? 0 : (mode == G_NODE_UPD ? 1 : 2);
}

// Variant (0 the default; the autotuner may pick another, see
// gnntrk_set_tuning): 0 = short tiles for calls whose rows fill at most one
// round of short tiles over the grid's warps, tall tiles above; 1 = tall tiles
// always; 2 = short tiles up to two rounds. The line of variant 0: up to one round every
// warp has one short tile, and a call's time is the time of one tile (one
// event of 2146 hits at hidden 64: node step 17.9 us against 31.0 us with tall
// tiles); with two rounds or more the short tiles' weight loads, one per row
// group and k instead of one for 8 rows, cost more than the idle warps
// (16 652 edges, 2.3 rounds: edge step 20.1 us against 17.1 us with tall
// tiles). Variant 2 goes no further than two rounds: a choice may be kept and applied
// to calls of any size, and short tiles at every size took 9.71 ms per call of 400
// events at hidden 32 and 23.7 ms for 100 at hidden 64 (variant 0: 4.03 and 8.40 ms).
//
// Shapes (GB300; edge steps and node steps of a call, against the kernels they
// replaced, whose warps of 4-warp blocks had 32 accumulators per lane):
//   hidden 32, 20 warps, 32-row tiles: 4.0 M edges x 4 steps 1.80 ms (2.42),
//     0.67 M hits x 4 steps 0.71 ms (0.95). 16 warps: 1.85 ms; 8 warps x 2
//     blocks: 1.99 ms; a 4-lane row group (half the LayerNorm work per row,
//     8-column lanes): 2.05 ms and more, fewer warps for the registers.
//   hidden 64, 12 warps, 32-row tiles (64 accumulators per lane): 1.76 M edges
//     x 8 steps 4.74 ms (6.58), 0.22 M hits x 8 steps 1.73 ms (2.27). 4 warps
//     x 3 blocks 5.42 ms; weights through L1 5.01 ms, through the ring 5.02 ms.
//   hidden 128, 12 warps, 16-row tiles, weights through the ring: 1.83 M listed
//     edges 2.35 ms (4.56), 0.74 M hits 2.83 ms (5.16). Before, one 16-byte
//     weight load fed 8 products and the L1 pipe was the bound; the six
//     matrices of the node step (384 KB) miss L1 (4.05 ms without the ring).
//     Short tiles of 8 rows: a warp reads a whole matrix from shared memory per
//     tile whatever its height (a 16-byte load takes 4 cycles of the pipe), so
//     half the rows per warp would read twice as much.
// Now 55 % (hidden 32) to 68 % (hidden 64) of the FP32 rate that packed FMAs
// reach alone (75 TFLOP/s); what is left is the row gathers and the LayerNorm
// between the products.
template <class X>
void launch_shape(GnnArgs a, int64_t rows_hint, cudaStream_t s) {
  const int v = g_f32_variant[X::H == 32 ? 0 : (X::H == 64 ? 1 : 2)][f32_family(X::MODE)].load(
      std::memory_order_relaxed);
  a.short_rounds = v == 0 ? 1 : v == 1 ? 0 : 2;
  const void* fn = (const void*)k_gnn_f32<X>;
  int grid = device_sms() * blocks_per_sm(fn, X::NW * 32, X::SMEM);
  // four short tiles per block before another block is used
  constexpr int kRowsPerBlock = 4 * X::Short::WR;
  grid = int(std::max<int64_t>(1, std::min<int64_t>(grid, (rows_hint + kRowsPerBlock - 1) / kRowsPerBlock)));
  launch_pdl(true, k_gnn_f32<X>, grid, X::NW * 32, X::SMEM, s, 1, a);
}

template <int H, int MODE>
void launch_gnn(const GnnArgs& a, int64_t rows_hint, cudaStream_t s) {
  if constexpr (H == 32)
    launch_shape<GnnShape<32, 8, 1, MODE, 20, W_BLOCK>>(a, rows_hint, s);
  else if constexpr (H == 64)
    launch_shape<GnnShape<64, 8, 1, MODE, 12, W_BLOCK>>(a, rows_hint, s);
  else
    launch_shape<GnnShape<128, 4, 2, MODE, 12, W_RING>>(a, rows_hint, s);
}

void launch_gnn_any(int h, int mode, const GnnArgs& a, int64_t rows_hint, cudaStream_t s) {
#define GNNTRK_M(HH)                                                                \
  switch (mode) {                                                                   \
    case G_NODE_ENC: launch_gnn<HH, G_NODE_ENC>(a, rows_hint, s); break;            \
    case G_EDGE_ENC: launch_gnn<HH, G_EDGE_ENC>(a, rows_hint, s); break;            \
    case G_NODE_UPD: launch_gnn<HH, G_NODE_UPD>(a, rows_hint, s); break;            \
    case G_EDGE_UPD: launch_gnn<HH, G_EDGE_UPD>(a, rows_hint, s); break;            \
    case G_EDGE_UPD_CLS: launch_gnn<HH, G_EDGE_UPD_CLS>(a, rows_hint, s); break;    \
    case G_CLS: launch_gnn<HH, G_CLS>(a, rows_hint, s); break;                      \
    case G_TRIP: launch_gnn<HH, G_TRIP>(a, rows_hint, s); break;                    \
  }
  if (h == 32) {
    GNNTRK_M(32)
  } else if (h == 64) {
    GNNTRK_M(64)
  } else {
    GNNTRK_M(128)
  }
#undef GNNTRK_M
}

GnnArgs gnn_args(const Batch& b, const Ws& w, Sel sel) {
  GnnArgs a{};
  a.b = b;
  a.w = w;
  a.sel = sel;
  return a;
}

}  // namespace

void launch_triplet_scores_f32(const Batch& b, const Ws& w, const TripletHeads& t, int h,
                               float cut_logit, cudaStream_t s) {
  GnnArgs a{};
  a.b = b;
  a.w = w;
  a.cut = cut_logit;
  a.sel = Sel{nullptr, nullptr};
  a.m = t.art;
  a.t1 = w.trip_a1;
  a.t2 = w.trip_a2;
  a.tn = w.counters + C_TRIP_A;
  a.tlogit = w.trip_alogit;
  a.tkeep = w.trip_akeep;
  launch_gnn_any(h, G_TRIP, a, triplet_rows_hint(b.n_hits), s);
  a.m = t.elb;
  a.t1 = w.trip_e1;
  a.t2 = w.trip_e2;
  a.tn = w.counters + C_TRIP_E;
  a.tlogit = w.trip_elogit;
  a.tkeep = w.trip_ekeep;
  launch_gnn_any(h, G_TRIP, a, triplet_rows_hint(b.n_hits), s);
}

void f32_set_variant(int h, int family, int v) {
  if ((h != 32 && h != 64 && h != 128) || family < 0 || family > 2) return;
  g_f32_variant[h == 32 ? 0 : (h == 64 ? 1 : 2)][family].store((v >= 0 && v <= 2) ? v : 0,
                                                                std::memory_order_relaxed);
}

namespace {
template <class X>
void launch_embed_tiles(const EmbedArgs& a, cudaStream_t s) {
  const int full = device_sms() * blocks_per_sm((const void*)k_embed_tiles<X>, X::NW * 32, X::SMEM);
  const int grid = std::max(1, std::min(full, div_up(a.b.n_hits, 4 * X::Short::WR)));
  launch_pdl(true, k_embed_tiles<X>, grid, X::NW * 32, X::SMEM, s, 1, a);
}

// The warp-tile kernel for one or two hidden layers W -> W of the usual widths
// 64 and 128 (two matrices at 128 come through the ring: copies of both would
// not fit beside the row buffers), the block kernel for any other shape. The
// block kernel keeps both activations of 128 rows in shared memory, at width
// 128 one block of 8 warps per SM, and one event fills a block per 128 hits.
// Embedding and node encoder together, block kernel -> warp tiles: 3-128-128-
// 128-8 on 219 k hits 1.46 -> 0.40 ms, on one event of 2146 hits 128 -> 45 us;
// 3-128-128-4 on 874 k hits 2.04 -> 0.92 ms; 3-64-64-4 on 1.68 M hits 0.59 ->
// 0.40 ms (of which the embedding runs at 51 TFLOP/s, 68 % of the FP32 rate).
void launch_embed_f32(const Batch& b, const Ws& w, const LayerF32* embed, int n_embed, int D,
                      const GraphParams& g, cudaStream_t s) {
  EmbedArgs a{};
  a.b = b;
  a.w = w;
  a.D = D;
  for (int i = 0; i < 3; ++i) a.fs[i] = g.fs[i];
  int maxw = 4;
  const int W = embed[0].out;
  bool tiles = n_embed >= 3;
  for (int l = 0; l < n_embed; ++l) {
    a.em.l[l] = embed[l];
    maxw = std::max(maxw, embed[l].ldo);
    tiles = tiles && (l + 1 == n_embed ? embed[l].ldo <= 16 : embed[l].out == W);
  }
  if (tiles && W == 64 && n_embed == 3) return launch_embed_tiles<EmbedShape<64, 8, 1, 12, W_BLOCK>>(a, s);
  if (tiles && W == 64 && n_embed == 4) return launch_embed_tiles<EmbedShape<64, 8, 2, 12, W_BLOCK>>(a, s);
  if (tiles && W == 128 && n_embed == 3) return launch_embed_tiles<EmbedShape<128, 4, 1, 12, W_BLOCK>>(a, s);
  if (tiles && W == 128 && n_embed == 4) return launch_embed_tiles<EmbedShape<128, 4, 2, 12, W_RING>>(a, s);
  const size_t smem = size_t(2) * maxw * kEmbedTM * sizeof(float);
  const int full = device_sms() * blocks_per_sm((const void*)k_embed_f32, kThreads, smem);
  const int grid = std::max(1, std::min(full, div_up(b.n_hits, kEmbedTM)));
  launch_pdl(true, k_embed_f32, grid, kThreads, smem, s, 1, b, w, a.em, n_embed, D, g, maxw);
}
}  // namespace

void launch_node_prep_f32(const Batch& b, const Ws& w, const LayerF32* embed, int n_embed,
                          const Mlp2F32& node_enc, const EdgeProj& proj, int D, int h,
                          const GraphParams& g, bool do_embed, bool do_node_enc, Sel sel,
                          cudaStream_t s) {
  if (b.n_hits <= 0) return;
  if (do_embed) launch_embed_f32(b, w, embed, n_embed, D, g, s);
  if (do_node_enc) {
    GnnArgs a = gnn_args(b, w, sel);
    a.m = node_enc;
    a.proj = proj;
    for (int i = 0; i < 6; ++i) a.fs[i] = g.fs[i];
    launch_gnn_any(h, G_NODE_ENC, a, b.n_hits, s);
  }
}

void launch_edge_enc_f32(const Batch& b, const Ws& w, const Mlp2F32& m, int h, Sel sel,
                         cudaStream_t s) {
  GnnArgs a = gnn_args(b, w, sel);
  a.m = m;
  launch_gnn_any(h, G_EDGE_ENC, a, edge_rows_hint(b.n_hits), s);
}

void launch_messages_f32(const Batch& b, const Ws& w, int h, Sel sel, cudaStream_t s) {
  if (b.n_hits <= 0) return;
  const int full = device_sms() * 8;
  const int grid = sel.rows ? full : std::max(1, std::min(full, div_up(b.n_hits, 256 / (h / 4))));
  launch_pdl(false, h == 32 ? k_msg_f32<32> : h == 64 ? k_msg_f32<64> : k_msg_f32<128>, grid, 256, 0,
             s, 1, b, w, sel);
}

void launch_node_update_f32(const Batch& b, const Ws& w, const Mlp2F32& m, const EdgeProj& proj,
                            int h, Sel sel, cudaStream_t s) {
  if (b.n_hits <= 0) return;
  GnnArgs a = gnn_args(b, w, sel);
  a.m = m;
  a.proj = proj;
  launch_gnn_any(h, G_NODE_UPD, a, b.n_hits, s);
}

void launch_edge_update_f32(const Batch& b, const Ws& w, const Mlp2F32& m, const Mlp2F32* cls,
                            int h, float cut_logit, bool rescore_only, float band_lo,
                            float band_hi, Sel sel, cudaStream_t s) {
  GnnArgs a = gnn_args(b, w, sel);
  a.m = m;
  if (cls) a.cls = *cls;
  a.cut = cut_logit;
  a.rescore_only = rescore_only;
  a.band_lo = band_lo;
  a.band_hi = band_hi;
  const int mode = cls == nullptr ? G_EDGE_UPD : (m.l1.WT == nullptr ? G_CLS : G_EDGE_UPD_CLS);
  launch_gnn_any(h, mode, a, edge_rows_hint(b.n_hits), s);
}

}  // namespace gnntrk
