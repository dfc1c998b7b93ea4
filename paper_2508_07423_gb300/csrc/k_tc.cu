// Tensor-core (tcgen05) kernels of the interaction network: BF16 or FP8-E4M3
// operands, FP32 accumulation in tensor memory.
//
// One CTA of 128 threads works on tiles of 128 rows (edges or hits); thread t
// owns row t of the tile and TMEM lane t (warp w reads lanes 32w..32w+31). Per
// tile:
//   1. gather: the pieces of the input rows ([e, h_src, h_dst], [h, sum_out e,
//      sum_in e], ...) come from global memory into the A tile in shared memory.
//      BF16: by cp.async, four lanes per 64 bytes of a row, into blocks of 32
//      columns in the 64-byte swizzle layout, during the tile before (see
//      Layout::SWZ). FP8 edge steps at hidden 128: by warpgroups of their own, see
//      p3_loader. The others: through registers into 8-row x
//      16-byte core matrices (K-major, no swizzle: row r, 16-byte chunk c at
//      ((r/8) * (K/epc) + c) * 128 + (r%8) * 16);
//   2. one thread issues the layer-1 MMAs (weights resident in shared memory,
//      loaded once per CTA by cp.async.bulk) and commits them to an mbarrier;
//   3. every thread reads its row of the accumulator back with tcgen05.ld,
//      adds the bias, applies LayerNorm and ReLU and writes the hidden row as
//      the next A tile; layer 2 follows the same way;
//   4. the epilogue adds the residual and stores the new state (BF16, the rows of
//      a warp through shared memory so that the stores are whole lines); at the
//      last step the edge classifier (a third MMA, LayerNorm, ReLU and a dot
//      product) and the cut run instead of the store.
// FP8: each input segment of layer 1 (e.g. e, h_src, h_dst) is quantised with
// its own per-row scale amax/448 and accumulated in its own TMEM block, so the
// epilogue can apply the scales (the edge steps at hidden 128: h_src and h_dst
// under one scale in one block, layer 1 in three passes, see Layout::P3);
// weights carry per-output-channel scales amax/448. Hidden rows are quantised per
// row as well. The K = 3 first layer of the node encoder and the 1-unit last layer
// of the classifier stay FP32.
#include <cuda_fp8.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "../../include/gnntrk.h"
#include "msg.cuh"
#include "tc.cuh"
#include "tc_ptx.cuh"

namespace gnntrk {

int device_sms();

namespace {

using namespace tc;

constexpr int kRows = 128;       // rows per tile = threads per CTA = TMEM lanes
constexpr long long kWaitCycles = 4000000000LL;  // bounded waits: about 2 s

enum Mode : int { M_NODE_ENC = 0, M_EDGE_ENC = 1, M_NODE_UPD = 2, M_EDGE_UPD = 3,
                  M_EDGE_UPD_CLS = 4, M_CLS = 5, M_TRIP = 6 };

struct TcArgs {
  Batch b;
  Ws w;
  const uint8_t* W1;  // layer-1 operand image (classifier layer 1 in M_CLS)
  const uint8_t* W2;  // layer-2 operand image
  const uint8_t* Wc;  // classifier layer-1 image (M_EDGE_UPD_CLS)
  const float* b1;
  const float* b2;
  const float* bc1;
  LayerF32 ne1;       // node encoder layer 1 (FP32, M_NODE_ENC)
  LayerF32 c2;        // classifier layer 2 (FP32, h -> 1)
  // M_TRIP: one triplet list (edge pairs, count on the device) and its outputs
  const int32_t* t1;
  const int32_t* t2;
  const int32_t* tn;
  float* tlogit;
  uint8_t* tkeep;
  float fs[6];
  float cut;
};

// A launch's arguments, and the host copies of its layers' biases and scales
struct TcCall : TcArgs {
  const LayerTC *l1 = nullptr, *l2 = nullptr, *lc = nullptr;
};

// Biases and FP8 weight scales of a launch as kernel arguments: the epilogues read
// them from the constant bank. (In shared memory each warp's 16-byte broadcast
// loads of them took a third of the shared memory pipe's cycles: BF16 edge step at
// hidden 32 on 10.1 M rows 340 -> 313 us, FP8 at 128 on 5.2 M 1.57 -> 1.48 ms.)
template <int H, bool FP8>
struct TcPar {
  float b1[H], b2[H], bc[H];
  float s1[FP8 ? H : 1], s2[FP8 ? H : 1], sc[FP8 ? H : 1];
};

__host__ __device__ constexpr int n_seg(int mode) {
  return (mode == M_EDGE_ENC || mode == M_TRIP)
             ? 2
             : ((mode == M_NODE_UPD || mode == M_EDGE_UPD || mode == M_EDGE_UPD_CLS) ? 3 : 1);
}
__host__ __device__ constexpr int align1k(int x) { return (x + 1023) & ~1023; }
__host__ __device__ constexpr int pow2_cols(int x) {
  return x <= 32 ? 32 : (x <= 64 ? 64 : (x <= 128 ? 128 : (x <= 256 ? 256 : 512)));
}

// Shared-memory layout of one CTA (byte offsets).
template <int H, bool FP8, int MODE>
struct Layout {
  static constexpr int ESZ = FP8 ? 1 : 2;
  static constexpr int NSEG = n_seg(MODE);
  // BF16 encoders carry the node encoding at about 16 significant bits: an
  // operand x enters the MMA as hi = bf16(x) and lo = bf16(x - hi) over a K
  // twice as long, against the weight image repeated along K (node encoder
  // layer 2: its hidden row; edge encoder layer 1: the FP32 rows h_src, h_dst).
  // The encoders see hit coordinates, whose useful precision (a 12 um
  // resolution over a 45 mm radius) is finer than BF16's 8-bit mantissa.
  static constexpr bool SPLIT = !FP8 && (MODE == M_NODE_ENC || MODE == M_EDGE_ENC);
  // at hidden 128 the split edge encoder runs layer 1 in four passes of K = H
  // over a one-segment tile (hi h_src, hi h_dst, lo h_src, lo h_dst, accumulated
  // into the same tensor memory) against the K halves of the plain weight image,
  // so that two tiles fit beside the weights
  static constexpr bool SPLIT2 = SPLIT && MODE == M_EDGE_ENC && H > 64;
  // FP8 edge steps at hidden 128 run layer 1 in three passes of K = H over
  // one-segment tiles (e, then h_src, then h_dst) against the K chunks of the
  // weight image; h_src and h_dst share one per-row scale and accumulate into
  // one tensor-memory block (e into the other), so that two tiles' accumulators
  // (256 columns each) fill an SM. Two warpgroups work on a tile each; two more,
  // the loaders, each load and quantise the rows of the next tile of one of them
  // into a ring of P3_SLOTS one-segment tiles meanwhile. (One warpgroup doing both
  // waited for its loads in each pass: 1.95 ms per launch on 5.2 M rows, 1.82 with
  // loaders that copied four lanes to a row, 1.57 with half a warp to a row.)
  static constexpr bool P3 = FP8 && H == 128 && (MODE == M_EDGE_UPD || MODE == M_EDGE_UPD_CLS);
  // FP8 node step at hidden 128: the next tile's rows are loaded during a tile, and
  // the three segments' accumulators take turns in two blocks of tensor memory (the
  // third starts once the first has been read), so that an SM works on two tiles
  static constexpr bool NODE8 = FP8 && H == 128 && MODE == M_NODE_UPD;
  static constexpr int P3_SLOTS = MODE == M_EDGE_UPD_CLS ? 2 : 3;
  static constexpr int K1 = (MODE == M_NODE_ENC) ? H : (SPLIT && !SPLIT2 ? 2 : 1) * NSEG * H;
  static constexpr int K2 = (SPLIT && MODE == M_NODE_ENC) ? 2 * H : H;
  static constexpr bool HAS_W1 = MODE != M_NODE_ENC;
  static constexpr bool HAS_W2 = MODE != M_CLS && MODE != M_TRIP;
  static constexpr bool HAS_WC = MODE == M_EDGE_UPD_CLS;
  static constexpr int W1 = 0;
  static constexpr int W1_BYTES = HAS_W1 ? H * K1 * ESZ : 0;
  static constexpr int W2 = align1k(W1 + W1_BYTES);
  static constexpr int W2_BYTES = HAS_W2 ? H * K2 * ESZ : 0;
  static constexpr int WC = align1k(W2 + W2_BYTES);
  static constexpr int WC_BYTES = HAS_WC ? H * H * ESZ : 0;
  // BF16 layer-1 inputs (but the three-pass forms' and the node encoder's) are
  // kept as blocks of 128 rows x 64 bytes in the 64-byte swizzle layout and filled
  // by cp.async with four lanes per row: one copy instruction then touches 8 lines
  // of global memory and 4 x 128 bytes of shared memory without bank conflicts.
  // With the canonical layout (8 rows x 16 bytes) either the loads touch 32 lines
  // or the stores conflict four ways, and the kernels were bound by the shared
  // memory pipe (82-87 % of its cycles). Hidden 32, 1024 events, us per launch
  // before and after: edge encoder (10.1 M rows) 638 -> 338, edge step 499 -> 340,
  // node step (1.7 M rows) 130 -> 68.
  static constexpr bool SWZ = !FP8 && MODE != M_NODE_ENC && !SPLIT2;
  // the next tile's rows load while this tile's layer 2 and epilogue run; the
  // hidden row then needs a tile of its own (in the edge encoder at hidden 64 that
  // would leave room for one CTA per SM instead of two)
  static constexpr bool PREF = SWZ && (H == 32 || !SPLIT);
  // tiles in flight per CTA, each worked on by a warpgroup of its own with its
  // own buffers and accumulators; they share the weights. Two at hidden 128, where
  // the weights leave room for one CTA per SM.
  static constexpr int G = SPLIT2 || P3 || NODE8 ? 2 : 1;
  static constexpr int THREADS = kRows * (P3 ? 2 * G : G);
  static constexpr int A = align1k(WC + WC_BYTES);
  static constexpr int A_BYTES =
      MODE == M_NODE_ENC ? 0 : kRows * (P3 ? P3_SLOTS * H : (SPLIT2 ? H : K1)) * ESZ;
  // hidden / classifier input: its own tile or over the layer-1 input
  static constexpr bool OWN_HA = MODE == M_NODE_ENC || (PREF && HAS_W2) || P3;
  static constexpr int HA = OWN_HA ? align1k(A + G * A_BYTES) : A;
  static constexpr int HA_BYTES = OWN_HA ? kRows * K2 * ESZ : 0;  // (per warpgroup)
  static_assert(G == 1 || (HA_BYTES % 1024 == 0 && A_BYTES % 1024 == 0), "a buffer per warpgroup");
  static constexpr int PAR = align1k(HA_BYTES > 0 ? HA + G * HA_BYTES : A + G * A_BYTES);
  // fp32 parameters: c2 weights and bias, ne1 (3 x H + H)
  static constexpr int PAR_FLOATS = 5 * H + 8;
  static constexpr int BAR = PAR + PAR_FLOATS * 4;
  // hidden 128: each warp's state rows pass through a staging block of 32 rows x
  // 64 bytes (80-byte stride) on their way in (residual) and out
  static constexpr bool COOP = H == 128 && MODE != M_CLS && MODE != M_TRIP;
  // BF16 at hidden 32 and 64: out through the hidden tile, which is free by then
  static constexpr bool OUT_STAGE = !FP8 && H <= 64 && MODE != M_CLS && MODE != M_TRIP && MODE != M_EDGE_UPD_CLS;
  static_assert(THREADS <= 512 && !(SWZ && (NODE8 || P3)) && !(OUT_STAGE && COOP), "one way in, one way out");
  // P3: full and empty barriers of the rings, and the rows' two scales (of two
  // tiles, by turns; written after the wait for the tile's first slot, see p3_loader)
  static constexpr int RING = BAR + 64;
  static constexpr int SCALES = RING + (P3 ? 128 : 0);
  static constexpr int STAGE = SCALES + (P3 ? G * 2 * kRows * 8 : 0);
  static constexpr int STAGE_ROW = 80;
  static constexpr int TOTAL = STAGE + (COOP ? G * kRows * STAGE_ROW : 0);
  // FP8: one accumulator block per layer-1 segment scale
  static constexpr int TSEG = P3 || NODE8 ? 2 : (FP8 ? NSEG : 1);
  static constexpr int TMEM_COLS = pow2_cols(TSEG * H);
  static_assert(G * TMEM_COLS <= 512, "tensor memory of one SM");
};

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t pack_e4m3x4(float a, float b, float c, float d) {
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3);
  return lo | (hi << 16);
}

// byte offset of (row, 16-byte chunk) in a canonical tile with `kchunks`
// chunks per row
__device__ __forceinline__ uint32_t tile_off(int row, int chunk, int kchunks) {
  return uint32_t(((row >> 3) * kchunks + chunk) * 128 + (row & 7) * 16);
}

// Write `n` (multiple of 16 for FP8, of 8 for BF16) FP32 values of this
// thread's row into the A tile starting at element k0, scaled by `inv` for FP8.
template <bool FP8>
__device__ __forceinline__ void put_row_f32(uint8_t* tile, int row, int kchunks, int k0,
                                            const float* v, int n, float inv) {
  if constexpr (FP8) {
    for (int c = 0; c < n / 16; ++c) {
      const float* q = v + 16 * c;
      uint4 u;
      u.x = pack_e4m3x4(q[0] * inv, q[1] * inv, q[2] * inv, q[3] * inv);
      u.y = pack_e4m3x4(q[4] * inv, q[5] * inv, q[6] * inv, q[7] * inv);
      u.z = pack_e4m3x4(q[8] * inv, q[9] * inv, q[10] * inv, q[11] * inv);
      u.w = pack_e4m3x4(q[12] * inv, q[13] * inv, q[14] * inv, q[15] * inv);
      *reinterpret_cast<uint4*>(tile + tile_off(row, (k0 >> 4) + c, kchunks)) = u;
    }
  } else {
    for (int c = 0; c < n / 8; ++c) {
      const float* q = v + 8 * c;
      uint4 u;
      u.x = pack_bf16(q[0], q[1]);
      u.y = pack_bf16(q[2], q[3]);
      u.z = pack_bf16(q[4], q[5]);
      u.w = pack_bf16(q[6], q[7]);
      *reinterpret_cast<uint4*>(tile + tile_off(row, (k0 >> 3) + c, kchunks)) = u;
    }
  }
}

// Quantise one BF16 row of H values from global memory into an E4M3 A tile (the
// per-row scale is returned). `keep` receives the raw row when not null.
template <int H>
__device__ __forceinline__ float put_row_e4m3(uint8_t* tile, int row, int kchunks, int k0,
                                              const __nv_bfloat16* src, uint4* keep) {
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4 r[H / 8];
  float amax = 0.f;
#pragma unroll
  for (int c = 0; c < H / 8; ++c) {
    r[c] = s4[c];
    if (keep) keep[c] = r[c];
    const uint32_t q[4] = {r[c].x, r[c].y, r[c].z, r[c].w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      amax = fmaxf(amax, fmaxf(fabsf(bf16_lo(q[j])), fabsf(bf16_hi(q[j]))));
  }
  const float scale = amax > 0.f ? amax / 448.f : 1.f;
  const float inv = amax > 0.f ? 448.f / amax : 1.f;
#pragma unroll
  for (int c = 0; c < H / 16; ++c) {
    const uint4 a = r[2 * c], b = r[2 * c + 1];
    uint4 u;
    u.x = pack_e4m3x4(bf16_lo(a.x) * inv, bf16_hi(a.x) * inv, bf16_lo(a.y) * inv, bf16_hi(a.y) * inv);
    u.y = pack_e4m3x4(bf16_lo(a.z) * inv, bf16_hi(a.z) * inv, bf16_lo(a.w) * inv, bf16_hi(a.w) * inv);
    u.z = pack_e4m3x4(bf16_lo(b.x) * inv, bf16_hi(b.x) * inv, bf16_lo(b.y) * inv, bf16_hi(b.y) * inv);
    u.w = pack_e4m3x4(bf16_lo(b.z) * inv, bf16_hi(b.z) * inv, bf16_lo(b.w) * inv, bf16_hi(b.w) * inv);
    *reinterpret_cast<uint4*>(tile + tile_off(row, (k0 >> 4) + c, kchunks)) = u;
  }
  return scale;
}

// Write n FP32 values (a multiple of 8) into a BF16 tile as two parts, hi =
// bf16(v) at element k_hi and lo = bf16(v - hi) at element k_lo.
__device__ __forceinline__ void put_row_split(uint8_t* tile, int row, int kchunks, int k_hi,
                                              int k_lo, const float* v, int n) {
  for (int c = 0; c < n / 8; ++c) {
    const float* q = v + 8 * c;
    float r[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) r[j] = q[j] - __bfloat162float(__float2bfloat16_rn(q[j]));
    *reinterpret_cast<uint4*>(tile + tile_off(row, (k_hi >> 3) + c, kchunks)) =
        make_uint4(pack_bf16(q[0], q[1]), pack_bf16(q[2], q[3]), pack_bf16(q[4], q[5]),
                   pack_bf16(q[6], q[7]));
    *reinterpret_cast<uint4*>(tile + tile_off(row, (k_lo >> 3) + c, kchunks)) =
        make_uint4(pack_bf16(r[0], r[1]), pack_bf16(r[2], r[3]), pack_bf16(r[4], r[5]),
                   pack_bf16(r[6], r[7]));
  }
}

__device__ __forceinline__ float amax_bf16(const uint4& v) {
  float m = 0.f;
  const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) m = fmaxf(m, fmaxf(fabsf(bf16_lo(q[j])), fabsf(bf16_hi(q[j]))));
  return m;
}

// the larger magnitudes of two pairs (a NaN gives way to the other, as in fmaxf)
__device__ __forceinline__ uint32_t max_abs_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  a &= 0x7fff7fffu;
  b &= 0x7fff7fffu;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// four BF16 values times f as E4M3 codes
__device__ __forceinline__ uint32_t e4m3x4_of_bf16(uint32_t a, uint32_t b, float f) {
  const float2 p = __fmul2_rn(make_float2(bf16_lo(a), bf16_hi(a)), make_float2(f, f));
  const float2 q = __fmul2_rn(make_float2(bf16_lo(b), bf16_hi(b)), make_float2(f, f));
  return pack_e4m3x4(p.x, p.y, q.x, q.y);
}

// ---- row copies at hidden 128 -------------------------------------------------
// A warp's 32 rows of 256 bytes (128 BF16 values, or two rows of 128 E4M3 codes),
// in registers between their load and their way into a tile, so that a load can be
// in flight during an MMA or the epilogue. Half a warp copies a row: a load reads
// whole lines, and a store into 128-byte rows of the 128-byte swizzle fills whole
// rows. (With a row per thread, or four lanes per row, every load touched 32 lines
// and the kernels were bound by the shared memory pipe: edge encoder on 5.2 M rows
// 1.52 -> 1.14 ms, node step on 0.87 M rows 0.41 -> 0.29 ms, the latter with the two
// tiles per SM of Layout::NODE8.)
// `id`: each lane's own row (lane l: row l of the warp); rows that do not exist read
// another (their results are not stored).
struct HalfRows {
  static constexpr int kBlock = kRows * 128;  // bytes of a tile's block of 128-byte rows
  uint4 v[16];
  __device__ __forceinline__ void load(const void* src, int id) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int row = __shfl_sync(0xffffffffu, id, 2 * i + (lane >> 4));
      v[i] = reinterpret_cast<const uint4*>(src)[size_t(max(row, 0)) * 16 + (lane & 15)];
    }
  }
  // as they are: the rows' two halves of 128 bytes into two blocks
  __device__ __forceinline__ void put(uint8_t* tile) const {
    const int lane = threadIdx.x & 31, piece = lane & 15, warp = (threadIdx.x & (kRows - 1)) >> 5;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int row = 32 * warp + 2 * i + (lane >> 4);
      *reinterpret_cast<uint4*>(tile + (piece >> 3) * kBlock + row * 128 + (((piece & 7) ^ (row & 7)) << 4)) = v[i];
    }
  }
  // as E4M3 codes under each row's own scale (the owner lane gets it)
  __device__ __forceinline__ float put_e4m3(uint8_t* tile) const {
    const int lane = threadIdx.x & 31, half = lane >> 4, piece = lane & 15;
    const int warp = (threadIdx.x & (kRows - 1)) >> 5;
    float m = 0.f;  // lane (half, piece): the maximum of row 2 piece + half
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      uint32_t q = max_abs_bf16x2(max_abs_bf16x2(v[i].x, v[i].y), max_abs_bf16x2(v[i].z, v[i].w));
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) q = max_abs_bf16x2(q, __shfl_xor_sync(0xffffffffu, q, d));
      if (piece == i) m = fmaxf(bf16_lo(q), bf16_hi(q));
    }
    const float iv = m > 0.f ? 448.f / m : 1.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float f = __shfl_sync(0xffffffffu, iv, 16 * half + i);
      const int row = 32 * warp + 2 * i + half;
      uint2 o;
      o.x = e4m3x4_of_bf16(v[i].x, v[i].y, f);
      o.y = e4m3x4_of_bf16(v[i].z, v[i].w, f);
      *reinterpret_cast<uint2*>(tile + row * 128 + (((piece >> 1) ^ (row & 7)) << 4) + (piece & 1) * 8) = o;
    }
    return __shfl_sync(0xffffffffu, m > 0.f ? m / 448.f : 1.f, (lane & 1) * 16 + (lane >> 1));
  }
};

// A warp's 32 state rows of H BF16 values, 32 columns (64 bytes) at a time,
// through its staging block: lane (row lane / 4 + 8 i, part lane % 4) moves 16
// bytes between global memory and the block, lane l reads and writes row l (rows
// STRIDE bytes apart: 80, or 64 with the parts swizzled).
template <int H, int STRIDE>
struct RowStage {
  uint8_t* blk;                // the warp's block
  const __nv_bfloat16* first;  // the warp's first row
  int n;                       // rows of the warp that exist
  uint4 v[4];

  __device__ __forceinline__ uint4* slot(int row, int part) const {
    return reinterpret_cast<uint4*>(blk + row * STRIDE + 16 * (STRIDE == 64 ? part ^ ((row >> 1) & 3) : part));
  }
  // columns 32 c .. 32 c + 31 of every row into registers (missing rows: row 0)
  __device__ __forceinline__ void fetch(int c) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = (lane >> 2) + 8 * i;
      v[i] = n > 0 ? *(reinterpret_cast<const uint4*>(first + size_t(row < n ? row : 0) * H + 32 * c) + (lane & 3))
                   : make_uint4(0, 0, 0, 0);
    }
  }
  // the fetched columns of this lane's row
  __device__ __forceinline__ void rows(uint4 (&out)[4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) *slot((lane >> 2) + 8 * i, lane & 3) = v[i];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = *slot(lane, j);
    __syncwarp();
  }
  // columns 32 c .. of this lane's row to global memory
  __device__ __forceinline__ void put(int c, const uint4 (&in)[4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j) *slot(lane, j) = in[j];
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = (lane >> 2) + 8 * i;
      if (row < n)
        *(reinterpret_cast<uint4*>(const_cast<__nv_bfloat16*>(first) + size_t(row) * H + 32 * c) + (lane & 3)) =
            *slot(row, lane & 3);
    }
    __syncwarp();
  }
};

// the lo parts of 32 columns, bf16(z - bf16(z)), packed
__device__ __forceinline__ void lo_parts(const float (&z)[32], uint4 (&o)[4]) {
  float l[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) l[j] = z[j] - __bfloat162float(__float2bfloat16_rn(z[j]));
#pragma unroll
  for (int q = 0; q < 4; ++q)
    o[q] = make_uint4(pack_bf16(l[8 * q], l[8 * q + 1]), pack_bf16(l[8 * q + 2], l[8 * q + 3]),
                      pack_bf16(l[8 * q + 4], l[8 * q + 5]), pack_bf16(l[8 * q + 6], l[8 * q + 7]));
}
// acc[0..7] += the 8 BF16 values of u
__device__ __forceinline__ void add_bf16x8(float* acc, const uint4& u) {
  acc[0] += bf16_lo(u.x);
  acc[1] += bf16_hi(u.x);
  acc[2] += bf16_lo(u.y);
  acc[3] += bf16_hi(u.y);
  acc[4] += bf16_lo(u.z);
  acc[5] += bf16_hi(u.z);
  acc[6] += bf16_lo(u.w);
  acc[7] += bf16_hi(u.w);
}

// x[j] = v[j] + b[j] (BF16) or fma(v[j], sc[j], b[j]) (FP8) for 32 columns,
// the parameters read as 16-byte broadcasts from shared memory
__device__ __forceinline__ void add_params(const float (&v)[32], const float* b, float (&x)[32]) {
  const float4* b4 = reinterpret_cast<const float4*>(b);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 bb = b4[q];
    x[4 * q] = v[4 * q] + bb.x;
    x[4 * q + 1] = v[4 * q + 1] + bb.y;
    x[4 * q + 2] = v[4 * q + 2] + bb.z;
    x[4 * q + 3] = v[4 * q + 3] + bb.w;
  }
}

// FP8 messages of a hit in the projection rows' memory ([h_cap][2H] floats): 2H
// codes [m_out | m_in] per hit from the start, then two scales per hit
template <int H>
__device__ __forceinline__ uint8_t* msg_codes(const Ws& w, int row) {
  return reinterpret_cast<uint8_t*>(w.pstate) + size_t(row) * 2 * H;
}
template <int H>
__device__ __forceinline__ float* msg_scales(const Ws& w, int row) {
  return w.pstate + size_t(w.h_cap) * (2 * H / 4) + size_t(row) * 2;
}

// Issue the MMAs of one layer: A tile (kchunks 16-byte chunks per row) times
// the weight image (H rows) over K elements. FP8 with segments: segment s
// (H columns of K) accumulates into TMEM columns [s*H, (s+1)*H).
template <int H, bool FP8>
__device__ __forceinline__ void issue_layer(uint32_t tmem, const uint8_t* A, const uint8_t* W,
                                            int K, int nseg_sep, bool accumulate = false) {
  constexpr int ESZ = FP8 ? 1 : 2;
  constexpr int KSTEP = FP8 ? 32 : 16;
  constexpr uint32_t IDESC = FP8 ? idesc_e4m3(kRows, H) : idesc_bf16(kRows, H);
  const int kchunks = K * ESZ / 16;
  const uint32_t sbo = uint32_t(kchunks) * 128;
  const uint32_t a0 = smem_u32(A), w0 = smem_u32(W);
  const int seg_len = nseg_sep > 1 ? K / nseg_sep : K;
  for (int k = 0; k < K; k += KSTEP) {
    const int seg = k / seg_len;
    const uint32_t byte_k = uint32_t(k * ESZ / 16) * 128;  // chunk index * 128
    const uint64_t ad = smem_desc(a0 + byte_k, 128, sbo);
    const uint64_t bd = smem_desc(w0 + byte_k, 128, sbo);
    const uint32_t d = tmem + uint32_t(nseg_sep > 1 ? seg * H : 0);
    const uint32_t acc = accumulate || (k % seg_len) != 0;
    if constexpr (FP8)
      mma_e4m3(d, ad, bd, IDESC, acc);
    else
      mma_bf16(d, ad, bd, IDESC, acc);
  }
}

// Layer 1 of a BF16 tile kept as swizzled blocks of 32 columns (K of them in all).
template <int H, int K>
__device__ __forceinline__ void issue_blocks_bf16(uint32_t tmem, const uint8_t* A, const uint8_t* W) {
  constexpr uint32_t IDESC = idesc_bf16(kRows, H);
  constexpr uint32_t SBO_W = uint32_t(K * 2 / 16) * 128;
  const uint32_t a0 = smem_u32(A), w0 = smem_u32(W);
#pragma unroll
  for (int k = 0; k < K; k += 16)
    mma_bf16(tmem, smem_desc_sw64(a0 + uint32_t((k / 32) * (kRows * 64) + (k % 32) * 2)),
             smem_desc(w0 + uint32_t(k * 2 / 16) * 128, 128, SBO_W), IDESC, k > 0 ? 1u : 0u);
}

// One pass of a three-pass FP8 layer 1 (K = 3H, H = 128): the one-segment A tile
// (E4M3, 128 bytes per row, 128-byte swizzle) times K chunk `pass` of the weight
// image (E4M3, 3H per row), starting its accumulator or adding to it.
template <int H>
__device__ __forceinline__ void issue_pass_e4m3(uint32_t tmem, const uint8_t* A, const uint8_t* W,
                                                int pass, bool add) {
  static_assert(H == 128, "a row of one segment is one 128-byte swizzle row");
  constexpr uint32_t IDESC = idesc_e4m3(kRows, H);
  constexpr uint32_t SBO_W = uint32_t(3 * H / 16) * 128;
  const uint32_t a0 = smem_u32(A), w0 = smem_u32(W) + uint32_t(pass * (H / 16)) * 128;
#pragma unroll
  for (int k = 0; k < H; k += 32)
    mma_e4m3(tmem, smem_desc_sw128(a0 + uint32_t(k)), smem_desc(w0 + uint32_t(k / 16) * 128, 128, SBO_W), IDESC,
             (add || k > 0) ? 1u : 0u);
}

// One pass of the split edge encoder's layer 1 at hidden 128 (K = 2H): the
// one-segment BF16 A tile (two blocks of 64 columns, 128-byte swizzle) times K half pass % 2 of the weight image; pass 0
// starts the accumulator, the others add to it.
template <int H>
__device__ __forceinline__ void issue_pass_bf16(uint32_t tmem, const uint8_t* A, const uint8_t* W,
                                                int pass) {
  constexpr uint32_t IDESC = idesc_bf16(kRows, H);
  constexpr uint32_t SBO_W = uint32_t(2 * H * 2 / 16) * 128;
  const uint32_t a0 = smem_u32(A), w0 = smem_u32(W) + uint32_t((pass & 1) * (H * 2 / 16)) * 128;
#pragma unroll
  for (int k = 0; k < H; k += 16) {
    const uint32_t byte_k = uint32_t(k * 2 / 16) * 128;
    mma_bf16(tmem, smem_desc_sw128(a0 + uint32_t((k / 64) * HalfRows::kBlock + (k % 64) * 2)),
             smem_desc(w0 + byte_k, 128, SBO_W), IDESC, (pass > 0 || k > 0) ? 1u : 0u);
  }
}

// Issue the cp.async copies of a warp's 32 rows of a BF16 tile's layer-1 input
// into the swizzled blocks of `A` (16-byte chunk c of row r at chunk
// c ^ ((r >> 1) & 3)): lane (row lane / 4 + 8 i, part lane % 4). Rows at or past
// `hi` are zero-filled. id_a, id_b: each lane's own row's two gathered rows.
template <int H, int MODE>
__device__ __forceinline__ void gather_blocks(uint8_t* A, const TcArgs& p, int row0, int hi, int warp,
                                              int id_a, int id_b) {
  using bf = __nv_bfloat16;
  constexpr int NS = MODE == M_EDGE_ENC ? 4 : n_seg(MODE);
  const Ws& w = p.w;
  const int lane = threadIdx.x & 31, part = lane & 3;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int wr = (lane >> 2) + 8 * i, rr = 32 * warp + wr, r = row0 + rr;
    const bool in = r < hi;
    const size_t row = size_t(in ? r : 0) * H;
    size_t ga = 0, gb = 0;
    if constexpr (MODE != M_NODE_UPD && MODE != M_CLS) {
      ga = size_t(max(__shfl_sync(0xffffffffu, id_a, wr), 0)) * H;
      gb = size_t(max(__shfl_sync(0xffffffffu, id_b, wr), 0)) * H;
    }
    const bf* src[4] = {};
    if constexpr (MODE == M_NODE_UPD) {
      src[0] = w.hstate16 + row;
      src[1] = reinterpret_cast<const bf*>(w.pstate) + 2 * row;
      src[2] = src[1] + H;
    } else if constexpr (MODE == M_EDGE_ENC) {
      const bf* hlo = reinterpret_cast<const bf*>(w.hstate);
      src[0] = w.hstate16 + ga;
      src[1] = w.hstate16 + gb;
      src[2] = hlo + ga;
      src[3] = hlo + gb;
    } else if constexpr (MODE == M_TRIP) {
      src[0] = w.estate16 + ga;
      src[1] = w.estate16 + gb;
    } else {
      src[0] = w.estate16 + row;
      src[1] = w.hstate16 + ga;
      src[2] = w.hstate16 + gb;
    }
    uint8_t* d = A + rr * 64 + ((part ^ ((rr >> 1) & 3)) << 4);
#pragma unroll
    for (int sg = 0; sg < NS; ++sg)
#pragma unroll
      for (int c = 0; c < H / 32; ++c)
        cp_async16(d + (sg * (H / 32) + c) * (kRows * 64), src[sg] + 32 * c + 8 * part, in ? 16u : 0u);
  }
}

// barrier of a tile's 128 threads: the CTA's, or with two warpgroups their own
template <int G>
__device__ __forceinline__ void group_sync(int wg) {
  if constexpr (G == 1)
    __syncthreads();
  else
    asm volatile("barrier.cta.sync.aligned %0, %1;" ::"r"(1 + wg), "n"(kRows) : "memory");
}
template <int G>
__device__ __forceinline__ bool group_sync_or(int wg, bool v) {
  if constexpr (G == 1) {
    return __syncthreads_or(v);
  } else {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred.aligned q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"(uint32_t(v)), "r"(1 + wg), "n"(kRows)
        : "memory");
    return r != 0;
  }
}

// The loaders of the FP8 edge steps at hidden 128: warpgroup `wg`'s tiles' rows,
// quantised into its ring of one-segment tiles (128-byte swizzle). A warp fills its
// own 32 rows of each in four steps of eight: half a warp copies a row, so that a
// load reads whole lines and a store fills whole rows; the loads run a step ahead
// (across segments and tiles: step 12 is the next tile's first). Rows that do not
// exist repeat another (their results are not stored).
// A wait that runs out ends the loader; the warpgroup's own wait then does too.
template <int H, bool FP8, int MODE>
__device__ __forceinline__ void p3_loader(const TcArgs& p, uint8_t* smem, int wg, int tid, int hi, int n_tiles) {
  using L = Layout<H, FP8, MODE>;
  const Ws& w = p.w;
  const int lane = tid & 31, half = lane >> 4, piece = lane & 15, row0 = tid & ~31;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::RING) + wg * 2 * L::P3_SLOTS;
  uint64_t* empty = full + L::P3_SLOTS;
  float2* scales = reinterpret_cast<float2*>(smem + L::SCALES) + wg * 2 * kRows;
  uint8_t* ring = smem + L::A + wg * L::A_BYTES;
  const int step = int(gridDim.x) * L::G;
  int slot = 0, uses = 0, turn = 0;
  int t = int(blockIdx.x) * L::G + wg;
  // the two hits of this lane's row of tile t
  auto row_of = [&](int t) { return min(t * kRows + tid, hi - 1); };
  if (t >= n_tiles) return;
  int id_s = w.src[row_of(t)], id_d = w.col[row_of(t)];
  float amax = fmaxf(w.hamax[id_s], w.hamax[id_d]);
  uint4 v[2][4];
  auto load_e = [&](uint4 (&v)[4], int t, int g) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      v[i] = reinterpret_cast<const uint4*>(
          w.estate16 + size_t(min(t * kRows + row0 + 8 * g + 2 * i + half, hi - 1)) * H)[piece];
  };
  auto load_h = [&](uint4 (&v)[4], int id, int g) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      v[i] = reinterpret_cast<const uint4*>(
          w.hstate16 + size_t(__shfl_sync(0xffffffffu, id, 8 * g + 2 * i + half)) * H)[piece];
  };
  // this lane's 8 bytes of rows 2 i + half of a step's eight
  uint32_t at[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    at[i] = uint32_t((row0 + 2 * i + half) * H + (((piece >> 1) ^ (2 * i + half)) << 4) + (piece & 1) * 8);
  load_e(v[0], t, 0);
  for (; t < n_tiles; t += step) {
    const int tn = min(t + step, n_tiles - 1);
    const int nid_s = w.src[row_of(tn)], nid_d = w.col[row_of(tn)];
    const float h_scale = amax > 0.f ? amax / 448.f : 1.f;
    const float hinv = 1.f / h_scale;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const int seg = k / 4, g = k % 4, n = k + 1;
      if (n < 4)
        load_e(v[n % 2], t, n);
      else if (n < 12)
        load_h(v[n % 2], n < 8 ? id_s : id_d, n % 4);
      else
        load_e(v[n % 2], tn, 0);
      if (k == 6) amax = fmaxf(w.hamax[nid_s], w.hamax[nid_d]);  // (the next tile's)
      if (g == 0) {  // (the slot's last MMA has read it)
        const bool free = uses == 0 || mbar_wait_bounded(&empty[slot], uint32_t(uses - 1) & 1u, kWaitCycles);
        if (!__all_sync(0xffffffffu, free)) return;
        // (the tile's first slot was last read by an MMA of the tile before, which the
        // warpgroup issues once all its threads have the scales of the tile before
        // that one: this tile's place)
        if (k == 0) scales[turn * kRows + tid].y = h_scale;
      }
      uint4 (&u)[4] = v[k % 2];
      float iv = hinv;
      if (seg == 0) {
        // the rows' own scales: lane `piece` i of a half takes row i's maximum
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t q = max_abs_bf16x2(max_abs_bf16x2(u[i].x, u[i].y), max_abs_bf16x2(u[i].z, u[i].w));
#pragma unroll
          for (int d = 8; d > 0; d >>= 1) q = max_abs_bf16x2(q, __shfl_xor_sync(0xffffffffu, q, d));
          if (piece == i) m = fmaxf(bf16_lo(q), bf16_hi(q));
        }
        iv = m > 0.f ? 448.f / m : 1.f;
        if (piece < 4) scales[turn * kRows + row0 + 8 * g + 2 * piece + half].x = m > 0.f ? m / 448.f : 1.f;
      }
      uint8_t* rows = ring + slot * (kRows * H) + 8 * g * H;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float f = __shfl_sync(0xffffffffu, iv, seg == 0 ? 16 * half + i : 8 * g + 2 * i + half);
        uint2 o;
        o.x = e4m3x4_of_bf16(u[i].x, u[i].y, f);
        o.y = e4m3x4_of_bf16(u[i].z, u[i].w, f);
        *reinterpret_cast<uint2*>(rows + at[i]) = o;
      }
      if (g == 3) {
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[slot]);
        if (++slot == L::P3_SLOTS) {
          slot = 0;
          ++uses;
        }
      }
    }
    id_s = nid_s;
    id_d = nid_d;
    turn ^= 1;
  }
}

// v (times the FP8 weight scale) plus the bias, columns 32 c .. 32 c + 31
template <bool FP8, int N, int M>
__device__ __forceinline__ void add_par(float (&v)[32], const float (&b)[N], const float (&sc)[M], int c) {
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    if constexpr (FP8)
      v[j] = fmaf(v[j], sc[c * 32 + j], b[c * 32 + j]);
    else
      v[j] += b[c * 32 + j];
  }
}

// (x - m, y - m) in one packed instruction, rounded like the scalar ones (packed
// subtractions, products and scales in the epilogues: FP8 edge step at hidden 128 on
// 5.2 M rows 1.478 -> 1.445 ms, no change at hidden 32)
__device__ __forceinline__ float2 sub2(float x, float y, float m) {
  return __fadd2_rn(make_float2(x, y), make_float2(-m, -m));
}

// Tiles per SM that the registers must allow: BF16 at hidden 32 as many as the
// shared memory holds (edge step on 10.1 M rows 356 us with four, 340 us with five;
// the node encoder would spill).
constexpr int min_ctas(int H, bool FP8, int MODE) { return !FP8 && H == 32 && MODE != M_NODE_ENC ? 5 : 1; }

template <int H, bool FP8, int MODE>
__global__ void __launch_bounds__((Layout<H, FP8, MODE>::THREADS), min_ctas(H, FP8, MODE)) k_tc(const TcArgs p, const __grid_constant__ TcPar<H, FP8> q) {
  using L = Layout<H, FP8, MODE>;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sW1 = smem + L::W1;
  uint8_t* sW2 = smem + L::W2;
  uint8_t* sWC = smem + L::WC;
  float* par = reinterpret_cast<float*>(smem + L::PAR);
  float* pc2 = par;          // classifier layer 2 weights [H] + bias
  float* pne = par + H + 4;  // node encoder layer 1: W[3][H], b[H]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::BAR);  // [0] weights, [1 + wg] mma
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + L::BAR + 48);

  constexpr int G = L::G;
  uint64_t* ring_bar = reinterpret_cast<uint64_t*>(smem + L::RING);
  (void)ring_bar;
  // warpgroup, row of its tile, warp of the warpgroup
  const int wg = G == 1 ? 0 : int(threadIdx.x) / kRows;
  const int tid = G == 1 ? int(threadIdx.x) : int(threadIdx.x) % kRows, warp = tid >> 5;
  uint64_t* mma_bar = bar + 1 + wg;
  const Ws& w = p.w;
  // ---- set-up: barriers, TMEM, weights --------------------------------------
  if (threadIdx.x == 0) {
    for (int i = 0; i < 1 + G; ++i) mbar_init(&bar[i], 1);
    if constexpr (L::P3)  // full: a loader's four warps; empty: a commit
      for (int i = 0; i < 2 * G * L::P3_SLOTS; ++i) mbar_init(&ring_bar[i], (i / L::P3_SLOTS) % 2 == 0 ? 4 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(tslot, G * L::TMEM_COLS);
    tmem_relinquish();
  }
  for (int i = tid; i < H; i += kRows) {
    if (MODE == M_EDGE_UPD_CLS || MODE == M_CLS || MODE == M_TRIP) pc2[i] = p.c2.WT[i * p.c2.ldo];
    if (MODE == M_NODE_ENC) {
      for (int j = 0; j < 3; ++j) pne[j * H + i] = p.ne1.WT[j * p.ne1.ldo + i];
      pne[3 * H + i] = p.ne1.b[i];
    }
  }
  if (tid == 0 && (MODE == M_EDGE_UPD_CLS || MODE == M_CLS || MODE == M_TRIP)) pc2[H] = p.c2.b[0];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tslot + uint32_t(wg * L::TMEM_COLS);
  const uint32_t tmem_lane = tmem_base + (uint32_t(warp * 32) << 16);

  if (threadIdx.x == 0) {
    uint32_t bytes = uint32_t(L::W1_BYTES + L::W2_BYTES + L::WC_BYTES);
    mbar_expect_tx(&bar[0], bytes);
    if (L::HAS_W1) bulk_g2s(sW1, MODE == M_CLS ? p.Wc : p.W1, L::W1_BYTES, &bar[0]);
    if (L::HAS_W2) bulk_g2s(sW2, p.W2, L::W2_BYTES, &bar[0]);
    if (L::HAS_WC) bulk_g2s(sWC, p.Wc, L::WC_BYTES, &bar[0]);
  }
  bool ok = mbar_wait_bounded(&bar[0], 0, kWaitCycles);
  uint32_t mma_phase = 0;
  bool mma_pending = false;  // an MMA commit not yet waited for
  const bool weights_late = __syncthreads_or(!ok);
  bool aborted = weights_late;

  pdl_begin();
  const bool edge_rows = MODE != M_NODE_ENC && MODE != M_NODE_UPD;
  int lo = 0, hi = 0;
  // no tiles after an input error (the triplet lists are only valid when the
  // triplet workspace held them)
  const int stop = MODE == M_TRIP ? (ST_INPUT | ST_CAPACITY) : ST_INPUT;
  if (!(*(volatile int32_t*)&w.counters[C_STATUS] & stop)) {
    const Batch& b = p.b;
    hi = edge_rows ? clamp_edges(w.counters, w.e_cap) : b.n_hits;
    if constexpr (MODE == M_TRIP) hi = min(*p.tn, int(w.t_cap));
  }
  const int n_tiles = (hi - lo + kRows - 1) / kRows;
  constexpr int K1 = L::K1;
  constexpr int KCH1 = K1 * L::ESZ / 16;  // 16-byte chunks per A row, layer 1
  constexpr int KCHH = H * L::ESZ / 16;   // 16-byte chunks per A row, K = H
  constexpr int KCH2 = L::K2 * L::ESZ / 16;  // 16-byte chunks per A row, layer 2

  // The node encoder leaves its encoding h in two parts, hi = bf16(h) in hstate16
  // and lo = bf16(h - hi) in the place of the FP32 states (which the re-score
  // computes anew); the edge encoder copies both into its tile.
  __nv_bfloat16* hlo = reinterpret_cast<__nv_bfloat16*>(w.hstate);
  (void)hlo;
  // wait for the MMAs committed so far; false on timeout (uniform across CTA)
  auto wait_mma = [&]() -> bool {
    mma_pending = true;
    bool good = mbar_wait_bounded(mma_bar, mma_phase, kWaitCycles);
    tc_fence_after();
    if (group_sync_or<G>(wg, !good)) return false;
    mma_phase ^= 1;
    mma_pending = false;
    return true;
  };

  const int t_first = int(blockIdx.x) * G + wg;
  HalfRows pre, pre_m;  // (pre_m: the 2H message codes of a hit)
  (void)pre;
  float n_scale[2] = {1.f, 1.f};
  (void)pre_m;
  (void)n_scale;
  int nid_s = -1, nid_d = -1;
  auto next_ids = [&](int t) {
    const int r = lo + t * kRows + tid;
    const bool in = t < n_tiles && r < hi;
    if constexpr (MODE == M_NODE_UPD || MODE == M_CLS) return;
    nid_s = in ? (MODE == M_TRIP ? p.t1 : w.src)[r] : -1;
    nid_d = in ? (MODE == M_TRIP ? p.t2 : w.col)[r] : -1;
  };
  auto node8_rows = [&](int t) {
    const int r = lo + t * kRows + tid;
    const bool in = t < n_tiles && r < hi;
    pre.load(w.hstate16, in ? r : -1);
    pre_m.load(msg_codes<H>(w, 0), in ? r : -1);
    const float2 sc = *reinterpret_cast<const float2*>(msg_scales<H>(w, in ? r : 0));
    n_scale[0] = in ? sc.x : 1.f;
    n_scale[1] = in ? sc.y : 1.f;
  };
  if constexpr (L::NODE8) node8_rows(t_first);
  // (the split edge encoder: the rows of a pass during the MMAs of the pass before)
  if constexpr (L::SPLIT2) {
    next_ids(t_first);
    pre.load(w.hstate16, nid_s);
  }
  if constexpr (L::P3) {
    // registers for the rows' passes, taken from the loaders
    if (wg >= G) {
      regs_lower<80>();
      if (!aborted) p3_loader<H, FP8, MODE>(p, smem, wg - G, tid, hi, n_tiles);
      __syncthreads();  // (the one before the clean-up)
      return;
    }
    regs_raise<176>();
  }
  int p3_slot = 0, p3_uses = 0, p3_turn = 0;
  (void)p3_slot;
  (void)p3_uses;
  (void)p3_turn;
  // BF16: rows of tile t into the blocks (its ids loaded a tile ahead)
  auto gather = [&](int t) {
    if (t < n_tiles) gather_blocks<H, MODE>(smem + L::A, p, lo + t * kRows, hi, warp, nid_s, nid_d);
    cp_async_commit();
  };
  (void)gather;
  if constexpr (L::SWZ) {
    next_ids(t_first);
    if constexpr (L::PREF) gather(t_first);
  }
  for (int t = t_first; t < n_tiles && !aborted; t += int(gridDim.x) * G) {
    const int r = lo + t * kRows + tid;
    const bool valid = r < hi;
    uint8_t* sA = smem + L::A + wg * L::A_BYTES;
    uint8_t* sHA = L::HA == L::A ? sA : smem + L::HA + wg * L::HA_BYTES;  // layer-2 input and classifier input
    float sa[3] = {1.f, 1.f, 1.f};  // FP8 per-row scales of the layer-1 segments
    int id_s = -1, id_d = -1;       // this row's source and target hit (hidden 128)
    (void)id_s;
    (void)id_d;
    uint4 keep_row[(H <= 64) ? H / 8 : 1];
    (void)keep_row;

    // ---- 1. gather ---------------------------------------------------------
    if constexpr (L::SWZ) {
      if constexpr (!L::PREF) {
        group_sync<G>(wg);  // every thread is done with the buffer
        gather(t);
      }
      next_ids(t + int(gridDim.x));
      cp_async_wait<0>();
    } else if constexpr (MODE == M_NODE_ENC) {
      // FP32 first layer (K = 3) in registers, then LayerNorm + ReLU into A
      float hid[H];
      if (valid) {
        const float4 q = w.pos[r];
        const float f0 = q.x / p.fs[3], f1 = q.y / p.fs[4], f2 = q.z / p.fs[5];
#pragma unroll
        for (int i = 0; i < H; ++i) {
          float a = pne[3 * H + i];
          a = fmaf(f0, pne[i], a);
          a = fmaf(f1, pne[H + i], a);
          a = fmaf(f2, pne[2 * H + i], a);
          hid[i] = a;
        }
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < H; ++i) s += hid[i];
        const float mean = s / float(H);
        float v = 0.f;
#pragma unroll
        for (int i = 0; i < H; ++i) {
          const float d = hid[i] - mean;
          v = fmaf(d, d, v);
        }
        const float inv = 1.0f / sqrtf(v / float(H) + kLnEps);
        float amax = 0.f;
#pragma unroll
        for (int i = 0; i < H; ++i) {
          hid[i] = fmaxf((hid[i] - mean) * inv, 0.f);
          amax = fmaxf(amax, hid[i]);
        }
        sa[0] = FP8 ? (amax > 0.f ? amax / 448.f : 1.f) : 1.f;
        if constexpr (L::SPLIT)
          put_row_split(sHA, tid, KCH2, 0, H, hid, H);
        else
          put_row_f32<FP8>(sHA, tid, KCHH, 0, hid, H, FP8 ? (amax > 0.f ? 448.f / amax : 1.f) : 1.f);
      } else {
#pragma unroll
        for (int i = 0; i < H; ++i) hid[i] = 0.f;
        for (int k = 0; k < L::K2; k += H) put_row_f32<FP8>(sHA, tid, KCH2, k, hid, H, 1.f);
      }
    } else if constexpr (L::NODE8) {
      // h under its own scale, the messages as the message kernel left them
      sa[1] = n_scale[0];
      sa[2] = n_scale[1];
      sa[0] = pre.put_e4m3(sA);
      pre_m.put(sA + HalfRows::kBlock);
    } else if constexpr (MODE == M_NODE_UPD) {
      // (FP8, hidden 32 and 64)
      if (valid) {
        sa[0] = put_row_e4m3<H>(sA, tid, KCH1, 0, w.hstate16 + size_t(r) * H,
                                H <= 64 ? keep_row : nullptr);
        const uint4* m4 = reinterpret_cast<const uint4*>(msg_codes<H>(w, r));
#pragma unroll
        for (int c = 0; c < 2 * H / 16; ++c)
          *reinterpret_cast<uint4*>(sA + tile_off(tid, H / 16 + c, KCH1)) = m4[c];
        sa[1] = msg_scales<H>(w, r)[0];
        sa[2] = msg_scales<H>(w, r)[1];
      } else {
        float z[16] = {};
        for (int k = 0; k < K1; k += 16) put_row_f32<FP8>(sA, tid, KCH1, k, z, 16, 1.f);
      }
    } else if constexpr (L::P3) {
      // (the loaders)
    } else if constexpr (L::SPLIT2) {
      // pass 0: hi(h_src)
      id_s = nid_s;
      id_d = nid_d;
      next_ids(t + int(gridDim.x) * G);
      pre.put(sA);
    } else {
      // (FP8) edge rows: [e], [h_src, h_dst], [e, h_src, h_dst]
      if (valid) {
        int seg = 0;
        if constexpr (MODE != M_EDGE_ENC) {
          sa[0] = put_row_e4m3<H>(sA, tid, KCH1, 0, w.estate16 + size_t(r) * H,
                                  (H <= 64 && MODE != M_CLS) ? keep_row : nullptr);
          seg = 1;
        }
        if constexpr (MODE != M_CLS) {
          sa[seg] = put_row_e4m3<H>(sA, tid, KCH1, seg * H, w.hstate16 + size_t(w.src[r]) * H, nullptr);
          sa[seg + 1] = put_row_e4m3<H>(sA, tid, KCH1, (seg + 1) * H, w.hstate16 + size_t(w.col[r]) * H,
                                        nullptr);
        }
      } else {
        float z[16] = {};
        for (int k = 0; k < K1; k += 16) put_row_f32<FP8>(sA, tid, KCH1, k, z, 16, 1.f);
      }
    }
    fence_proxy_async();
    tc_fence_before();
    group_sync<G>(wg);

    float hid_scale = 1.f;  // FP8 per-row scale of the layer-2 input
    if constexpr (MODE != M_NODE_ENC) {
      // ---- 2. layer 1 ------------------------------------------------------
      bool late = false;
      if (tid == 0) {
        tc_fence_after();
        if constexpr (L::P3) {
          // e, h_src, h_dst as the loaders fill their slots (after a wait that ran
          // out: no commit, and wait_mma runs out too)
          uint64_t* full = ring_bar + wg * 2 * L::P3_SLOTS;
          bool filled = true;
          for (int pass = 0; pass < 3 && filled; ++pass) {
            const int sl = (p3_slot + pass) % L::P3_SLOTS;
            const int use = p3_uses + (p3_slot + pass) / L::P3_SLOTS;
            filled = mbar_wait_bounded(&full[sl], uint32_t(use) & 1u, kWaitCycles);
            if (!filled) break;
            issue_pass_e4m3<H>(tmem_base + uint32_t(pass > 0 ? H : 0), sA + sl * (kRows * H), sW1, pass, pass == 2);
            mma_commit(&full[L::P3_SLOTS + sl]);
          }
          late = !filled;
        } else if constexpr (L::NODE8) {
          issue_pass_e4m3<H>(tmem_base, sA, sW1, 0, false);
          issue_pass_e4m3<H>(tmem_base + uint32_t(H), sA + HalfRows::kBlock, sW1, 1, false);
        } else if constexpr (L::SPLIT2)
          issue_pass_bf16<H>(tmem_base, sA, sW1, 0);
        else if constexpr (L::SWZ)
          issue_blocks_bf16<H, K1>(tmem_base, sA, sW1);
        else
          issue_layer<H, FP8>(tmem_base, sA, sW1, K1, FP8 ? L::NSEG : 1);
        if (!late) mma_commit(mma_bar);
      }
      if constexpr (L::SPLIT2) pre.load(w.hstate16, id_d);
      if (!wait_mma()) {
        aborted = true;
        break;
      }
      if constexpr (L::P3) {
        // (the barrier in wait_mma orders the loader's scales before these reads)
        const float2 sc = reinterpret_cast<const float2*>(smem + L::SCALES)[(wg * 2 + p3_turn) * kRows + tid];
        sa[0] = sc.x;
        sa[1] = sc.y;
        p3_turn ^= 1;
        p3_uses += (p3_slot + 3) / L::P3_SLOTS;
        p3_slot = (p3_slot + 3) % L::P3_SLOTS;
      }
      if constexpr (L::SPLIT2) {
        // hi(h_dst), lo(h_src), lo(h_dst) into the same tile, accumulated
        for (int pass = 1; pass <= 3 && !aborted; ++pass) {
          pre.put(sA);
          fence_proxy_async();
          tc_fence_before();
          group_sync<G>(wg);
          if (tid == 0) {
            tc_fence_after();
            issue_pass_bf16<H>(tmem_base, sA, sW1, pass);
            mma_commit(mma_bar);
          }
          if (pass < 3) pre.load(hlo, pass == 1 ? id_s : id_d);
          if (!wait_mma()) aborted = true;
        }
        if (aborted) break;
      }
      if constexpr (L::SWZ && L::HAS_W2 && MODE != M_EDGE_ENC) {
        // the residual: this row's first segment, before the buffer is refilled
        constexpr int NK = H <= 64 ? H / 8 : 1;
#pragma unroll
        for (int c = 0; c < NK; ++c)
          keep_row[c] = *reinterpret_cast<const uint4*>(sA + (c / 4) * (kRows * 64) + tid * 64 +
                                                        (((c & 3) ^ ((tid >> 1) & 3)) << 4));
      }
      if constexpr (L::PREF && !L::HAS_W2) gather(t + int(gridDim.x));
      // ---- 3. bias + LayerNorm + ReLU (-> A as the next operand, or the
      //         classifier output for M_CLS) -------------------------------
      // x[n] = s_w[n] * sum_seg s_a[seg] * acc_seg[n] + b[n]  (FP8)
      //      = acc[n] + b[n]                                   (BF16)
      auto xval_ld = [&](int c, float (&v)[32]) {
        tmem_ld32(tmem_lane + uint32_t(c * 32), v);
        if constexpr (FP8) {
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float2 y = __fmul2_rn(make_float2(v[j], v[j + 1]), make_float2(sa[0], sa[0]));
            v[j] = y.x;
            v[j + 1] = y.y;
          }
#pragma unroll
          for (int s = 1; s < L::TSEG; ++s) {
            float u[32];
            tmem_ld32(tmem_lane + uint32_t(s * H + c * 32), u);
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const float2 y = __ffma2_rn(make_float2(u[j], u[j + 1]), make_float2(sa[s], sa[s]), make_float2(v[j], v[j + 1]));
              v[j] = y.x;
              v[j + 1] = y.y;
            }
          }
        }
        tmem_wait_ld();
        add_par<FP8>(v, q.b1, q.s1, c);
      };
      // the row is read from tensor memory once and kept in registers (at h = 128
      // the three passes over it waited on tcgen05.ld each time: FP8 edge step on
      // 5.2 M rows 2.22 -> 1.95 ms, node step on 0.87 M rows 0.52 -> 0.42 ms)
      float xc[H / 32][32];
      if constexpr (L::NODE8) {
        auto add_block = [&](int block, float f, bool first) {
#pragma unroll
          for (int c = 0; c < H / 32; ++c) {
            float u[32];
            tmem_ld32(tmem_lane + uint32_t(block * H + c * 32), u);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) xc[c][j] = first ? u[j] * f : fmaf(u[j], f, xc[c][j]);
          }
        };
        add_block(0, sa[0], true);
        tc_fence_before();
        group_sync<G>(wg);
        if (tid == 0) {
          tc_fence_after();
          issue_pass_e4m3<H>(tmem_base, sA + 2 * HalfRows::kBlock, sW1, 2, false);
          mma_commit(mma_bar);
        }
        add_block(1, sa[1], false);
        if (!wait_mma()) {
          aborted = true;
          break;
        }
        add_block(0, sa[2], false);
#pragma unroll
        for (int c = 0; c < H / 32; ++c) add_par<FP8>(xc[c], q.b1, q.s1, c);
      } else {
#pragma unroll
        for (int c = 0; c < H / 32; ++c) xval_ld(c, xc[c]);
      }
      auto xval = [&](int c, float (&x)[32]) {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = xc[c][j];
      };
      float sum = 0.f, xmax = -INFINITY;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        xval(c, x);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          sum += x[j];
          xmax = fmaxf(xmax, x[j]);
        }
      }
      const float mean = sum / float(H);
      float var = 0.f;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        xval(c, x);
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 d = sub2(x[j], x[j + 1], mean);
          var = fmaf(d.x, d.x, var);
          var = fmaf(d.y, d.y, var);
        }
      }
      const float inv = 1.0f / sqrtf(var / float(H) + kLnEps);
      if constexpr (MODE == M_CLS || MODE == M_TRIP) {
        float logit = pc2[H];
#pragma unroll
        for (int c = 0; c < H / 32; ++c) {
          float x[32];
          xval(c, x);
#pragma unroll
          for (int j = 0; j < 32; ++j) logit = fmaf(fmaxf((x[j] - mean) * inv, 0.f), pc2[c * 32 + j], logit);
        }
        if (valid) {
          if constexpr (MODE == M_TRIP) {
            p.tlogit[r] = logit;
            p.tkeep[r] = logit >= p.cut ? 1 : 0;
          } else {
            w.logit[r] = logit;
            w.keep[r] = logit >= p.cut ? 1 : 0;
          }
        }
        tc_fence_before();
        continue;
      }
      const float hmax = fmaxf((xmax - mean) * inv, 0.f);
      hid_scale = FP8 ? (hmax > 0.f ? hmax / 448.f : 1.f) : 1.f;
      const float hinv = FP8 ? (hmax > 0.f ? 448.f / hmax : 1.f) : 1.f;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        xval(c, x);
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 y = __fmul2_rn(sub2(x[j], x[j + 1], mean), make_float2(inv, inv));
          x[j] = fmaxf(y.x, 0.f);
          x[j + 1] = fmaxf(y.y, 0.f);
        }
        put_row_f32<FP8>(sHA, tid, KCHH, c * 32, x, 32, hinv);
      }
      fence_proxy_async();
      tc_fence_before();
      group_sync<G>(wg);
    } else {
      hid_scale = sa[0];
    }

    // the warp's state rows on their way out (and in, the residual, at hidden 128) through
    // its staging block: the forms of Layout::OUT_STAGE and COOP
    constexpr bool NODE_ROWS = MODE == M_NODE_ENC || MODE == M_NODE_UPD;
    const int row0 = r - (tid & 31);
    RowStage<H, L::OUT_STAGE ? 64 : L::STAGE_ROW> st{
        L::OUT_STAGE ? sHA + warp * 32 * L::K2 * 2 : smem + L::STAGE + (wg * kRows + warp * 32) * L::STAGE_ROW,
        (NODE_ROWS ? w.hstate16 : w.estate16) + size_t(row0) * H, min(max(hi - row0, 0), 32), {}};
    (void)st;
    // ---- 4. layer 2 ----------------------------------------------------------
    if (tid == 0) {
      tc_fence_after();
      issue_layer<H, FP8>(tmem_base, sHA, sW2, L::K2, 1);
      mma_commit(mma_bar);
    }
    // (every thread has its residual and is past the barrier above)
    if constexpr (L::PREF) gather(t + int(gridDim.x));
    if constexpr (L::P3) st.fetch(0);
    if constexpr (L::NODE8) node8_rows(t + int(gridDim.x) * G);
    if constexpr (L::SPLIT2) pre.load(w.hstate16, nid_s);
    if (!wait_mma()) {
      aborted = true;
      break;
    }
    // z[n] = s_w2[n] * s_h * acc[n] + b2[n] (FP8) or acc[n] + b2[n]
    auto zval = [&](int c, float (&v)[32]) {
      tmem_ld32(tmem_lane + uint32_t(c * 32), v);
      tmem_wait_ld();
      if constexpr (FP8) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] *= hid_scale;
      }
      add_par<FP8>(v, q.b2, q.s2, c);
    };
    // ZB chunks of 32 columns from chunk c on, their loads in flight together
    constexpr int ZB = L::P3 ? 2 : 1;
    auto zvals = [&](int c, float (*z)[32]) {
#pragma unroll
      for (int i = 0; i < ZB; ++i) tmem_ld32(tmem_lane + uint32_t((c + i) * 32), z[i]);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < ZB; ++i) {
        if constexpr (FP8) {
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float2 y = __fmul2_rn(make_float2(z[i][j], z[i][j + 1]), make_float2(hid_scale, hid_scale));
            z[i][j] = y.x;
            z[i][j + 1] = y.y;
          }
        }
        add_par<FP8>(z[i], q.b2, q.s2, c + i);
      }
    };
    (void)zvals;
    // residual input row (BF16) for the update modes
    auto resid = [&](int c, float (&z)[32]) {
      if constexpr (L::COOP && MODE == M_EDGE_UPD_CLS) {
        uint4 e[4];
        st.rows(e);
        if (c + 1 < H / 32) st.fetch(c + 1);
#pragma unroll
        for (int q = 0; q < 4; ++q) add_bf16x8(z + 8 * q, e[q]);
      } else if constexpr (MODE == M_NODE_UPD || MODE == M_EDGE_UPD || MODE == M_EDGE_UPD_CLS) {
        const __nv_bfloat16* rowp = (MODE == M_NODE_UPD ? w.hstate16 : w.estate16) + size_t(r) * H;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 u = (H <= 64) ? keep_row[c * 4 + q] : reinterpret_cast<const uint4*>(rowp)[c * 4 + q];
          add_bf16x8(z + 8 * q, u);
        }
      }
    };

    if constexpr (MODE != M_EDGE_UPD_CLS) {
      // ---- 5. store the new state (BF16) -----------------------------------
      __nv_bfloat16* dst = (NODE_ROWS ? w.hstate16 : w.estate16) + size_t(r) * H;
      float row_max = 0.f;  // largest |stored value| of a node row
      auto st_lo = st;  // (node encoder: the lo parts)
      if constexpr (MODE == M_NODE_ENC) st_lo.first = hlo + size_t(row0) * H;
      (void)st_lo;
      if constexpr (L::OUT_STAGE) {
#pragma unroll
        for (int c = 0; c < H / 32; ++c) {
          float z[32];
          zval(c, z);
          if constexpr (MODE == M_NODE_UPD || MODE == M_EDGE_UPD) resid(c, z);
          uint4 o[4];
          if constexpr (MODE == M_NODE_ENC) {
            lo_parts(z, o);
            st_lo.put(c, o);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            o[q] = make_uint4(pack_bf16(z[8 * q], z[8 * q + 1]), pack_bf16(z[8 * q + 2], z[8 * q + 3]),
                              pack_bf16(z[8 * q + 4], z[8 * q + 5]), pack_bf16(z[8 * q + 6], z[8 * q + 7]));
          st.put(c, o);
        }
      } else if constexpr (L::COOP) {
        constexpr bool RESID = MODE == M_NODE_UPD || MODE == M_EDGE_UPD;
        if constexpr (RESID && !L::P3) st.fetch(0);
        float zb[ZB][32];
#pragma unroll
        for (int c = 0; c < H / 32; ++c) {
          if (c % ZB == 0) zvals(c, zb);
          float (&z)[32] = zb[c % ZB];
          if constexpr (RESID) {
            uint4 e[4];
            st.rows(e);
            if (c + 1 < H / 32) st.fetch(c + 1);
#pragma unroll
            for (int q = 0; q < 4; ++q) add_bf16x8(z + 8 * q, e[q]);
          }
          uint4 o[4];
          if constexpr (L::SPLIT && MODE == M_NODE_ENC) {
            lo_parts(z, o);
            st_lo.put(c, o);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            o[q] = make_uint4(pack_bf16(z[8 * q], z[8 * q + 1]), pack_bf16(z[8 * q + 2], z[8 * q + 3]),
                              pack_bf16(z[8 * q + 4], z[8 * q + 5]), pack_bf16(z[8 * q + 6], z[8 * q + 7]));
            if constexpr (NODE_ROWS) row_max = fmaxf(row_max, amax_bf16(o[q]));
          }
          st.put(c, o);
        }
      } else {
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float z[32];
        zval(c, z);
        if (valid) {
          resid(c, z);
          uint4* d4 = reinterpret_cast<uint4*>(dst) + c * 4;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 u = make_uint4(pack_bf16(z[8 * q], z[8 * q + 1]), pack_bf16(z[8 * q + 2], z[8 * q + 3]),
                                       pack_bf16(z[8 * q + 4], z[8 * q + 5]), pack_bf16(z[8 * q + 6], z[8 * q + 7]));
            d4[q] = u;
          }
        }
      }
      }
      // (read by the FP8 edge steps at hidden 128 for their shared h scale)
      if constexpr (NODE_ROWS && H == 128)
        if (valid && w.hamax != nullptr) w.hamax[r] = row_max;
      tc_fence_before();
    } else {
      // ---- 5'. classifier on the new edge state, then the cut ---------------
      float zc[H / 32][32];  // the new state
#pragma unroll
      for (int c = 0; c < H / 32; c += ZB) zvals(c, zc + c);
      float emax = 0.f;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        resid(c, zc[c]);
        if constexpr (FP8) {
#pragma unroll
          for (int j = 0; j < 32; ++j) emax = fmaxf(emax, fabsf(zc[c][j]));
        }
      }
      const float es = FP8 ? (emax > 0.f ? emax / 448.f : 1.f) : 1.f;
      const float einv = FP8 ? (emax > 0.f ? 448.f / emax : 1.f) : 1.f;
      // rounded to BF16 as it would be stored, then fed on
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float (&z)[32] = zc[c];
#pragma unroll
        for (int j = 0; j < 32; ++j) z[j] = __bfloat162float(__float2bfloat16_rn(z[j]));
        put_row_f32<FP8>(sHA, tid, KCHH, c * 32, z, 32, einv);
      }
      fence_proxy_async();
      tc_fence_before();
      group_sync<G>(wg);
      if (tid == 0) {
        tc_fence_after();
        issue_layer<H, FP8>(tmem_base, sHA, sWC, H, 1);
        mma_commit(mma_bar);
      }
      if (!wait_mma()) {
        aborted = true;
        break;
      }
      auto cval_ld = [&](int c, float (&v)[32]) {
        tmem_ld32(tmem_lane + uint32_t(c * 32), v);
        tmem_wait_ld();
        if constexpr (FP8) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] *= es;
        }
        add_par<FP8>(v, q.bc, q.sc, c);
      };
      float cc[H / 32][32];
#pragma unroll
      for (int c = 0; c < H / 32; ++c) cval_ld(c, cc[c]);
      auto cval = [&](int c, float (&x)[32]) {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = cc[c][j];
      };
      float sum = 0.f;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        cval(c, x);
#pragma unroll
        for (int j = 0; j < 32; ++j) sum += x[j];
      }
      const float mean = sum / float(H);
      float var = 0.f;
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        cval(c, x);
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 d = sub2(x[j], x[j + 1], mean);
          var = fmaf(d.x, d.x, var);
          var = fmaf(d.y, d.y, var);
        }
      }
      const float inv = 1.0f / sqrtf(var / float(H) + kLnEps);
      float logit = pc2[H];
#pragma unroll
      for (int c = 0; c < H / 32; ++c) {
        float x[32];
        cval(c, x);
#pragma unroll
        for (int j = 0; j < 32; ++j) logit = fmaf(fmaxf((x[j] - mean) * inv, 0.f), pc2[c * 32 + j], logit);
      }
      if (valid) {
        w.logit[r] = logit;
        w.keep[r] = logit >= p.cut ? 1 : 0;
      }
      tc_fence_before();
    }
  }

  // ---- clean-up: on a timeout, give the outstanding MMAs one more bounded
  //      wait, then free the tensor memory -----------------------------------
  if constexpr (L::SWZ) cp_async_wait<0>();  // no copy may land after the exit
  if (aborted) {
    if (tid == 0) set_status(w.counters, ST_TIMEOUT);
    if (weights_late) mbar_wait_bounded(&bar[0], 0, kWaitCycles);
    if (mma_pending) mbar_wait_bounded(mma_bar, mma_phase, kWaitCycles);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_dealloc(tmem_base, G * L::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// BF16 edge step with TMA-staged tiles (hidden 32). Same arithmetic as
// k_tc<32, BF16, M_EDGE_UPD / M_EDGE_UPD_CLS> (the MMAs see the same operand
// values in the same K order), but the layer-1 input [e, h_src, h_dst] of a
// tile is never touched by the threads:
//   * segment 0 (e rows, contiguous edges) is one 2-D TMA box of 128 rows;
//   * segments 1 and 2 (h_src, h_dst rows) are TMA row gathers, four rows per
//     instruction, one instruction per lane of warp 0 and segment;
// each segment lands as 128 rows x 64 bytes in the 64-byte swizzle layout
// (8 KB, 1024-byte aligned), which the MMA reads through swizzled
// descriptors. One tile buffer: once layer 1 has read it and every thread has
// taken its residual row into registers, the next tile's rows load while
// layer 2 and the epilogue run. The hidden row and the classifier input are
// written by the threads into a no-swizzle tile as in k_tc.
// ---------------------------------------------------------------------------
template <int H, bool CLS>
struct TmaLayout {
  static constexpr int SEG = kRows * H * 2;  // one segment: 128 rows x 64 bytes
  static constexpr int K1 = 3 * H;
  static constexpr int W1 = 0;
  static constexpr int W1_BYTES = H * K1 * 2;
  static constexpr int W2 = align1k(W1 + W1_BYTES);
  static constexpr int W2_BYTES = H * H * 2;
  static constexpr int WC = align1k(W2 + W2_BYTES);
  static constexpr int WC_BYTES = CLS ? H * H * 2 : 0;
  static constexpr int A = align1k(WC + WC_BYTES);
  static constexpr int ABUF = 3 * SEG;
  static constexpr int HA = align1k(A + ABUF);
  static constexpr int HA_BYTES = kRows * H * 2;
  static constexpr int PAR = HA + HA_BYTES;
  static constexpr int PAR_FLOATS = 4 * H + 4;  // b1, b2, bc1, c2 weights + bias
  static constexpr int BAR = PAR + PAR_FLOATS * 4;  // [0] weights [1] mma [2] tile
  static constexpr int TOTAL = BAR + 64;
  static constexpr int ALLOC = TOTAL + 1024;  // room to align the base to 1024 bytes
};

// (registers capped so that five CTAs fit an SM, as their shared memory does)
template <int H, bool CLS>
__global__ void __launch_bounds__(kRows, 5)
    k_tc_edge_tma(const TcArgs p, const __grid_constant__ CUtensorMap map_e,
                  const __grid_constant__ CUtensorMap map_h) {
  static_assert(H == 32, "one BF16 row segment of 32 elements is one 64-byte swizzle row");
  using L = TmaLayout<H, CLS>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sW1 = smem + L::W1;
  uint8_t* sW2 = smem + L::W2;
  uint8_t* sWC = smem + L::WC;
  uint8_t* sHA = smem + L::HA;
  float* par = reinterpret_cast<float*>(smem + L::PAR);
  float* pb1 = par;
  float* pb2 = par + H;
  float* pbc = par + 2 * H;
  float* pc2 = par + 3 * H;  // classifier layer 2: H weights, then the bias
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::BAR);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + L::BAR + 32);
  constexpr int KCHH = H * 2 / 16;  // 16-byte chunks per row of the hidden tile
  constexpr int MODE = CLS ? M_EDGE_UPD_CLS : M_EDGE_UPD;
  (void)MODE;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Ws& w = p.w;
  pdl_wait();
  if (*(volatile int32_t*)&w.counters[C_STATUS] & ST_INPUT) return;

  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(&bar[i], 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tslot, 32);
    tmem_relinquish();
  }
  for (int i = tid; i < H; i += kRows) {
    pb1[i] = p.b1[i];
    pb2[i] = p.b2[i];
    pbc[i] = CLS ? p.bc1[i] : 0.f;
    pc2[i] = CLS ? p.c2.WT[i * p.c2.ldo] : 0.f;
  }
  if (tid == 0) pc2[H] = CLS ? p.c2.b[0] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tslot;
  pdl_trigger();  // (not before this block has its tensor memory)
  const uint32_t tmem_lane = tmem_base + (uint32_t(warp * 32) << 16);

  if (tid == 0) {
    mbar_expect_tx(&bar[0], uint32_t(L::W1_BYTES + L::W2_BYTES + L::WC_BYTES));
    bulk_g2s(sW1, p.W1, L::W1_BYTES, &bar[0]);
    bulk_g2s(sW2, p.W2, L::W2_BYTES, &bar[0]);
    if (CLS) bulk_g2s(sWC, p.Wc, L::WC_BYTES, &bar[0]);
  }
  const bool wok = mbar_wait_bounded(&bar[0], 0, kWaitCycles);
  const bool weights_late = __syncthreads_or(!wok);
  bool aborted = weights_late;
  uint32_t mma_phase = 0, a_phase = 0;
  bool mma_pending = false, a_pending = false;

  const int hi = clamp_edges(w.counters, w.e_cap);
  const int n_tiles = (hi + kRows - 1) / kRows;
  uint8_t* A = smem + L::A;

  // warp 0: the node indices of the four rows 4 lane .. 4 lane + 3 of tile t
  // (rows past the last edge gather node 0 and are never stored), loaded a
  // phase ahead of their use
  int sv[4] = {0, 0, 0, 0}, dv[4] = {0, 0, 0, 0};
  auto load_idx = [&](int t) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = t * kRows + 4 * lane + i;
      sv[i] = r < hi ? w.src[r] : 0;
      dv[i] = r < hi ? w.col[r] : 0;
    }
  };
  // warp 0: the loads of tile t (expect-tx first, then the box of e rows and
  // each lane's two four-row gathers)
  auto issue = [&](int t) {
    if (lane == 0) {
      mbar_expect_tx(&bar[2], uint32_t(3 * L::SEG));
      tma_load_2d(A, &map_e, 0, t * kRows, &bar[2]);
    }
    __syncwarp();
    tma_gather4(A + L::SEG + 4 * lane * (H * 2), &map_h, 0, sv[0], sv[1], sv[2], sv[3], &bar[2]);
    tma_gather4(A + 2 * L::SEG + 4 * lane * (H * 2), &map_h, 0, dv[0], dv[1], dv[2], dv[3],
                &bar[2]);
  };
  auto wait_mma = [&]() -> bool {
    mma_pending = true;
    const bool good = mbar_wait_bounded(&bar[1], mma_phase, kWaitCycles);
    tc_fence_after();
    if (__syncthreads_or(!good)) return false;
    mma_phase ^= 1;
    mma_pending = false;
    return true;
  };

  if (!aborted && int(blockIdx.x) < n_tiles) {
    if (warp == 0) {
      load_idx(blockIdx.x);
      issue(blockIdx.x);
    }
    a_pending = true;
  }
  for (int t = blockIdx.x; t < n_tiles && !aborted; t += gridDim.x) {
    const int tn = t + int(gridDim.x);
    if (warp == 0 && tn < n_tiles) load_idx(tn);  // used after layer 1
    const bool got = mbar_wait_bounded(&bar[2], a_phase, kWaitCycles);
    if (__syncthreads_or(!got)) {
      aborted = true;
      break;
    }
    a_phase ^= 1;
    a_pending = false;
    const int r = t * kRows + tid;
    const bool valid = r < hi;

    // ---- layer 1: [e, h_src, h_dst] x W1 (K = 3H, 16 per instruction) --------
    if (tid == 0) {
      tc_fence_after();
      constexpr uint32_t IDESC = idesc_bf16(kRows, H);
      constexpr uint32_t SBO_W = uint32_t(L::K1 * 2 / 16) * 128;
      const uint32_t a0 = smem_u32(A), w0 = smem_u32(sW1);
#pragma unroll
      for (int k = 0; k < L::K1; k += 16) {
        const int seg = k / H, j = (k % H) / 16;
        const uint64_t ad = smem_desc_sw64(a0 + uint32_t(seg * L::SEG + j * 32));
        const uint64_t bd = smem_desc(w0 + uint32_t(k * 2 / 16) * 128, 128, SBO_W);
        mma_bf16(tmem_base, ad, bd, IDESC, k > 0 ? 1u : 0u);
      }
      mma_commit(&bar[1]);
    }
    if (!wait_mma()) {
      aborted = true;
      break;
    }
    // the residual: this row's e from segment 0 (64-byte swizzle), kept in
    // registers so that the buffer is free once the barrier below is passed
    uint4 e_row[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      e_row[q] = *reinterpret_cast<const uint4*>(A + tid * (H * 2) + ((q ^ ((tid >> 1) & 3)) << 4));
    // ---- bias + LayerNorm + ReLU -> hidden tile --------------------------------
    float x[32];
    {
      float v[32];
      tmem_ld32(tmem_lane, v);
      tmem_wait_ld();
      add_params(v, pb1, x);
    }
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) sum += x[j];
    const float mean = sum / float(H);
    float var = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const float d = x[j] - mean;
      var = fmaf(d, d, var);
    }
    const float inv = 1.0f / sqrtf(var / float(H) + kLnEps);
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = fmaxf((x[j] - mean) * inv, 0.f);
    put_row_f32<false>(sHA, tid, KCHH, 0, x, 32, 1.f);
    fence_proxy_async();  // hidden tile (MMA operand) and the reads of A done
    tc_fence_before();
    __syncthreads();
    // the tile buffer is free: the next tile's rows load during layer 2
    if (tn < n_tiles) {
      if (warp == 0) issue(tn);
      a_pending = true;
    }

    // ---- layer 2 ----------------------------------------------------------------
    if (tid == 0) {
      tc_fence_after();
      issue_layer<H, false>(tmem_base, sHA, sW2, H, 1);
      mma_commit(&bar[1]);
    }
    if (!wait_mma()) {
      aborted = true;
      break;
    }
    float z[32];
    {
      float v[32];
      tmem_ld32(tmem_lane, v);
      tmem_wait_ld();
      add_params(v, pb2, z);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 u = e_row[q];
      z[8 * q + 0] += bf16_lo(u.x);
      z[8 * q + 1] += bf16_hi(u.x);
      z[8 * q + 2] += bf16_lo(u.y);
      z[8 * q + 3] += bf16_hi(u.y);
      z[8 * q + 4] += bf16_lo(u.z);
      z[8 * q + 5] += bf16_hi(u.z);
      z[8 * q + 6] += bf16_lo(u.w);
      z[8 * q + 7] += bf16_hi(u.w);
    }
    if constexpr (!CLS) {
      if (valid) {
        uint4* d4 = reinterpret_cast<uint4*>(w.estate16 + size_t(r) * H);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          d4[q] = make_uint4(pack_bf16(z[8 * q], z[8 * q + 1]), pack_bf16(z[8 * q + 2], z[8 * q + 3]),
                             pack_bf16(z[8 * q + 4], z[8 * q + 5]), pack_bf16(z[8 * q + 6], z[8 * q + 7]));
      }
      tc_fence_before();
      __syncthreads();  // every thread has read the tensor memory of this tile
    } else {
      // ---- classifier on the new edge state (rounded to BF16 as stored) -------
#pragma unroll
      for (int j = 0; j < 32; ++j) z[j] = __bfloat162float(__float2bfloat16_rn(z[j]));
      put_row_f32<false>(sHA, tid, KCHH, 0, z, 32, 1.f);
      fence_proxy_async();
      tc_fence_before();
      __syncthreads();
      if (tid == 0) {
        tc_fence_after();
        issue_layer<H, false>(tmem_base, sHA, sWC, H, 1);
        mma_commit(&bar[1]);
      }
      if (!wait_mma()) {
        aborted = true;
        break;
      }
      float c[32];
      {
        float v[32];
        tmem_ld32(tmem_lane, v);
        tmem_wait_ld();
        add_params(v, pbc, c);
      }
      float cs = 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) cs += c[j];
      const float cmean = cs / float(H);
      float cvar = 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float d = c[j] - cmean;
        cvar = fmaf(d, d, cvar);
      }
      const float cinv = 1.0f / sqrtf(cvar / float(H) + kLnEps);
      float logit = pc2[H];
#pragma unroll
      for (int j = 0; j < 32; ++j) logit = fmaf(fmaxf((c[j] - cmean) * cinv, 0.f), pc2[j], logit);
      if (valid) {
        w.logit[r] = logit;
        w.keep[r] = logit >= p.cut ? 1 : 0;
      }
      tc_fence_before();
      __syncthreads();  // the hidden tile and the tensor memory are reused
    }
  }

  // ---- clean-up: on a timeout, give what is still in flight one more bounded
  //      wait, then free the tensor memory ---------------------------------------
  if (aborted) {
    if (tid == 0) set_status(w.counters, ST_TIMEOUT);
    if (weights_late) mbar_wait_bounded(&bar[0], 0, kWaitCycles);
    if (a_pending) mbar_wait_bounded(&bar[2], a_phase, kWaitCycles);
    if (mma_pending) mbar_wait_bounded(&bar[1], mma_phase, kWaitCycles);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 32);
  }
}

// ---------------------------------------------------------------------------
// BF16 edge step at hidden 32, warp-specialised (tuning form 2): same
// operands, K order and epilogue arithmetic as k_tc<32, BF16, M_EDGE_UPD /
// M_EDGE_UPD_CLS>, with several tiles in flight per CTA:
//   * warp 0 (producer) fills a ring of kWsStages tile buffers by TMA (box of
//     128 e rows, row gathers of h_src and h_dst, as in k_tc_edge_tma);
//   * warp 1 (one lane issues) runs the MMAs: layer 1 of tile i + 1 into one
//     of two tensor-memory accumulators while the epilogue works on tile i in
//     the other, then layer 2 (and the classifier) of tile i once its hidden
//     tile is written;
//   * two epilogue warpgroups (warps 2-5 and 6-9) take alternate tiles:
//     bias, LayerNorm, ReLU, the hidden tile, the residual e read from the
//     tile buffer (which then goes back to the producer), the new state or
//     the classifier and the cut.
// Hand-offs are mbarriers (full / empty per tile buffer; accumulator, hidden
// tile and accumulator-free per accumulator). Every wait is bounded; a wait
// that runs out raises a shared abort flag on which every other wait gives
// up too, and the kernel latches ST_TIMEOUT.
// ---------------------------------------------------------------------------
constexpr int kWsStages = 3;
constexpr int kWsThreads = 320;  // producer, MMA, two epilogue warpgroups

template <bool CLS>
struct WsLayout {
  static constexpr int H = 32;
  static constexpr int SEG = kRows * H * 2;
  static constexpr int K1 = 3 * H;
  static constexpr int W1 = 0;
  static constexpr int W1_BYTES = H * K1 * 2;
  static constexpr int W2 = align1k(W1 + W1_BYTES);
  static constexpr int W2_BYTES = H * H * 2;
  static constexpr int WC = align1k(W2 + W2_BYTES);
  static constexpr int WC_BYTES = CLS ? H * H * 2 : 0;
  static constexpr int A = align1k(WC + WC_BYTES);
  static constexpr int ABUF = 3 * SEG;
  static constexpr int HA = A + kWsStages * ABUF;  // two hidden tiles
  static constexpr int HA_BYTES = kRows * H * 2;
  static constexpr int PAR = HA + 2 * HA_BYTES;
  static constexpr int PAR_FLOATS = 4 * H + 4;
  // barriers: full[S], empty[S], then per accumulator acc1, hid, acc2, cin,
  // acc3, free (2 each)
  static constexpr int BAR = PAR + PAR_FLOATS * 4;
  static constexpr int NBAR = 2 * kWsStages + 12;
  static constexpr int FLAG = BAR + NBAR * 8;  // abort flag, TMEM address
  static constexpr int TOTAL = FLAG + 16;
  static constexpr int ALLOC = TOTAL + 1024;
};

// Bounded wait that also gives up when another role has raised the abort flag.
__device__ __forceinline__ bool ws_wait(uint64_t* m, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait(m, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(m, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > kWaitCycles) {
      *abort = 1;
      return false;
    }
  }
  return true;
}

template <bool CLS>
__global__ void __launch_bounds__(kWsThreads, 2)
    k_tc_edge_ws(const TcArgs p, const __grid_constant__ CUtensorMap map_e,
                 const __grid_constant__ CUtensorMap map_h) {
  constexpr int H = 32;
  using L = WsLayout<CLS>;
  constexpr int S = kWsStages;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint8_t* sW1 = smem + L::W1;
  uint8_t* sW2 = smem + L::W2;
  uint8_t* sWC = smem + L::WC;
  float* par = reinterpret_cast<float*>(smem + L::PAR);
  float* pb1 = par;
  float* pb2 = par + H;
  float* pbc = par + 2 * H;
  float* pc2 = par + 3 * H;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::BAR);
  uint64_t* full = bar;            // [S] tile loaded
  uint64_t* empty = bar + S;       // [S] tile buffer free (128 arrivals)
  uint64_t* acc1 = bar + 2 * S;    // [2] layer-1 accumulator ready
  uint64_t* hid = acc1 + 2;        // [2] hidden tile written (128)
  uint64_t* acc2 = acc1 + 4;       // [2] layer-2 accumulator ready
  uint64_t* cin = acc1 + 6;        // [2] classifier input written (128)
  uint64_t* acc3 = acc1 + 8;       // [2] classifier accumulator ready
  uint64_t* tfree = acc1 + 10;     // [2] accumulator read out (128)
  volatile int* abort = reinterpret_cast<volatile int*>(smem + L::FLAG);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + L::FLAG + 4);
  constexpr int KCHH = H * 2 / 16;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Ws& w = p.w;
  pdl_wait();
  if (*(volatile int32_t*)&w.counters[C_STATUS] & ST_INPUT) return;

  if (tid == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kRows);
    }
    for (int d = 0; d < 2; ++d) {
      mbar_init(&acc1[d], 1);
      mbar_init(&hid[d], kRows);
      mbar_init(&acc2[d], 1);
      mbar_init(&cin[d], kRows);
      mbar_init(&acc3[d], 1);
      mbar_init(&tfree[d], kRows);
    }
    *abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tslot, 64);  // two accumulators of 32 columns
    tmem_relinquish();
  }
  for (int i = tid; i < H; i += kWsThreads) {
    pb1[i] = p.b1[i];
    pb2[i] = p.b2[i];
    pbc[i] = CLS ? p.bc1[i] : 0.f;
    pc2[i] = CLS ? p.c2.WT[i * p.c2.ldo] : 0.f;
  }
  if (tid == 0) pc2[H] = CLS ? p.c2.b[0] : 0.f;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tslot;
  pdl_trigger();  // (not before this block has its tensor memory)

  // the weights come with the first tile: their bytes are counted on the
  // first full barrier, which the MMA warp waits for before its first MMA
  const int hi = clamp_edges(w.counters, w.e_cap);
  const int n_tiles = (hi + kRows - 1) / kRows;
  const int n_local = int(blockIdx.x) < n_tiles ? (n_tiles - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x) : 0;
  // a whole warp waits; it goes on only if every lane saw the phase complete
  // (so that the warp-collective instructions after it never diverge)
  auto wait_warp = [&](uint64_t* m, uint32_t parity) -> bool {
    const bool ok = ws_wait(m, parity, abort);
    return __all_sync(0xffffffffu, ok);
  };

  if (warp == 0) {
    // ---- producer ----------------------------------------------------------
    for (int i = 0; i < n_local; ++i) {
      const int t = int(blockIdx.x) + i * int(gridDim.x);
      const int s = i % S, u = i / S;
      if (u > 0 && !wait_warp(&empty[s], uint32_t((u - 1) & 1))) break;
      int sv[4], dv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = t * kRows + 4 * lane + q;
        sv[q] = r < hi ? w.src[r] : 0;
        dv[q] = r < hi ? w.col[r] : 0;
      }
      uint8_t* A = smem + L::A + s * L::ABUF;
      if (lane == 0) {
        const uint32_t wbytes = i == 0 ? uint32_t(L::W1_BYTES + L::W2_BYTES + L::WC_BYTES) : 0u;
        mbar_expect_tx(&full[s], uint32_t(3 * L::SEG) + wbytes);
        if (i == 0) {
          bulk_g2s(sW1, p.W1, L::W1_BYTES, &full[s]);
          bulk_g2s(sW2, p.W2, L::W2_BYTES, &full[s]);
          if (CLS) bulk_g2s(sWC, p.Wc, L::WC_BYTES, &full[s]);
        }
        tma_load_2d(A, &map_e, 0, t * kRows, &full[s]);
      }
      __syncwarp();
      tma_gather4(A + L::SEG + 4 * lane * (H * 2), &map_h, 0, sv[0], sv[1], sv[2], sv[3], &full[s]);
      tma_gather4(A + 2 * L::SEG + 4 * lane * (H * 2), &map_h, 0, dv[0], dv[1], dv[2], dv[3],
                  &full[s]);
    }
  } else if (warp == 1) {
    // ---- MMA issuer (lane 0; the other lanes wait for it at the warp barrier)
    if (lane == 0) {
      constexpr uint32_t IDESC = idesc_bf16(kRows, H);
      constexpr uint32_t SBO_W = uint32_t(L::K1 * 2 / 16) * 128;
      auto layer1 = [&](int i) -> bool {
        const int s = i % S, d = i & 1;
        if (!ws_wait(&full[s], uint32_t((i / S) & 1), abort)) return false;
        if (i >= 2 && !ws_wait(&tfree[d], uint32_t(((i >> 1) - 1) & 1), abort)) return false;
        tc_fence_after();
        const uint32_t a0 = smem_u32(smem + L::A + s * L::ABUF), w0 = smem_u32(sW1);
#pragma unroll
        for (int k = 0; k < L::K1; k += 16) {
          const int seg = k / H, j = (k % H) / 16;
          const uint64_t ad = smem_desc_sw64(a0 + uint32_t(seg * L::SEG + j * 32));
          const uint64_t bd = smem_desc(w0 + uint32_t(k * 2 / 16) * 128, 128, SBO_W);
          mma_bf16(tmem_base + uint32_t(32 * d), ad, bd, IDESC, k > 0 ? 1u : 0u);
        }
        mma_commit(&acc1[d]);
        return true;
      };
      bool ok = n_local == 0 || layer1(0);
      for (int i = 0; i < n_local && ok; ++i) {
        const int d = i & 1;
        const uint32_t ph = uint32_t((i >> 1) & 1);
        if (i + 1 < n_local && !layer1(i + 1)) break;
        uint8_t* HA = smem + L::HA + d * L::HA_BYTES;
        if (!ws_wait(&hid[d], ph, abort)) break;
        tc_fence_after();
        issue_layer<H, false>(tmem_base + uint32_t(32 * d), HA, sW2, H, 1);
        mma_commit(&acc2[d]);
        if constexpr (CLS) {
          if (!ws_wait(&cin[d], ph, abort)) break;
          tc_fence_after();
          issue_layer<H, false>(tmem_base + uint32_t(32 * d), HA, sWC, H, 1);
          mma_commit(&acc3[d]);
        }
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue warpgroups: g takes tiles i = g, g + 2, ... ---------------
    const int g = (warp - 2) >> 2;
    const int row = 32 * (warp & 3) + lane;  // TMEM lane of this thread
    const uint32_t tmem_row = tmem_base + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(32 * g);
    uint8_t* HA = smem + L::HA + g * L::HA_BYTES;
    for (int i = g; i < n_local; i += 2) {
      const int t = int(blockIdx.x) + i * int(gridDim.x);
      const int s = i % S;
      const uint32_t ph = uint32_t((i >> 1) & 1);
      const int r = t * kRows + row;
      const bool valid = r < hi;
      const uint8_t* A = smem + L::A + s * L::ABUF;
      if (!wait_warp(&acc1[g], ph)) break;
      tc_fence_after();
      float x[32];
      {
        float v[32];
        tmem_ld32(tmem_row, v);
        tmem_wait_ld();
        add_params(v, pb1, x);
      }
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) sum += x[j];
      const float mean = sum / float(H);
      float var = 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const float dd = x[j] - mean;
        var = fmaf(dd, dd, var);
      }
      const float inv = 1.0f / sqrtf(var / float(H) + kLnEps);
#pragma unroll
      for (int j = 0; j < 32; ++j) x[j] = fmaxf((x[j] - mean) * inv, 0.f);
      put_row_f32<false>(HA, row, KCHH, 0, x, 32, 1.f);
      uint4 e_row[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        e_row[q] = *reinterpret_cast<const uint4*>(A + row * (H * 2) + ((q ^ ((row >> 1) & 3)) << 4));
      fence_proxy_async();  // hidden tile to the MMA; the reads of A before its refill
      mbar_arrive(&hid[g]);
      mbar_arrive(&empty[s]);
      if (!wait_warp(&acc2[g], ph)) break;
      tc_fence_after();
      float z[32];
      {
        float v[32];
        tmem_ld32(tmem_row, v);
        tmem_wait_ld();
        add_params(v, pb2, z);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 u = e_row[q];
        z[8 * q + 0] += bf16_lo(u.x);
        z[8 * q + 1] += bf16_hi(u.x);
        z[8 * q + 2] += bf16_lo(u.y);
        z[8 * q + 3] += bf16_hi(u.y);
        z[8 * q + 4] += bf16_lo(u.z);
        z[8 * q + 5] += bf16_hi(u.z);
        z[8 * q + 6] += bf16_lo(u.w);
        z[8 * q + 7] += bf16_hi(u.w);
      }
      if constexpr (!CLS) {
        if (valid) {
          uint4* d4 = reinterpret_cast<uint4*>(w.estate16 + size_t(r) * H);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            d4[q] = make_uint4(pack_bf16(z[8 * q], z[8 * q + 1]), pack_bf16(z[8 * q + 2], z[8 * q + 3]),
                               pack_bf16(z[8 * q + 4], z[8 * q + 5]),
                               pack_bf16(z[8 * q + 6], z[8 * q + 7]));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) z[j] = __bfloat162float(__float2bfloat16_rn(z[j]));
        put_row_f32<false>(HA, row, KCHH, 0, z, 32, 1.f);  // layer 2 has read HA
        fence_proxy_async();
        mbar_arrive(&cin[g]);
        if (!wait_warp(&acc3[g], ph)) break;
        tc_fence_after();
        float c[32];
        {
          float v[32];
          tmem_ld32(tmem_row, v);
          tmem_wait_ld();
          add_params(v, pbc, c);
        }
        float cs = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) cs += c[j];
        const float cmean = cs / float(H);
        float cvar = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float dd = c[j] - cmean;
          cvar = fmaf(dd, dd, cvar);
        }
        const float cinv = 1.0f / sqrtf(cvar / float(H) + kLnEps);
        float logit = pc2[H];
#pragma unroll
        for (int j = 0; j < 32; ++j) logit = fmaf(fmaxf((c[j] - cmean) * cinv, 0.f), pc2[j], logit);
        if (valid) {
          w.logit[r] = logit;
          w.keep[r] = logit >= p.cut ? 1 : 0;
        }
      }
      tc_fence_before();
      mbar_arrive(&tfree[g]);  // this accumulator's tensor memory is read out
    }
  }

  // ---- end: after an abort, let copies and MMAs in flight drain (bounded
  //      sleep), then free the tensor memory -------------------------------------
  __syncthreads();
  if (*abort) {
    if (tid == 0) set_status(w.counters, ST_TIMEOUT);
    const long long t0 = clock64();
    while (clock64() - t0 < 20000000LL) {
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 64);
  }
}

// ---------------------------------------------------------------------------
// messages of the node step (msg.cuh) from the BF16 edge states, P[v] = [m_out |
// m_in], as the node step's operand: rounded to BF16 (BF16 path), or E4M3 codes
// under one scale amax / 448 per sum (FP8 path: a quarter of the FP32 sums' bytes
// to write and to read), rows of 2H codes and two scales (msg_codes, msg_scales)
// ---------------------------------------------------------------------------
template <int H, bool FP8>
struct MsgBf16 {
  static constexpr int LANES = H / 8;
  using Chunk = uint4;
  struct Acc {
    float2 s[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f),
                   make_float2(0.f, 0.f)};
    float amax = 0.f;
    __device__ __forceinline__ void add(const uint4& v) {
      s[0] = __fadd2_rn(s[0], make_float2(bf16_lo(v.x), bf16_hi(v.x)));
      s[1] = __fadd2_rn(s[1], make_float2(bf16_lo(v.y), bf16_hi(v.y)));
      s[2] = __fadd2_rn(s[2], make_float2(bf16_lo(v.z), bf16_hi(v.z)));
      s[3] = __fadd2_rn(s[3], make_float2(bf16_lo(v.w), bf16_hi(v.w)));
    }
    // FP8: the largest |sum| of the row, over the lanes of its group
    __device__ __forceinline__ void finish() {
      if constexpr (FP8) {
        amax = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) amax = fmaxf(amax, fmaxf(fabsf(s[c].x), fabsf(s[c].y)));
#pragma unroll
        for (int o = 1; o < LANES; o *= 2) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      }
    }
  };
  static __device__ __forceinline__ uint4 load(const Ws& w, int e, int q) {
    return __ldg(reinterpret_cast<const uint4*>(w.estate16 + size_t(e) * H) + q);
  }
  static __device__ __forceinline__ void store(const Ws& w, int row, int side, int q, const Acc& a) {
    if constexpr (FP8) {
      const float inv = a.amax > 0.f ? 448.f / a.amax : 1.f;
      *(reinterpret_cast<uint2*>(msg_codes<H>(w, row) + side * H) + q) =
          make_uint2(pack_e4m3x4(a.s[0].x * inv, a.s[0].y * inv, a.s[1].x * inv, a.s[1].y * inv),
                     pack_e4m3x4(a.s[2].x * inv, a.s[2].y * inv, a.s[3].x * inv, a.s[3].y * inv));
      if (q == 0) msg_scales<H>(w, row)[side] = a.amax > 0.f ? a.amax / 448.f : 1.f;
    } else {
      *(reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(w.pstate) + size_t(row) * 2 * H +
                                 side * H) + q) =
          make_uint4(pack_bf16(a.s[0].x, a.s[0].y), pack_bf16(a.s[1].x, a.s[1].y),
                     pack_bf16(a.s[2].x, a.s[2].y), pack_bf16(a.s[3].x, a.s[3].y));
    }
  }
};

template <int H, bool FP8>
__global__ void __launch_bounds__(256, 4) k_msg_bf16(Batch b, Ws w) {
  pdl_begin();
  if (*(volatile int32_t*)&w.counters[C_STATUS] & ST_INPUT) return;
  message_sums<MsgBf16<H, FP8>>(w, Sel{nullptr, nullptr}, 0, b.n_hits);
}

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
// CTAs per SM of one kernel: the occupancy query, capped so that the CTAs of an
// SM fit in its 512 tensor-memory columns; computed once per instantiation.
template <int H, bool FP8, int MODE>
int tc_blocks_per_sm() {
  using L = Layout<H, FP8, MODE>;
  // computed once per instantiation (thread-safe initialisation of a local static)
  static const int per_sm = [] {
    cudaError_t e = cudaFuncSetAttribute(k_tc<H, FP8, MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, L::TOTAL);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tc<H, FP8, MODE>,
                               cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    int n = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_tc<H, FP8, MODE>, L::THREADS, L::TOTAL);
    // the same bound from the kernel's resources: registers (allocated per warp
    // in units of 256), shared memory (228 KB per SM, 1 KB reserved per CTA),
    // 2048 threads per SM. CTAs never wait on one another, so a bound above
    // what fits only queues CTAs.
    cudaFuncAttributes fa{};
    int est = 16;
    if (cudaFuncGetAttributes(&fa, k_tc<H, FP8, MODE>) == cudaSuccess && fa.numRegs > 0) {
      const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;
      est = std::min(est, 65536 / (regs_warp * (L::THREADS / 32)));
    }
    est = std::min(est, 233472 / (L::TOTAL + 1024));
    if (e != cudaSuccess) cudaGetLastError();
    if (getenv("GNNTRK_VERBOSE"))
      fprintf(stderr, "gnntrk: k_tc<%d,%d,%d> occupancy query %d (%s), resource bound %d\n", H,
              int(FP8), MODE, n, cudaGetErrorString(e), est);
    n = std::max(n, est);
    n = n < 1 ? 1 : n;
    while (n > 1 && n * L::G * L::TMEM_COLS > 512) --n;
    if (getenv("GNNTRK_VERBOSE"))
      fprintf(stderr, "gnntrk: k_tc<%d,%d,%d> smem %d B, %d CTAs/SM\n", H, int(FP8), MODE,
              L::TOTAL, n);
    return n;
  }();
  return per_sm;
}

// Resident CTAs per SM chosen by the autotuner, per (FP8, hidden, kernel
// family); 0 = the resource bound. Families: 0 node encoder, 1 edge encoder,
// 2 node step, 3 edge step and classifier.
std::atomic<int> g_tuned[2][3][4] = {};

constexpr int family_of(int mode) {
  return mode == M_NODE_ENC ? 0 : mode == M_EDGE_ENC ? 1 : mode == M_NODE_UPD ? 2 : 3;
}
static_assert(family_of(M_TRIP) == 3, "triplet classifier tunes with the edge family");
constexpr int hidx(int h) { return h == 32 ? 0 : (h == 64 ? 1 : 2); }

// BF16 edge step at hidden 32: 0 cp.async row copies, 1 TMA-staged tiles, 2
// warp-specialised with TMA-staged tiles
std::atomic<int> g_edge_form{0};

// CTAs per SM of the TMA edge step: shared memory and tensor memory bound
template <bool CLS>
int tma_blocks_per_sm() {
  using L = TmaLayout<32, CLS>;
  static const int per_sm = [] {
    cudaError_t e = cudaFuncSetAttribute(k_tc_edge_tma<32, CLS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, L::ALLOC);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tc_edge_tma<32, CLS>,
                               cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) cudaGetLastError();
    int n = 233472 / (L::ALLOC + 1024);
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, k_tc_edge_tma<32, CLS>) == cudaSuccess && fa.numRegs > 0) {
      const int regs_warp = ((fa.numRegs * 32 + 255) / 256) * 256;
      n = std::min(n, 65536 / (regs_warp * (kRows / 32)));
    }
    n = std::max(1, std::min(n, 512 / 32));
    if (getenv("GNNTRK_VERBOSE"))
      fprintf(stderr, "gnntrk: k_tc_edge_tma<32,%d> smem %d B, %d CTAs/SM\n", int(CLS), L::ALLOC, n);
    return n;
  }();
  return per_sm;
}

template <bool CLS>
void launch_edge_tma(const TcArgs& a, const TcModel& m, cudaStream_t s) {
  using L = TmaLayout<32, CLS>;
  const int grid = device_sms() * tma_blocks_per_sm<CLS>();
  launch_pdl(a.b.n_hits <= kEarlyTcHits, k_tc_edge_tma<32, CLS>, grid, kRows, L::ALLOC, s, 1, a, m.map_e, m.map_h);
}

// CTAs per SM of the warp-specialised edge step (shared memory bound)
template <bool CLS>
int ws_blocks_per_sm() {
  using L = WsLayout<CLS>;
  static const int per_sm = [] {
    cudaError_t e = cudaFuncSetAttribute(k_tc_edge_ws<CLS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, L::ALLOC);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tc_edge_ws<CLS>, cudaFuncAttributePreferredSharedMemoryCarveout,
                               100);
    if (e != cudaSuccess) cudaGetLastError();
    int n = std::max(1, std::min(2, 233472 / (L::ALLOC + 1024)));
    if (getenv("GNNTRK_VERBOSE"))
      fprintf(stderr, "gnntrk: k_tc_edge_ws<%d> smem %d B, %d CTAs/SM\n", int(CLS), L::ALLOC, n);
    return n;
  }();
  return per_sm;
}

template <bool CLS>
void launch_edge_ws(const TcArgs& a, const TcModel& m, cudaStream_t s) {
  using L = WsLayout<CLS>;
  const int grid = device_sms() * ws_blocks_per_sm<CLS>();
  launch_pdl(a.b.n_hits <= kEarlyTcHits, k_tc_edge_ws<CLS>, grid, kWsThreads, L::ALLOC, s, 1, a, m.map_e, m.map_h);
}

template <int H, bool FP8, int MODE>
void launch_mode(const TcCall& a, cudaStream_t s, int64_t rows_hint) {
  using L = Layout<H, FP8, MODE>;
  TcPar<H, FP8> q{};
  const LayerTC* l1 = MODE == M_CLS ? a.lc : a.l1;
  for (int i = 0; i < H; ++i) {
    if (MODE != M_NODE_ENC) q.b1[i] = l1->hb[i];
    if (L::HAS_W2) q.b2[i] = a.l2->hb[i];
    if (L::HAS_WC) q.bc[i] = a.lc->hb[i];
    if constexpr (FP8) {
      if (MODE != M_NODE_ENC) q.s1[i] = l1->hs[i];
      if (L::HAS_W2) q.s2[i] = a.l2->hs[i];
      if (L::HAS_WC) q.sc[i] = a.lc->hs[i];
    }
  }
  int per_sm = tc_blocks_per_sm<H, FP8, MODE>();
  const int tuned = g_tuned[FP8 ? 1 : 0][hidx(H)][family_of(MODE)].load(std::memory_order_relaxed);
  if (tuned > 0 && tuned < per_sm) per_sm = tuned;
  int grid = device_sms() * per_sm;
  grid = int(std::max<int64_t>(1, std::min<int64_t>(grid, (rows_hint + kRows * L::G - 1) / (kRows * L::G))));
  launch_pdl(!FP8 && a.b.n_hits <= kEarlyTcHits, k_tc<H, FP8, MODE>, grid, L::THREADS, L::TOTAL, s, 1, static_cast<const TcArgs&>(a), q);
}

template <int H, bool FP8>
void launch_h(int mode, const TcCall& a, cudaStream_t s, int64_t rows_hint) {
  switch (mode) {
    case M_NODE_ENC: launch_mode<H, FP8, M_NODE_ENC>(a, s, rows_hint); break;
    case M_EDGE_ENC: launch_mode<H, FP8, M_EDGE_ENC>(a, s, rows_hint); break;
    case M_TRIP:
      if constexpr (!FP8) launch_mode<H, false, M_TRIP>(a, s, rows_hint);
      break;
    default: break;
  }
  // (hidden 128 has BF16 encoders and triplets only: its steps' tiles and weights
  // exceed the shared memory)
  if constexpr (FP8 || H <= 64) switch (mode) {
    case M_NODE_UPD: launch_mode<H, FP8, M_NODE_UPD>(a, s, rows_hint); break;
    case M_EDGE_UPD: launch_mode<H, FP8, M_EDGE_UPD>(a, s, rows_hint); break;
    case M_EDGE_UPD_CLS: launch_mode<H, FP8, M_EDGE_UPD_CLS>(a, s, rows_hint); break;
    case M_CLS: launch_mode<H, FP8, M_CLS>(a, s, rows_hint); break;
    default: break;
  }
}

template <bool FP8>
constexpr int smem_total(int H, int mode) {
#define GNNTRK_LT(HH)                                                                 \
  (mode == M_NODE_ENC ? Layout<HH, FP8, M_NODE_ENC>::TOTAL                            \
   : mode == M_EDGE_ENC ? Layout<HH, FP8, M_EDGE_ENC>::TOTAL                          \
   : mode == M_NODE_UPD ? Layout<HH, FP8, M_NODE_UPD>::TOTAL                          \
   : mode == M_EDGE_UPD ? Layout<HH, FP8, M_EDGE_UPD>::TOTAL                          \
   : mode == M_EDGE_UPD_CLS ? Layout<HH, FP8, M_EDGE_UPD_CLS>::TOTAL                  \
   : mode == M_TRIP ? Layout<HH, FP8, M_TRIP>::TOTAL                                  \
                            : Layout<HH, FP8, M_CLS>::TOTAL)
  return H == 32 ? GNNTRK_LT(32) : (H == 64 ? GNNTRK_LT(64) : GNNTRK_LT(128));
#undef GNNTRK_LT
}

void launch_any(int H, bool fp8, int mode, const TcCall& a, cudaStream_t s, int64_t rows_hint) {
  if (fp8) {
    if (H == 32) launch_h<32, true>(mode, a, s, rows_hint);
    else if (H == 64) launch_h<64, true>(mode, a, s, rows_hint);
    else launch_h<128, true>(mode, a, s, rows_hint);
  } else {
    if (H == 32) launch_h<32, false>(mode, a, s, rows_hint);
    else if (H == 64) launch_h<64, false>(mode, a, s, rows_hint);
    else launch_h<128, false>(mode, a, s, rows_hint);
  }
}

constexpr int kMaxSmem = 232448;  // 227 KB of dynamic shared memory per CTA

// ---------------------------------------------------------------------------
// host: weight packing
// ---------------------------------------------------------------------------
uint16_t bf16_bits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7fffffffu) > 0x7f800000u) return uint16_t((u >> 16) | 0x40);  // quiet NaN
  u += 0x7fffu + ((u >> 16) & 1u);  // round to nearest even
  return uint16_t(u >> 16);
}

}  // namespace

// E4M3 (1 sign, 4 exponent bits with bias 7, 3 mantissa bits, no infinities,
// largest finite 448) of a float, rounding to nearest even and saturating to
// +-448; NaN maps to 0x7F.
uint8_t e4m3_from_float(float f) {
  if (std::isnan(f)) return 0x7f;
  const uint8_t sign = std::signbit(f) ? 0x80 : 0x00;
  double a = std::fabs(double(f));
  if (a >= 448.0) return sign | 0x7e;
  // candidates: subnormals k * 2^-9 (k = 0..7), normals (1 + m/8) * 2^(e-7)
  int e = 0;
  if (a < std::ldexp(1.0, -6)) {
    double k = a / std::ldexp(1.0, -9);
    double fl = std::floor(k), r = k - fl;
    int q = int(fl);
    if (r > 0.5 || (r == 0.5 && (q & 1))) ++q;
    return sign | uint8_t(q);  // q == 8 is the smallest normal (0x08)
  }
  std::frexp(a, &e);  // a = f * 2^e, f in [0.5, 1)
  int E = e - 1;      // a in [2^E, 2^(E+1))
  double m = a / std::ldexp(1.0, E) - 1.0;  // [0, 1)
  double k = m * 8.0;
  double fl = std::floor(k), r = k - fl;
  int q = int(fl);
  if (r > 0.5 || (r == 0.5 && (q & 1))) ++q;
  if (q == 8) {
    q = 0;
    ++E;
  }
  int be = E + 7;
  uint8_t code = uint8_t((be << 3) | q);
  if (code > 0x7e) code = 0x7e;
  return sign | code;
}

float e4m3_to_float(uint8_t c) {
  const float s = (c & 0x80) ? -1.f : 1.f;
  const int be = (c >> 3) & 0xf, m = c & 7;
  if (be == 0xf && m == 7) return NAN;
  if (be == 0) return s * std::ldexp(float(m), -9);
  return s * std::ldexp(1.f + float(m) / 8.f, be - 7);
}

namespace {

// Operand image of W[out][in] for the tensor cores: K-major rows of `out`,
// core matrices of 8 rows x 16 bytes, chunks of a row contiguous per 8-row
// group. FP8: per-output-channel scale amax/448 applied before encoding.
void pack_layer(const HostLayer& l, bool fp8, std::vector<uint8_t>& img, std::vector<float>& scale) {
  const int N = l.out, K = l.in;
  const int esz = fp8 ? 1 : 2, epc = 16 / esz;
  const int kch = K / epc;
  img.assign(size_t(N) * K * esz, 0);
  scale.assign(N, 1.f);
  for (int n = 0; n < N; ++n) {
    float amax = 0.f;
    for (int k = 0; k < K; ++k) amax = std::max(amax, std::fabs(l.W[size_t(n) * K + k]));
    if (fp8) scale[n] = amax > 0.f ? amax / 448.f : 1.f;
    for (int k = 0; k < K; ++k) {
      const size_t off = size_t((n / 8) * kch + k / epc) * 128 + (n % 8) * 16 + (k % epc) * esz;
      const float v = l.W[size_t(n) * K + k];
      if (fp8) {
        img[off] = e4m3_from_float(v / scale[n]);
      } else {
        const uint16_t b = bf16_bits(v);
        img[off] = uint8_t(b & 0xff);
        img[off + 1] = uint8_t(b >> 8);
      }
    }
  }
}

}  // namespace

int tc_upload(TcModel& m, const HostLayer* L, int n_layers, int n_embed, int h, int K,
              int precision, void** dmem, std::string& err) {
  const bool fp8 = precision == GNNTRK_FP8_E4M3;
  // which layers: node enc l2, edge enc l1/l2, per step node l1/l2 edge l1/l2, cls l1
  // (BF16: the node encoder's layer 2 and the edge encoder's layer 1 take
  // split operands, so their images repeat W along K)
  // (FP8: the encoders run as the BF16 split-operand kernels, whose images
  // are packed in BF16 as well; E4M3 cannot carry the node encoding the
  // encoders consume)
  struct Item {
    int layer;
    LayerTC* dst;
    bool repeat_k = false;
    bool bf16 = false;  // a BF16 image on an FP8 handle
  };
  std::vector<Item> items;
  int c = n_embed;
  items.push_back({c + 1, &m.node_enc.l2, !fp8});
  items.push_back({c + 2, &m.edge_enc.l1, !fp8});
  items.push_back({c + 3, &m.edge_enc.l2});
  m.enc16 = fp8;
  if (m.enc16) {
    items.push_back({c + 1, &m.node_enc16.l2, true, true});
    items.push_back({c + 2, &m.edge_enc16.l1, h <= 64, true});  // h 128: four passes, plain image
    items.push_back({c + 3, &m.edge_enc16.l2, false, true});
  }
  c += 4;
  for (int k = 0; k < K; ++k) {
    items.push_back({c, &m.node[k].l1});
    items.push_back({c + 1, &m.node[k].l2});
    items.push_back({c + 2, &m.edge[k].l1});
    items.push_back({c + 3, &m.edge[k].l2});
    c += 4;
  }
  items.push_back({c, &m.cls.l1});
  if (c + 2 != n_layers) {
    err = "tensor-core packing: unexpected layer count";
    return GNNTRK_ERR_WEIGHTS;
  }
  // shared-memory budget of the largest kernel (FP8: its encoders are BF16)
  for (int mode : {M_EDGE_UPD, M_NODE_UPD, M_EDGE_ENC, M_NODE_ENC}) {
    const bool enc = mode == M_EDGE_ENC || mode == M_NODE_ENC;
    const bool as_fp8 = fp8 && !(enc && m.enc16);
    if ((as_fp8 ? smem_total<true>(h, mode) : smem_total<false>(h, mode)) > kMaxSmem) {
      err = "tensor-core kernels do not fit shared memory at this hidden size";
      return GNNTRK_ERR_UNSUPPORTED;
    }
  }
  std::vector<uint8_t> blob;
  std::vector<size_t> off_img(items.size()), off_b(items.size()), off_s(items.size()), n_scales(items.size());
  auto align = [&](size_t a) { blob.resize((blob.size() + a - 1) / a * a, 0); };
  for (size_t i = 0; i < items.size(); ++i) {
    std::vector<uint8_t> img;
    std::vector<float> sc;
    if (items[i].repeat_k) {
      const HostLayer& l = L[items[i].layer];
      HostLayer r2;
      r2.in = 2 * l.in;
      r2.out = l.out;
      r2.b = l.b;
      r2.W.resize(size_t(r2.out) * r2.in);
      for (int n = 0; n < l.out; ++n)
        for (int k = 0; k < r2.in; ++k) r2.W[size_t(n) * r2.in + k] = l.W[size_t(n) * l.in + k % l.in];
      pack_layer(r2, fp8 && !items[i].bf16, img, sc);
    } else {
      pack_layer(L[items[i].layer], fp8 && !items[i].bf16, img, sc);
    }
    align(1024);
    off_img[i] = blob.size();
    blob.insert(blob.end(), img.begin(), img.end());
    align(16);
    off_b[i] = blob.size();
    const auto& bb = L[items[i].layer].b;
    blob.resize(blob.size() + 4 * bb.size());
    std::memcpy(blob.data() + off_b[i], bb.data(), 4 * bb.size());
    align(16);
    off_s[i] = blob.size();
    n_scales[i] = sc.size();
    blob.resize(blob.size() + 4 * sc.size());
    std::memcpy(blob.data() + off_s[i], sc.data(), 4 * sc.size());
  }
  void* d = nullptr;
  if (cudaMalloc(&d, blob.size()) != cudaSuccess) {
    cudaGetLastError();
    err = "cudaMalloc of the tensor-core weights failed";
    return GNNTRK_ERR_OOM;
  }
  if (cudaMemcpy(d, blob.data(), blob.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(d);
    err = "tensor-core weight upload failed";
    return GNNTRK_ERR_CUDA;
  }
  *dmem = d;
  const uint8_t* base = static_cast<const uint8_t*>(d);
  for (size_t i = 0; i < items.size(); ++i) {
    const HostLayer& l = L[items[i].layer];
    *items[i].dst = LayerTC{base + off_img[i], reinterpret_cast<const float*>(base + off_b[i]),
                            reinterpret_cast<const float*>(base + off_s[i]),
                            items[i].repeat_k ? 2 * l.in : l.in, l.out, {}, {}};
    std::memcpy(items[i].dst->hb, l.b.data(), 4 * l.b.size());
    std::memcpy(items[i].dst->hs, blob.data() + off_s[i], 4 * n_scales[i]);
  }
  m.precision = precision;
  m.h = h;
  m.K = K;
  m.n_embed = n_embed;
  return GNNTRK_OK;
}

int tc_upload_triplets(TcModel& m, const HostLayer& art1, const HostLayer& elb1, void** dmem,
                       std::string& err) {
  std::vector<uint8_t> ia, ie;
  std::vector<float> sa, se;
  pack_layer(art1, false, ia, sa);
  pack_layer(elb1, false, ie, se);
  const size_t off_e = (ia.size() + 1023) / 1024 * 1024;
  std::vector<uint8_t> blob(off_e + ie.size());
  std::memcpy(blob.data(), ia.data(), ia.size());
  std::memcpy(blob.data() + off_e, ie.data(), ie.size());
  void* d = nullptr;
  if (cudaMalloc(&d, blob.size()) != cudaSuccess) {
    cudaGetLastError();
    err = "cudaMalloc of the triplet-classifier weights failed";
    return GNNTRK_ERR_OOM;
  }
  if (cudaMemcpy(d, blob.data(), blob.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(d);
    err = "triplet-classifier weight upload failed";
    return GNNTRK_ERR_CUDA;
  }
  *dmem = d;
  const uint8_t* base = static_cast<const uint8_t*>(d);
  m.art1 = LayerTC{base, nullptr, nullptr, art1.in, art1.out, {}, {}};
  m.elb1 = LayerTC{base + off_e, nullptr, nullptr, elb1.in, elb1.out, {}, {}};
  std::memcpy(m.art1.hb, art1.b.data(), 4 * art1.b.size());
  std::memcpy(m.elb1.hb, elb1.b.data(), 4 * elb1.b.size());
  m.has_trip = true;
  return GNNTRK_OK;
}

namespace {
TcCall base_args(const Batch& b, const Ws& w, const GraphParams& g) {
  TcCall a{};
  a.b = b;
  a.w = w;
  for (int i = 0; i < 6; ++i) a.fs[i] = g.fs[i];
  a.cut = g.cut_logit;
  return a;
}
}  // namespace

void tc_node_prep(const Batch& b, const Ws& w, const TcModel& m, const LayerF32* embed_f32,
                  int n_embed, int D, int h, const GraphParams& g, const LayerF32& ne1_f32,
                  cudaStream_t s, bool do_embed) {
  // embedding in FP32: its output feeds the threshold d^2 < r^2
  const Sel all{nullptr, nullptr};
  if (do_embed)
    launch_node_prep_f32(b, w, embed_f32, n_embed, Mlp2F32{}, EdgeProj{}, D, h, g, true, false,
                         all, s);
  TcCall a = base_args(b, w, g);
  a.ne1 = ne1_f32;
  const Mlp2TC& ne = m.enc16 ? m.node_enc16 : m.node_enc;
  a.W2 = static_cast<const uint8_t*>(ne.l2.B);
  a.b2 = ne.l2.b;
  a.l2 = &ne.l2;
  launch_any(h, m.precision == GNNTRK_FP8_E4M3 && !m.enc16, M_NODE_ENC, a, s, b.n_hits);
}

void tc_messages(const Batch& b, const Ws& w, int h, bool fp8, cudaStream_t s) {
  const int grid = std::max(1, std::min(device_sms() * 8, div_up(b.n_hits, 256 / (h / 8))));
  if (h == 32)
    launch_pdl(false, fp8 ? k_msg_bf16<32, true> : k_msg_bf16<32, false>, grid, 256, 0, s, 1, b, w);
  else if (h == 64)
    launch_pdl(false, fp8 ? k_msg_bf16<64, true> : k_msg_bf16<64, false>, grid, 256, 0, s, 1, b, w);
  else
    launch_pdl(false, fp8 ? k_msg_bf16<128, true> : k_msg_bf16<128, false>, grid, 256, 0, s, 1, b, w);
}

namespace {
// (a second tile per block costs a small call a whole tile's latency: twice the
// edges per hit that the FP32 kernels' grids are sized for)
int64_t tc_rows(int64_t n_hits) { return 2 * edge_rows_hint(n_hits); }
}  // namespace

void tc_gnn(const Batch& b, const Ws& w, const TcModel& m, int h, int K, const GraphParams& g,
            const LayerF32& cls2_f32, cudaStream_t s, int stage, bool store_final) {
  const bool fp8 = m.precision == GNNTRK_FP8_E4M3;
  TcCall a = base_args(b, w, g);
  a.c2 = cls2_f32;
  a.Wc = static_cast<const uint8_t*>(m.cls.l1.B);
  a.bc1 = m.cls.l1.b;
  a.lc = &m.cls.l1;
  const bool fuse = !store_final &&
                    (fp8 ? smem_total<true>(h, M_EDGE_UPD_CLS) : smem_total<false>(h, M_EDGE_UPD_CLS)) <= kMaxSmem;
  auto set = [&](const Mlp2TC& mm) {
    a.W1 = static_cast<const uint8_t*>(mm.l1.B);
    a.b1 = mm.l1.b;
    a.W2 = static_cast<const uint8_t*>(mm.l2.B);
    a.b2 = mm.l2.b;
    a.l1 = &mm.l1;
    a.l2 = &mm.l2;
  };
  // stage < 0: everything; otherwise 0 = edge encoder, 1 + 2k = node step k,
  // 2 + 2k = edge step k (with the classifier at the last step)
  if (stage < 0 || stage == 0) {
    if (m.enc16) {
      set(m.edge_enc16);
      launch_any(h, false, M_EDGE_ENC, a, s, tc_rows(b.n_hits));
    } else {
      set(m.edge_enc);
      launch_any(h, fp8, M_EDGE_ENC, a, s, tc_rows(b.n_hits));
    }
  }
  for (int k = 0; k < K; ++k) {
    if (stage < 0) tc_messages(b, w, h, fp8, s);
    if (stage < 0 || stage == 1 + 2 * k) {
      set(m.node[k]);
      launch_any(h, fp8, M_NODE_UPD, a, s, b.n_hits);
    }
    if (stage < 0 || stage == 2 + 2 * k) {
      set(m.edge[k]);
      const bool last = k + 1 == K;
      const int form = (!fp8 && h == 32 && m.maps) ? g_edge_form.load(std::memory_order_relaxed) : 0;
      if (form == 1 && last && fuse)
        launch_edge_tma<true>(a, m, s);
      else if (form == 1)
        launch_edge_tma<false>(a, m, s);
      else if (form == 2 && last && fuse)
        launch_edge_ws<true>(a, m, s);
      else if (form == 2)
        launch_edge_ws<false>(a, m, s);
      else
        launch_any(h, fp8, last && fuse ? M_EDGE_UPD_CLS : M_EDGE_UPD, a, s, tc_rows(b.n_hits));
      if (last && !fuse) launch_any(h, fp8, M_CLS, a, s, tc_rows(b.n_hits));
    }
  }
  if (K == 0 && (stage < 0 || stage == 1)) launch_any(h, fp8, M_CLS, a, s, tc_rows(b.n_hits));
}

void tc_set_edge_form(int form) {
  g_edge_form.store(form >= 0 && form <= 2 ? form : 0, std::memory_order_relaxed);
}
int tc_get_edge_form() { return g_edge_form.load(std::memory_order_relaxed); }

void tc_make_maps(TcModel& m, const Ws& w, int h) {
  m.maps = false;
  if (h != 32 || w.estate16 == nullptr || w.hstate16 == nullptr) return;
  // the CUDA driver API encoder, looked up through the runtime (the library does not
  // link libcuda, so it loads on machines without a GPU driver)
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      fn = nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }();
  if (encode == nullptr) return;
  const cuuint32_t es[2] = {1, 1};
  const cuuint64_t dim_e[2] = {cuuint64_t(h), cuuint64_t(w.e_cap)};
  const cuuint64_t dim_h[2] = {cuuint64_t(h), cuuint64_t(w.h_cap)};
  const cuuint64_t stride[1] = {cuuint64_t(h) * 2};  // bytes between rows
  const cuuint32_t box_e[2] = {cuuint32_t(h), cuuint32_t(kRows)};
  const cuuint32_t box_h[2] = {cuuint32_t(h), 1};  // one row high: row gathers
  CUresult r1 = encode(&m.map_e, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                       static_cast<void*>(w.estate16), dim_e, stride, box_e, es,
                                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                       CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CUresult r2 = encode(&m.map_h, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                                       static_cast<void*>(w.hstate16), dim_h, stride, box_h, es,
                                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                                       CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  m.maps = r1 == CUDA_SUCCESS && r2 == CUDA_SUCCESS;
}

void tc_set_ctas(int precision, int h, int family, int n) {
  if (family < 0 || family > 3 || (h != 32 && h != 64 && h != 128)) return;
  g_tuned[precision == GNNTRK_FP8_E4M3 ? 1 : 0][hidx(h)][family].store(n < 0 ? 0 : n,
                                                                       std::memory_order_relaxed);
}

int tc_get_ctas(int precision, int h, int family) {
  if (family < 0 || family > 3 || (h != 32 && h != 64 && h != 128)) return 0;
  return g_tuned[precision == GNNTRK_FP8_E4M3 ? 1 : 0][hidx(h)][family].load(
      std::memory_order_relaxed);
}

void tc_triplet_scores(const Batch& b, const Ws& w, const TcModel& m, int h, const LayerF32& art2,
                       const LayerF32& elb2, float cut_logit, cudaStream_t s) {
  GraphParams g{};
  g.cut_logit = cut_logit;
  TcCall a = base_args(b, w, g);
  // articulations
  a.W1 = static_cast<const uint8_t*>(m.art1.B);
  a.l1 = &m.art1;
  a.c2 = art2;
  a.t1 = w.trip_a1;
  a.t2 = w.trip_a2;
  a.tn = w.counters + C_TRIP_A;
  a.tlogit = w.trip_alogit;
  a.tkeep = w.trip_akeep;
  launch_any(h, false, M_TRIP, a, s, triplet_rows_hint(b.n_hits));
  // elbows
  a.W1 = static_cast<const uint8_t*>(m.elb1.B);
  a.l1 = &m.elb1;
  a.c2 = elb2;
  a.t1 = w.trip_e1;
  a.t2 = w.trip_e2;
  a.tn = w.counters + C_TRIP_E;
  a.tlogit = w.trip_elogit;
  a.tkeep = w.trip_ekeep;
  launch_any(h, false, M_TRIP, a, s, triplet_rows_hint(b.n_hits));
}

bool tc_cls_fused(int h, int precision) {
  const bool fp8 = precision == GNNTRK_FP8_E4M3;
  return (fp8 ? smem_total<true>(h, M_EDGE_UPD_CLS) : smem_total<false>(h, M_EDGE_UPD_CLS)) <= kMaxSmem;
}


namespace {
// Tensor-core throughput probe: one CTA per SM, one thread issuing BF16 MMAs
// M = 128, N = NN, K = 64 (four K = 16 instructions) back to back from shared
// memory (zeros, no-swizzle layout) into one tensor-memory accumulator, one
// commit at the end (bounded wait). Measures what the tensor pipe sustains at
// the narrow N of the interaction-network layers.
template <int NN>
__global__ void __launch_bounds__(32, 1) k_tc_probe(int64_t iters, int32_t* flag) {
  constexpr int K = 64;
  __shared__ __align__(1024) uint8_t sA[kRows * K * 2];
  __shared__ __align__(1024) uint8_t sB[NN * K * 2];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tslot;
  for (int i = threadIdx.x * 16; i < kRows * K * 2; i += 32 * 16)
    *reinterpret_cast<uint4*>(sA + i) = make_uint4(0, 0, 0, 0);
  for (int i = threadIdx.x * 16; i < NN * K * 2; i += 32 * 16)
    *reinterpret_cast<uint4*>(sB + i) = make_uint4(0, 0, 0, 0);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  tmem_alloc(&tslot, NN < 32 ? 32 : NN);
  tmem_relinquish();
  fence_proxy_async();
  tc_fence_before();
  __syncwarp();
  tc_fence_after();
  const uint32_t tmem = tslot;
  if (threadIdx.x == 0) {
    constexpr uint32_t IDESC = idesc_bf16(kRows, NN);
    constexpr uint32_t SBO = uint32_t(K * 2 / 16) * 128;
    const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
    for (int64_t it = 0; it < iters; ++it) {
#pragma unroll
      for (int k = 0; k < K; k += 16) {
        const uint32_t off = uint32_t(k * 2 / 16) * 128;
        mma_bf16(tmem, smem_desc(a0 + off, 128, SBO), smem_desc(b0 + off, 128, SBO), IDESC,
                 (it > 0 || k > 0) ? 1u : 0u);
      }
    }
    mma_commit(&bar);
    if (!mbar_wait_bounded(&bar, 0, kWaitCycles)) atomicExch(flag, 1);
  }
  tc_fence_before();
  __syncwarp();
  tc_fence_after();
  tmem_dealloc(tmem, NN < 32 ? 32 : NN);
}
}  // namespace

int tc_probe(int n, int64_t iters, double* ms) {
  int32_t* flag = nullptr;
  if (cudaMalloc(&flag, sizeof(int32_t)) != cudaSuccess) return GNNTRK_ERR_OOM;
  cudaMemset(flag, 0, sizeof(int32_t));
  cudaEvent_t a, b;
  cudaEventCreate(&a);
  cudaEventCreate(&b);
  const int grid = device_sms();
  auto go = [&](int64_t its) {
    if (n == 32) k_tc_probe<32><<<grid, 32>>>(its, flag);
    else if (n == 64) k_tc_probe<64><<<grid, 32>>>(its, flag);
    else if (n == 128) k_tc_probe<128><<<grid, 32>>>(its, flag);
    else k_tc_probe<256><<<grid, 32>>>(its, flag);
  };
  go(16);  // warm-up
  cudaEventRecord(a);
  go(iters);
  cudaEventRecord(b);
  cudaError_t e = cudaEventSynchronize(b);
  float t = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&t, a, b);
  int32_t hflag = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&hflag, flag, sizeof(int32_t), cudaMemcpyDeviceToHost);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(flag);
  if (e != cudaSuccess) return GNNTRK_ERR_CUDA;
  if (hflag) return GNNTRK_ERR_TIMEOUT;
  *ms = double(t);
  return GNNTRK_OK;
}

namespace {
// Self-test of the bounded waits: one thread waits on an mbarrier that no
// thread ever arrives on, through the same bounded wait the tensor-core
// kernels use, and latches ST_TIMEOUT when it runs out, as they do.
__global__ void k_wait_selftest(int32_t* counters, long long max_cycles) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait_bounded(&bar, 0, max_cycles)) set_status(counters, ST_TIMEOUT);
}
}  // namespace

void tc_wait_selftest(int32_t* counters, long long max_cycles, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(counters, max_cycles);
}

}  // namespace gnntrk

// ---------------------------------------------------------------------------
// E4M3 conversion entry points (host packing routine, device activation
// conversion), for checks of both against an independent codec
// ---------------------------------------------------------------------------
namespace gnntrk {
namespace {
__global__ void k_e4m3_encode(const float* in, uint8_t* out, int64_t n) {
  const int64_t pairs = (n + 1) / 2;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < pairs;
       i += int64_t(gridDim.x) * blockDim.x) {
    const float a = in[2 * i];
    const float b = 2 * i + 1 < n ? in[2 * i + 1] : 0.f;
    const uint32_t c = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
    out[2 * i] = uint8_t(c & 0xff);
    if (2 * i + 1 < n) out[2 * i + 1] = uint8_t(c >> 8);
  }
}
}  // namespace
void set_global_error(const std::string& msg);
}  // namespace gnntrk

extern "C" gnntrk_status gnntrk_e4m3_encode(const float* in, uint8_t* out, int64_t n,
                                            int32_t on_device, void* stream) {
  using namespace gnntrk;
  if (n < 0 || (n > 0 && (in == nullptr || out == nullptr))) {
    set_global_error("gnntrk_e4m3_encode: bad arguments");
    return GNNTRK_ERR_INVALID_ARG;
  }
  if (n == 0) return GNNTRK_OK;
  if (!on_device) {
    for (int64_t i = 0; i < n; ++i) out[i] = e4m3_from_float(in[i]);
    return GNNTRK_OK;
  }
  const int64_t pairs = (n + 1) / 2;
  const int grid = int(std::min<int64_t>(int64_t(device_sms()) * 8, (pairs + 255) / 256));
  k_e4m3_encode<<<grid, 256, 0, static_cast<cudaStream_t>(stream)>>>(in, out, n);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_global_error(std::string("gnntrk_e4m3_encode: ") + cudaGetErrorString(e));
    return GNNTRK_ERR_CUDA;
  }
  return GNNTRK_OK;
}

extern "C" gnntrk_status gnntrk_tc_throughput(int32_t n, int64_t iters, double* ms) {
  using namespace gnntrk;
  if (!ms || (n != 32 && n != 64 && n != 128 && n != 256) || iters < 1 || iters > (int64_t(1) << 30)) {
    set_global_error("gnntrk_tc_throughput: n must be 32, 64, 128 or 256, iters 1..2^30, ms not NULL");
    return GNNTRK_ERR_INVALID_ARG;
  }
  const int st = tc_probe(n, iters, ms);
  if (st != GNNTRK_OK) set_global_error("gnntrk_tc_throughput: the probe failed or timed out");
  return gnntrk_status(st);
}

extern "C" gnntrk_status gnntrk_e4m3_decode(const uint8_t* in, float* out, int64_t n) {
  using namespace gnntrk;
  if (n < 0 || (n > 0 && (in == nullptr || out == nullptr))) {
    set_global_error("gnntrk_e4m3_decode: bad arguments");
    return GNNTRK_ERR_INVALID_ARG;
  }
  for (int64_t i = 0; i < n; ++i) out[i] = e4m3_to_float(in[i]);
  return GNNTRK_OK;
}
