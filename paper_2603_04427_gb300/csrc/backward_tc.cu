// Gradient kernel of thin-key attention on the 5th-generation tensor cores:
// tcgen05.mma with accumulators in tensor memory, operands staged in shared
// memory by TMA.
//
// Paper: Section 2.1, Eqs. 1-4 (the forward being differentiated); training
// with thin keys is Sections 3.2-3.3.  Per head, with p = softmax(scale q k^T)
// (masked) and dL/d(out) = dO:
//     dV = p^T dO,  dP = dO v^T,  dS = p * (dP - D),  D_i = sum_c dO_ic out_ic,
//     dQ = scale dS k,  dK = scale dS^T q.
// The preprocessing pass (backward.cu) has written -lse log2(e) and -D for
// every query row, padded to a multiple of 128 rows (-inf and 0 on the
// padding: such rows get weight 0), and zeroed dQ.
//
// One CTA per (sequence, kv head g, 128-key tile j).  Keys are the MMA's M
// dimension and the TMEM lanes: thread t of a 4-warp group owns key t.  The
// CTA visits every 128-query tile i (i >= j when causal) of each of the G
// query heads of g, as two 64-query halves h:
//   warp 21 (one lane): TMA loads of K_j, V_j (once) and, per half tile, of
//       Q, dO and the rows' statistics into a ring.
//   warps 20 and 22 (whole warp, one elected lane issues): per tile and half
//       S^T_h  = K Q_h^T     (M=128 keys, N=64 queries, K=r)
//       dP^T_h = V dO_h^T    (M=128, N=64, K=d_v)
//       dV    += P^T_h dO_h  (N=d_v, K=64; P^T_h read from TMEM)
//       dK    += dS^T_h Q_h  (N=r,   K=64; dS^T_h from shared memory, K-major)
//     and per tile  dQ_i = dS K  (M=128 queries, N=r, K=128 keys; dS from the
//     same shared-memory tile read MN-major), completion on mbarriers through
//     tcgen05.commit.  Where TMEM has room for P^T in columns of its own and
//     shared memory for two dS tiles (the EARLY schedule), warp 20 issues the next
//     tile's S / dP products of a half as soon as the half's softmax warps have
//     read S / dP into registers, and warp 22 all others as their operands arrive;
//     otherwise warp 20 issues everything, each half's products after its softmax.
//   warps 0-15 (warps 8 h .. 8 h + 7: half h, 32 of its queries each group of four):
//       read their part of S^T_h and dP^T_h from TMEM 16 columns at a time, form
//       P^T = exp2(S^T scale log2e - lse log2e) (masked) and
//       dS^T = P^T (dP^T - D) in packed fp32 pairs, write P^T as bf16 into
//       TMEM and dS^T as bf16 into the swizzled shared-memory tile.  At the end they
//       store dV.
//   warps 16-19 (thread: one query): read dQ of each tile from TMEM and add it into
//       global dq, staged in shared memory, by TMA tensor reduce-adds
//       (cp.reduce.async.bulk.tensor .add).  At the end they store dK (times scale).
// What bounds it: the tensor pipe is busy for about 60 % of a tile's time (44 small
// products, 2000 cycles, those with N = 64 or r limited by reading A from shared
// memory), the rest are handoffs.  What brought it there (7B shape, B=2, H=32,
// S=8192, r=32, d_v=128, causal, preprocessing included): dQ read back by warps of
// its own instead of by the softmax warps (1987 -> 1743 us), sixteen softmax warps
// with 80 registers instead of eight with 168 and dK / dV through TMA stores
// (1655), the statistics apart from the tiles and two staging places for dQ (1608),
// warp-uniform waits of the softmax warps (1601).
// One product of N = 128 for both halves' S^T and dP^T needs fewer reads of K and
// V, but the halves then run in step and wait together: 1820 us.
//
// TMEM columns: [0,64) S^T_0, [64,128) dP^T_0, [128,192) S^T_1,
// [192,256) dP^T_1, then dV (d_v), dK (r), dQ (r), and where they fit P^T_0,
// P^T_1 (32 columns each; otherwise P^T_h sits in S^T_h, each group of four warps'
// 16 columns over the first half of the 32 it has read itself).
// At r = 128, dV, dK and dQ do not fit beside the score tiles: dQ_i is then
// computed over S^T_1 / dP^T_1 once the half-1 softmax has consumed them,
// warps 16-19 read it back at once, and the next half-1 scores follow.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "split.h"
#include "tc05.cuh"

namespace tk {
namespace {

constexpr int kKeys = 128;         // keys per CTA (MMA M, TMEM lanes)
constexpr int kQT = 128;           // queries per tile
constexpr int kHalfQ = 64;         // queries per S / dP half
// Warps 0-15: softmax gradient, four groups of four: query half 0 / 1, 32 of its
// 64 queries each; 16-19: dQ; 20: MMA; 21: TMA; 22: the gradients' MMAs where
// scores are issued early.
constexpr int kTcThreads = 736;
constexpr int kTcBound = 768;      // six warps per sub-partition: 80 registers per thread
constexpr int kWarpDq = 16, kWarpMma = 20, kWarpTma = 21, kWarpMma2 = 22;
constexpr int kTmemColsTc = 512;
constexpr int kBoxB = 128 * 128;   // one 64-column (128-byte) box of a 128-row tile

constexpr int align1k(int x) { return (x + 1023) / 1024 * 1024; }

template <int R, int DV>
struct TCfg {
  // Q / K rows are r bf16 = 2r bytes: one swizzle span of min(2r, 128) bytes,
  // in QK_NBOX boxes of QK_BOXW columns (two 128-byte boxes at r = 128)
  static constexpr int QK_SW = 2 * R < 128 ? 2 * R : 128;
  static constexpr int QK_NBOX = 2 * R / QK_SW;
  static constexpr int QK_BOXW = QK_SW / 2;
  static constexpr uint32_t QK_LAYOUT = QK_SW == 32 ? 6u : (QK_SW == 64 ? 4u : 2u);
  static constexpr int KSTEP_PER_BOX = QK_SW / 32;  // 16-column K steps per box
  static constexpr int KBOX = kKeys * QK_SW;        // one box of the K tile
  static constexpr int KB = QK_NBOX * KBOX;         // K tile
  static constexpr int VB = kKeys * DV * 2;         // V tile (DV / 64 boxes)
  // Q / dO arrive in 64-query half tiles through a ring of slots: a slot is
  // released as soon as its half's dV / dK products have read it
  static constexpr int QHBOX = kHalfQ * QK_SW;      // one box of a Q half tile
  static constexpr int QHB = QK_NBOX * QHBOX;       // Q half tile
  static constexpr int OHB = kHalfQ * DV * 2;       // dO half tile (DV / 64 boxes)
  static constexpr int OBOX = kHalfQ * 128;         // one 64-column box of a dO half tile
  static constexpr int SL_Q = 0, SL_O = align1k(QHB);
  static constexpr int SLOT = SL_O + OHB;
  static constexpr int STATS = 2 * kHalfQ * 4;      // a slot's -lse log2 e, then -D, apart from the tiles
  static constexpr int DSB = kKeys * kQT * 2;       // dS^T tile: [2 halves][128 keys][64 queries]
  // dQ of a tile in TMEM: in columns of its own where they fit (r <= 64), else
  // over S^T_1 / dP^T_1 once the half-1 softmax has consumed them (r = 128)
  static constexpr bool DQ_OWN = 256 + DV + 2 * R <= kTmemColsTc;
  // dQ read back by the dQ warps and staged for the TMA reduce-add in boxes of
  // DQ_W fp32 columns x 32 rows (one warp's) swizzled over DQ_SW bytes; where
  // shared memory holds a whole dQ tile (R <= 64) each box has its own place
  static constexpr int DQ_W = R < 32 ? R : 32;
  static constexpr int DQ_SW = DQ_W * 4;
  static constexpr int DQ_BOX = 32 * DQ_SW;
  static constexpr int DQ_PLACES = DQ_OWN ? R / DQ_W : 2;   // per warp
  static constexpr int DQ_LD = DQ_OWN ? DQ_W : 64;          // columns read at a time
  static constexpr int DQB = 4 * DQ_PLACES * DQ_BOX;
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = align1k(KB);
  static constexpr int OFF_SL = OFF_V + VB;
  // without the dS tiles: K, V, a ring of n slots, the dQ stage, barriers, alignment slack
  static constexpr int fixed(int n) { return OFF_SL + n * (SLOT + STATS) + DQB + 256 + 1024; }
  static constexpr int NDS = fixed(4) + 2 * DSB <= 227 * 1024 ? 2 : 1;   // dS^T tiles in flight
  // half-tile slots: 4 (a fifth, where it fits, measured slower), 3 where 4 do not fit
  static constexpr int NSLOT = fixed(4) + NDS * DSB <= 227 * 1024 ? 4 : 3;
  static constexpr int OFF_DS = OFF_SL + NSLOT * SLOT;
  static constexpr int OFF_DQ = OFF_DS + NDS * DSB;
  static constexpr int OFF_ST = OFF_DQ + DQB;
  static constexpr int OFF_BAR = OFF_ST + NSLOT * STATS;
  static constexpr int SMEM = std::max(OFF_BAR + 256 + 1024, kOneCtaSmem);
  static_assert(OFF_BAR + 256 + 1024 <= 227 * 1024, "shared memory");
  static_assert(OFF_DQ - OFF_SL >= kWarpDq * 4096 + 4 * 8192, "staging places of the epilogue");
  // TMEM columns
  static constexpr int T_S = 0;          // + 128 h: S^T_h
  static constexpr int T_DP = 64;        // + 128 h: dP^T_h
  static constexpr int T_DV = 256, T_DK = 256 + DV, T_DQ = DQ_OWN ? 256 + DV + R : 128;
  static_assert(T_DK + R <= kTmemColsTc && (!DQ_OWN || T_DQ + R <= kTmemColsTc), "TMEM columns");
  static constexpr bool P_OWN = DQ_OWN && T_DQ + R + 2 * (kHalfQ / 2) <= kTmemColsTc;  // P^T in columns of its own
  static constexpr int T_P = P_OWN ? T_DQ + R : T_S;   // + (P_OWN ? 32 : 128) h: P^T_h
  static constexpr int P_STRIDE = P_OWN ? kHalfQ / 2 : 128;
  // With P^T in its own columns and two dS tiles, the next tile's scores of a
  // half are issued as soon as the half's softmax warps have read S / dP into
  // registers, and a tile's dQ product one step later; otherwise the products
  // follow the softmax of each half.
  static constexpr bool EARLY = P_OWN && NDS == 2;
  // instruction descriptors
  static constexpr uint32_t ID_S = instr_desc(kKeys, kHalfQ, false);       // S^T, dP^T
  static constexpr uint32_t ID_DV = instr_desc(kKeys, DV, true);           // A = P^T (TMEM), B = dO MN-major
  static constexpr uint32_t ID_DK = instr_desc(kKeys, R, true);            // A = dS^T K-major, B = Q MN-major
  static constexpr uint32_t ID_DQ = instr_desc(kQT, R, true, true);        // A = dS MN-major, B = K MN-major
};

struct TcMaps {
  CUtensorMap q, k, v, d_out, dq, dk, dv;
};

// TMA tensor reduce-add of a shared-memory box into global memory (bulk group).
__device__ __forceinline__ void tma_reduce_add_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
  asm volatile(
      "cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(smem_addr(src)), "r"(x), "r"(y), "r"(z)
      : "memory");
}


// 16 consecutive columns at each of two TMEM addresses, one wait.
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, "
      "%27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : TK_R8(0), TK_R8(8), TK_R8(16), TK_R8(24)
      : "r"(ta), "r"(tb)
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), TK_W8(0)
               : "memory");
}
// N consecutive 32-bit columns (N = 16, 32 or 64).
template <int N>
__device__ __forceinline__ void tmem_ld_n(uint32_t taddr, uint32_t* v) {
  if constexpr (N == 16) tmem_ld16(taddr, v);
  else if constexpr (N == 32) tmem_ld32(taddr, v);
  else tmem_ld64(taddr, v);
}

__device__ __forceinline__ uint32_t pack2(float2 x) {
  __nv_bfloat162 v = __floats2bfloat162_rn(x.x, x.y);  // low half = x.x
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 f2(uint32_t a, uint32_t b) {
  return make_float2(__uint_as_float(a), __uint_as_float(b));
}

// Stages W fp32 columns of a warp's 32 rows (thread: one row) times `mul` as a
// box of 4 W bytes per row in the matching swizzle, for a TMA store or reduce.
template <int W>
__device__ __forceinline__ void stage_rows(unsigned char* box, const uint32_t* w, float mul, int lane) {
  constexpr int SW = W * 4, SHIFT = SW == 128 ? 0 : 1;
  static_assert(SW == 128 || SW == 64, "boxes of 32 or 16 columns");
#pragma unroll
  for (int c = 0; c < SW / 16; ++c) {
    const int pc = c ^ ((lane >> SHIFT) & (SW / 16 - 1));
    *reinterpret_cast<float4*>(box + lane * SW + pc * 16) =
        make_float4(__uint_as_float(w[4 * c]) * mul, __uint_as_float(w[4 * c + 1]) * mul,
                    __uint_as_float(w[4 * c + 2]) * mul, __uint_as_float(w[4 * c + 3]) * mul);
  }
  fence_proxy_async_smem();
  __syncwarp();
}

// N TMEM columns of a warp's 32 rows, times `mul`, to columns x .. x + N of rows
// row .. row + 31 of a plane by TMA stores of W columns each (rows past the
// tensor are cut off), staged in two places of 4 KB in turn.  Per-thread row
// stores instead touch 32 lines each (64 x 32 planes of S = 256: 339 us against 286).
template <int N, int W>
__device__ __forceinline__ void store_cols(const CUtensorMap* map, uint32_t taddr, unsigned char* places, float mul,
                                           int x, int row, int plane, int lane) {
#pragma unroll
  for (int c0 = 0; c0 < N; c0 += W) {
    uint32_t w[W];
    tmem_ld_n<W>(taddr + c0, w);
    if (c0 >= 2 * W) {   // the store before last has read this place
      if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      __syncwarp();
    }
    unsigned char* box = places + (c0 / W & 1) * 4096;
    stage_rows<W>(box, w, mul, lane);
    if (lane == 0) {
      tma_store_3d(map, box, x + c0, row, plane);
      bulk_commit();
    }
  }
}

// Where the CTAs of a split key tile leave their dK and dV, from the start of shared
// memory: per key R + DV floats in 16-byte pieces, swizzled by the key.
template <int R, int DV>
struct KeyPartial {
  static constexpr int PIECES = (R + DV) / 4, ROW = (PIECES + 7) / 8 * 8;
  static constexpr int BYTES = kKeys * ROW * 16;
  __device__ static int piece(int key, int c) { return (key * ROW + (c ^ (key & 7))) * 16; }
};

// W TMEM columns of this thread's key as pieces c0 .. of its partial.
template <int R, int DV, int W>
__device__ __forceinline__ void put_partial(uint32_t taddr, unsigned char* smem, int key, int c0) {
  uint32_t w[W];
  tmem_ld_n<W>(taddr, w);
#pragma unroll
  for (int c = 0; c < W / 4; ++c)
    *reinterpret_cast<uint4*>(smem + KeyPartial<R, DV>::piece(key, c0 + c)) =
        make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// This CTA's share of the tile's keys (rank, rank + C, ...) summed over the CTAs
// that have tiles (bit c of `have`), in their order, and written out by the 512
// softmax threads.
template <int R, int DV, int C>
__device__ __forceinline__ void sum_split(const BackwardParams& p, unsigned char* smem, int rank, uint32_t have, int key0,
                                          size_t plane, int tid) {
  using K = KeyPartial<R, DV>;
  constexpr int U = 8 / C;
  const int n = (min(kKeys, p.S - key0) - rank + C - 1) / C * K::PIECES;
  const uint32_t base = smem_addr(smem);
  for (int q0 = tid; q0 < n; q0 += 512 * U) {
    float4 y[U][C];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = min(q0 + 512 * u, n - 1);
      const uint32_t at = base + K::piece(rank + q / K::PIECES * C, q % K::PIECES);
#pragma unroll
      for (int c = 0; c < C; ++c) y[u][c] = ld_cluster_f32x4(cluster_addr(at, c));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + 512 * u, c4 = q % K::PIECES;
      if (q >= n) continue;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if ((have >> c) & 1u) {
          a.x += y[u][c].x;
          a.y += y[u][c].y;
          a.z += y[u][c].z;
          a.w += y[u][c].w;
        }
      }
      const size_t row = plane * p.S + key0 + rank + q / K::PIECES * C;
      if (c4 < R / 4) {
        a = make_float4(a.x * p.scale, a.y * p.scale, a.z * p.scale, a.w * p.scale);
        *reinterpret_cast<float4*>(p.dk + row * R + 4 * c4) = a;
      } else {
        *reinterpret_cast<float4*>(p.dv + row * DV + 4 * c4 - R) = a;
      }
    }
  }
}

// SPLIT: the CTAs of a cluster share a key tile's query tiles and add up their dK
// and dV through distributed shared memory at the end; for launches whose key tiles
// are too few or too uneven to keep the SMs busy alone (backward_split).
template <int R, int DV, bool SPLIT>
__global__ void __launch_bounds__(kTcBound, 1)
bwd_tc_kernel(const __grid_constant__ TcMaps maps, const BackwardParams p) {
  using C = TCfg<R, DV>;
  constexpr int NDS = C::NDS;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint64_t* kv_full = bars + 0;
  uint64_t* sl_full = bars + 1;      // [NSLOT] half-tile slot loaded
  uint64_t* sl_empty = bars + 6;     // [NSLOT] half-tile slot consumed
  uint64_t* s_full = bars + 11;      // [2] S^T_h, dP^T_h in TMEM
  uint64_t* p_ready = bars + 13;     // [2] P^T_h in TMEM, dS^T_h in shared memory
  uint64_t* p_free = bars + 15;      // [2] P^T_h read by the dV product (P in its own columns)
  uint64_t* ds_free = bars + 17;     // [NDS] dS^T tile read by its last product
  uint64_t* dq_full = bars + 19;
  uint64_t* dq_empty = bars + 20;
  uint64_t* acc_full = bars + 21;
  uint64_t* s_free = bars + 22;      // [2] S^T_h, dP^T_h read into registers (EARLY schedule)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 24);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = p.S, G = p.Hq / p.Hkv;
  const int n_kt = (S + kKeys - 1) / kKeys;
  const int n_qt = (S + kQT - 1) / kQT;
  // CTA order: (sequence, kv head) major, so that the CTAs at work read the same
  // queries, or key tile major where all queries stay in L2 anyway; the key tiles with
  // most work first
  const uint32_t work = SPLIT ? blockIdx.x / p.split : blockIdx.x;
  const int rank = SPLIT ? static_cast<int>(blockIdx.x % p.split) : 0;   // = the rank in the cluster
  const int j = static_cast<int>(p.tile_major ? work / (p.B * p.Hkv) : work % n_kt);
  const int bg = static_cast<int>(p.tile_major ? work % (p.B * p.Hkv) : work / n_kt);
  const int b = bg / p.Hkv, g = bg % p.Hkv;
  const int i0 = p.causal ? j : 0;     // kKeys == kQT: query tiles i >= j see key tile j
  const int per_head = n_qt - i0;
  // this CTA's tiles: t0 .. t0 + n_tiles - 1 of the key tile's, counted from t0
  const int all_tiles = G * per_head;
  auto first_tile = [&](int c) { return SPLIT ? all_tiles * c / p.split : 0; };
  const int t0 = first_tile(rank), n_tiles = SPLIT ? first_tile(rank + 1) - t0 : all_tiles;
  auto tile_head = [&](int t) { return g * G + (t0 + t) / per_head; };
  auto tile_q = [&](int t) { return i0 + (t0 + t) % per_head; };
  // half tile u = 2 t + h lives in slot u % NSLOT, its (u / NSLOT)-th use of the slot
  auto slot_of = [](int t, int h) { return (2 * t + h) % C::NSLOT; };
  auto slot_par = [](int t, int h) { return static_cast<uint32_t>(((2 * t + h) / C::NSLOT) & 1); };

  if (tid == 0) {
    mbar_init(kv_full, 1);
    for (int s = 0; s < C::NSLOT; ++s) {
      mbar_init(&sl_full[s], 1);
      mbar_init(&sl_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&s_full[s], 1);
      mbar_init(&p_ready[s], 256);
      mbar_init(&p_free[s], 1);
      mbar_init(&s_free[s], 256);
    }
    for (int s = 0; s < NDS; ++s) mbar_init(&ds_free[s], 1);
    mbar_init(dq_full, 1);
    mbar_init(dq_empty, 128);
    mbar_init(acc_full, 1);
    fence_barrier_init();
  }
  if (warp == kWarpMma) {
    tmem_alloc(tmem_slot, kTmemColsTc);
    tmem_relinquish();
  }
  if (warp == kWarpTma && lane == 0) {
    prefetch_map(&maps.q);
    prefetch_map(&maps.k);
    prefetch_map(&maps.v);
    prefetch_map(&maps.d_out);
  }
  // the set-up above reads no global memory: it runs while the previous kernel finishes
  pdl_wait();
  __syncthreads();
  // after the barrier, so that every CTA of this grid holds its TMEM before a
  // CTA of the next kernel can ask for some
  pdl_trigger();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (SPLIT && n_tiles == 0) {
    // fewer tiles than CTAs: this one only takes its share of the sums below
  } else if (warp == kWarpTma) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const int kv_plane = b * p.Hkv + g;
      mbar_arrive_expect_tx(kv_full, C::KB + C::VB);
      for (int x = 0; x < C::QK_NBOX; ++x)
        tma_load_3d(smem + C::OFF_K + x * C::KBOX, &maps.k, x * C::QK_BOXW, j * kKeys, kv_plane, kv_full);
      for (int x = 0; x < DV / 64; ++x)
        tma_load_3d(smem + C::OFF_V + x * kBoxB, &maps.v, 64 * x, j * kKeys, kv_plane, kv_full);
      int issued = 0;
      for (int u = 0; u < 2 * n_tiles; ++u) {
        const int sl = u % C::NSLOT;
        if (u >= C::NSLOT && !mbar_wait(&sl_empty[sl], ((u / C::NSLOT) - 1) & 1, p.err)) break;
        const int t = u >> 1, h = u & 1;
        const int bh = b * p.Hq + tile_head(t), row = tile_q(t) * kQT + h * kHalfQ;
        unsigned char* sb = smem + C::OFF_SL + sl * C::SLOT;
        mbar_arrive_expect_tx(&sl_full[sl], C::QHB + C::OHB + 2 * kHalfQ * 4);
        for (int x = 0; x < C::QK_NBOX; ++x)
          tma_load_3d(sb + C::SL_Q + x * C::QHBOX, &maps.q, x * C::QK_BOXW, row, bh, &sl_full[sl]);
        for (int x = 0; x < DV / 64; ++x)
          tma_load_3d(sb + C::SL_O + x * C::OBOX, &maps.d_out, 64 * x, row, bh, &sl_full[sl]);
        const size_t srow = static_cast<size_t>(bh) * p.S_pad + row;
        bulk_g2s(smem + C::OFF_ST + sl * C::STATS, p.nl2 + srow, kHalfQ * 4, &sl_full[sl]);
        bulk_g2s(smem + C::OFF_ST + sl * C::STATS + kHalfQ * 4, p.nd + srow, kHalfQ * 4, &sl_full[sl]);
        issued = u + 1;
      }
      // no copy may still be landing in shared memory when the CTA exits
      // (normally all were consumed; after a timed-out wait, bounded waits)
      mbar_wait(kv_full, 0, p.err);
      for (int u = std::max(0, issued - C::NSLOT); u < issued; ++u)
        mbar_wait(&sl_full[u % C::NSLOT], (u / C::NSLOT) & 1, p.err);
    }
  } else if (warp == kWarpMma || (C::EARLY && warp == kWarpMma2)) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t s_base = smem_addr(smem);
    // one descriptor serves a tile read K-major and MN-major: SBO is the stride of
    // 8-row groups either way, LBO the stride of MN atoms (unused when N fits one)
    const Desc dK_d = make_desc(s_base + C::OFF_K, C::KBOX, 8 * C::QK_SW, C::QK_LAYOUT);  // K
    const Desc dV_a = make_desc(s_base + C::OFF_V, 16, 1024, 2u);                         // V, K-major
    const Desc dQ_b = make_desc(s_base + C::OFF_SL + C::SL_Q, C::QHBOX, 8 * C::QK_SW, C::QK_LAYOUT);  // Q_h
    const Desc dO_bk = make_desc(s_base + C::OFF_SL + C::SL_O, 16, 1024, 2u);             // dO_h, K-major
    const Desc dO_bm = make_desc(s_base + C::OFF_SL + C::SL_O, C::OBOX, 1024, 2u);        // dO_h, MN-major
    const Desc dS_ak = make_desc(s_base + C::OFF_DS, 16, 1024, 2u);                       // dS^T, K-major
    const Desc dS_am = make_desc(s_base + C::OFF_DS, C::DSB / 2, 1024, 2u);               // dS, MN-major
    auto issue_sdp = [&](int t, int h) {   // S^T_h, dP^T_h of tile t
      const uint32_t so = slot_of(t, h) * C::SLOT;
#pragma unroll
      for (int k = 0; k < R / 16; ++k) {
        const uint32_t kb = (k / C::KSTEP_PER_BOX), ko = (k % C::KSTEP_PER_BOX) * 32;
        mma_ss_e(tmem + C::T_S + 128 * h, dK_d.at(kb * C::KBOX + ko), dQ_b.at(so + kb * C::QHBOX + ko), C::ID_S,
                 k > 0);
      }
#pragma unroll
      for (int k = 0; k < DV / 64; ++k)
        mma_ss4_e(tmem + C::T_DP + 128 * h, dV_a.at(k * kBoxB), 32, dO_bk.at(so + k * C::OBOX), 32, C::ID_S, k > 0);
      tc_commit_e(&s_full[h]);
    };
    auto issue_dvdk = [&](int t, int h) {  // dV += P^T_h dO_h, dK += dS^T_h Q_h; the slot is then free
      const uint32_t so = slot_of(t, h) * C::SLOT;
      const uint32_t dso = (t % NDS) * C::DSB + h * (C::DSB / 2);
      static_assert(kHalfQ == 64, "four K steps per half");
      const uint32_t acc = (t > 0 || h > 0) ? 1u : 0u;
      mma_ts4_e(tmem + C::T_DV, tmem + C::T_P + C::P_STRIDE * h, dO_bm.at(so), 16 * 128, C::ID_DV, acc,
                C::P_OWN ? 16 : 32);
      if (C::P_OWN) tc_commit_e(&p_free[h]);
      mma_ss4_e(tmem + C::T_DK, dS_ak.at(dso), 32, dQ_b.at(so), 16 * C::QK_SW, C::ID_DK, acc);
      tc_commit_e(&sl_empty[slot_of(t, h)]);
    };
    auto issue_dq = [&](int t) {           // dQ_t = dS K over the 128 keys
      const uint32_t dso = (t % NDS) * C::DSB;
#pragma unroll
      for (int k = 0; k < kKeys / 64; ++k)
        mma_ss4_e(tmem + C::T_DQ, dS_am.at(dso + k * 64 * 128), 16 * 128, dK_d.at(k * 64 * C::QK_SW), 16 * C::QK_SW,
                  C::ID_DQ, k > 0);
      tc_commit_e(dq_full);
      tc_commit_e(&ds_free[t % NDS]);
    };
    auto wait_all = [&](uint64_t* bar, uint32_t parity) {
      return mbar_wait_warp(bar, parity, p.err);
    };
    bool ok = true;
    if (warp == kWarpMma) {
      ok = wait_all(kv_full, 0) && wait_all(&sl_full[0], 0);
      if (ok) {
        tc_fence_after();
        issue_sdp(0, 0);
        ok = wait_all(&sl_full[1], 0);
        tc_fence_after();
        if (ok) issue_sdp(0, 1);
      }
    }
    if constexpr (C::EARLY) {
      // Two issuing warps, so that neither waits for what only the other needs.
      // One: the next tile's scores of each half as soon as its softmax warps
      // release S / dP.  The other: a tile's dV / dK products when P / dS arrive
      // (its Q and dO half tiles have landed: its scores were computed), then its
      // dQ product.
      if (warp == kWarpMma) {
        for (int t = 1; ok && t < n_tiles; ++t) {
          for (int h = 0; ok && h < 2; ++h) {
            if (!(ok = wait_all(&sl_full[slot_of(t, h)], slot_par(t, h)) && wait_all(&s_free[h], (t - 1) & 1))) break;
            tc_fence_after();
            issue_sdp(t, h);
          }
        }
        ok = false;   // the other warp commits the accumulators
      } else {
        for (int t = 0; ok && t < n_tiles; ++t) {
          for (int h = 0; ok && h < 2; ++h) {
            if (!(ok = wait_all(&p_ready[h], t & 1))) break;
            tc_fence_after();
            issue_dvdk(t, h);
          }
          if (!ok || (t > 0 && !(ok = wait_all(dq_empty, (t - 1) & 1)))) break;
          tc_fence_after();
          issue_dq(t);
        }
      }
    } else {
      for (int t = 0; ok && t < n_tiles; ++t) {
        const bool next = t + 1 < n_tiles;
        for (int h = 0; ok && h < 2; ++h) {
          if (!(ok = wait_all(&p_ready[h], t & 1))) break;
          if (next && !(ok = wait_all(&sl_full[slot_of(t + 1, h)], slot_par(t + 1, h)))) break;
          tc_fence_after();
          // P^T_h in columns of its own: the next tile's scores of this half go
          // first; otherwise P^T_h overlays S^T_h and its dV product goes first
          if (C::P_OWN && next) issue_sdp(t + 1, h);
          issue_dvdk(t, h);
          if (h == 1) {
            // dQ before the next tile's half-1 scores: with one dS tile the next
            // tile's half-0 dS waits for it, and without columns of its own dQ
            // occupies S^T_1 / dP^T_1 until the dQ warps have read it
            if (C::DQ_OWN && t > 0 && !(ok = wait_all(dq_empty, (t - 1) & 1))) break;
            tc_fence_after();
            issue_dq(t);
            if (!C::DQ_OWN && next) {
              if (!(ok = wait_all(dq_empty, t & 1))) break;
              tc_fence_after();
            }
          }
          if (!C::P_OWN && next) issue_sdp(t + 1, h);
        }
      }
    }
    if (ok) tc_commit_e(acc_full);
  } else if (warp >= kWarpDq && warp < kWarpDq + 4) {
    // ------------------------------------------------------------------ dQ warps
    // dQ of every tile (thread: query 32 w + lane of the tile, its TMEM lane) read
    // from TMEM, scaled, staged in shared memory and added into global dq by one
    // TMA tensor reduce-add per box, so that no warp waits for another.
    const int w4 = warp & 3;
    const uint32_t lane_off = static_cast<uint32_t>(w4 * 32) << 16;
    unsigned char* place = smem + C::OFF_DQ + w4 * (C::DQ_PLACES * C::DQ_BOX);
    bool pending = false;
    for (int t = 0; t < n_tiles; ++t) {
      if (!mbar_wait_warp(dq_full, t & 1, p.err)) break;
      tc_fence_after();
      const int row0 = tile_q(t) * kQT + w4 * 32;   // first query of this warp's rows
#pragma unroll
      for (int c0 = 0; c0 < R; c0 += C::DQ_LD) {
        uint32_t w[C::DQ_LD];
        tmem_ld_n<C::DQ_LD>(tmem + C::T_DQ + c0 + lane_off, w);
        if (c0 + C::DQ_LD == R) {
          tc_fence_before();
          mbar_arrive(dq_empty);
        }
        if (row0 >= S) continue;
        if (c0 % (C::DQ_PLACES * C::DQ_W) == 0) {   // the previous reduce-adds have read their boxes
          if (lane == 0 && pending) bulk_wait_read_all();
          __syncwarp();
        }
#pragma unroll
        for (int x = 0; x < C::DQ_LD; x += C::DQ_W) {
          unsigned char* box = place + (c0 + x) / C::DQ_W % C::DQ_PLACES * C::DQ_BOX;
          stage_rows<C::DQ_W>(box, w + x, p.scale, lane);
          if (lane == 0) {
            tma_reduce_add_3d(&maps.dq, box, c0 + x, row0, b * p.Hq + tile_head(t));
            bulk_commit();
            pending = true;
          }
        }
      }
    }
    // dK of the CTA's keys (these warps are done before the softmax warps are)
    const int key0 = j * kKeys + w4 * 32;
    if (SPLIT) {
      if (mbar_wait_warp(acc_full, 0, p.err)) {
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < R; c0 += C::DQ_W)
          put_partial<R, DV, C::DQ_W>(tmem + C::T_DK + c0 + lane_off, smem, w4 * 32 + lane, c0 / 4);
      }
    } else if (mbar_wait_warp(acc_full, 0, p.err) && key0 < S) {
      tc_fence_after();
      store_cols<R, C::DQ_W>(&maps.dk, tmem + C::T_DK + lane_off, smem + C::OFF_SL + kWarpDq * 4096 + w4 * 8192, p.scale, 0, key0,
                             b * p.Hkv + g, lane);
    }
    if (lane == 0) bulk_wait_read_all();
  } else if (warp < kWarpDq) {
    // ------------------------------------------------------------------ softmax gradient warps
    const int h = warp >> 3;                      // query half
    const int cg = (warp >> 2) & 1;               // which 32 of its queries
    const int kt = (warp & 3) * 32 + lane;        // key of this thread within the tile (TMEM lane)
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + C::T_S + 128 * h + lane_off, tD = tmem + C::T_DP + 128 * h + lane_off;
    const uint32_t tP = tmem + C::T_P + C::P_STRIDE * h + lane_off;
    const bool kvalid = j * kKeys + kt < S;
    const float sl2 = p.scale * 1.4426950408889634f;
    const float2 sl2x2 = make_float2(sl2, sl2);
    bool ok = true;
    for (int t = 0; t < n_tiles; ++t) {
      const int sl = slot_of(t, h), buf = t % NDS;
      if (ok) {
        ok = mbar_wait_warp(&s_full[h], t & 1, p.err) && mbar_wait_warp(&sl_full[sl], slot_par(t, h), p.err);
        // (with one dS tile its buffer is asked for as late as possible, below)
        if (NDS > 1 && ok && t >= NDS) ok = mbar_wait_warp(&ds_free[buf], ((t / NDS) - 1) & 1, p.err);
      }
      if (ok) {
        tc_fence_after();
        const float* nl2 = reinterpret_cast<const float*>(smem + C::OFF_ST + sl * C::STATS);
        const float* nd = nl2 + kHalfQ;
        unsigned char* ds_row = smem + C::OFF_DS + buf * C::DSB + h * (C::DSB / 2) + kt * 128;
        // keys past S, and keys after the query on the diagonal tile, get weight 0
        const int qlim = (p.causal && tile_q(t) == j) ? kt - h * kHalfQ : 0;  // visible iff column >= qlim
        // warp-uniform choice: both paths issue warp-collective TMEM loads and stores
        const bool masked = __any_sync(0xffffffffu, !kvalid || qlim > 0);
        auto chunk = [&](auto mask_tag, int c) {   // queries 16 c .. 16 c + 15 of the half
          constexpr bool kMask = decltype(mask_tag)::value;
          uint32_t v[32];   // [0, 16): S^T, [16, 32): dP^T
          tmem_ld16x2(tS + 16 * c, tD + 16 * c, v);
          if (C::EARLY && (c & 1)) {   // these columns of S^T_h, dP^T_h may be overwritten
            tc_fence_before();
            mbar_arrive(&s_free[h]);
          }
          uint32_t pk[8], dk[8];
#pragma unroll
          for (int e2 = 0; e2 < 8; ++e2) {
            // (pairs: a broadcast 16-byte shared load takes twice the wavefronts per byte)
            const int col = 16 * c + 2 * e2;
            float2 x = ffma2(f2(v[2 * e2], v[2 * e2 + 1]), sl2x2, *reinterpret_cast<const float2*>(nl2 + col));
            if (kMask) {
              if (!kvalid || col < qlim) x.x = -INFINITY;
              if (!kvalid || col + 1 < qlim) x.y = -INFINITY;
            }
            const float2 pr = make_float2(fast_exp2(x.x), fast_exp2(x.y));
            const float2 dsv = fmul2(pr, fadd2(f2(v[16 + 2 * e2], v[17 + 2 * e2]),
                                               *reinterpret_cast<const float2*>(nd + col)));
            pk[e2] = pack2(pr);
            dk[e2] = pack2(dsv);
          }
          // P^T_h may overwrite the previous tile's only once its dV product has read
          // it, dS^T_h its buffer's last tile once its dK and dQ products have
          if (!(c & 1) && t > 0 && (C::P_OWN || NDS == 1)) {
            if (C::P_OWN && !mbar_wait_warp(&p_free[h], (t - 1) & 1, p.err)) ok = false;
            if (NDS == 1 && !mbar_wait_warp(&ds_free[0], (t - 1) & 1, p.err)) ok = false;
          }
          // over scores that this warp itself has read, where P^T has no columns of its own
          tmem_st8(tP + (C::P_OWN ? 8 * c : 32 * (c >> 1) + 8 * (c & 1)), pk);
          // dS^T row kt, queries 16 c .. 16 c + 15 of the half: two 16-byte pieces, SW128 swizzle
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int chunk_i = (2 * c + m) ^ (kt & 7);
            *reinterpret_cast<uint4*>(ds_row + chunk_i * 16) =
                make_uint4(dk[4 * m], dk[4 * m + 1], dk[4 * m + 2], dk[4 * m + 3]);
          }
        };
#pragma unroll
        for (int c = 2 * cg; c < 2 * cg + 2; ++c) {
          if (masked) chunk(std::true_type{}, c);
          else chunk(std::false_type{}, c);
        }
        tmem_wait_st();
        fence_proxy_async_smem();
        tc_fence_before();
        mbar_arrive(&p_ready[h]);
      }
    }
    // dV of the CTA's keys, 32 columns each group of four warps; the ring and the dS
    // tiles are free: every product has read them
    const int key0 = j * kKeys + (warp & 3) * 32, x0 = 32 * (warp >> 2);
    if (ok) ok = mbar_wait(acc_full, 0, p.err);
    if (SPLIT) {
      if (__all_sync(0xffffffffu, ok) && x0 < DV) {
        tc_fence_after();
        put_partial<R, DV, 32>(tmem + C::T_DV + x0 + lane_off, smem, kt, (R + x0) / 4);
      }
    } else if (__all_sync(0xffffffffu, ok) && key0 < S && x0 < DV) {
      tc_fence_after();
      store_cols<32, 32>(&maps.dv, tmem + C::T_DV + x0 + lane_off, smem + C::OFF_SL + warp * 4096, 1.f, x0, key0,
                         b * p.Hkv + g, lane);
    }
    if (lane == 0) bulk_wait_read_all();
  }
  if constexpr (SPLIT) {
    static_assert(KeyPartial<R, DV>::BYTES <= C::OFF_DQ, "partials over K, V, the ring and the dS tiles");
    cluster_sync();
    if (warp < kWarpDq) {
      uint32_t have = 0;
      for (int c = 0; c < p.split; ++c) have |= (first_tile(c + 1) > first_tile(c) ? 1u : 0u) << c;
      const size_t plane = static_cast<size_t>(b) * p.Hkv + g;
      if (p.split == 2) sum_split<R, DV, 2>(p, smem, rank, have, j * kKeys, plane, tid);
      else if (p.split == 4) sum_split<R, DV, 4>(p, smem, rank, have, j * kKeys, plane, tid);
      else sum_split<R, DV, 8>(p, smem, rank, have, j * kKeys, plane, tid);
    }
    cluster_sync();  // no CTA leaves while others read its shared memory
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemColsTc);
  }
}

template <int R, int DV>
cudaError_t launch_tc(const BackwardParams& p, cudaStream_t stream) {
  using C = TCfg<R, DV>;
  TcMaps maps;
  if (!make_map(&maps.q, p.q, R, p.S, p.B * p.Hq, C::QK_BOXW, kHalfQ, C::QK_SW) ||
      !make_map(&maps.k, p.k, R, p.S, p.B * p.Hkv, C::QK_BOXW, kKeys, C::QK_SW) ||
      !make_map(&maps.v, p.v, DV, p.S, p.B * p.Hkv, 64, kKeys, 128) ||
      !make_map(&maps.d_out, p.d_out, DV, p.S, p.B * p.Hq, 64, kHalfQ, 128) ||
      !make_map(&maps.dq, p.dq, R, p.S, p.B * p.Hq, C::DQ_W, 32, C::DQ_SW, true) ||
      !make_map(&maps.dk, p.dk, R, p.S, p.B * p.Hkv, C::DQ_W, 32, C::DQ_SW, true) ||
      !make_map(&maps.dv, p.dv, DV, p.S, p.B * p.Hkv, 32, 32, 128, true))
    return cudaErrorInvalidValue;
  const long long n_kt = (p.S + kKeys - 1) / kKeys;
  const long long grid = static_cast<long long>(p.B) * p.Hkv * n_kt;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  BackwardParams pp = p;
  pp.split = backward_split(p.B, p.Hq, p.Hkv, p.S, p.causal != 0, p.num_sms);
  pp.tile_major = backward_tile_major(p.B, p.Hq, p.S, R, DV);
  auto kern = pp.split > 1 ? bwd_tc_kernel<R, DV, true> : bwd_tc_kernel<R, DV, false>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  return launch_pdl_cluster(kern, dim3(static_cast<unsigned>(grid * pp.split)), dim3(kTcThreads), C::SMEM, stream,
                            pp.split, maps, pp);
}

template <int R>
cudaError_t tc_by_dv(const BackwardParams& p, cudaStream_t s, int* uns) {
  switch (p.DV) {
    case 64: return launch_tc<R, 64>(p, s);
    case 128: return launch_tc<R, 128>(p, s);
  }
  *uns = 1;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_backward_tc(const BackwardParams& p, cudaStream_t stream, int* unsupported) {
  switch (p.R) {
    case 16: return tc_by_dv<16>(p, stream, unsupported);
    case 32: return tc_by_dv<32>(p, stream, unsupported);
    case 64: return tc_by_dv<64>(p, stream, unsupported);
    case 128: return tc_by_dv<128>(p, stream, unsupported);
  }
  *unsupported = 1;
  return cudaSuccess;
}

}  // namespace tk
