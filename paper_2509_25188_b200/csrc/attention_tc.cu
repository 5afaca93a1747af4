// Bidirectional (non-causal) multi-head attention on the 5th-generation tensor cores, head size 128.
// Flash style: one pass over the keys in tiles of 128 with a running row max and row sum, so the
// [queries x keys] scores never leave the SM.  Every query of a sequence sees keys [0, kv_len) of
// that sequence: there is no mask, only the ragged tail of the last key tile.
//
// An item is 128 query rows of one head; a persistent CTA per SM takes items in turn.  Two groups of four softmax warps take
// the CTA's key tiles alternately, three score buffers keep the tensor pipe ahead of them.  Per key tile T of 128 keys
// (counted over all items of the CTA: group T mod 2, buffer b = T mod 3):
//     S_b  = Q K_T^T            tcgen05.mma, Q and K_T K-major in shared memory (TMA, 128-byte swizzle), fp32 scores in
//                               tensor memory
//     P_b  = exp2(S_b c - m)    a softmax thread owns a row: no exchange within a tile.  Packed bf16 pairs go over the
//                               scores' first 64 columns, where the second product reads them as its A operand
//     O   += P_b V_T            tcgen05.mma, A from tensor memory, V_T read MN-major from shared memory (rows of V are
//                               keys = the K dimension); O stays in tensor memory for the whole item
// m is the row's reference maximum.  It follows the running maximum lazily: only when the maximum has grown by more than 8 (a
// factor 256) does the thread rescale O.  Both groups take probabilities against the same m: the thread that has fixed it for
// a tile hands it to the other group's thread of the same row before its exponentials, so the hand-over is half a tile old
// when it is looked for.  With it go the sums of the group's tile before, so that the row sums grow in the order of the tiles.
// One warp issues all products in the order S(0) S(1) S(2) PV(0) S(3) PV(1) ..., running on into the next item: the tensor
// pipe keeps that order, so S(T + 3) cannot overtake the PV(T) that still reads the probabilities it overwrites, and scores of
// a group's next tile, of the next item too, are complete while it is still at the exponentials of its last one.  K and V
// travel through one ring in the order of their use, five tiles of 32 KB deep.
//
// What bounds it: for a 128 x 128 tile the exponentials take the SM's special-function units 1024 cycles, the two products
// the tensor pipe 1032, and their operands with the tiles' arrival shared memory 1280; measured 1240 a tile, 1900 with every
// SM busy for long.  A CTA per item spent 9000 cycles on its start, first loads, first scores and last product, the time of
// seven tiles, and 2000 on storing rows 16 bytes at a time: hence the persistent loop and the staged output.  One head-set of
// eight sequences of 1024 rows (256 heads): 197 -> 148 us (928 TFLOP/s); four of 2048: 320 -> 255 us (1077); 512 rows, one
// item to a CTA: 11.3 -> 10.5 us.  Few query rows: the stream of K and V; warps without rows only keep the barriers.  32
// rows on 2048 keys, eight sequences: 52 -> 44.5 us, 6.0 TB/s.
//
// Warp roles (384 threads): 0 = TMA producer, 1 = MMA issuer (owns tensor memory), 4-7 and 8-11 = softmax groups 0 and 1 and
// output (group g writes head dimensions 64 g .. 64 g + 63).
// Tensor memory (512 columns): S_b at 128 b, O at 384.
// Every wait is bounded; a wait that runs out sets the status word and the CTA leaves normally.
#include <math.h>

#include "common.cuh"
#include "ptx.cuh"

namespace l2pd {

namespace {

constexpr int BQ = 128, BKV = 128, DH = 128;
constexpr uint32_t HALF_BYTES = 128 * 128;        // 128 rows x 64 bf16: one swizzled half tile
constexpr uint32_t TILE_BYTES = 2 * HALF_BYTES;   // 128 x 128 bf16
constexpr int RING = 5, NS = 3;
constexpr uint32_t STAGE_BYTES = 32 * 64;         // a warp's output staging: 32 rows x 32 bf16
constexpr int SMEM_BYTES = (1 + RING) * TILE_BYTES + 8 * STAGE_BYTES + 1024;   // Q, the ring, staging (+ alignment slack)
constexpr int REGS_LEAN = 56, REGS_SOFTMAX = 224;            // 384 x 168 = 128 x 56 + 256 x 224

struct AttnTcParams {
  bf16 *out;
  const SeqMeta *meta;
  SeqMeta single;
  int use_single;
  int64_t out_stride;
  float scale_log2;
  int kv_rows_per_seq;   // rows between two sequences in the key/value tensor maps
  int kv_row_base;       // first row of this layer's store in the key/value tensor maps
  int H, n_qt, n_items;  // items: [sequence slot][head][query tile], query tiles fastest
  int kv_packed;         // keys / values are the packed activation rows: row = row0 of the sequence + key
  int32_t *status;
};

enum { B_QFULL = 0, B_QFREE = 1, B_FULL = 2, B_EMPTY = B_FULL + RING, B_SFULL = B_EMPTY + RING, B_PFULL = B_SFULL + NS, B_PV = B_PFULL + NS,
       B_OFULL = B_PV + 2, B_OFREE = B_OFULL + 1, B_MREF = B_OFREE + 1, B_MEET = B_MREF + 8, B_COUNT = B_MEET + 4 };
constexpr float RESCALE_STEP = 8.0f;   // log2 units the row maximum may run ahead of the reference maximum

__device__ __forceinline__ void fail(int32_t *status, int code) {
  if (status) atomicCAS(status, 0, code);
}

__global__ void __launch_bounds__(384, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const AttnTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[B_COUNT];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sRing = base + TILE_BYTES;
  // [group][row]: reference maximum of the group's last tile; sums (two halves of 64 keys) and factor of the one before
  __shared__ float4 hand[2][BQ];
  // [item parity][group][row]: sums and factor of the group's last tile of an item; the row sums two tiles before it
  __shared__ float4 fin[2][2][BQ];
  __shared__ float2 fin_l[2][2][BQ];
  const uint32_t bar0 = ptx::smem_u32(bars);
  auto bar = [&](int i) { return bar0 + 8u * i; };

  if (threadIdx.x == 0) {
    ptx::mbar_init(bar(B_QFULL), 1);
    ptx::mbar_init(bar(B_QFREE), 1);
    for (int i = 0; i < RING; ++i) { ptx::mbar_init(bar(B_FULL + i), 1); ptx::mbar_init(bar(B_EMPTY + i), 1); }
    for (int i = 0; i < NS; ++i) { ptx::mbar_init(bar(B_SFULL + i), 1); ptx::mbar_init(bar(B_PFULL + i), 4); }
    for (int i = 0; i < 2; ++i) ptx::mbar_init(bar(B_PV + i), 1);
    for (int i = 0; i < 8; ++i) ptx::mbar_init(bar(B_MREF + i), 1);
    ptx::mbar_init(bar(B_OFULL), 1);
    ptx::mbar_init(bar(B_OFREE), 8);
    for (int i = 0; i < 4; ++i) ptx::mbar_init(bar(B_MEET + i), 2);
    abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmQ); ptx::prefetch_tensormap(&tmK); ptx::prefetch_tensormap(&tmV);
  }
  if (warp == 1) { ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), 512); ptx::tmem_relinquish(); }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = tmem_slot;
  const uint32_t tS = tmem_base, tO = tmem_base + NS * BKV;
  grid_dep_launch();
  grid_dep_wait();

  int32_t *const status = p.status;
  // One item's coordinates; n_tiles = 0: nothing to do (the same answer in every role)
  struct Item { int q0, h, row0, n_rows, kv_len, krow, n_tiles; };
  auto item_at = [&](int i) {
    Item w;
    const int per_slot = p.H * p.n_qt, z = i / per_slot, y = i - z * per_slot;
    const SeqMeta m = p.use_single ? p.single : p.meta[z];
    w.h = y / p.n_qt;
    w.q0 = (y - w.h * p.n_qt) * BQ;
    w.row0 = m.row0; w.n_rows = m.n_rows; w.kv_len = m.kv_len;
    w.krow = p.kv_row_base + (p.kv_packed ? m.row0 : m.seq * p.kv_rows_per_seq);
    w.n_tiles = w.q0 < w.n_rows ? (w.kv_len + BKV - 1) / BKV : 0;
    return w;
  };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LEAN));
    if (warp == 0) {
      // ------------------------------------------------------------------ TMA producer: Q, then K0 K1 K2 V0 K3 V1 ..., where
      // "next" runs on into the following item: its first keys go ahead of this item's last values
      uint32_t dst = sRing, full = bar(B_FULL), par = 1, qpar = 1;
      int slot = 0;
      auto load = [&](const CUtensorMap *tm, int col, int row, uint64_t pol) {
        const bool ok = ptx::mbar_wait_or_abort(full + 8u * RING, par, &abort_flag, status, DEV_TIMEOUT_PRODUCER);
        if (ptx::elect_one() && ok) {
          ptx::mbar_arrive_expect_tx(full, TILE_BYTES);
          ptx::tma_load_2d_hint(dst, tm, full, col, row, pol);
          ptx::tma_load_2d_hint(dst + HALF_BYTES, tm, full, col + 64, row, pol);
        }
        dst += TILE_BYTES; full += 8u;
        if (++slot == RING) { slot = 0; dst = sRing; full = bar(B_FULL); par ^= 1u; }
      };
      int col1 = 0, row1 = -1, col2 = 0, row2 = -1;   // the values of the last tile and of the one before, not loaded yet
      uint64_t pol1 = 0, pol2 = 0;
      for (int i = blockIdx.x; i < p.n_items; i += gridDim.x) {
        const Item w = item_at(i);
        if (w.n_tiles == 0) continue;
        // K and V of a head are re-read by every other query tile; read once when there is only this one
        const uint64_t pol = w.n_rows > BQ ? ptx::policy_evict_last() : ptx::policy_evict_first();
        const bool ok = ptx::mbar_wait_or_abort(bar(B_QFREE), qpar, &abort_flag, status, DEV_TIMEOUT_PRODUCER);
        qpar ^= 1u;
        if (ptx::elect_one() && ok) {
          ptx::mbar_arrive_expect_tx(bar(B_QFULL), TILE_BYTES);
          ptx::tma_load_2d(sQ, &tmQ, bar(B_QFULL), w.h * DH, w.row0 + w.q0);
          ptx::tma_load_2d(sQ + HALF_BYTES, &tmQ, bar(B_QFULL), w.h * DH + 64, w.row0 + w.q0);
        }
        for (int t = 0; t < w.n_tiles; ++t) {
          load(&tmK, w.h * DH, w.krow + t * BKV, pol);
          if (row2 >= 0) load(&tmV, col2, row2, pol2);
          col2 = col1; row2 = row1; pol2 = pol1;
          col1 = w.h * DH; row1 = w.krow + t * BKV; pol1 = pol;
        }
      }
      if (row2 >= 0) load(&tmV, col2, row2, pol2);
      if (row1 >= 0) load(&tmV, col1, row1, pol1);
    } else if (warp == 1) {
      // ------------------------------------------------------------------ MMA issuer
      const uint32_t idesc_s = ptx::idesc_bf16(BQ, BKV), idesc_o = ptx::idesc_bf16_b_mn(BQ, DH);
      const uint64_t qd = ptx::smem_desc_sw128(sQ);
      uint32_t src = sRing, full = bar(B_FULL), par = 0;
      int slot = 0;
      auto next = [&]() {
        src += TILE_BYTES; full += 8u;
        if (++slot == RING) { slot = 0; src = sRing; full = bar(B_FULL); par ^= 1u; }
      };
      int sb = 0, pb = 0;           // score buffer of the next S, of the next PV
      uint32_t ppar = 0, qpar = 0, opar = 1, pv = 0;
      auto scores = [&](bool last) {
        const bool ok = ptx::mbar_wait_or_abort(full, par, &abort_flag, status, DEV_TIMEOUT_MMA);
        ptx::tc_fence_after_sync();
        const uint64_t kd = ptx::smem_desc_sw128(src);
        if (ptx::elect_one() && ok) {
#pragma unroll
          for (int k = 0; k < DH / 16; ++k) {
            const uint32_t off = (k >> 2) * (HALF_BYTES >> 4) + 2u * (k & 3);
            ptx::mma_bf16_ss(tS + sb * BKV, qd + off, kd + off, idesc_s, k ? 1u : 0u);
          }
          ptx::mma_commit(full + 8u * RING);
          ptx::mma_commit(bar(B_SFULL + sb));
          if (last) ptx::mma_commit(bar(B_QFREE));
        }
        next();
        if (++sb == NS) sb = 0;
      };
      enum { TILE = 1, FIRST = 2, LAST = 4 };
      auto output = [&](int flags) {
        bool ok = ptx::mbar_wait_or_abort(full, par, &abort_flag, status, DEV_TIMEOUT_MMA);
        if (flags & FIRST) {          // the item before has been read out of O
          ok = ptx::mbar_wait_or_abort(bar(B_OFREE), opar, &abort_flag, status, DEV_TIMEOUT_MMA) && ok;
          opar ^= 1u;
        }
        ok = ptx::mbar_wait_or_abort(bar(B_PFULL + pb), ppar, &abort_flag, status, DEV_TIMEOUT_MMA) && ok;
        ptx::tc_fence_after_sync();
        const uint64_t vd = ptx::smem_desc_sw128_mn(src, HALF_BYTES);
        const uint32_t add = (flags & FIRST) ? 0u : 1u;
        if (ptx::elect_one() && ok) {
#pragma unroll
          for (int k = 0; k < BKV / 16; ++k)   // 16 keys per instruction: 8 columns of P, two 8-row groups of the V tile
            ptx::mma_bf16_ts(tO, tS + pb * BKV + k * 8, vd + k * (2048u >> 4), idesc_o, k ? 1u : add);
          ptx::mma_commit(full + 8u * RING);
          ptx::mma_commit(bar(B_PV) + 8u * pv);
          if (flags & LAST) ptx::mma_commit(bar(B_OFULL));
        }
        next();
        pv ^= 1u;
        if (++pb == NS) { pb = 0; ppar ^= 1u; }
      };
      int f1 = 0, f2 = 0;             // the last tile and the one before, whose second product is still to come
      for (int i = blockIdx.x; i < p.n_items; i += gridDim.x) {
        const int n_tiles = item_at(i).n_tiles;
        if (n_tiles == 0) continue;
        ptx::mbar_wait_or_abort(bar(B_QFULL), qpar, &abort_flag, status, DEV_TIMEOUT_MMA);
        qpar ^= 1u;
        for (int t = 0; t < n_tiles; ++t) {
          scores(t == n_tiles - 1);
          if (f2) output(f2);
          f2 = f1;
          f1 = TILE | (t == 0 ? FIRST : 0) | (t == n_tiles - 1 ? LAST : 0);
        }
      }
      if (f2) output(f2);
      if (f1) output(f1);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
    // ------------------------------------------------------------------ softmax and output
    const int g = (warp >> 2) - 1, q = warp & 3;
    const int row = q * 32 + lane;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const uint32_t tOr = tO + lane_base;
    const uint32_t mine = bar(B_MREF + g * 4 + q), theirs = bar(B_MREF + (g ^ 1) * 4 + q);
    const uint32_t stage = sRing + RING * TILE_BYTES + (warp - 4) * STAGE_BYTES;
    const float c = p.scale_log2;
    bool ok = true;
    int T0 = 0;                       // key tiles before this item, over all items of the CTA: they fix group and buffer
    uint32_t ipar = 0;
    for (int i = blockIdx.x; i < p.n_items && ok; i += gridDim.x) {
      const Item w = item_at(i);
      if (w.n_tiles == 0) continue;
      const bool rows = w.q0 + q * 32 < w.n_rows;            // this warp has rows (warp-uniform)
      float m_ref = -INFINITY;
      float2 l = {0.f, 0.f}, sum = {0.f, 0.f};               // row sums of two tiles ago; sums of this group's last tile ...
      float fac = 1.f;                                       // ... and the factor its reference maximum put on what came before
      for (int t = (g ^ T0) & 1; t < w.n_tiles && ok; t += 2) {
        const int T = T0 + t, T3 = T / NS, b = T - NS * T3;
        ok = ptx::mbar_wait_warp(bar(B_SFULL + b), (uint32_t)T3 & 1u);
        if (!ok) break;
        if (!rows) {
          if (T > 0) ok = ptx::mbar_wait_warp(theirs, (uint32_t)((T - 1) >> 1) & 1u);
          if (lane == 0) ptx::mbar_arrive(mine);
        } else {
          const uint32_t tSg = tS + lane_base + b * BKV;
          ptx::tc_fence_after_sync();
          uint32_t r[128];
#pragma unroll
          for (int i = 0; i < 4; ++i) ptx::tmem_ld_x32(tSg + 32 * i, r + 32 * i);
          ptx::tmem_ld_wait();
          const int n_valid = w.kv_len - t * BKV;              // this tile's columns that are keys
          if (n_valid < BKV) {                                 // ragged last tile only
#pragma unroll
            for (int i = 0; i < 128; ++i) if (i >= n_valid) r[i] = 0xff800000u;   // -inf
          }
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int i = 0; i < 128; i += 8) {
#pragma unroll
            for (int e = 0; e < 4; ++e) mx[e] = fmaxf(mx[e], fmaxf(__uint_as_float(r[i + e]), __uint_as_float(r[i + 4 + e])));
          }
          // waited for in an item's first tile too: the slot and the barrier stay one tile apart
          if (T > 0) ok = ptx::mbar_wait_warp(theirs, (uint32_t)((T - 1) >> 1) & 1u);
          float m_prev = -INFINITY;
          if (t > 0) {
            const float4 x = hand[g ^ 1][row];                 // sums of tile t - 3, then this group's own of tile t - 2
            m_prev = x.x;
            l.x = fmaf(fmaf(l.x, x.w, x.y), fac, sum.x);
            l.y = fmaf(fmaf(l.y, x.w, x.z), fac, sum.y);
          }
          const float m_new = fmaxf(m_prev, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * c);
          const bool rescale = m_new > m_prev + RESCALE_STEP;
          m_ref = rescale ? m_new : m_prev;
          hand[g][row] = make_float4(m_ref, sum.x, sum.y, fac);
          fac = rescale ? ptx::ex2(m_prev - m_ref) : 1.0f;     // first tile: 0
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(mine);
          // probabilities, packed two to a column; the first half goes out while the second is computed
          const float neg_m = -m_ref;
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            float rs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 64 * hf; i < 64 * hf + 64; i += 2) {
              const float p0 = ptx::ex2(fmaf(__uint_as_float(r[i]), c, neg_m));
              const float p1 = ptx::ex2(fmaf(__uint_as_float(r[i + 1]), c, neg_m));
              rs[(i >> 1) & 3] += p0 + p1;
              __nv_bfloat162 b2 = __floats2bfloat162_rn(p0, p1);
              r[i >> 1] = *reinterpret_cast<uint32_t *>(&b2);
            }
            ptx::tmem_st_x32(tSg + 32 * hf, r + 32 * hf);
            (hf ? sum.y : sum.x) = (rs[0] + rs[1]) + (rs[2] + rs[3]);
          }
          // tensor-memory loads and stores are warp-wide instructions: if any row of the warp moves its reference maximum, the
          // whole warp rewrites its rows of O (rows that keep theirs scale by 1), once the product of the tile before is
          // complete; this tile's follows the probabilities
          if (__any_sync(0xffffffffu, rescale && t > 0)) {
            ok = ptx::mbar_wait_warp(bar(B_PV) + 8u * ((T - 1) & 1), (uint32_t)((T - 1) >> 1) & 1u) && ok;
            ptx::tc_fence_after_sync();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              ptx::tmem_ld_x32(tOr + 32 * i, r + 64);
              ptx::tmem_ld_wait();
#pragma unroll
              for (int e = 64; e < 96; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * fac);
              ptx::tmem_st_x32(tOr + 32 * i, r + 64);
            }
          }
          ptx::tmem_st_wait();
          ptx::tc_fence_before_sync();
          __syncwarp();
        }
        if (lane == 0) ptx::mbar_arrive(bar(B_PFULL + b));
      }
      if (!ok) break;
      // the groups' last tiles meet: the row sums are carried on in the order of the tiles
      fin[ipar][g][row] = make_float4(sum.x, sum.y, fac, 0.f);
      fin_l[ipar][g][row] = l;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(bar(B_MEET + q));
      ok = ptx::mbar_wait_warp(bar(B_MEET + q), ipar);
      const int gl = (T0 + w.n_tiles - 1) & 1;                 // group of the last tile
      const float4 xa = fin[ipar][gl ^ 1][row], xb = fin[ipar][gl][row];
      l = fin_l[ipar][gl][row];
      const float inv = 1.0f / (fmaf(fmaf(l.x, xa.z, xa.x), xb.z, xb.x) + fmaf(fmaf(l.y, xa.z, xa.y), xb.z, xb.y));
      ok = ptx::mbar_wait_warp(bar(B_OFULL), ipar) && ok;
      ptx::tc_fence_after_sync();
      uint32_t o[64];
      if (rows) {
        ptx::tmem_ld_x32(tOr + g * 64, o);
        ptx::tmem_ld_x32(tOr + g * 64 + 32, o + 32);
        ptx::tmem_ld_wait();
        ptx::tc_fence_before_sync();
        __syncwarp();
      }
      if (lane == 0) ptx::mbar_arrive(bar(B_OFREE));
      if (rows && ok) {
        // a lane holds a row; through the staging a store instruction writes 64 contiguous bytes of each of eight rows
        // instead of 16 bytes of each of 32.  16-byte chunk j of row r lies at chunk j ^ (r >> 1 & 3): no bank conflicts
        bf16 *og = p.out + (int64_t)(w.row0 + w.q0 + q * 32) * p.out_stride + w.h * DH + g * 64;
        const int n_here = w.n_rows - (w.q0 + q * 32);
#pragma unroll
        for (int i = 0; i < 64; i += 32) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint4 pk;
            uint32_t *pw = reinterpret_cast<uint32_t *>(&pk);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const uint32_t *e = o + i + 8 * j + 2 * u;
              __nv_bfloat162 v = __floats2bfloat162_rn(__uint_as_float(e[0]) * inv, __uint_as_float(e[1]) * inv);
              pw[u] = *reinterpret_cast<uint32_t *>(&v);
            }
            ptx::st_shared_v4(stage + lane * 64 + ((j ^ (lane >> 1 & 3)) << 4), pk);
          }
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int r = u * 8 + (lane >> 2), j = lane & 3;
            const uint4 pk = ptx::ld_shared_v4(stage + r * 64 + ((j ^ (r >> 1 & 3)) << 4));
            if (r < n_here) *reinterpret_cast<uint4 *>(og + (int64_t)r * p.out_stride + i + 8 * j) = pk;
          }
          __syncwarp();
        }
      }
      T0 += w.n_tiles;
      ipar ^= 1u;
    }
    if (!ok) { fail(status, DEV_TIMEOUT_EPILOGUE); abort_flag = 1; }
  }

  // ---------------------------------------------------------------------- teardown
  __syncwarp();
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (abort_flag) {
    // A wait ran out: give copies still in flight time to land before the CTA's shared memory goes away.
    const uint64_t t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

bool attention_tc_supported(int dh, int64_t q_stride, int64_t kv_row_stride, int64_t out_stride) {
  return dh == DH && (q_stride % 8) == 0 && (kv_row_stride % 8) == 0 && (out_stride % 8) == 0;
}

cudaError_t launch_attention_tc(cudaStream_t st, const TmaDesc &tq, const TmaDesc &tk, const TmaDesc &tv,
                                const SeqMeta *meta, bf16 *out, int64_t out_stride, int kv_rows_per_seq,
                                int kv_row_base, int kv_packed, int n_slots, int max_q_rows, int H, int num_sms,
                                int32_t *status) {
  AttnTcParams p;
  p.out = out; p.meta = meta; p.use_single = 0; p.out_stride = out_stride;
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)DH);
  p.kv_rows_per_seq = kv_rows_per_seq; p.kv_row_base = kv_row_base; p.kv_packed = kv_packed; p.status = status;
  if (meta == nullptr) {
    // stand-alone call: one sequence, max_q_rows queries, n_slots carries the key count
    p.use_single = 1;
    p.single.seq = 0; p.single.row0 = 0; p.single.n_rows = max_q_rows; p.single.pos0 = 0;
    p.single.kv_len = n_slots; p.single.blk_start = 0; p.single.n_blk_rows = 0; p.single.block = 0;
    n_slots = 1;
  }
  if (max_q_rows <= 0 || n_slots <= 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(attention_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
  if (e != cudaSuccess) return e;
  p.H = H; p.n_qt = ceil_div(max_q_rows, BQ); p.n_items = p.n_qt * H * n_slots;
  dim3 grid(p.n_items < num_sms ? p.n_items : num_sms);
  return launch_kernel(attention_tc_kernel, grid, dim3(384), (size_t)SMEM_BYTES, st, tq.map, tk.map, tv.map, p);
}

}  // namespace l2pd
