// bf16 GEMM on the 5th-generation tensor cores with the weights on the M side:  acc[feature, row] = W[feature, K] * A[row, K]^T,
// the transpose of gemm_tcgen05.cu's accumulator.  An MMA's M is 128 or 256 whatever the problem has, its N any multiple of 16:
// weight matrices are multiples of 128 rows, a step's rows are any number, so here a step pays for its rows rounded up to 16 a
// tile where the other orientation pays for whole slabs of 128 or 256.
//
// The accumulator's lanes are output features.  An epilogue warp passes 32 features x 16 rows at a time through shared memory
// and then holds consecutive features of a row: rows leave in whole sectors to any address, so nothing here needs an output
// map, and a row of q, k or v goes to wherever the attention reads it.
//
// Epilogues
//   EPI_STORE     C (bf16)  = acc
//   EPI_QKV_ROPE  q, k rotated by the row's position (pairs (i, i + dh/2) of a head), v as it is; each part has a pointer of its
//                 own, k and v go to row kv_row[row] of theirs (the key/value store).  round_first: q and k are rounded to bf16 ahead
//                 of the rotation too, so that the result is that of the two kernels this replaces, bit for bit
//   EPI_RESIDUAL  X (fp32) += acc; K slices either add (atomics), store partial sums for a later sum in slice order, or are the
//                 CTAs of a cluster, which exchange their sums through shared memory: each adds a share of the rows, in slice order
//   EPI_SWIGLU    H (bf16)  = silu(acc_gate) * acc_up
// A rotary pair, or a gate and its up row, must meet in one warp: the weight tile's rows are interleaved in groups of eight
// (eight rows of the first half, eight of the second) by a 5-D tensor map over the matrix as it is.
//
// RMSNorm between two projections (p.n): the residual epilogue leaves bf16(x g) and the row's sum of squares per feature tile;
// the projection that follows multiplies its accumulators by 1 / sqrt(mean x^2 + eps).  The factor is common to a row, so it
// commutes with the product; bf16 has the same relative rounding with it or without.
//
// What bounds it: many rows, the tensor pipe and, beside it, shared memory, which the epilogue's staging takes some 6 % of; few
// rows, the weights' way from HBM and what lies between two projections (32 rows: 1.3 us from a kernel's end to the next one's
// release, 1.2 to its first MMA, the weights at 6.7 TB/s for gate/up, then 1.5 to 2 us of epilogue).  Stand-alone, rows on the M
// side -> here (us, back to back): 1029 rows QKV 91.4 -> 74.4, gate/up 167 -> 149, down 92.1 -> 83.7; 512 rows, which are whole
// slabs, QKV 48.1 -> 50.2, gate/up 89.6 -> 94.0.  Why 128-row weight tiles (96 or 64 where the plan finds them to share the
// last round better, gate/up of 32 rows: 3 % of a step): the MMA's M.  The cluster exchange replaced partial sums in global memory
// that the CTA arriving last added (5 us behind the last accumulator at 32 rows, 10 at 125).
//
// Warp roles (384 threads): 0 = TMA producer of the weight tiles (before the previous kernel has ended), 1 = MMA issuer (owns
// tensor memory), 2 = TMA producer of the activation tiles, 4-11 = epilogue (warp w: lanes 32 (w % 4) .., two warps a quarter
// take alternate chunks of 16 rows).  The loops of the issuing warps follow gemm_tcgen05.cu.
#include <math.h>

#include "common.cuh"
#include "gemm_device.cuh"
#include "ptx.cuh"

namespace l2pd {

using gemm_dev::silu_mul;

namespace {

constexpr int MMA_ROWS = 128;                     // weight rows an MMA takes from a CTA
constexpr int BK = 64;
constexpr int STAGES_MAX = 12;
constexpr int ACC = 256;                          // columns of an accumulator buffer; two of them
constexpr int CH = 16;                            // rows of a chunk
constexpr int ROW_F = 36;                         // floats between two rows of a chunk: eight rows' 16-byte pieces lie in different banks
constexpr int EPI_WARPS = 8;
constexpr int STAGING = EPI_WARPS * CH * ROW_F * 4;
constexpr int THREADS = 384;
constexpr int SMEM_MAX = 227 * 1024;
constexpr int EXCHANGE_ROWS = 128;                // rows of a tile whose K slices are exchanged: a share is at most 64, eight to an epilogue warp
constexpr int EXCHANGE_ROW_BYTES = MMA_ROWS * 4;

enum { RES_ADD = 0, RES_ATOMIC = 1, RES_PART = 2, RES_CLUSTER = 3 };

struct Params {
  int T, N, K, tile_t, n_stages, w_stage_bytes, x_stage_bytes, staging_off;
  int w_rows, w_tiles, t_tiles, k_splits, group_t;   // weight tiles of w_rows * CG rows
  int up_first;                                   // SwiGLU: the first of two interleaved groups is the up projection's
  bf16 *out; int64_t out_stride;                  // STORE, SWIGLU
  bf16 *q, *k, *v; int64_t q_stride, kv_stride;   // QKV
  const int32_t *kv_row, *row_pos; const float2 *cs;
  int hd, dh, natural, round_first;
  int res_mode;
  float *x, *part; int64_t part_stride;
  bf16 *n; const float *gain; float *ss_out;      // n != null: leave bf16(x gain) and the sums of squares
  const float *ss_in; int ss_n, ss_stride;        // > 0: scale rows by 1 / sqrt(sum / width + eps)
  float eps, inv_width;
  int32_t *status;
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&t);
}
__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory"); }

template <int EPI, int CG>
__global__ void __launch_bounds__(THREADS, 1)
gemm_wm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmX,
               const __grid_constant__ Params p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * STAGES_MAX + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float s_inv[EPI == EPI_RESIDUAL ? 1 : EPI_WARPS][EPI == EPI_RESIDUAL ? 1 : ACC / 2];   // a warp's chunks: at most 8 of 16 rows
  __shared__ int s_pos[EPI == EPI_QKV_ROPE ? EPI_WARPS : 1][EPI == EPI_QKV_ROPE ? ACC / 2 : 1], s_kv[EPI == EPI_QKV_ROPE ? EPI_WARPS : 1][EPI == EPI_QKV_ROPE ? ACC / 2 : 1];
  __shared__ float s_sq[EPI == EPI_RESIDUAL ? 4 : 1][EPI == EPI_RESIDUAL ? ACC : 1];

  const int warp = ptx::warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? ptx::cluster_ctarank() : 0u;
  const bool leader = rank == 0;
  const int group = CG == 2 ? blockIdx.x >> 1 : blockIdx.x;
  const int n_groups = CG == 2 ? gridDim.x >> 1 : gridDim.x;
  const bool clustered = EPI == EPI_RESIDUAL && CG == 1 && p.res_mode == RES_CLUSTER;   // one unit to a cluster, a CTA to a slice
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sW = base, sX = base + p.n_stages * p.w_stage_bytes;
  const uint32_t bar0 = ptx::smem_u32(bars);
  auto tfull = [&](int b) { return bar0 + 8u * (2 * STAGES_MAX + b); };
  auto tempty = [&](int b) { return bar0 + 8u * (2 * STAGES_MAX + 2 + b); };
  const uint32_t recv_bar = bar0 + 8u * (2 * STAGES_MAX + 4);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.n_stages; ++s) { ptx::mbar_init(bar0 + 8u * s, 1); ptx::mbar_init(bar0 + 8u * (STAGES_MAX + s), 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(tfull(b), 1); ptx::mbar_init(tempty(b), EPI_WARPS * CG); }
    ptx::mbar_init(recv_bar, 1);
    abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::fence_proxy_async();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tensormap(&tmW); ptx::prefetch_tensormap(&tmX);
    if (EPI == EPI_QKV_ROPE) ptx::prefetch_tensormap(&tmV);
  }
  if (warp == 1) {
    if (CG == 2) { ptx::tmem_alloc_pair(ptx::smem_u32(&tmem_slot), 2 * ACC); ptx::tmem_relinquish_pair(); }
    else { ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), 2 * ACC); ptx::tmem_relinquish(); }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (CG == 2) ptx::cluster_sync();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = tmem_slot;
  grid_dep_launch();

  const int num_units = p.w_tiles * p.t_tiles * p.k_splits;
  const int num_kb = (p.K + BK - 1) / BK, kb_per = (num_kb + p.k_splits - 1) / p.k_splits;
  // unit -> (weight tile, row tile, K slice): within a K slice, groups of group_t row tiles (activations sized to a share of
  // L2); inside a group the row tiles of one weight tile are adjacent, so that the weights come from memory once
  auto decode = [&](int u, int &wt, int &tt, int &ks) {
    const int per_slice = p.w_tiles * p.t_tiles;
    int r;
    if (clustered) { r = u / p.k_splits; ks = u - r * p.k_splits; }
    else { ks = u / per_slice; r = u - ks * per_slice; }
    const int per_group = p.group_t * p.w_tiles, g = r / per_group, w = r - g * per_group;
    const int gt = min(p.group_t, p.t_tiles - g * p.group_t);
    wt = w / gt;
    tt = g * p.group_t + (w - wt * gt);
  };
  int32_t *const status = p.status;
  const int n_stages = p.n_stages;
  auto produce = [&](uint32_t dst0, uint32_t stage_bytes, auto &&unit_begin, auto &&load) {
    uint32_t par = 1, full = bar0, dst = dst0;
    int stage = 0;
    for (int u = group; u < num_units; u += n_groups) {
      int wt, tt, ks;
      decode(u, wt, tt, ks);
      unit_begin(wt, tt);
      const int k_end = min(num_kb, (ks + 1) * kb_per) * BK;
      for (int k = ks * kb_per * BK; k < k_end; k += BK) {
        const bool ok = ptx::mbar_wait_or_abort(full + 8u * STAGES_MAX, par, &abort_flag, status, DEV_TIMEOUT_PRODUCER);
        if (ptx::elect_one() && ok) load(full, dst, k);
        full += 8u; dst += stage_bytes;
        if (++stage == n_stages) { stage = 0; full = bar0; dst = dst0; par ^= 1u; }
      }
    }
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ weight tiles: no kernel writes them
    const uint64_t pol = ptx::policy_evict_first();
    const uint32_t to_leader = CG == 2 ? ptx::mapa(bar0, 0) - bar0 : 0;
    const uint32_t tx = CG * (uint32_t)(p.w_stage_bytes + p.x_stage_bytes);
    int row = 0, c3 = 0, c4 = 0;
    bool plain = true;
    auto unit_begin = [&](int wt, int) {
      const int tile = wt * CG + (int)rank;
      row = tile * p.w_rows;
      if (EPI == EPI_SWIGLU) c3 = row >> 4;
      if (EPI == EPI_QKV_ROPE) {
        plain = row >= 2 * p.hd;
        c4 = row / p.dh;                          // a tile holds one head of 128 or two of 64
        if (plain) row -= 2 * p.hd;
      }
    };
    auto load = [&](uint32_t full, uint32_t dst, int k) {
      if (leader) ptx::mbar_arrive_expect_tx(full, tx);
      if (EPI == EPI_STORE || EPI == EPI_RESIDUAL || (EPI == EPI_QKV_ROPE && plain)) {
        const CUtensorMap *const m = EPI == EPI_QKV_ROPE ? &tmV : &tmW;
        if (CG == 2) ptx::tma_load_2d_pair_hint(dst, m, full + to_leader, k, row, pol);
        else ptx::tma_load_2d_hint(dst, m, full, k, row, pol);
      } else {
        if (CG == 2) ptx::tma_load_5d_pair_hint(dst, &tmW, full + to_leader, k, 0, 0, c3, c4, pol);
        else ptx::tma_load_5d_hint(dst, &tmW, full, k, 0, 0, c3, c4, pol);
      }
    };
    produce(sW, (uint32_t)p.w_stage_bytes, unit_begin, load);
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (leader CTA only when paired)
    if (leader) {
      const uint32_t idesc = ptx::idesc_bf16(MMA_ROWS * CG, (uint32_t)p.tile_t);
      const uint32_t w_step = (uint32_t)p.w_stage_bytes >> 4, x_step = (uint32_t)p.x_stage_bytes >> 4;
      const uint64_t w_desc0 = ptx::smem_desc_sw128(sW), x_desc0 = ptx::smem_desc_sw128(sX);
      uint32_t par = 0, full = bar0;
      uint64_t w_desc = w_desc0, x_desc = x_desc0;
      int lt = 0, stage = 0;
      for (int u = group; u < num_units; u += n_groups, ++lt) {
        int wt, tt, ks;
        decode(u, wt, tt, ks);
        const int ab = lt & 1;
        const uint32_t d_tmem = tmem_base + ab * ACC;
        bool ok = ptx::mbar_wait_or_abort(tempty(ab), ((uint32_t)(lt >> 1) & 1u) ^ 1u, &abort_flag, status, DEV_TIMEOUT_MMA);
        ptx::tc_fence_after_sync();
        uint32_t acc = 0;
        const int k1 = min(num_kb, (ks + 1) * kb_per);
        for (int i = ks * kb_per; i < k1; ++i) {
          ok = ptx::mbar_wait_or_abort(full, par, &abort_flag, status, DEV_TIMEOUT_MMA);
          ptx::tc_fence_after_sync();
          if (ptx::elect_one() && ok) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              if (CG == 2) ptx::mma_bf16_ss_pair(d_tmem, w_desc + 2u * k, x_desc + 2u * k, idesc, k ? 1u : acc);
              else ptx::mma_bf16_ss(d_tmem, w_desc + 2u * k, x_desc + 2u * k, idesc, k ? 1u : acc);
            }
            if (CG == 2) ptx::mma_commit_pair(full + 8u * STAGES_MAX, 3);
            else ptx::mma_commit(full + 8u * STAGES_MAX);
          }
          acc = 1;
          full += 8u; w_desc += w_step; x_desc += x_step;
          if (++stage == n_stages) { stage = 0; full = bar0; w_desc = w_desc0; x_desc = x_desc0; par ^= 1u; }
        }
        if (ptx::elect_one() && ok) {
          if (CG == 2) ptx::mma_commit_pair(tfull(ab), 3);
          else ptx::mma_commit(tfull(ab));
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ activation tiles
    const uint64_t pol = ptx::policy_evict_last();
    const uint32_t to_leader = CG == 2 ? ptx::mapa(bar0, 0) - bar0 : 0;
    grid_dep_wait();
    int row = 0;
    auto unit_begin = [&](int, int tt) { row = tt * p.tile_t + (CG == 2 ? (int)rank * (p.tile_t >> 1) : 0); };
    auto load = [&](uint32_t full, uint32_t dst, int k) {
      if (CG == 2) ptx::tma_load_2d_pair_hint(dst, &tmX, full + to_leader, k, row, pol);
      else ptx::tma_load_2d_hint(dst, &tmX, full, k, row, pol);
    };
    produce(sX, (uint32_t)p.x_stage_bytes, unit_begin, load);
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3, half = (warp - 4) >> 2, ew = warp - 4;
    const uint32_t stg = base + p.staging_off + (uint32_t)ew * (CH * ROW_F * 4);
    const int n_feat = EPI == EPI_SWIGLU ? 2 * p.N : p.N;   // rows of the weight matrix as tiled
    int lt = 0, row_tt = -1;
    grid_dep_wait();
    for (int u = group; u < num_units; u += n_groups, ++lt) {
      int wt, tt, ks;
      decode(u, wt, tt, ks);
      const int t0 = tt * p.tile_t, t_end = min(p.tile_t, p.T - t0);       // rows of this unit
      const int tile = wt * CG + (int)rank, f0 = tile * p.w_rows + quarter * 32;
      const bool feats = quarter * 32 < p.w_rows && f0 < n_feat;
      if (EPI != EPI_RESIDUAL && tt != row_tt) {
        // the rows' factors and places, 16 rows at a time; two lanes share a row's sums of squares
        for (int c = half; c * CH < t_end; c += 2) {
          const int t = c * CH + (lane & 15), at = (c >> 1) * CH + (lane & 15), row = t0 + (t < t_end ? t : 0);
          if (EPI == EPI_QKV_ROPE && lane < 16) {
            s_pos[ew][at] = p.row_pos[row];
            s_kv[ew][at] = p.kv_row ? p.kv_row[row] : row;
          }
          if (p.ss_n > 0) {
            float a = 0.f;
            const float *ss = p.ss_in + row;
#pragma unroll 16
            for (int i = lane >> 4; i < p.ss_n; i += 2) a += ss[(int64_t)i * p.ss_stride];
            a += __shfl_xor_sync(0xffffffffu, a, 16);
            if (lane < 16) s_inv[ew][at] = 1.0f / sqrtf(a * p.inv_width + p.eps);
          }
        }
        __syncwarp();
        row_tt = tt;
      }
      const bool rope = EPI == EPI_QKV_ROPE && f0 < 2 * p.hd;               // (warp-uniform)
      const int head0 = EPI == EPI_QKV_ROPE ? f0 - f0 % p.dh : 0, dim0 = EPI == EPI_QKV_ROPE ? (f0 - head0) / 2 + (lane >> 3) * 4 : 0;
      // what a chunk reads from memory is asked for one chunk ahead: residual rows, angles
      float4 ahead[4];
      auto ask = [&](int c) {
        if (EPI == EPI_RESIDUAL && p.res_mode == RES_ADD) {
          const int f = f0 + (lane & 7) * 4;
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            const int t = c * CH + it * 4 + (lane >> 3);
            ahead[it] = feats && f < p.N && t < t_end ? *reinterpret_cast<const float4 *>(p.x + (int64_t)(t0 + t) * p.N + f) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
        if (rope) {
#pragma unroll
          for (int it = 0; it < 2; ++it) {
            const float4 *cs = reinterpret_cast<const float4 *>(p.cs + (int64_t)s_pos[ew][(c >> 1) * CH + it * 8 + (lane & 7)] * (p.dh >> 1) + dim0);
            ahead[2 * it] = __ldg(cs); ahead[2 * it + 1] = __ldg(cs + 1);
          }
        }
      };
      if (half * CH < t_end) ask(half);
      const int ab = lt & 1;
      const bool ok = ptx::mbar_wait_idle_or_abort(tfull(ab), (uint32_t)(lt >> 1) & 1u, 20, &abort_flag, status, DEV_TIMEOUT_EPILOGUE);
      ptx::tc_fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + ab * ACC;
      if (clustered) {
        // this slice's sums, [row][feature] over the ring, which is idle: the unit is the CTA's only one
        if (ok && feats) {
          for (int c = half; c * CH < t_end; c += 2) {
            uint32_t v[CH];
            ptx::tmem_ld_x16(taddr + c * CH, v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < CH; ++i)
              asm volatile("st.shared.b32 [%0], %1;" ::"r"(base + (uint32_t)((c * CH + i) * MMA_ROWS + quarter * 32 + lane) * 4u), "r"(v[i]) : "memory");
          }
        }
        ptx::fence_proxy_async();
        break;
      }
      if (ok && feats) {
        // a chunk's columns are asked for as soon as the ones before have left the registers for shared memory; nothing reads the
        // registers between a load and its wait (they are undefined until then)
        uint32_t v[CH];
        if (half * CH < t_end) ptx::tmem_ld_x16(taddr + half * CH, v);
        for (int c = half; c * CH < t_end; c += 2) {
          ptx::tmem_ld_wait();
          const bool more = (c + 2) * CH < t_end;
          float4 now[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) now[i] = ahead[i];
          if (more) ask(c + 2);
#pragma unroll
          for (int i = 0; i < CH; ++i)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(stg + (uint32_t)(i * ROW_F + lane) * 4u), "r"(v[i]) : "memory");
          if (more) ptx::tmem_ld_x16(taddr + (c + 2) * CH, v);
          __syncwarp();
          const int tc = c * CH, n_rows = t_end - tc;       // rows of this chunk (>= 16: all)
          if (EPI == EPI_RESIDUAL) {
            const int f = f0 + (lane & 7) * 4;
            const bool on = f < p.N;
            float4 g4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p.n && on) g4 = __ldg(reinterpret_cast<const float4 *>(p.gain + f));
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const int r = it * 4 + (lane >> 3);
              const bool live = on && r < n_rows;
              float4 a = lds4(stg + (uint32_t)(r * ROW_F + (lane & 7) * 4) * 4u);
              const int64_t at = (int64_t)(t0 + tc + r) * p.N + f;
              if (p.res_mode == RES_ADD) {
                a.x += now[it].x; a.y += now[it].y; a.z += now[it].z; a.w += now[it].w;
                if (live) *reinterpret_cast<float4 *>(p.x + at) = a;
                if (p.n) {
                  if (live) *reinterpret_cast<uint2 *>(p.n + at) = make_uint2(pack2(a.x * g4.x, a.y * g4.y), pack2(a.z * g4.z, a.w * g4.w));
                  float s = live ? (a.x * a.x + a.y * a.y) + (a.z * a.z + a.w * a.w) : 0.f;
#pragma unroll
                  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                  if ((lane & 7) == 0) s_sq[quarter][tc + r] = s;
                }
              } else if (live) {
                if (p.res_mode == RES_ATOMIC) ptx::red_add_v4(p.x + at, a.x, a.y, a.z, a.w);
                else *reinterpret_cast<float4 *>(p.part + (int64_t)ks * p.part_stride + at) = a;
              }
            }
          } else if (EPI == EPI_STORE || (EPI == EPI_QKV_ROPE && !rope)) {
            // four lanes a row, eight features each
            const int f = f0 + (lane >> 3) * 8;
#pragma unroll
            for (int it = 0; it < 2; ++it) {
              const int r = it * 8 + (lane & 7);
              const uint32_t at = stg + (uint32_t)(r * ROW_F + (lane >> 3) * 8) * 4u;
              const float4 a = lds4(at), b = lds4(at + 16u);
              if (r < n_rows && f < p.N) {
                const int i = (c >> 1) * CH + r;
                const float s = p.ss_n > 0 ? s_inv[ew][i] : 1.0f;
                bf16 *const dst = EPI == EPI_STORE ? p.out + (int64_t)(t0 + tc + r) * p.out_stride + f
                                                   : p.v + (int64_t)s_kv[ew][EPI == EPI_QKV_ROPE ? i : 0] * p.kv_stride + (f - 2 * p.hd);
                *reinterpret_cast<uint4 *>(dst) = make_uint4(pack2(a.x * s, a.y * s), pack2(a.z * s, a.w * s), pack2(b.x * s, b.y * s), pack2(b.z * s, b.w * s));
              }
            }
          } else {
            // interleaved halves: lanes of a row take four features of the first and the same four of the second
            const int j = lane >> 3, off = (j >> 1) * 16 + (j & 1) * 4;
#pragma unroll
            for (int it = 0; it < 2; ++it) {
              const int r = it * 8 + (lane & 7), i = (c >> 1) * CH + r;
              const uint32_t at = stg + (uint32_t)(r * ROW_F + off) * 4u;
              float4 a = lds4(at), b = lds4(at + 32u);
              if (r < n_rows) {
                const float s = p.ss_n > 0 ? s_inv[ew][i] : 1.0f;
                const int t = t0 + tc + r;
                if (EPI == EPI_SWIGLU) {
                  const int f = (f0 >> 1) + j * 4;
                  if (p.up_first) { const float4 w = a; a = b; b = w; }
                  if (f < p.N)
                    *reinterpret_cast<uint2 *>(p.out + (int64_t)t * p.out_stride + f) =
                        make_uint2(pack2(silu_mul(a.x * s, b.x * s), silu_mul(a.y * s, b.y * s)), pack2(silu_mul(a.z * s, b.z * s), silu_mul(a.w * s, b.w * s)));
                } else {
                  // dimensions dim0 .. dim0 + 3 and their partners
                  const float4 c01 = now[2 * it], c23 = now[2 * it + 1];
                  float xa[4] = {a.x * s, a.y * s, a.z * s, a.w * s}, xb[4] = {b.x * s, b.y * s, b.z * s, b.w * s};
                  if (p.round_first) {   // as a projection that stores bf16 and a rotation kernel behind it
#pragma unroll
                    for (int e = 0; e < 4; ++e) { xa[e] = __bfloat162float(__float2bfloat16_rn(xa[e])); xb[e] = __bfloat162float(__float2bfloat16_rn(xb[e])); }
                  }
                  const float co[4] = {c01.x, c01.z, c23.x, c23.z}, si[4] = {c01.y, c01.w, c23.y, c23.w};
                  float ya[4], yb[4];
#pragma unroll
                  for (int e = 0; e < 4; ++e) { ya[e] = xa[e] * co[e] - xb[e] * si[e]; yb[e] = xb[e] * co[e] + xa[e] * si[e]; }
                  bf16 *const dst = f0 < p.hd ? p.q + (int64_t)t * p.q_stride + head0 : p.k + (int64_t)s_kv[ew][i] * p.kv_stride + (head0 - p.hd);
                  if (p.natural) {
                    *reinterpret_cast<uint2 *>(dst + dim0) = make_uint2(pack2(ya[0], ya[1]), pack2(ya[2], ya[3]));
                    *reinterpret_cast<uint2 *>(dst + (p.dh >> 1) + dim0) = make_uint2(pack2(yb[0], yb[1]), pack2(yb[2], yb[3]));
                  } else {   // pairs adjacent
                    *reinterpret_cast<uint4 *>(dst + 2 * dim0) = make_uint4(pack2(ya[0], yb[0]), pack2(ya[1], yb[1]), pack2(ya[2], yb[2]), pack2(ya[3], yb[3]));
                  }
                }
              }
            }
          }
          __syncwarp();
        }
      }
      ptx::tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (CG == 2) ptx::mbar_arrive_cluster(ptx::mapa(tempty(ab), 0));
        else ptx::mbar_arrive(tempty(ab));
      }
      if (EPI == EPI_RESIDUAL && p.n) {
        // sums of squares of this tile's features, quarter after quarter
        epi_barrier();
        const int t = threadIdx.x - 128;
        if (t < t_end && tile * p.w_rows < p.N) {
          const int nq = (min(p.w_rows, p.N - tile * p.w_rows) + 31) / 32;
          float s = s_sq[0][t];
          for (int i = 1; i < nq; ++i) s += s_sq[i][t];
          p.ss_out[(int64_t)tile * p.ss_stride + t0 + t] = s;
        }
        epi_barrier();
      }
    }
  }

  if (clustered) {
    // The slices of a tile.  CTA j of the cluster takes rows j * share ..: once all of the cluster's accumulators are complete every
    // CTA copies its sums of those rows into j's shared memory, [slice][row][feature] behind the rows of its own, and j adds them
    // to X in the order of the slices.
    int wt, tt, ks;
    decode(group, wt, tt, ks);
    const int t0 = tt * p.tile_t, t_end = min(p.tile_t, p.T - t0), share = (t_end + p.k_splits - 1) / p.k_splits;
    const int r0 = ks * share, mine = max(0, min(t_end - r0, share)), f = wt * MMA_ROWS + lane * 4;
    const uint32_t recv = base + EXCHANGE_ROWS * EXCHANGE_ROW_BYTES;
    const bool on = f < p.N;
    constexpr int AHEAD = EXCHANGE_ROWS / 2 / EPI_WARPS;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 g4 = warp >= 4 && on && p.n ? __ldg(reinterpret_cast<const float4 *>(p.gain + f)) : zero;
    float4 xv[AHEAD];
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) {
      const int r = (warp - 4) + i * EPI_WARPS;
      xv[i] = warp >= 4 && on && r < mine ? *reinterpret_cast<const float4 *>(p.x + (int64_t)(t0 + r0 + r) * p.N + f) : zero;
    }
    if (threadIdx.x == 128) ptx::mbar_arrive_expect_tx(recv_bar, (uint32_t)(p.k_splits * mine) * EXCHANGE_ROW_BYTES);
    __syncwarp();
    ptx::tc_fence_before_sync();
    ptx::cluster_sync();
    bool ok = true;
    if (warp >= 4) {
      if (warp == 4 && lane < p.k_splits && !abort_flag) {
        const int rows = max(0, min(t_end - lane * share, share));
        if (rows > 0)
          ptx::bulk_copy_to_cta(ptx::mapa(recv + (uint32_t)(ks * rows) * EXCHANGE_ROW_BYTES, (uint32_t)lane), base + (uint32_t)(lane * share) * EXCHANGE_ROW_BYTES,
                                (uint32_t)rows * EXCHANGE_ROW_BYTES, ptx::mapa(recv_bar, (uint32_t)lane));
      }
      __syncwarp();
      ok = ptx::mbar_wait_idle_or_abort(recv_bar, 0, 20, &abort_flag, status, DEV_TIMEOUT_EPILOGUE);
#pragma unroll
      for (int i = 0; i < AHEAD; ++i) {
        const int r = (warp - 4) + i * EPI_WARPS;
        if (r < mine && ok) {
          float4 a = xv[i];
          for (int s = 0; s < p.k_splits; ++s) {
            const float4 b = lds4(recv + (uint32_t)((s * mine + r) * MMA_ROWS + lane * 4) * 4u);
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
          }
          const int64_t at = (int64_t)(t0 + r0 + r) * p.N + f;
          if (on) *reinterpret_cast<float4 *>(p.x + at) = a;
          if (p.n) {
            if (on) *reinterpret_cast<uint2 *>(p.n + at) = make_uint2(pack2(a.x * g4.x, a.y * g4.y), pack2(a.z * g4.z, a.w * g4.w));
            float q2 = on ? (a.x * a.x + a.y * a.y) + (a.z * a.z + a.w * a.w) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) q2 += __shfl_xor_sync(0xffffffffu, q2, o);
            if (lane == 0) p.ss_out[(int64_t)wt * p.ss_stride + t0 + r0 + r] = q2;
          }
        }
      }
    }
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
  if (CG == 2 || clustered) ptx::cluster_sync();   // the others' copies out of or into this CTA's shared memory are complete
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    if (CG == 2) ptx::tmem_dealloc_pair(tmem_base, 2 * ACC);
    else ptx::tmem_dealloc(tmem_base, 2 * ACC);
  }
}

// what the kernel declares itself: barriers, factors, places (QKV), sums of squares
constexpr int static_smem(int epi) { return epi == EPI_QKV_ROPE ? 13 * 1024 : 5 * 1024; }

template <int EPI, int CG>
cudaError_t launch(cudaStream_t st, const WmArgs &g, const Params &p, int grid, size_t smem) {
  const unsigned cluster = CG == 2 ? 2 : EPI == EPI_RESIDUAL && p.res_mode == RES_CLUSTER ? (unsigned)p.k_splits : 1;
  auto kernel = gemm_wm_kernel<EPI, CG>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX - static_smem(EPI));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (cluster > 1) { at[n].id = cudaLaunchAttributeClusterDimension; at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1; ++n; }
  if (pdl_enabled()) { at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[n].val.programmaticStreamSerializationAllowed = 1; ++n; }
  cfg.attrs = at;
  cfg.numAttrs = n;
  const CUtensorMap &wv = g.wv ? g.wv->map : g.w->map;
  return cudaLaunchKernelEx(&cfg, kernel, g.w->map, wv, g.x->map, p);
}

}  // namespace

// The exchange takes a cluster of single CTAs with one unit each; its shares and slices have room for EXCHANGE_ROWS rows.
bool wm_slices_in_cluster(const WmPlan &pl, int T, int N, int num_sms) {
  return pl.cta_group == 1 && pl.w_rows == MMA_ROWS && (pl.k_splits == 2 || pl.k_splits == 4) && pl.tile_t <= EXCHANGE_ROWS &&
         ceil_div(N, pl.w_rows) * ceil_div(T, pl.tile_t) * pl.k_splits <= num_sms;
}

// Modelled cycles, in the terms of plan_cost (gemm_tcgen05.cu): a k-block takes the largest of the tensor pipe's 2 * tile_t cycles,
// its issuer's 250, the bytes a CTA takes in at 95 a cycle, and the CTAs' weights out of memory at 3450 a cycle of the whole chip
// (read once for all row tiles); a share of the bytes' time on top; drains overlap the next unit.  The units go round in order,
// so in the last round fewer CTAs share the memory.
// A step plans its four projections ahead of its first launch, which nothing hides: a row tile that several counts of tiles come
// to is looked at once, and a tile whose k-blocks alone take longer than the best so far not at all (the plans are the same; 1024
// rows: 95 -> 7 us, 306 rows 25 -> 7).
WmPlan plan_gemm_wm(int epi, int T, int N, int K, int num_sms, int max_k_splits, bool in_cluster, double limit) {
  WmPlan best{0, 0, 1, MMA_ROWS, limit};
  const int rows = epi == EPI_SWIGLU ? 2 * N : N;
  const int max_ks = epi == EPI_RESIDUAL ? (max_k_splits < 4 ? max_k_splits : 4) : 1;
  const double traffic = T >= 4096 ? 0.45 : 0.15;
  const int k_blocks = ceil_div(K, BK);
  if (8000.0 + 20.0 * 16 + 250.0 * k_blocks / max_ks >= limit) return best;   // no tile is below this
  for (int cg = 1; cg <= 2; ++cg) {
    if (cg == 2 && num_sms < 2) continue;
    const int groups = num_sms / cg;
    for (int wr = MMA_ROWS; wr >= (epi == EPI_QKV_ROPE ? MMA_ROWS : 64); wr -= 32) {
      const int w_tiles = ceil_div(rows, wr * cg);
      for (int nt = ceil_div(T, 256), last = 0;; ++nt) {
        const int tt = (ceil_div(T, nt) + 15) / 16 * 16;
        if (nt > ceil_div(T, 256) && (tt < 32 || nt > ceil_div(T, 256) + 64)) break;
        if (tt == last) continue;   // the same tiles again
        last = tt;
        const int t_tiles = ceil_div(T, tt);
        const double bytes = 128.0 * wr + 128.0 * tt / cg, pipe = 2.0 * tt * (cg == 1 ? 1.13 : 1.0);
        const double k_block = fmax(fmax(pipe, 250.0), bytes / 95.0) + traffic * bytes / 95.0, fixed = 8000.0 + 20.0 * tt;
        // no split of K takes less than all k-blocks spread evenly over the CTAs, nor than one unit
        if (k_block * k_blocks * fmax((double)w_tiles * t_tiles / groups, 1.0 / max_ks) + fixed >= best.cost) continue;
        for (int ks = 1; ks <= max_ks; ++ks) {
          if (ks > 1 && (k_blocks < 8 * ks || effective_k_splits(K, ks) != ks)) break;
          if (in_cluster && ks > 1 && !wm_slices_in_cluster(WmPlan{cg, tt, ks, wr, 0.0}, T, N, num_sms)) continue;
          const int kb = ceil_div(k_blocks, ks);
          auto unit = [&](int active) {
            return kb * fmax(k_block, 128.0 * wr * cg * active / t_tiles / 3450.0 + traffic * bytes / 95.0) + 400.0;
          };
          const int units = w_tiles * t_tiles * ks, q = units / groups, r = units % groups;
          double c = (q ? q * unit(groups) : 0.0) + (r ? unit(r) : 0.0) + fixed;
          if (ks > 1 && in_cluster) c += 2000.0;
          else if (ks > 1) c += 8.0 * ks * (double)T * N / 2000.0 * (T > 128 ? 1.0 : 0.25);
          if (c < best.cost - 1e-9) best = WmPlan{cg, tt, ks, wr, c};
        }
      }
    }
  }
  return best;
}

// The rotating epilogue takes 82 cycles a row of the tile (measured, d = 512, cycles a unit: 32 rows 3440, 96 8500, 176 14600), where
// the plan reckons with 20, and hides only behind the next unit's k-blocks.  With few of them (a narrow model) it is what the
// projection takes: 4096 rows at d = 512 16 us on the other side, 27 here; 2048 at d = 1024 19 and 29; 1029 at d = 4096 110 and 87.
// A decision between the sides that knows of it, four layers, rows in one to sixteen sequences of 257 to 8192, against one that does
// not: d = 512, heads of 64, 770 rows 238 -> 218 us, 4096 rows 433 -> 418; d = 1024, 4096 rows 735 -> 707, heads of 128 with a cache
// 623 -> 594; d = 4096 as before.  (The tiles stay those of the plan.)
double wm_exposed_drain(int epi, const WmPlan &pl, int T, int N, int K, int num_sms) {
  if (epi != EPI_QKV_ROPE) return 0.0;
  const int rounds = ceil_div(ceil_div(N, pl.w_rows * pl.cta_group) * ceil_div(T, pl.tile_t), num_sms / pl.cta_group);
  const double drain = 82.0 * pl.tile_t, bytes = 128.0 * pl.w_rows + 128.0 * pl.tile_t / pl.cta_group;
  const double loop = ceil_div(K, BK) * (fmax(fmax(2.0 * pl.tile_t * (pl.cta_group == 1 ? 1.13 : 1.0), 250.0), bytes / 95.0) + (T >= 4096 ? 0.45 : 0.15) * bytes / 95.0) + 400.0;
  return (rounds - 1) * fmax(0.0, drain - loop) + drain - 20.0 * pl.tile_t;
}

l2pd_status make_tma_halves(TmaDesc *out, const void *ptr, int64_t K, int64_t half_bytes, int64_t groups, int box_groups, int64_t outer,
                            int64_t outer_bytes, int box_outer) {
  TmaEncodeFn fn = tma_encode_fn();
  if (!fn) return L2PD_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (K % 8) || half_bytes <= 0 || (half_bytes % 16) || half_bytes >= (1ll << 40) || (outer_bytes % 16) || groups < 1)
    return L2PD_ERR_SHAPE;
  cuuint64_t dims[5] = {(cuuint64_t)K, 8, 2, (cuuint64_t)groups, (cuuint64_t)outer};
  cuuint64_t strides[4] = {(cuuint64_t)K * 2, (cuuint64_t)half_bytes, (cuuint64_t)K * 16, (cuuint64_t)outer_bytes};
  cuuint32_t box[5] = {(cuuint32_t)BK, 8, 2, (cuuint32_t)box_groups, (cuuint32_t)box_outer};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = fn(&out->map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? L2PD_OK : L2PD_ERR_CUDA;
}

l2pd_status make_tma_gate_up(TmaDesc *out, const void *gate, const void *up, int64_t F, int64_t K, int box_rows, int *up_first) {
  const intptr_t d = reinterpret_cast<intptr_t>(up) - reinterpret_cast<intptr_t>(gate);
  *up_first = d < 0;
  return make_tma_halves(out, d < 0 ? up : gate, K, d < 0 ? -d : d, F / 8, box_rows / 16, 1, F * K * 2, 1);
}

cudaError_t launch_gemm_wm(cudaStream_t st, const WmArgs &g, int num_sms) {
  const int cg = g.plan.cta_group == 2 ? 2 : 1, tt = g.plan.tile_t, ks = g.plan.k_splits > 1 ? g.plan.k_splits : 1;
  if (tt < 16 || tt > 256 || (tt % 16) || g.T < 1 || (ks > 1 && g.epi != EPI_RESIDUAL) || effective_k_splits(g.K, ks) != ks) return cudaErrorInvalidValue;
  Params p = {};
  p.T = g.T; p.N = g.N; p.K = g.K; p.tile_t = tt;
  p.w_rows = g.plan.w_rows;
  if (p.w_rows < 32 || p.w_rows > MMA_ROWS || (p.w_rows % 32) || (p.w_rows != MMA_ROWS && g.epi == EPI_QKV_ROPE)) return cudaErrorInvalidValue;
  // fewer weight rows than the MMA takes: it reads on into the next stages and, from the last ones, into the activation ring behind
  // (16 KB at least from the last weight stage on), into accumulator lanes that nobody reads
  p.w_stage_bytes = p.w_rows * BK * 2;
  p.x_stage_bytes = tt / cg * 128;
  p.n_stages = (SMEM_MAX - static_smem(g.epi) - 1024 - STAGING) / (p.w_stage_bytes + p.x_stage_bytes);
  if (p.n_stages > STAGES_MAX) p.n_stages = STAGES_MAX;
  if (p.n_stages < 2 || p.w_stage_bytes + p.n_stages * p.x_stage_bytes < MMA_ROWS * BK * 2) return cudaErrorInvalidValue;
  p.staging_off = p.n_stages * (p.w_stage_bytes + p.x_stage_bytes);
  p.w_tiles = ceil_div(g.epi == EPI_SWIGLU ? 2 * g.N : g.N, p.w_rows * cg);
  p.t_tiles = ceil_div(g.T, tt);
  p.k_splits = ks;
  {
    int gt = (int)(46.0e6 / ((double)tt * ((double)g.K / ks) * 2.0));   // as gemm_tcgen05.cu's group_m
    p.group_t = gt < 1 ? 1 : gt > p.t_tiles ? p.t_tiles : gt;
  }
  p.up_first = g.up_first;
  p.out = g.out; p.out_stride = g.out_stride;
  p.q = g.q; p.k = g.k; p.v = g.v; p.q_stride = g.q_stride; p.kv_stride = g.kv_stride; p.kv_row = g.kv_row; p.row_pos = g.row_pos;
  p.cs = g.cs_table; p.hd = g.hd; p.dh = g.dh; p.natural = g.natural; p.round_first = g.round_first;
  p.x = g.xres; p.part = g.part; p.part_stride = g.part_stride;
  p.n = g.n; p.gain = g.gain; p.ss_out = g.ss_out; p.ss_in = g.ss_in; p.ss_n = g.ss_in ? g.ss_n : 0; p.ss_stride = g.ss_stride;
  p.eps = g.eps; p.inv_width = g.width > 0 ? 1.0f / (float)g.width : 0.f;
  p.status = g.status;
  p.res_mode = ks == 1 ? RES_ADD : g.in_cluster ? RES_CLUSTER : g.part ? RES_PART : RES_ATOMIC;
  if (p.res_mode == RES_CLUSTER && (!wm_slices_in_cluster(g.plan, g.T, g.N, num_sms) || p.staging_off < 2 * EXCHANGE_ROWS * EXCHANGE_ROW_BYTES)) return cudaErrorInvalidValue;
  if (g.epi == EPI_RESIDUAL && g.n && (!g.gain || !g.ss_out || (ks > 1 && !g.in_cluster))) return cudaErrorInvalidValue;
  if (g.epi == EPI_QKV_ROPE && ((g.dh != 64 && g.dh != 128) || g.N != 3 * g.hd || !g.wv || !g.cs_table || !g.row_pos)) return cudaErrorInvalidValue;
  const int units = p.w_tiles * p.t_tiles * ks, groups = num_sms / cg;
  const int grid = cg * (units < groups ? units : groups);
  const size_t smem = (size_t)p.staging_off + STAGING + 1024;
#define L2PD_WM(E) case E: return cg == 2 ? launch<E, 2>(st, g, p, grid, smem) : launch<E, 1>(st, g, p, grid, smem);
  switch (g.epi) {
    L2PD_WM(EPI_STORE) L2PD_WM(EPI_QKV_ROPE) L2PD_WM(EPI_RESIDUAL) L2PD_WM(EPI_SWIGLU)
    default: return cudaErrorInvalidValue;
  }
#undef L2PD_WM
}

}  // namespace l2pd
