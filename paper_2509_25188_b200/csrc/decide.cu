// Decision kernel: everything of a denoising step that follows M(X).
//   * merges the LM head's per-vocabulary-tile (max, sum-exp, argmax) records into the greedy
//     prediction (Eq. 3) and its confidence (Eq. 4);
//   * runs the filter f_theta on the block's s confidences, z = W2 relu(W1 c + b1) + b2,
//     p = sigmoid(z) (Section 3.2);
//   * Algorithm 2: every masked position with p > tau (strict) is committed in place; if none
//     passes, the masked position with the highest confidence is committed so the loop advances;
//     (comparison policies of Section 3.1 replace the test: confidence above a fixed threshold, or
//     Extremely Greedy Parallel, prediction == reference token; an EGP step in which nothing
//     matches commits the reference token at the most confident masked position);
//   * EoTP (Section 3.3): the earliest committed [EoT] cuts the sequence; later positions leave
//     the mask set and read as [EoT];
//   * block advance / stop (Algorithm 3: no block after one that holds [EoT]).
// One thread block per sequence taking part in the step.  What took longest was the merge (988 records of 32 rows in a step of
// the 8B shape, 380 KB): a warp to a row read a 32-byte sector for each 4-byte value it wanted, eight times the bytes through one
// SM; with lanes along the rows the kernel takes 16.0 us where it took 36.6.  Besides, it is bound by its chain of latencies: the
// two-layer filter's weights come to shared memory before the wait for the LM head, the tile records and the sequence's
// description leave together, its state follows at once.  The summary and the device status go straight to pinned host memory,
// so that nothing is left to copy behind the step's last kernel.  With the descriptions of a step's sequences as an argument of
// its first kernel, a step of 306 rows at d = 512: 212 -> 202 us.
#include "common.cuh"

namespace l2pd {

namespace {

constexpr int MAX_S = 64;

// folds the record (om, os, oi) into (mx, sum, ix); the lowest id on ties
__device__ __forceinline__ void fold(float &mx, float &sum, int &ix, float om, float os, int oi) {
  const float nm = fmaxf(mx, om);
  sum = (mx == -INFINITY ? 0.f : sum * expf(mx - nm)) + (om == -INFINITY ? 0.f : os * expf(om - nm));
  ix = (om > mx || (om == mx && oi < ix)) ? oi : ix;
  mx = nm;
}

__global__ void __launch_bounds__(1024) decide_kernel(const __grid_constant__ DecideArgs a) {
  extern __shared__ float recs[];                                // records of the merge: max, sum exp, argmax
  __shared__ float s_w[2][MAX_S * (MAX_S + 1)], s_b[2][MAX_S];   // the two-layer filter, rows of s + 1
  __shared__ float s_conf[MAX_S];
  __shared__ int s_pred[MAX_S];
  __shared__ float s_c[MAX_S];
  __shared__ float s_h[MAX_S];
  __shared__ float s_t[MAX_S];
  __shared__ float s_p[MAX_S];
  __shared__ int s_masked[MAX_S];
  __shared__ int s_unmask[MAX_S];
  __shared__ int s_commit[MAX_S];
  __shared__ int s_any, s_forced, s_e, s_left;

  grid_dep_launch();
  const int slot = blockIdx.x;
  const int s = a.s;
  const bool two_layers = a.use_filter && a.rule == 0 && a.n_filter_layers == 0;
  if (two_layers) {
    for (int i = threadIdx.x; i < s * s; i += blockDim.x) {
      const int j = i / s, at = j * (s + 1) + (i - j * s);
      s_w[0][at] = a.w1[i];
      s_w[1][at] = a.w2[i];
    }
    if (threadIdx.x < s) { s_b[0][threadIdx.x] = a.b1[threadIdx.x]; s_b[1][threadIdx.x] = a.b2[threadIdx.x]; }
  }
  grid_dep_wait();
  const SeqMeta m = a.meta[slot];
  const int seq = m.seq;
  const int g0 = m.block * s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;

  // ---- confidence head: merge tile records, row r = slot*s + j -------------------------------
  // Lanes take rows, which are adjacent in memory, and the warps (half warps for up to 16 rows) take turns along the tiles; their
  // records then meet in shared memory, where a warp folds those of a row.
  {
    const int rl = s > 16 ? 32 : 16, row = lane & (rl - 1), sub = warp * (32 / rl) + lane / rl, n_sub = n_warps * (32 / rl);
    float *const rec_m = recs, *const rec_s = recs + n_sub * (rl + 1);
    int *const rec_i = reinterpret_cast<int *>(recs + 2 * n_sub * (rl + 1));
    const int n_rec = n_sub < a.n_tiles ? n_sub : a.n_tiles;
    for (int j0 = 0; j0 < s; j0 += rl) {
      // rows beyond the block's (padding of the records) are folded in too and dropped below: no wait for m
      const bool on = j0 + row < s;
      const int64_t r = (int64_t)slot * s + (on ? j0 + row : 0);
      float mx = -INFINITY, sum = 0.f;
      int ix = 0x7fffffff;
      constexpr int U = 8;   // records requested before the first is folded in
      for (int t0 = sub; t0 < a.n_tiles; t0 += n_sub * U) {
        float tm[U], ts[U];
        int ti[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int t = t0 + n_sub * u;
          const bool in = on && t < a.n_tiles;
          const int64_t o = (int64_t)(in ? t : t0) * a.rows_padded + r;
          tm[u] = in ? a.part_m[o] : -INFINITY;
          ts[u] = in ? a.part_s[o] : 0.f;
          ti[u] = in ? a.part_i[o] : 0x7fffffff;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (t0 + n_sub * u >= a.n_tiles) break;
          if (tm[u] > mx) { sum = sum * expf(mx - tm[u]) + ts[u]; mx = tm[u]; ix = ti[u]; }
          else { sum += ts[u] * expf(tm[u] - mx); if (tm[u] == mx && ti[u] < ix) ix = ti[u]; }
        }
      }
      if (j0 > 0) __syncthreads();   // the records of the rows before have been read
      rec_m[sub * (rl + 1) + row] = mx; rec_s[sub * (rl + 1) + row] = sum; rec_i[sub * (rl + 1) + row] = ix;
      __syncthreads();
      for (int j = warp; j < rl && j0 + j < s; j += n_warps) {
        mx = -INFINITY; sum = 0.f; ix = 0x7fffffff;
        for (int g = lane; g < n_rec; g += 32) fold(mx, sum, ix, rec_m[g * (rl + 1) + j], rec_s[g * (rl + 1) + j], rec_i[g * (rl + 1) + j]);
        for (int o = 16; o > 0; o >>= 1) {
          const float om = __shfl_xor_sync(0xffffffffu, mx, o), os = __shfl_xor_sync(0xffffffffu, sum, o);
          const int oi = __shfl_xor_sync(0xffffffffu, ix, o);
          fold(mx, sum, ix, om, os, oi);
        }
        if (lane == 0) {
          const bool live = j0 + j < m.n_blk_rows;
          s_conf[j0 + j] = live ? 1.0f / sum : 0.f;
          s_pred[j0 + j] = live ? ix : -1;
        }
      }
    }
  }
  int e = a.st.eot_pos[seq], l_eff = a.st.l_eff[seq], steps = 0, n_forced = 0;
  if (threadIdx.x == 0) { steps = a.st.steps[seq]; n_forced = a.st.forced[seq]; }
  if (threadIdx.x < s) {
    int j = threadIdx.x;
    s_masked[j] = a.masked[(int64_t)seq * a.G + g0 + j];
    s_unmask[j] = 0;
  }
  if (threadIdx.x == 0) { s_any = 0; s_forced = 0; s_e = 0x7fffffff; s_left = 0; }
  __syncthreads();

  // ---- filter ----------------------------------------------------------------------------------
  if (threadIdx.x < s) {
    int j = threadIdx.x;
    float c = (j < m.n_blk_rows) ? s_conf[j] : 1.0f;       // positions cut off by EoTP read as finished
    if (a.committed_conf_mode == 1 && !s_masked[j]) c = 1.0f;
    s_c[j] = c;
  }
  __syncthreads();
  if (a.use_filter && a.rule == 0 && a.n_filter_layers > 0) {
    // depth variants: x <- W_k x + b_k with ReLU between consecutive layers; s_h / s_t alternate as output
    // (s_c, the filter's input, stays intact for the sample sink)
    float *src = s_c, *dst = s_h;
    for (int k = 0; k < a.n_filter_layers; ++k) {
      if (threadIdx.x < s) {
        const int j = threadIdx.x;
        float z = a.fb[k][j];
        for (int i = 0; i < s; ++i) z = fmaf(a.fw[k][j * s + i], k > 0 ? fmaxf(src[i], 0.f) : src[i], z);
        dst[j] = z;
        if (k + 1 == a.n_filter_layers) s_p[j] = 1.0f / (1.0f + expf(-z));
      }
      __syncthreads();
      src = dst; dst = (dst == s_h) ? s_t : s_h;
    }
  } else if (two_layers) {
    if (threadIdx.x < s) {
      int j = threadIdx.x;
      float h = s_b[0][j];
#pragma unroll 8
      for (int i = 0; i < s; ++i) h = fmaf(s_w[0][j * (s + 1) + i], s_c[i], h);
      s_h[j] = fmaxf(h, 0.f);
    }
    __syncthreads();
    if (threadIdx.x < s) {
      int j = threadIdx.x;
      float z = s_b[1][j];
#pragma unroll 8
      for (int i = 0; i < s; ++i) z = fmaf(s_w[1][j * (s + 1) + i], s_h[i], z);
      s_p[j] = 1.0f / (1.0f + expf(-z));
    }
  } else if (threadIdx.x < s) {
    s_p[threadIdx.x] = 0.f;
  }
  __syncthreads();

  // ---- threshold, progress fallback ------------------------------------------------------------------
  if (threadIdx.x < s) {
    int j = threadIdx.x;
    bool pass;
    if (a.rule == 0) pass = s_p[j] > a.tau;
    else if (a.rule == 1) pass = s_conf[j] > a.conf_threshold;
    else pass = s_pred[j] == a.ref[(int64_t)seq * a.G + g0 + j];   // dead rows hold -1, never a token id
    s_commit[j] = s_pred[j];
    if (s_masked[j] && pass) { s_unmask[j] = 1; s_any = 1; }
  }
  __syncthreads();
  // Nothing passed: thread 0 commits the most confident masked position.  s_any is not written after the barrier
  // above, and every thread takes the barrier below, so all warps run the same number of barriers whatever they read.
  if (threadIdx.x == 0 && s_any == 0) {
    int best = -1;
    float bc = -1.f;
    for (int j = 0; j < s; ++j)
      if (s_masked[j] && s_conf[j] > bc) { bc = s_conf[j]; best = j; }
    if (best >= 0) {
      s_unmask[best] = 1; s_forced = 1;
      if (a.rule == 2) s_commit[best] = a.ref[(int64_t)seq * a.G + g0 + best];
    }
  }
  __syncthreads();
  const int forced = s_forced;

  // ---- commit in place ----------------------------------------------------------------------------
  if (threadIdx.x < s) {
    int j = threadIdx.x;
    if (s_unmask[j]) {
      a.tokens[(int64_t)seq * a.tok_stride + m.blk_start + j] = s_commit[j];
      a.masked[(int64_t)seq * a.G + g0 + j] = 0;
      s_masked[j] = 0;
      if (a.use_eotp && s_commit[j] == a.eot_id) atomicMin(&s_e, g0 + j);
    }
    if (a.collect_c) {   // stage 1 of Algorithm 1: the filter's input and the target y_j = [pred_j == r_j]
      const int64_t row = a.collect_base + slot;
      a.collect_c[row * s + j] = s_c[j];
      a.collect_y[row * s + j] = (a.rule == 2 && s_pred[j] == a.ref[(int64_t)seq * a.G + g0 + j]) ? 1 : 0;
    }
    if (a.o_conf) a.o_conf[(int64_t)seq * s + j] = s_conf[j];
    if (a.o_pred) a.o_pred[(int64_t)seq * s + j] = s_pred[j];
    if (a.o_p) a.o_p[(int64_t)seq * s + j] = s_p[j];
    if (a.o_unmask) a.o_unmask[(int64_t)seq * s + j] = (uint8_t)s_unmask[j];
  }
  __syncthreads();

  // ---- EoTP -------------------------------------------------------------------------------------
  if (a.use_eotp && s_e != 0x7fffffff && (e < 0 || s_e < e)) {
    e = s_e;
    l_eff = a.P + e + 1;
    for (int g = e + 1 + threadIdx.x; g < a.G; g += blockDim.x) {
      a.masked[(int64_t)seq * a.G + g] = 0;
      a.tokens[(int64_t)seq * a.tok_stride + a.P + g] = a.eot_id;
    }
    if (threadIdx.x < s && g0 + threadIdx.x > e) s_masked[threadIdx.x] = 0;
  }
  __syncthreads();
  if (threadIdx.x < s && s_masked[threadIdx.x]) atomicAdd(&s_left, 1);
  __syncthreads();

  // ---- block advance / stop -------------------------------------------------------------------------
  if (threadIdx.x == 0) {
    int cur = m.block, done = 0;
    if (s_left == 0) {
      if (e >= 0 || cur + 1 == a.n_blocks) done = 1;
      else cur += 1;
    }
    a.st.cur_block[seq] = cur;
    a.st.l_eff[seq] = l_eff;
    a.st.eot_pos[seq] = e;
    a.st.done[seq] = done;
    a.st.steps[seq] = steps + 1;
    a.st.forced[seq] = n_forced + forced;
    StepSummary sm;
    sm.block = m.block; sm.masks_left = s_left; sm.l_eff = l_eff; sm.done = done;
    sm.forced = forced; sm.cur_block = cur;
    a.summary[seq] = sm;
    if (slot == 0) *a.status_out = *a.status;   // every kernel that may set it is complete
  }
}

}  // namespace

cudaError_t launch_decide(cudaStream_t st, const DecideArgs &a, int n_slots) {
  // a warp per block row: up to 32 take turns along the tile records (the merge is the longest part)
  int threads = 32 * a.s;
  threads = threads < 256 ? 256 : (threads > 1024 ? 1024 : threads);
  const int rl = a.s > 16 ? 32 : 16;
  const size_t smem = sizeof(float) * 3 * (threads / rl) * (rl + 1);
  // beside the kernel's own arrays within what any launch may have: a limit set here would hold for every thread's launches
  static_assert(sizeof(float) * (2 * MAX_S * (MAX_S + 1) + 11 * MAX_S + 4) + sizeof(float) * 3 * 32 * 33 <= 48 * 1024, "shared memory of the decision kernel");
  return launch_kernel(decide_kernel, dim3(n_slots), dim3(threads), smem, st, a);
}

}  // namespace l2pd
