// Filter training, stage 2 of Algorithm 1: minimise Eq. 6, the mean binary cross-entropy between
// sigmoid(f_theta(conf)) and the EGP targets, over the weights of the filter (Section 3.2: two Linear(s, s)
// layers; Section 4.4: one to four, ReLU between consecutive layers) with AdamW (Section 4.1: learning rate 0.001).
//
// filter_train_kernel runs some 100 us of updates in one cooperative launch.  One update:
//   gradient   every block walks tiles of T samples held in shared memory: forward through the layers, dz = sigmoid(z) - y,
//              delta of the layers below (delta_{k-1} = (delta_k W_k) [x_k > 0]), then dW_k += delta_k^T x_k into
//              accumulators its threads own; it ends by writing its sums (not yet divided by the batch's element count) and its loss sum to its own
//              row of `gpart`;
//   meeting    all blocks meet at a counter in global memory (cooperative launch: all are resident; bounded wait; the
//              counter runs on from launch to launch);
//   AdamW      a block takes 8, 32 or all its threads' number of parameters at a time, the threads of one parameter shares
//              of the rows, whose sums are then added in order (a run is bit-reproducible on a given GPU), scales by
//              1 / (samples * s) and applies the update: decoupled weight decay, bias-corrected moments;
//   meeting    and every block reads the new weights.
// K = s <= 64 is too short a contraction, and fp32 too wide a type, for the tensor cores; what bounds the kernel is the
// fp32 pipe (432 M multiply-adds for 84,480 samples of 32: 12 us) and, for small batches, the two meetings (~2 us each) and
// the phases' latency.  A thread computes 4 samples x C positions (dW: 4 x 4 elements) from 16-byte shared-memory
// vectors, 16 C multiply-adds for 4 + C loads; rows are padded to 4 mod 32 words and positions dealt out so that the
// vectors of a warp lie in different banks.  The next tile arrives (cp.async) while one is worked on.
// Measured, one update, two launches of per-sample warps before -> this: 84,480 samples of 32 positions, two layers 100 -> 40 us
// (tiles 30 us, which are bound by shared-memory loads at 40 % of the fp32 pipe); 1,024 samples of 64, four layers
// 72 -> 20 us; a call without updates 0.80 -> 0.10 ms.  Batches of at most 300 samples of s <= 24 are 1 to 2 us an update
// slower than those two launches (300 of 8, one layer: 6.3 -> 7.4), which had no meetings.
#include "common.cuh"
#include "ptx.cuh"

namespace l2pd {

namespace {

constexpr int MAX_LAYERS = 4;
constexpr int MAX_S = 64;

struct TrainArgs {
  const float *C;          // [N, s] filter inputs
  const uint8_t *Y;        // [N, s] targets (0 / 1)
  int64_t N, batch;        // samples; samples per update (the last batch of an epoch may be shorter)
  int64_t u0, u1;          // this launch's updates
  int64_t per_epoch;       // updates per epoch
  int s, n_layers, P;      // P parameters
  float *theta, *m, *v;    // packed per layer: W_k [s*s], b_k [s]
  float *gpart;            // a row per block: gradient sums, then the loss sum
  float *losses;           // [updates]: the batch's loss, measured before the update
  float lr, beta1, beta2, eps, weight_decay;
  double p1, p2;           // beta1^u0, beta2^u0
  unsigned *bar;           // meeting counter, `arrivals` at launch
  unsigned arrivals;
  int32_t *status;
  uint64_t limit_ns;       // bound of a meeting's wait
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All blocks of the launch meet: `target` arrivals on the counter.  False (for the whole block) when the wait ran out.
__device__ __forceinline__ bool meet(unsigned *bar, unsigned target, int32_t *status, uint64_t limit_ns, int *s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
    int ok = 1;
    const uint64_t t0 = ptx::globaltimer();
    uint32_t spins = 0;
    while ((int)(ld_acquire(bar) - target) < 0) {
      if ((++spins & 0x3fu) == 0) {
        if (*reinterpret_cast<volatile int32_t *>(status) != DEV_OK) { ok = 0; break; }
        if (ptx::globaltimer() - t0 > limit_ns) { atomicCAS(status, 0, DEV_TIMEOUT_EPILOGUE); ok = 0; break; }
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// Words of the tile buffers: X[0] twice (the next tile arrives while this one is worked on), X[1 .. L - 1], and the deltas of
// the layer being differentiated and of the one below.  They also hold the end of an update's sums (4096 + 256 words where
// threads share a gradient).
template <int S, int T>
__host__ __device__ constexpr int train_tile_floats(int L) {
  return (L + 1 + (L < 2 ? L : 2)) * T * (S + 4) < 4096 + 256 ? 4096 + 256 : (L + 1 + (L < 2 ? L : 2)) * T * (S + 4);
}
template <int S, int T>
constexpr int train_smem_floats(int L) { return L * (S * (S + 4) + S) + train_tile_floats<S, T>(L) + 2 * T * S / 4 + 64; }

__device__ __forceinline__ void cp_async16(void *dst, const void *src, int bytes) {   // the rest of the 16 bytes is zero
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}

// S: positions padded to 32 or 64; T: samples per tile; LM: most layers (accumulators in registers); TH threads per block,
// OCC blocks per SM.
template <int S, int T, int LM, int TH, int OCC>
__global__ void __launch_bounds__(TH, OCC) filter_train_kernel(const TrainArgs a) {
  constexpr int TRAIN_THREADS = TH, TRAIN_WARPS = TH / 32;
  constexpr int C = T * S / (4 * TRAIN_THREADS);      // positions per thread (x 4 samples)
  constexpr int NCG = S / C, NSG = T / 4;
  static_assert(C >= 1 && NCG % 8 == 0 && NCG * NSG == TRAIN_THREADS, "thread tiling");
  constexpr int RS = S + 4;                           // row stride of every matrix: 4 mod 32 words
  constexpr int G = 16 * TH / (S * S);                  // groups of threads that share a gradient, each with T / G of the samples
  constexpr int GT = TRAIN_THREADS / G, GA = S / 4;   // threads per group = GA x GA
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_ok;
  const int s = a.s, L = a.n_layers, per = s * s + s, P = a.P, gs = filter_train_row_floats(P), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float *W = sm;                          // [L][S][RS]
  float *Bv = W + L * S * RS;             // [L][S]
  float *X0 = Bv + L * S;                 // [2][T][RS]: inputs of this tile and the next
  float *X1 = X0 + 2 * T * RS;            // [L - 1][T][RS]: relu(output of layer k - 1) at k - 1
  float *D = X1 + (L - 1) * T * RS;       // [min(L, 2)][T][RS]: gradient of the loss with respect to a layer's output
  float *X = X0;                          // (the sums at the end of an update)
  uint8_t *Ys = reinterpret_cast<uint8_t *>(X0 + train_tile_floats<S, T>(L));   // [2][T][S]
  float *red = reinterpret_cast<float *>(Ys + 2 * T * S);                       // [64]
  // outputs of a thread: samples sg + NSG e, positions cg + NCG c (forward) or C cg + c (backward); a warp has 8 position
  // groups x 4 sample groups
  const int cg = (tid & 7) + 8 * (tid / (8 * NSG)), sg = (tid >> 3) % NSG;
  const int grp = tid / GT, ga = (tid % GT) / GA, gb_ = tid % GA;            // dW: elements (4 ga + r, 4 gb_ + q) of group grp
  constexpr int DBP = TRAIN_THREADS / S;                                     // db: position tid % S, one of DBP parts of the samples
  // rows that fill their padded width and start on 16 bytes come by cp.async
  const bool vec = s == S && ((reinterpret_cast<uintptr_t>(a.C) | reinterpret_cast<uintptr_t>(a.Y)) & 15) == 0;
  double p1 = a.p1, p2 = a.p2;
  unsigned target = a.arrivals;
  // a meeting of an earlier launch ran out: the parameters are part old, part new, and nothing may be made of them
  if (*reinterpret_cast<volatile int32_t *>(a.status) != DEV_OK) return;

  for (int64_t u = a.u0; u < a.u1; ++u) {
    const int64_t n0 = (u % a.per_epoch) * a.batch, nb = a.N - n0 < a.batch ? a.N - n0 : a.batch;
    const int64_t n_tiles = (nb + T - 1) / T;
    const int rows = (int)(n_tiles < gridDim.x ? n_tiles : gridDim.x);       // blocks that have tiles
    if (blockIdx.x < rows) {
      if (s == S) {
        for (int k = 0; k < L; ++k) {
          constexpr int NV = S * S / 4 / TRAIN_THREADS;     // 16-byte vectors per thread and layer, all in flight together
          float4 t[NV];
#pragma unroll
          for (int q = 0; q < NV; ++q) t[q] = __ldcg(reinterpret_cast<const float4 *>(a.theta + k * per) + tid + q * TRAIN_THREADS);
#pragma unroll
          for (int q = 0; q < NV; ++q) {
            const int e = 4 * (tid + q * TRAIN_THREADS);
            *reinterpret_cast<float4 *>(W + (k * S + e / S) * RS + e % S) = t[q];
          }
        }
      } else {
#pragma unroll 8
        for (int e = tid; e < L * S * S; e += TRAIN_THREADS) {
          const int k = e / (S * S), j = (e / S) % S, i = e % S;
          W[(k * S + j) * RS + i] = (j < s && i < s) ? __ldcg(a.theta + k * per + j * s + i) : 0.f;
        }
      }
      for (int e = tid; e < L * S; e += TRAIN_THREADS) Bv[e] = (e % S) < s ? __ldcg(a.theta + (e / S) * per + s * s + e % S) : 0.f;
      float acc[LM][16], gb[LM], loss = 0.f;
#pragma unroll
      for (int k = 0; k < LM; ++k) {
        gb[k] = 0.f;
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[k][q] = 0.f;
      }
      auto fetch = [&](int64_t tile, int buf) {
        const int64_t base = n0 + tile * T;
        const int live = (int)(nb - tile * T < T ? nb - tile * T : T);
        float *xd = X0 + buf * T * RS;
        uint8_t *yd = Ys + buf * T * S;
        if (vec) {
          for (int e = tid; e < T * S / 4; e += TRAIN_THREADS) {
            const int n = e / (S / 4), i = 4 * (e % (S / 4));
            const bool in = n < live;
            cp_async16(xd + n * RS + i, a.C + (in ? (base + n) * s + i : 0), in ? 16 : 0);
          }
          for (int e = tid; e < T * S / 16; e += TRAIN_THREADS) {
            const bool in = 16 * e < live * S;
            cp_async16(yd + 16 * e, a.Y + (in ? base * s + 16 * e : 0), in ? 16 : 0);
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
        } else {
          for (int e = tid; e < T * S; e += TRAIN_THREADS) {
            const int n = e / S, i = e % S;
            const bool in = n < live && i < s;
            xd[n * RS + i] = in ? a.C[(base + n) * s + i] : 0.f;
            yd[e] = in ? a.Y[(base + n) * s + i] : 0;
          }
        }
      };
      int buf = 0;
      fetch(blockIdx.x, 0);
      for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, buf ^= 1) {
        const int live = (int)(nb - tile * T < T ? nb - tile * T : T);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                   // this tile has arrived; the previous one is no longer read
        if (tile + gridDim.x < n_tiles) fetch(tile + gridDim.x, buf ^ 1);
        float *const x0 = X0 + buf * T * RS;
        // forward: layer k maps X[k] to X[k + 1] = relu(.), the last layer to dz = sigmoid(z) - y in D
        for (int k = 0; k < L; ++k) {
          const float *xin = (k ? X1 + (k - 1) * T * RS : x0) + sg * RS, *wk = W + (k * S + cg) * RS;
          float o[C][4];
#pragma unroll
          for (int c = 0; c < C; ++c) o[c][0] = o[c][1] = o[c][2] = o[c][3] = Bv[k * S + cg + NCG * c];
#pragma unroll 4
          for (int i = 0; i < S; i += 4) {
            float4 w[C], x[4];
#pragma unroll
            for (int c = 0; c < C; ++c) w[c] = *reinterpret_cast<const float4 *>(wk + NCG * c * RS + i);
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = *reinterpret_cast<const float4 *>(xin + NSG * e * RS + i);
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
              for (int e = 0; e < 4; ++e)
                o[c][e] = fmaf(w[c].w, x[e].w, fmaf(w[c].z, x[e].z, fmaf(w[c].y, x[e].y, fmaf(w[c].x, x[e].x, o[c][e]))));
          }
          if (k + 1 < L) {
            float *xo = X1 + k * T * RS + sg * RS + cg;
#pragma unroll
            for (int c = 0; c < C; ++c)
#pragma unroll
              for (int e = 0; e < 4; ++e) xo[NSG * e * RS + NCG * c] = fmaxf(o[c][e], 0.f);
          } else {
            // loss = max(z, 0) - z y + log(1 + t), t = exp(-|z|): the logarithms of this thread's outputs are taken as one,
            // of the product of the (1 + t), carried as pm = product - 1
            float pm = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int n = sg + NSG * e;
#pragma unroll
              for (int c = 0; c < C; ++c) {
                const int j = cg + NCG * c;
                const bool on = n < live && j < s;
                const float z = o[c][e], y = Ys[(buf * T + n) * S + j] ? 1.f : 0.f;
                const float t = expf(-fabsf(z)), sig = __fdividef(z >= 0.f ? 1.f : t, 1.f + t);
                if (on) { loss += fmaxf(z, 0.f) - z * y; pm = fmaf(pm, t, pm + t); }
                D[n * RS + j] = on ? sig - y : 0.f;
              }
            }
            loss += log1pf(pm);
          }
          __syncthreads();
        }
        // backward, layer by layer: dW_k += D[k]^T X[k], db_k += sum D[k], D[k - 1] = (D[k] W_k) [X[k] > 0]
        float *dcur = D, *dnxt = D + T * RS;
#pragma unroll
        for (int kk = 0; kk < LM; ++kk) {                  // acc[kk] belongs to layer L - 1 - kk
          const int k = L - 1 - kk;
          if (k < 0) break;
          const float *xin = k ? X1 + (k - 1) * T * RS : x0;
          const float *dk = dcur + grp * (T / G) * RS + 4 * ga, *xk = xin + grp * (T / G) * RS + 4 * gb_;
#pragma unroll 4
          for (int n = 0; n < T / G; ++n) {
            const float4 dv = *reinterpret_cast<const float4 *>(dk + n * RS), xv = *reinterpret_cast<const float4 *>(xk + n * RS);
            const float dr[4] = {dv.x, dv.y, dv.z, dv.w}, xr[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int q = 0; q < 4; ++q) acc[kk][4 * r + q] = fmaf(dr[r], xr[q], acc[kk][4 * r + q]);
          }
          const float *db = dcur + (tid / S) * (T / DBP) * RS + tid % S;
#pragma unroll
          for (int n = 0; n < T / DBP; ++n) gb[kk] += db[n * RS];
          if (k > 0) {
            const float *din = dcur + sg * RS, *wk = W + k * S * RS + C * cg;
            float o[C][4];
#pragma unroll
            for (int c = 0; c < C; ++c) o[c][0] = o[c][1] = o[c][2] = o[c][3] = 0.f;
#pragma unroll 2
            for (int j = 0; j < S; j += 4) {
              float4 d[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) d[e] = *reinterpret_cast<const float4 *>(din + NSG * e * RS + j);
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                float w[C];
                if constexpr (C == 4) *reinterpret_cast<float4 *>(w) = *reinterpret_cast<const float4 *>(wk + (j + r) * RS);
                else if constexpr (C == 2) *reinterpret_cast<float2 *>(w) = *reinterpret_cast<const float2 *>(wk + (j + r) * RS);
                else w[0] = wk[(j + r) * RS];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float dr = r == 0 ? d[e].x : r == 1 ? d[e].y : r == 2 ? d[e].z : d[e].w;
#pragma unroll
                  for (int c = 0; c < C; ++c) o[c][e] = fmaf(w[c], dr, o[c][e]);
                }
              }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
              for (int c = 0; c < C; ++c) {
                const int at = (sg + NSG * e) * RS + C * cg + c;
                dnxt[at] = xin[at] > 0.f ? o[c][e] : 0.f;
              }
            __syncthreads();
            float *t = dcur; dcur = dnxt; dnxt = t;
          }
        }
      }
      // the block's sums: groups and parts are added in order through shared memory (over the tile buffers)
      float *out = a.gpart + (int64_t)blockIdx.x * gs;
#pragma unroll
      for (int kk = 0; kk < LM; ++kk) {
        const int k = L - 1 - kk;
        if (k < 0) break;
        __syncthreads();
        if (G > 1) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            *reinterpret_cast<float4 *>(X + (grp * S + 4 * ga + r) * S + 4 * gb_) =
                make_float4(acc[kk][4 * r], acc[kk][4 * r + 1], acc[kk][4 * r + 2], acc[kk][4 * r + 3]);
        }
        X[G * S * S * (G > 1) + tid] = gb[kk];
        __syncthreads();
        if (G > 1) {
          // (the groups' sums lie as [group][position][position])
#pragma unroll
          for (int q = 0; q < S * S / TRAIN_THREADS; ++q) {
            const int e = tid + q * TRAIN_THREADS, j = e / S, i = e % S;
            float t = X[e];
#pragma unroll
            for (int g = 1; g < G; ++g) t += X[g * S * S + e];
            if (j < s && i < s) __stcg(out + k * per + j * s + i, t);
          }
        } else {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (s == S)
              __stcg(reinterpret_cast<float4 *>(out + k * per + (4 * ga + r) * S + 4 * gb_),
                     make_float4(acc[kk][4 * r], acc[kk][4 * r + 1], acc[kk][4 * r + 2], acc[kk][4 * r + 3]));
            else
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int j = 4 * ga + r, i = 4 * gb_ + q;
              if (j < s && i < s) __stcg(out + k * per + j * s + i, acc[kk][4 * r + q]);
            }
        }
        if (tid < s) {
          float t = 0.f;
#pragma unroll
          for (int q = 0; q < DBP; ++q) t += X[G * S * S * (G > 1) + q * S + tid];
          __stcg(out + k * per + s * s + tid, t);
        }
      }
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if (lane == 0) red[warp] = loss;
      __syncthreads();
      if (tid == 0) {
        float t = 0.f;
        for (int w = 0; w < TRAIN_WARPS; ++w) t += red[w];
        __stcg(out + P, t);
      }
    }
    target += gridDim.x;
    if (!meet(a.bar, target, a.status, a.limit_ns, &s_ok)) return;

    // AdamW; entry P is the loss
    p1 *= (double)a.beta1; p2 *= (double)a.beta2;
    const float bc1 = (float)(1.0 - p1), bc2 = (float)(1.0 - p2), inv_count = (float)(1.0 / ((double)nb * s));
    // A block's pass: PW parameters x RG shares of the rows.  Few parameters and many rows: a sector of a row per load and
    // many shares; many parameters: wider passes, whose number costs more than their length.
    const int PW = P < 16 * (int)gridDim.x ? 8 : rows > 64 ? 32 : TRAIN_THREADS, RG = TRAIN_THREADS / PW;
    const int pl = tid % PW, rg = tid / PW, share = (rows + RG - 1) / RG, b0 = rg * share, b1 = min(rows, b0 + share);
    for (int c = blockIdx.x; c * PW <= P; c += gridDim.x) {
      const int p = c * PW + pl;
      float g = 0.f;
      if (p <= P) {
        // up to 16 rows in flight; added by halves, as a chain of 64 rows cost a batch of 1,024 half its accuracy
        for (int b = b0; b < b1; b += 16) {
          float t[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) t[i] = b + i < b1 ? __ldcg(a.gpart + (int64_t)(b + i) * gs + p) : 0.f;
#pragma unroll
          for (int h = 8; h > 0; h >>= 1)
#pragma unroll
            for (int i = 0; i < h; ++i) t[i] += t[i + h];
          g += t[0];
        }
      }
      if (RG > 1) {
        __syncthreads();
        X[tid] = g;
        __syncthreads();
      }
      if (tid < PW && p <= P) {
        for (int w = 1; w < RG; ++w) g += X[w * PW + tid];
        g *= inv_count;
        if (p == P) {
          a.losses[u] = g;
        } else {
          const float th = __ldcg(a.theta + p) * (1.0f - a.lr * a.weight_decay);
          const float m = a.beta1 * a.m[p] + (1.0f - a.beta1) * g;
          const float v = a.beta2 * a.v[p] + (1.0f - a.beta2) * g * g;
          a.m[p] = m; a.v[p] = v;
          __stcg(a.theta + p, th - a.lr * (m / bc1) / (sqrtf(v / bc2) + a.eps));
        }
      }
    }
    if (u + 1 < a.u1) {
      target += gridDim.x;
      if (!meet(a.bar, target, a.status, a.limit_ns, &s_ok)) return;
    }
  }
}

struct PackArgs { float *w[MAX_LAYERS], *b[MAX_LAYERS]; float *theta; int s, n_layers; };

// The caller's arrays -> theta, moments 0, status and meeting counter 0 (pack), and theta -> the caller's arrays, which stay as they were when a
// meeting ran out (blocks leave it at different points, so theta is then part old, part new).
__global__ void filter_pack_kernel(PackArgs a, int pack, int32_t *status, unsigned *bar) {
  if (!pack && *status != DEV_OK) return;
  const int per = a.s * a.s + a.s, P = a.n_layers * per;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < P; e += gridDim.x * blockDim.x) {
    const int k = e / per, r = e - k * per;
    float *q = r < a.s * a.s ? a.w[k] + r : a.b[k] + (r - a.s * a.s);
    if (pack) { a.theta[e] = *q; a.theta[P + e] = 0.f; a.theta[2 * P + e] = 0.f; }
    else *q = a.theta[e];
  }
  if (pack && blockIdx.x == 0 && threadIdx.x == 0) { *status = DEV_OK; *bar = 0; }
}

template <int S, int T, int LM, int TH, int OCC>
cudaError_t launch_train(cudaStream_t st, TrainArgs &a, int sms, int *blocks) {
  const size_t smem = sizeof(float) * (size_t)train_smem_floats<S, T>(a.n_layers);
  // the limit of the deepest filter of this form: it belongs to the kernel, and another thread may be preparing another depth
  cudaError_t e = cudaFuncSetAttribute(filter_train_kernel<S, T, LM, TH, OCC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(sizeof(float) * (size_t)train_smem_floats<S, T>(LM)));
  if (e != cudaSuccess) return e;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, filter_train_kernel<S, T, LM, TH, OCC>, TH, smem);
  if (e != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  if (occ > OCC) occ = OCC;
  const int64_t tiles = ((a.N < a.batch ? a.N : a.batch) + T - 1) / T;
  // one block per SM at least takes part in the parameters' update, tiles or not; more only for their own tiles
  int grid = sms * occ;
  if (tiles < grid) grid = (int)(tiles > sms ? tiles : sms);
  void *args[] = {&a};
  *blocks = grid;
  return cudaLaunchCooperativeKernel((const void *)filter_train_kernel<S, T, LM, TH, OCC>, dim3(grid), dim3(TH), args, smem, st);
}

}  // namespace

cudaError_t launch_filter_pack(cudaStream_t st, float *const *w, float *const *b, int s, int n_layers, float *theta, int32_t *status, unsigned *bar, bool pack) {
  PackArgs a = {};
  for (int k = 0; k < n_layers; ++k) { a.w[k] = w[k]; a.b[k] = b[k]; }
  a.theta = theta; a.s = s; a.n_layers = n_layers;
  filter_pack_kernel<<<(n_layers * (s * s + s) + 255) / 256, 256, 0, st>>>(a, pack ? 1 : 0, status, bar);
  return cudaGetLastError();
}

int filter_train_max_rows(int64_t batch, int sms) { return (int)(ceil_div64(batch, 16) < 3 * sms ? ceil_div64(batch, 16) : 3 * sms); }

// A launch occupies every SM, and a kernel of another stream waits for it, so a launch takes about 100 us of updates, by a
// model of their time that holds within a fifth (the fixed part: meetings and phases).  Beside training at 84,480 x 32, two
// layers, a decode step of the tiny model (20 kernels, 0.12 ms alone) takes 0.48 ms and the 512-row step of four 8B layers
// (0.85 ms alone) 2.5 ms; with launches of 400 us 2.0 and 9.1 ms, of 80 ms each stands still for a launch or two.  The
// training itself pays 2 % (38.9 -> 39.9 us an update), 5 % of a call of 60 updates of 20 us (1.30 -> 1.37 ms).
int64_t filter_train_updates_per_launch(int64_t batch, int s, int n_layers) {
  const double S = s <= 32 ? 32.0 : 64.0, macs = (double)batch * S * S * (3 * n_layers - 1);
  const double us = 5.0 + 3.0 * n_layers + macs / 14.4e6;
  const int64_t n = (int64_t)(100.0 / us);
  return n < 1 ? 1 : n;
}

cudaError_t launch_filter_train(cudaStream_t st, FilterTrainArgs &f, int64_t u0, int64_t u1, double p1, double p2, int sms) {
  if (f.n_layers < 1 || f.n_layers > MAX_LAYERS || f.s < 1 || f.s > MAX_S) return cudaErrorInvalidValue;
  TrainArgs a;
  a.C = f.C; a.Y = f.Y; a.N = f.N; a.batch = f.batch; a.u0 = u0; a.u1 = u1;
  a.per_epoch = (f.N + f.batch - 1) / f.batch;
  a.s = f.s; a.n_layers = f.n_layers; a.P = f.n_layers * (f.s * f.s + f.s);
  a.theta = f.theta; a.m = f.m; a.v = f.v; a.gpart = f.gpart; a.losses = f.losses;
  a.lr = f.h.lr; a.beta1 = f.h.beta1; a.beta2 = f.h.beta2; a.eps = f.h.eps; a.weight_decay = f.h.weight_decay;
  a.p1 = p1; a.p2 = p2; a.bar = f.bar; a.arrivals = f.arrivals; a.status = f.status; a.limit_ns = f.limit_ns;
  const int64_t nb = f.N < f.batch ? f.N : f.batch;
  // Large batches: tiles of 64 samples, 4 x 4 outputs per thread.  With fewer than one such tile for every SM smaller tiles
  // spread the batch over more blocks (1,024 samples of 64, four layers: tiles of 16 take 19.5 k cycles, of 32 30 k; 84,480
  // of 32: 128 threads with 4 x 4 outputs 56 k, 256 threads with 2 x 4 65 k).
  const bool small = nb < (int64_t)(f.s <= 32 ? 64 : 32) * sms;
  int blocks = 0;
  cudaError_t e;
  if (f.s <= 32) {
    if (f.n_layers <= 2) e = small ? launch_train<32, 32, 2, 256, 2>(st, a, sms, &blocks) : launch_train<32, 64, 2, 128, 3>(st, a, sms, &blocks);
    else e = small ? launch_train<32, 32, 4, 256, 1>(st, a, sms, &blocks) : launch_train<32, 64, 4, 128, 2>(st, a, sms, &blocks);
  } else {
    if (f.n_layers <= 2) e = small ? launch_train<64, 16, 2, 256, 2>(st, a, sms, &blocks) : launch_train<64, 64, 2, 256, 1>(st, a, sms, &blocks);
    else e = small ? launch_train<64, 16, 4, 256, 1>(st, a, sms, &blocks) : launch_train<64, 64, 4, 256, 1>(st, a, sms, &blocks);
  }
  f.arrivals += (unsigned)blocks * (unsigned)(2 * (u1 - u0) - 1);   // two meetings an update, but for the launch's last one
  return e;
}

}  // namespace l2pd
