// CUDA-core kernels: the GEMM and attention of fp32 configurations (tcgen05 has no fp32
// kind, and TF32 would not reach 1e-4 relative accuracy).  Their models are small: a projection is a few
// dozen MFLOP, so what bounds it is latency.  gemm_f32_kernel and attention_f32_kernel keep everything a
// block needs in flight at once (cp.async) and spread a step over as many blocks as its sizes allow.
// The plain templates simt_gemm_kernel / simt_attention_kernel serve bf16 storage, as an independent
// cross-check of the tensor-core kernels, and fp32 matrices that do not start on 16 bytes.
#include "common.cuh"
#include "ptx.cuh"

#include <type_traits>

namespace l2pd {

namespace {

constexpr int BM = 64, BN = 64, BK = 16;
constexpr int MAX_GRID_YZ = 65535;   // blocks along the y and z of a grid

// C[M,N] = A[M,K] * W[N,K]^T with fp32 accumulation in k order; 256 threads, 4x4 outputs each.
//   EPI_STORE      C (T)    = acc
//   EPI_RESIDUAL   X (fp32) += acc
//   EPI_SWIGLU     H (T)    = silu(acc_gate) * acc_up  (W = gate rows, W2 = up rows)
//   EPI_STORE_F32  C (fp32) = acc + bias[col]
template <typename T, int EPI>
__global__ void __launch_bounds__(256) simt_gemm_kernel(const T *__restrict__ A, const T *__restrict__ W,
                                                        const T *__restrict__ W2, void *Cv,
                                                        const float *__restrict__ bias, int M, int N, int K) {
  grid_dep_launch();
  grid_dep_wait();
  __shared__ float As[BK][BM + 1];
  __shared__ float Ws[BK][BN + 1];
  __shared__ float W2s[EPI == EPI_SWIGLU ? BK : 1][BN + 1];
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  float acc[4][4] = {}, acc2[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += BK) {
    for (int i = threadIdx.x; i < BM * BK; i += 256) {
      int r = i / BK, c = i - r * BK;
      int gm = m0 + r, gk = k0 + c;
      As[c][r] = (gm < M && gk < K) ? to_f32(A[(int64_t)gm * K + gk]) : 0.f;
      int gn = n0 + r;
      Ws[c][r] = (gn < N && gk < K) ? to_f32(W[(int64_t)gn * K + gk]) : 0.f;
      if (EPI == EPI_SWIGLU) W2s[c][r] = (gn < N && gk < K) ? to_f32(W2[(int64_t)gn * K + gk]) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[4], b[4], b2[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = As[k][ty * 4 + i];
        b[i] = Ws[k][tx * 4 + i];
        if (EPI == EPI_SWIGLU) b2[i] = W2s[k][tx * 4 + i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
          if (EPI == EPI_SWIGLU) acc2[i][j] = fmaf(a[i], b2[j], acc2[i][j]);
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gm = m0 + ty * 4 + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gn = n0 + tx * 4 + j;
      if (gn >= N) continue;
      int64_t o = (int64_t)gm * N + gn;
      float v = acc[i][j];
      if (EPI == EPI_STORE) {
        reinterpret_cast<T *>(Cv)[o] = from_f32<T>(v);
      } else if (EPI == EPI_RESIDUAL) {
        reinterpret_cast<float *>(Cv)[o] += v;
      } else if (EPI == EPI_SWIGLU) {
        float sg = v / (1.0f + expf(-v));
        reinterpret_cast<T *>(Cv)[o] = from_f32<T>(sg * acc2[i][j]);
      } else {
        reinterpret_cast<float *>(Cv)[o] = v + (bias ? bias[gn] : 0.f);
      }
    }
  }
}

// One block per (query row, head): scores over all visible keys, softmax, weighted sum of values.
// No causal mask: every query sees keys [0, kv_len) of its own sequence.
template <typename T>
__global__ void simt_attention_kernel(const T *__restrict__ q, const T *__restrict__ kc,
                                      const T *__restrict__ vc, const SeqMeta *meta,
                                      const int32_t *row_slot, T *out, int64_t kv_seq_stride, int H,
                                      int dh) {
  grid_dep_launch();
  grid_dep_wait();
  extern __shared__ float sm[];
  float *qs = sm;          // [dh]
  float *sc = sm + dh;     // [kv_len]
  __shared__ float red[32];
  int row = blockIdx.x, h = blockIdx.y;
  SeqMeta m = meta[row_slot[row]];
  int hd = H * dh;
  const T *qr = q + (int64_t)row * hd + h * dh;
  for (int i = threadIdx.x; i < dh; i += blockDim.x) qs[i] = to_f32(qr[i]);
  __syncthreads();
  const T *kb = kc + (int64_t)m.seq * kv_seq_stride + h * dh;
  const T *vb = vc + (int64_t)m.seq * kv_seq_stride + h * dh;
  float scale = 1.0f / sqrtf((float)dh);
  float mx = -INFINITY;
  for (int j = threadIdx.x; j < m.kv_len; j += blockDim.x) {
    const T *kr = kb + (int64_t)j * hd;
    float a = 0.f;
    for (int c = 0; c < dh; ++c) a = fmaf(qs[c], to_f32(kr[c]), a);
    a *= scale;
    sc[j] = a;
    mx = fmaxf(mx, a);
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (l == 0) red[w] = mx;
  __syncthreads();
  mx = (l < nw) ? red[l] : -INFINITY;
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float sum = 0.f;
  for (int j = threadIdx.x; j < m.kv_len; j += blockDim.x) {
    float e = expf(sc[j] - mx);
    sc[j] = e;
    sum += e;
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  __syncthreads();
  if (l == 0) red[w] = sum;
  __syncthreads();
  sum = (l < nw) ? red[l] : 0.f;
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  float inv = 1.0f / sum;
  T *orow = out + (int64_t)row * hd + h * dh;
  for (int c = threadIdx.x; c < dh; c += blockDim.x) {
    float a = 0.f;
    for (int j = 0; j < m.kv_len; ++j) a = fmaf(sc[j], to_f32(vb[(int64_t)j * hd + c]), a);
    orow[c] = from_f32<T>(a * inv);
  }
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in) {   // zeros where `in` is false
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// C[M,N] = A[M,K] * W[N,K]^T in fp32, epilogues as simt_gemm_kernel.  A block computes a B x B tile with 256 threads: KG
// groups of threads hold the whole tile, 4 x 4 outputs each, and take turns along K (16-deep shares of a 64-deep stage for
// B = 32, 4-deep ones for B = 16); the groups' sums are added in order at the end, by all threads.  Four stages in flight:
// K = 256 is requested whole before the first multiply.  Rows are 68 words apart and dealt out interleaved, so the 16-byte
// loads of a warp do not collide.
// Measured at 96 rows of the tiny model (d 256, 688), one launch between events, 64 x 64 blocks with 16-deep unpipelined
// stages before -> now (us, some 5 of them the events): QKV 34 -> 9, O 38 -> 8, gate/up 43 -> 11, down 103 -> 9, LM head 22 -> 10.
constexpr int F_BK = 64, F_ROW = F_BK + 4, F_STAGES = 4, F_THREADS = 256;
template <int EPI, int B>
__global__ void __launch_bounds__(F_THREADS) gemm_f32_kernel(const float *__restrict__ A, const float *__restrict__ W,
                                                             const float *__restrict__ W2, float *out, const float *__restrict__ bias,
                                                             int M, int N, int K) {
  constexpr int TG = (B / 4) * (B / 4), KG = F_THREADS / TG, KS = F_BK / KG;   // threads per group, groups, k per group and stage
  constexpr int MATS = EPI == EPI_SWIGLU ? 3 : 2, MAT = B * F_ROW;
  static_assert(KG >= 1 && KS % 4 == 0, "tiling");
  extern __shared__ __align__(16) float sm[];   // [F_STAGES][MATS][B][F_ROW]; the groups' sums at the end
  const int tid = threadIdx.x, grp = tid / TG, t = tid % TG, tx = t % (B / 4), ty = t / (B / 4);
  const int m0 = blockIdx.y * B, n0 = blockIdx.x * B, n_st = (K + F_BK - 1) / F_BK;
  auto load = [&](int st, bool act, bool wts) {
    float *d = sm + (st % F_STAGES) * MATS * MAT;
    for (int e = tid; e < B * (F_BK / 4); e += F_THREADS) {
      const int r = e / (F_BK / 4), c = 4 * (e % (F_BK / 4)), k = st * F_BK + c;
      if (act) cp_async16(d + r * F_ROW + c, A + (m0 + r < M && k < K ? (int64_t)(m0 + r) * K + k : 0), m0 + r < M && k < K);
      if (wts) {
        const bool in = n0 + r < N && k < K;
        const int64_t o = in ? (int64_t)(n0 + r) * K + k : 0;
        cp_async16(d + MAT + r * F_ROW + c, W + o, in);
        if (EPI == EPI_SWIGLU) cp_async16(d + 2 * MAT + r * F_ROW + c, W2 + o, in);
      }
    }
  };
  grid_dep_launch();
  // no kernel writes weights: the first stages' are requested before the previous kernel has completed
  for (int st = 0; st < F_STAGES - 1 && st < n_st; ++st) load(st, false, true);
  grid_dep_wait();
  for (int st = 0; st < F_STAGES - 1; ++st) {
    if (st < n_st) load(st, true, false);
    cp_async_commit();                          // (the weights requested above belong to the first group)
  }
  float acc[4][4] = {}, acc2[EPI == EPI_SWIGLU ? 4 : 1][4] = {};
  for (int st = 0; st < n_st; ++st) {
    cp_async_wait<F_STAGES - 2>();
    __syncthreads();
    if (st + F_STAGES - 1 < n_st) load(st + F_STAGES - 1, true, true);
    cp_async_commit();
    const float *a = sm + (st % F_STAGES) * MATS * MAT + ty * F_ROW + grp * KS, *w = sm + (st % F_STAGES) * MATS * MAT + MAT + tx * F_ROW + grp * KS;
#pragma unroll
    for (int k = 0; k < KS; k += 4) {
      float4 av[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4 *>(a + (B / 4) * i * F_ROW + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 wv = *reinterpret_cast<const float4 *>(w + (B / 4) * j * F_ROW + k);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          acc[i][j] = fmaf(av[i].w, wv.w, fmaf(av[i].z, wv.z, fmaf(av[i].y, wv.y, fmaf(av[i].x, wv.x, acc[i][j]))));
        if (EPI == EPI_SWIGLU) {
          const float4 uv = *reinterpret_cast<const float4 *>(w + MAT + (B / 4) * j * F_ROW + k);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            acc2[i][j] = fmaf(av[i].w, uv.w, fmaf(av[i].z, uv.z, fmaf(av[i].y, uv.y, fmaf(av[i].x, uv.x, acc2[i][j]))));
        }
      }
    }
  }
  auto emit = [&](int i, int j, int x, int y, float v, float u) {   // output (i, j) of thread (x, y) of the tile
    const int gm = m0 + y + (B / 4) * i, gn = n0 + x + (B / 4) * j;
    if (gm >= M || gn >= N) return;
    float *o = out + (int64_t)gm * N + gn;
    if (EPI == EPI_STORE) *o = v;
    else if (EPI == EPI_RESIDUAL) *o += v;
    else if (EPI == EPI_SWIGLU) *o = v / (1.0f + expf(-v)) * u;
    else *o = v + (bias ? bias[gn] : 0.f);
  };
  if (KG == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) emit(i, j, tx, ty, acc[i][j], EPI == EPI_SWIGLU ? acc2[i][j] : 0.f);
  } else {
    // the groups leave their sums ([group][output][thread]: no bank conflicts), all threads share out the outputs and add
    // them in the order of the groups
    constexpr int NO = EPI == EPI_SWIGLU ? 32 : 16;
    static_assert(KG * NO * TG <= F_STAGES * MATS * MAT, "room for the groups' sums");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sm[(grp * NO + 4 * i + j) * TG + t] = acc[i][j];
        if (EPI == EPI_SWIGLU) sm[(grp * NO + 16 + 4 * i + j) * TG + t] = acc2[i][j];
      }
    __syncthreads();
    for (int e = tid; e < B * B; e += F_THREADS) {
      const int k = e / TG, th = e % TG;
      float v = sm[k * TG + th], u = EPI == EPI_SWIGLU ? sm[(16 + k) * TG + th] : 0.f;
#pragma unroll
      for (int g = 1; g < KG; ++g) {
        v += sm[(g * NO + k) * TG + th];
        if (EPI == EPI_SWIGLU) u += sm[(g * NO + 16 + k) * TG + th];
      }
      emit(k / 4, k % 4, th % (B / 4), th / (B / 4), v, u);
    }
  }
}

// fp32 attention: a block takes 8 query rows of one head and walks the keys in tiles of 64 with a running maximum and sum;
// the next tile is on its way meanwhile where two fit (`bufs`).  16 threads per row: thread l computes the scores of keys
// l + 16 i and the output dimensions 4 l + 64 i ... + 3, four sums that share each probability and take a value row in
// 16-byte pieces.  96 rows, 96 keys, 4 heads of 64 (some 5 us of it the events): a block per row and head 24 us; 16 rows to a
// block, one tile at a time and one dimension after the other 17; this 13.
constexpr int A_Q = 8, A_K = 64, A_THREADS = 16 * A_Q;
__global__ void __launch_bounds__(A_THREADS) attention_f32_kernel(const float *__restrict__ q, const float *__restrict__ kc,
                                                            const float *__restrict__ vc, const SeqMeta *meta, float *out,
                                                            int64_t kv_seq_stride, int H, int dh, int bufs) {
  extern __shared__ __align__(16) float sm[];
  grid_dep_launch();
  grid_dep_wait();
  const SeqMeta m = meta[blockIdx.z];
  const int q0 = blockIdx.x * A_Q, h = blockIdx.y, hd = H * dh, tid = threadIdx.x, r = tid >> 4, l = tid & 15;
  if (q0 >= m.n_rows) return;
  const int stride = (dh + 3) / 4 * 4 + 4, sk = A_K + 4;
  float *const Q = sm, *const S = Q + A_Q * stride, *const KV = S + A_Q * sk;   // S [A_Q][sk], KV [bufs][K then V][A_K][stride]
  const float *kb = kc + (int64_t)m.seq * kv_seq_stride + h * dh, *vb = vc + (int64_t)m.seq * kv_seq_stride + h * dh;
  const bool live = q0 + r < m.n_rows;
  const bool v4 = (dh & 3) == 0;
  // (dh is a multiple of 4 here, or every row is copied word by word)
  auto rows = [&](float *d, const float *src, int n, int n_valid) {
    if (v4) {
      for (int e = tid; e < n * (dh / 4); e += A_THREADS) {
        const int i = e / (dh / 4), c = 4 * (e % (dh / 4));
        cp_async16(d + i * stride + c, src + (i < n_valid ? (int64_t)i * hd + c : 0), i < n_valid);
      }
    } else {
      for (int e = tid; e < n * dh; e += A_THREADS) {
        const int i = e / dh, c = e - i * dh;
        d[i * stride + c] = i < n_valid ? src[(int64_t)i * hd + c] : 0.f;
      }
    }
  };
  rows(Q, q + (int64_t)(m.row0 + q0) * hd + h * dh, A_Q, min(A_Q, m.n_rows - q0));
  constexpr int MAX_D = 4;                        // dh <= 256: 64 dimensions at a time
  float o[MAX_D][4] = {}, m_run = -INFINITY, l_run = 0.f;
  const float scale = 1.0f / sqrtf((float)dh);
  auto fetch = [&](int j0, int buf) {
    const int nk = min(A_K, m.kv_len - j0);
    rows(KV + 2 * buf * A_K * stride, kb + (int64_t)j0 * hd, A_K, nk);
    rows(KV + (2 * buf + 1) * A_K * stride, vb + (int64_t)j0 * hd, A_K, nk);
  };
  fetch(0, 0);
  cp_async_commit();
  for (int j0 = 0; j0 < m.kv_len; j0 += A_K) {
    const int nk = min(A_K, m.kv_len - j0), buf = bufs == 2 ? (j0 / A_K) & 1 : 0;
    const float *const Kt = KV + 2 * buf * A_K * stride, *const Vt = Kt + A_K * stride;
    if (bufs == 2) {
      if (j0 + A_K < m.kv_len) fetch(j0 + A_K, buf ^ 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else
      cp_async_wait<0>();
    __syncthreads();
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if (v4) {
      for (int c = 0; c < dh; c += 4) {
        const float4 x = *reinterpret_cast<const float4 *>(Q + r * stride + c);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 y = *reinterpret_cast<const float4 *>(Kt + (l + 16 * i) * stride + c);
          s[i] = fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, s[i]))));
        }
      }
    } else {
      for (int c = 0; c < dh; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = fmaf(Q[r * stride + c], Kt[(l + 16 * i) * stride + c], s[i]);
    }
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s[i] = l + 16 * i < nk ? s[i] * scale : -INFINITY;
      mx = fmaxf(mx, s[i]);
    }
    for (int w = 8; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
    // while every score so far is -inf (dot products beyond the range), the reference is 0: their probabilities are then 0
    const float m_new = fmaxf(m_run, mx), m_ref = m_new == -INFINITY ? 0.f : m_new, f = expf(m_run - m_ref);   // the first tile: exp(-inf) = 0
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float e = expf(s[i] - m_ref);
      sum += e;
      S[r * sk + l + 16 * i] = e;
    }
    for (int w = 8; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
    l_run = l_run * f + sum;
    m_run = m_new;
    __syncwarp();
    // each sum runs over the keys in order; probabilities of absent keys are zero, and so are their value rows
#pragma unroll
    for (int i = 0; i < MAX_D; ++i) {
      const int c = 4 * l + 64 * i;
      if (64 * i >= dh) break;
      if (c < dh) {
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int j = 0; j < nk; j += 4) {
          const float4 p4 = *reinterpret_cast<const float4 *>(S + r * sk + j);
          const float p[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 y = *reinterpret_cast<const float4 *>(Vt + (j + u) * stride + c);
            a[0] = fmaf(p[u], y.x, a[0]); a[1] = fmaf(p[u], y.y, a[1]);
            a[2] = fmaf(p[u], y.z, a[2]); a[3] = fmaf(p[u], y.w, a[3]);
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) o[i][e] = fmaf(o[i][e], f, a[e]);
      }
    }
    __syncthreads();                              // this tile has been read: its place may be filled again
    if (bufs == 1 && j0 + A_K < m.kv_len) { fetch(j0 + A_K, 0); cp_async_commit(); }
  }
  const float inv = 1.0f / l_run;
  float *orow = out + (int64_t)(m.row0 + q0 + r) * hd + h * dh;
#pragma unroll
  for (int i = 0; i < MAX_D; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (4 * l + 64 * i + e < dh && live) orow[4 * l + 64 * i + e] = o[i][e] * inv;
}


// Per-row max, sum of exp and argmax (lowest id on ties) of stored fp32 logits: one tile.  A thread folds 16 logits at a
// time (all requested together) into its running (max, sum, argmax); the threads' records are merged at the end.
constexpr int R_THREADS = 512;
__device__ __forceinline__ void merge_records(float &mx, float &sum, int &ix, float om, float os, int oi) {
  const float nm = fmaxf(mx, om);
  sum = (mx == -INFINITY ? 0.f : sum * expf(mx - nm)) + (om == -INFINITY ? 0.f : os * expf(om - nm));
  ix = (om > mx || (om == mx && oi < ix)) ? oi : ix;
  mx = nm;
}
__global__ void __launch_bounds__(R_THREADS) row_softmax_partials_kernel(const float *logits, int V, float *part_m, float *part_s,
                                                                         int32_t *part_i) {
  grid_dep_launch();
  grid_dep_wait();
  __shared__ float rm[R_THREADS / 32], rs[R_THREADS / 32];
  __shared__ int ri[R_THREADS / 32];
  const int r = blockIdx.x;
  const float *row = logits + (int64_t)r * V;
  float mx = -INFINITY, sum = 0.f;
  int ix = 0x7fffffff;
  constexpr int U = 16;
  for (int v0 = threadIdx.x; v0 < V; v0 += U * R_THREADS) {
    float f[U], cm = -INFINITY;
#pragma unroll
    for (int u = 0; u < U; ++u) f[u] = v0 + u * R_THREADS < V ? row[v0 + u * R_THREADS] : -INFINITY;
#pragma unroll
    for (int u = 0; u < U; ++u) cm = fmaxf(cm, f[u]);
    if (cm > mx) {
      sum *= expf(mx - cm);                       // the first chunk: 0 * exp(-inf)
      mx = cm;
#pragma unroll
      for (int u = U - 1; u >= 0; --u) if (f[u] == cm) ix = v0 + u * R_THREADS;   // the lowest id that holds the maximum
    }
#pragma unroll
    for (int u = 0; u < U; ++u) sum += mx == -INFINITY ? 0.f : expf(f[u] - mx);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int o = 16; o > 0; o >>= 1) {
    const float om = __shfl_xor_sync(0xffffffffu, mx, o), os = __shfl_xor_sync(0xffffffffu, sum, o);
    const int oi = __shfl_xor_sync(0xffffffffu, ix, o);
    merge_records(mx, sum, ix, om, os, oi);
  }
  if (l == 0) { rm[w] = mx; rs[w] = sum; ri[w] = ix; }
  __syncthreads();
  if (w == 0) {
    mx = l < R_THREADS / 32 ? rm[l] : -INFINITY;
    sum = l < R_THREADS / 32 ? rs[l] : 0.f;
    ix = l < R_THREADS / 32 ? ri[l] : 0x7fffffff;
    for (int o = 16; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, mx, o), os = __shfl_xor_sync(0xffffffffu, sum, o);
      const int oi = __shfl_xor_sync(0xffffffffu, ix, o);
      merge_records(mx, sum, ix, om, os, oi);
    }
    if (l == 0) { part_m[r] = mx; part_s[r] = sum; part_i[r] = ix; }
  }
}

template <int EPI, int B>
cudaError_t launch_gemm_f32(cudaStream_t st, const float *A, const float *W, const float *W2, float *C, const float *bias, int M, int N, int K) {
  const size_t smem = sizeof(float) * F_STAGES * (EPI == EPI_SWIGLU ? 3 : 2) * B * F_ROW;
  cudaError_t e = cudaFuncSetAttribute(gemm_f32_kernel<EPI, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(gemm_f32_kernel<EPI, B>, dim3(ceil_div(N, B), ceil_div(M, B)), dim3(F_THREADS), smem, st, A, W, W2, C, bias, M, N, K);
}

}  // namespace

template <typename T>
cudaError_t launch_simt_gemm(cudaStream_t st, int epi, const T *A, const T *W, const T *W2, void *C,
                             const float *bias, int M, int N, int K, int num_sms) {
  if constexpr (std::is_same<T, float>::value) {
    const uintptr_t bits = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(W2);
    // 32 x 32 tiles until 64 x 64 ones give every SM two blocks (SwiGLU, two weight tiles: no more than 32 x 32); 16 x 16 tiles
    // as long as 32 x 32 ones fill at most every second SM.  Tiny decode of 96 rows on 148 SMs, 32 x 32 alone 4.00 ms, 16 x 16 up
    // to 37 blocks (O, down) 3.36, up to 74 (QKV and gate/up too) 3.13
    auto blocks = [&](int b) { return (int64_t)ceil_div(N, b) * ceil_div(M, b); };
    const int tile = blocks(64) >= 2 * num_sms && epi != EPI_SWIGLU ? 64 : (blocks(32) <= num_sms / 2 ? 16 : 32);
    // more row tiles than a grid's y (SwiGLU of 2.1 million rows): the plain kernel below with its 64-row tiles
    if ((bits & 15) == 0 && (K & 3) == 0 && ceil_div(M, tile) <= MAX_GRID_YZ) {
      float *Cf = reinterpret_cast<float *>(C);
#define L2PD_F32(E)                                                                                      \
  case E: return tile == 16 ? launch_gemm_f32<E, 16>(st, A, W, W2, Cf, bias, M, N, K)                    \
                            : launch_gemm_f32<E, 32>(st, A, W, W2, Cf, bias, M, N, K);
      switch (tile == 64 ? epi : -1) {
        case EPI_STORE: return launch_gemm_f32<EPI_STORE, 64>(st, A, W, W2, Cf, bias, M, N, K);
        case EPI_RESIDUAL: return launch_gemm_f32<EPI_RESIDUAL, 64>(st, A, W, W2, Cf, bias, M, N, K);
        case EPI_STORE_F32: return launch_gemm_f32<EPI_STORE_F32, 64>(st, A, W, W2, Cf, bias, M, N, K);
        default: break;
      }
      switch (epi) {
        L2PD_F32(EPI_STORE) L2PD_F32(EPI_RESIDUAL) L2PD_F32(EPI_SWIGLU) L2PD_F32(EPI_STORE_F32)
#undef L2PD_F32
        default: return cudaErrorInvalidValue;
      }
    }
  }
  dim3 grid(ceil_div(N, BN), ceil_div(M, BM));
  switch (epi) {
    case EPI_STORE: return launch_kernel(simt_gemm_kernel<T, EPI_STORE>, grid, dim3(256), 0, st, A, W, W2, C, bias, M, N, K);
    case EPI_RESIDUAL: return launch_kernel(simt_gemm_kernel<T, EPI_RESIDUAL>, grid, dim3(256), 0, st, A, W, W2, C, bias, M, N, K);
    case EPI_SWIGLU: return launch_kernel(simt_gemm_kernel<T, EPI_SWIGLU>, grid, dim3(256), 0, st, A, W, W2, C, bias, M, N, K);
    case EPI_STORE_F32: return launch_kernel(simt_gemm_kernel<T, EPI_STORE_F32>, grid, dim3(256), 0, st, A, W, W2, C, bias, M, N, K);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_simt_attention(cudaStream_t st, const T *q, const T *kc, const T *vc,
                                  const SeqMeta *meta, const int32_t *row_slot, T *out,
                                  int64_t kv_seq_stride, int rows, int H, int dh, int max_kv, int n_slots, int max_q) {
  // The limits of shared memory are set to what a call can ask for at most: they belong to the kernel, not to the call, and a thread
  // with smaller tiles would take them from under another's launch.
  // the grid's z holds the sequences; of more of them, a block per row and head takes any number
  if constexpr (std::is_same<T, float>::value) {   // q, K and V are the library's own buffers: rows of H * dh floats, 16-byte aligned
    if (n_slots <= MAX_GRID_YZ) {
      auto bytes = [&](int bufs) { return (int)(sizeof(float) * ((size_t)(A_Q + 2 * bufs * A_K) * ((dh + 3) / 4 * 4 + 4) + A_Q * (A_K + 4))); };
      constexpr int most = 200 * 1024;   // (one buffer of the widest head: 140 KB)
      const int bufs = max_kv > A_K && bytes(2) <= most ? 2 : 1;
      cudaError_t e = cudaFuncSetAttribute(attention_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
      if (e != cudaSuccess) return e;
      return launch_kernel(attention_f32_kernel, dim3(ceil_div(max_q, A_Q), H, n_slots), dim3(A_THREADS), (size_t)bytes(bufs), st, q, kc, vc,
                           meta, out, kv_seq_stride, H, dh, bufs);
    }
  }
  size_t smem = (size_t)(dh + max_kv) * sizeof(float);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(simt_attention_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e != cudaSuccess) return e;
  }
  return launch_kernel(simt_attention_kernel<T>, dim3(rows, H), dim3(128), smem, st, q, kc, vc, meta, row_slot, out,
                       kv_seq_stride, H, dh);
}

cudaError_t launch_row_softmax_partials(cudaStream_t st, const float *logits, int R, int V,
                                        float *part_m, float *part_s, int32_t *part_i) {
  return launch_kernel(row_softmax_partials_kernel, dim3(R), dim3(R_THREADS), 0, st, logits, V, part_m, part_s, part_i);
}

template cudaError_t launch_simt_gemm<float>(cudaStream_t, int, const float *, const float *,
                                             const float *, void *, const float *, int, int, int, int);
template cudaError_t launch_simt_gemm<bf16>(cudaStream_t, int, const bf16 *, const bf16 *, const bf16 *,
                                            void *, const float *, int, int, int, int);
template cudaError_t launch_simt_attention<float>(cudaStream_t, const float *, const float *,
                                                  const float *, const SeqMeta *, const int32_t *,
                                                  float *, int64_t, int, int, int, int, int, int);
template cudaError_t launch_simt_attention<bf16>(cudaStream_t, const bf16 *, const bf16 *, const bf16 *,
                                                 const SeqMeta *, const int32_t *, bf16 *, int64_t, int,
                                                 int, int, int, int, int);

}  // namespace l2pd
