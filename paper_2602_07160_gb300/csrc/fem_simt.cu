// The FEM read on CUDA cores, exact to fp32 rounding: fp32 inputs of any head
// dimension up to 256, and bf16 inputs of head dimension 16 or 32 (too narrow
// for the tensor-core read's 64-channel tiles to pay; here every product and
// sum is fp32).  fem_row_kernel runs few short rows, the tiles of
// fem_f32_tile.cu longer sequences (use_tile below), fem_simt_kernel the rest:
// many short rows, and d > 128.
//
// fem_simt_kernel: one warp per output row t, four consecutive rows of one (b, h) per block;
// lane l owns channels l, l+32, ...  The block stages the keys' K and V rows
// in shared memory, a tile of fem_simt_tile(d) keys at a time (as fp32), so the
// walk below reads them with shared-memory latency.  For every key
// i in the support the warp forms s_{t,i} = q_t . k_i / sqrt(d) (lane-partial
// dot product, butterfly sum) and folds key i into
//   L   = sum_i P_i,                          P_i = exp(s_i - m)
//   A_j = sum_i P_i exp(beta_j (v_ij - c_j))
//   W_j = sum_i P_i expm1(beta_j (v_ij - c_j)) / beta_j   (v_ij - c_j at beta 0)
// with a running row maximum m and an exact running per-channel maximum c_j
// of the visible values (the per-channel stabilisation of App. E, per row).
// When m grows by dm, L, A and W scale by exp(-dm); when c_j grows to c',
// with r = exp(beta (c - c')), A <- r A and W <- r W + expm1(beta (c - c'))/beta L
// (the joint rescale of the two running shifts).  The read is then
//   o = c + log1p(beta W / L) / beta   when beta W / L > -1/2 (no cancellation),
//   o = c + log(A / L) / beta          otherwise,
//   o = c + W / L                      at beta = 0 (the prior mean),
// which is (1/beta) log sum_i p_t(i) exp(beta v_ij) (Sec. 2.3).  An A / L below kSumGuard or not finite
// (fp32's range could then hide terms that count: the largest value under a tiny weight) is summed again
// around the largest s_i + beta v_i.
#include "fem_common.cuh"
#include "fem_launch.h"

namespace fem {

constexpr int kSimtMaxPerLane = 8;  // d <= 256

constexpr float kSumGuard = 0x1p-84f;

// rows up to which a row gets a block of its own (its keys split over the warps)
constexpr long long kSimtSplitRows = 2048;

// keys per staged tile: K and V of a tile take 32 KB at most (8 KB at d = 16)
inline __host__ __device__ int fem_simt_tile(int d) {
  const int kt = 4096 / d;
  return kt > 64 ? 64 : (kt < 8 ? 8 : kt);
}

__device__ __forceinline__ float expm1_over_beta(float b, float x) {
  // expm1(b x) / b, continuous at b = 0
  return b != 0.f ? expm1f(b * x) / b : x;
}

__device__ __forceinline__ float ld_in(const float *p) { return *p; }
__device__ __forceinline__ float ld_in(const __nv_bfloat16 *p) { return __bfloat162float(*p); }

// The warp's row again for the channel slots of `redo` (a mask per lane): the keys in turn, first for the
// largest s_i + beta v_i, then for the sum around it.
template <typename In, int PER>
__device__ __noinline__ void simt_exact(const In *qr, const In *kb, const In *vb, const float *beta, int n, int d,
                                        float m, float L, unsigned redo, float *orow) {
  const int lane = threadIdx.x & 31;
  const float inv_sqrt_d = rsqrtf(static_cast<float>(d));
  float top[PER], sum[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    top[u] = -INFINITY;
    sum[u] = 0.f;
  }
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = 0; i < n; ++i) {
      const In *kr = kb + static_cast<long long>(i) * d, *vr = vb + static_cast<long long>(i) * d;
      float s = 0.f;
      for (int j = lane; j < d; j += 32) s = fmaf(ld_in(qr + j), ld_in(kr + j), s);
#pragma unroll
      for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      s *= inv_sqrt_d;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        if (!((redo >> u) & 1u)) continue;
        const int j = lane + 32 * u;
        const float y = fmaf(beta[j], ld_in(vr + j), s);
        if (pass == 0)
          top[u] = fmaxf(top[u], y);
        else
          sum[u] += expf(y - top[u]);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = lane + 32 * u;
    if ((redo >> u) & 1u) orow[j] = ((top[u] - m) + (logf(sum[u]) - logf(L))) / beta[j];
  }
}

// PER: channel slots per lane, d <= 32 PER (the unrolled per-slot code costs
// issue slots even where a slot is empty).  SPLIT (few rows): one row per
// block, each warp folding a quarter of every staged tile's keys from an empty
// state, the four states merged at the end (each scaled to the common row
// maximum, each channel's moved to the larger shift as when a key raises it),
// so that a row's dependent chain is a quarter as long.
template <typename In, int PER, bool SPLIT>
__global__ void __launch_bounds__(128) fem_simt_kernel(const In *__restrict__ q, const In *__restrict__ k,
                                                        const In *__restrict__ v, const float *__restrict__ beta,
                                                        float *__restrict__ out, float *__restrict__ lse, int H,
                                                        int T, int d, int causal) {
  extern __shared__ float simt_smem[];  // [tile][d] K, then [tile][d] V
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bpr = SPLIT ? T : (T + 3) / 4;  // blocks per (b, h)
  const long long bh = blockIdx.x / bpr;
  const int t0 = static_cast<int>(blockIdx.x % bpr) * (SPLIT ? 1 : 4), t = SPLIT ? t0 : t0 + warp;
  const bool valid = t < T;
  const long long row = bh * T + t;
  const int h = static_cast<int>(bh % H);
  const int n = !valid ? 0 : (causal ? t + 1 : T);                // keys this row sees
  const int n_blk = SPLIT ? n : (causal ? min(T, t0 + 4) : T);    // keys any row of the block sees
  const int per = (d + 31) / 32;  // <= PER
  const int tile = fem_simt_tile(d);
  const float inv_sqrt_d = rsqrtf(static_cast<float>(d));
  const In *kb = k + bh * T * d;
  const In *vb = v + bh * T * d;
  float *sk = simt_smem, *sv = simt_smem + tile * d;

  float qv[PER], bj[PER], c[PER], A[PER], W[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = lane + 32 * u;
    const bool ok = valid && u < per && j < d;
    qv[u] = ok ? ld_in(q + row * d + j) : 0.f;
    bj[u] = ok ? normal_beta(beta[h * d + j]) : 0.f;
    c[u] = -INFINITY;
    A[u] = 0.f;
    W[u] = 0.f;
  }
  float m = -INFINITY, L = 0.f;

  for (int i0 = 0; i0 < n_blk; i0 += tile) {
    const int nt = min(tile, n_blk - i0);
    __syncthreads();  // the previous tile is consumed
    for (int e = tid; e < nt * d; e += 128) {
      sk[e] = ld_in(kb + static_cast<long long>(i0) * d + e);
      sv[e] = ld_in(vb + static_cast<long long>(i0) * d + e);
    }
    __syncthreads();
    const int n_here = min(nt, n - i0);  // this row's keys in the tile
    // SPLIT: this warp's quarter of them
    const int quarter = (n_here + 3) / 4;
    const int ii0 = SPLIT ? min(n_here, warp * quarter) : 0, ii1 = SPLIT ? min(n_here, ii0 + quarter) : n_here;
    for (int ii = ii0; ii < ii1; ++ii) {
      const float *kr = sk + ii * d;
      float part = 0.f;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = lane + 32 * u;
        if (u < per && j < d) part = fmaf(qv[u], kr[j], part);
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
      const float s = part * inv_sqrt_d;
      if (s > m) {
        const float alpha = expf(m - s);  // 0 when m = -inf
        L *= alpha;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          A[u] *= alpha;
          W[u] *= alpha;
        }
        m = s;
      }
      const float p = expf(s - m);
      const float *vr = sv + ii * d;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = lane + 32 * u;
        if (!(u < per && j < d)) continue;
        const float x = vr[j];
        const float b = bj[u];
        if (x > c[u]) {
          if (c[u] != -INFINITY) {
            const float r = expf(b * (c[u] - x));
            W[u] = r * W[u] + expm1_over_beta(b, c[u] - x) * L;
            A[u] *= r;
          }
          c[u] = x;
        }
        A[u] += p * expf(b * (x - c[u]));
        W[u] += p * expm1_over_beta(b, x - c[u]);
      }
      L += p;
    }
  }
  if (SPLIT) {
    // warps 1..3 leave their states in shared memory (m, L, then c, A, W per channel); warp 0
    // folds them into its own in key order
    __syncthreads();  // the last tile is consumed
    float *st = simt_smem + (warp - 1) * (2 + 3 * d);
    if (warp > 0) {
      if (lane == 0) {
        st[0] = m;
        st[1] = L;
      }
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = lane + 32 * u;
        if (!(u < per && j < d)) continue;
        st[2 + j] = c[u];
        st[2 + d + j] = A[u];
        st[2 + 2 * d + j] = W[u];
      }
    }
    __syncthreads();
    if (warp > 0) return;
    for (int w = 1; w < 4; ++w) {
      const float *sw = simt_smem + (w - 1) * (2 + 3 * d);
      const float m2 = sw[0], L2 = sw[1];
      if (m2 == -INFINITY) continue;  // a warp that saw no key
      if (m == -INFINITY) {           // this one saw none: take the other state
        m = m2;
        L = L2;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int j = lane + 32 * u;
          if (!(u < per && j < d)) continue;
          c[u] = sw[2 + j];
          A[u] = sw[2 + d + j];
          W[u] = sw[2 + 2 * d + j];
        }
        continue;
      }
      const float mn = fmaxf(m, m2), a1 = expf(m - mn), a2 = expf(m2 - mn);
      const float L1 = L * a1, Ls = L2 * a2;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = lane + 32 * u;
        if (!(u < per && j < d)) continue;
        const float b = bj[u], c2 = sw[2 + j];
        float A1 = A[u] * a1, W1 = W[u] * a1, A2 = sw[2 + d + j] * a2, W2 = sw[2 + 2 * d + j] * a2;
        if (c2 > c[u]) {
          const float r = expf(b * (c[u] - c2));
          W1 = r * W1 + expm1_over_beta(b, c[u] - c2) * L1;
          A1 *= r;
          c[u] = c2;
        } else if (c2 < c[u]) {
          const float r = expf(b * (c2 - c[u]));
          W2 = r * W2 + expm1_over_beta(b, c2 - c[u]) * Ls;
          A2 *= r;
        }
        A[u] = A1 + A2;
        W[u] = W1 + W2;
      }
      L = L1 + Ls;
      m = mn;
    }
  }
  if (!valid) return;

  unsigned redo = 0;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = lane + 32 * u;
    if (!(u < per && j < d)) continue;
    const float b = bj[u];
    float o;
    if (b == 0.f) {
      o = c[u] + W[u] / L;
    } else {
      const float z = b * W[u] / L, r = A[u] / L;
      o = z > -0.5f ? c[u] + log1pf(z) / b : c[u] + logf(r) / b;
      if (!(z > -0.5f) && !(r >= kSumGuard && r < INFINITY)) redo |= 1u << u;
    }
    if (!((redo >> u) & 1u)) out[row * d + j] = o;
  }
  if (__any_sync(0xffffffffu, redo != 0u))
    simt_exact<In, PER>(q + row * d, kb, vb, beta + static_cast<size_t>(h) * d, n, d, m, L, redo, out + row * d);
  if (lse && lane == 0) lse[row] = m + logf(L);
}

// Few rows of few keys: a block per row with every visible key in shared memory, so that nothing is
// folded in turn.  Thread = key for the scores (K padded by one float a row: no bank conflicts), then
// thread = channel j and key group g (C channels, 128 / C groups): the channel's largest value, then
// sums at it over the group's keys, the groups combined through shared memory.
//   L = sum_i P_i,  A_j = sum_i P_i exp(beta_j (v_ij - c_j)),  X_j = sum_i P_i expm1(beta_j (v_ij - c_j))
// (X of the plain differences at beta = 0), read as above with X = beta W, a rejected A / L summed again
// likewise.  What bounds it is latency: one
// round of loads, two block reductions and a group's exponentials.  us in a graph, four warps folding key
// after key / this: B1 H1 T64 d16 12.5 / 4.9, B1 H1 T40 d128 26.9 / 9.4, B4 H8 T47 d64 32.1 / 14.3, B16 H4
// T30 d128 49.7 / 21.0, B1 H1 T5 d16 3.8 / 3.2.
constexpr int kRowThreads = 128, kRowMaxKeys = 128;
constexpr size_t kRowSmem = 48 * 1024 - 4096;  // beside the static arrays, without an opt-in

__host__ __device__ inline size_t row_floats(int T, int d) { return static_cast<size_t>(T) * (2 * d + 1) + d; }

static bool row_fits(long long rows, int T, int d) {
  return rows <= kSimtSplitRows && T <= kRowMaxKeys && row_floats(T, d) * sizeof(float) <= kRowSmem;
}

template <typename In>
__global__ void __launch_bounds__(kRowThreads) fem_row_kernel(const In *__restrict__ q, const In *__restrict__ k,
                                                               const In *__restrict__ v,
                                                               const float *__restrict__ beta, float *__restrict__ out,
                                                               float *__restrict__ lse, int H, int T, int d, int C,
                                                               int causal) {
  extern __shared__ float simt_smem[];
  __shared__ float s_p[kRowMaxKeys], s_s[kRowMaxKeys], s_red[2][4], s_g[3][kRowThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long row = blockIdx.x, bh = row / T;
  const int t = static_cast<int>(row % T), n = causal ? t + 1 : T, ldk = d + 1;
  float *sk = simt_smem, *sv = sk + n * ldk, *sq = sv + n * d;
  const In *kb = k + bh * T * d, *vb = v + bh * T * d;
  for (int e = tid; e < n * d; e += kRowThreads) {
    const int i = e / d;
    sk[e + i] = ld_in(kb + e);
    sv[e] = ld_in(vb + e);
  }
  for (int e = tid; e < d; e += kRowThreads) sq[e] = ld_in(q + row * d + e);
  __syncthreads();
  // ---- scores, their maximum, P and its sum
  float s = -INFINITY;
  if (tid < n) {
    const float *kr = sk + tid * ldk;
    float s0 = 0.f, s1 = 0.f;
    int e = 0;
#pragma unroll 4
    for (; e + 1 < d; e += 2) {
      s0 = fmaf(sq[e], kr[e], s0);
      s1 = fmaf(sq[e + 1], kr[e + 1], s1);
    }
    if (e < d) s0 = fmaf(sq[e], kr[e], s0);
    s = (s0 + s1) * rsqrtf(static_cast<float>(d));
  }
  float m = s;
#pragma unroll
  for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if (lane == 0) s_red[0][warp] = m;
  __syncthreads();
  m = fmaxf(fmaxf(s_red[0][0], s_red[0][1]), fmaxf(s_red[0][2], s_red[0][3]));
  float p = tid < n ? expf(s - m) : 0.f;
  s_p[tid] = p;
  s_s[tid] = s;
#pragma unroll
  for (int off = 16; off; off >>= 1) p += __shfl_xor_sync(0xffffffffu, p, off);
  if (lane == 0) s_red[1][warp] = p;
  // ---- channels, C at a time
  const int G = kRowThreads / C, jl = tid % C, g = tid / C, h = static_cast<int>(bh % H);
  for (int j0 = 0; j0 < d; j0 += C) {
    const int j = j0 + jl;
    const bool on = j < d;
    const float b = on ? normal_beta(beta[static_cast<size_t>(h) * d + j]) : 0.f;
    float c = -INFINITY;
    if (on) {
#pragma unroll 4
      for (int i = g; i < n; i += G) c = fmaxf(c, sv[i * d + j]);
    }
    s_g[0][tid] = c;
    __syncthreads();  // also: P and its partial sums
    for (int u = 0; u < G; ++u) c = fmaxf(c, s_g[0][u * C + jl]);
    float A = 0.f, X = 0.f;
    if (on) {
#pragma unroll 4
      for (int i = g; i < n; i += G) {
        const float x = sv[i * d + j] - c, y = b * x, pi = s_p[i];
        A = fmaf(pi, expf(y), A);
        X = fmaf(pi, b != 0.f ? expm1f(y) : x, X);
      }
    }
    s_g[1][tid] = A;
    s_g[2][tid] = X;
    __syncthreads();
    const float L = (s_red[1][0] + s_red[1][1]) + (s_red[1][2] + s_red[1][3]);
    if (g == 0 && on) {
      for (int u = 1; u < G; ++u) {
        A += s_g[1][u * C + jl];
        X += s_g[2][u * C + jl];
      }
      const float z = X / L, r = A / L;
      float o = b == 0.f ? c + z : z > -0.5f ? c + log1pf(z) / b : c + logf(r) / b;
      if (b != 0.f && !(z > -0.5f) && !(r >= kSumGuard && r < INFINITY)) {
        float top = -INFINITY, sum = 0.f;
        for (int i = 0; i < n; ++i) top = fmaxf(top, fmaf(b, sv[i * d + j], s_s[i]));
        for (int i = 0; i < n; ++i) sum += expf(fmaf(b, sv[i * d + j], s_s[i]) - top);
        o = ((top - m) + (logf(sum) - logf(L))) / b;
      }
      out[row * d + j] = o;
    }
    if (j0 == 0 && tid == 0 && lse) lse[row] = m + logf(L);
  }
}

template <typename In>
static cudaError_t launch_simt(const In *q, const In *k, const In *v, const float *beta, float *out, float *lse, int B,
                               int H, int T, int d, int causal, cudaStream_t stream) {
  if (d > 32 * kSimtMaxPerLane) return cudaErrorInvalidValue;
  // few rows: a block per row, its keys split over the four warps (the merge area of three
  // states fits in the staging space: 3 (2 + 3 d) <= 2 tile d floats)
  const long long rows = static_cast<long long>(B) * H * T;
  const bool split = rows <= kSimtSplitRows;
  if (row_fits(rows, T, d)) {
    int C = 16;
    while (C < d && C < kRowThreads) C *= 2;
    fem_row_kernel<In><<<static_cast<unsigned>(rows), kRowThreads, row_floats(T, d) * sizeof(float), stream>>>(
        q, k, v, beta, out, lse, H, T, d, C, causal);
    return cudaGetLastError();
  }
  const unsigned blocks = static_cast<unsigned>(split ? rows : static_cast<long long>(B) * H * ((T + 3) / 4));
  const size_t smem = 2 * static_cast<size_t>(fem_simt_tile(d)) * d * sizeof(float);
  const int per = (d + 31) / 32;
#define FEM_SIMT_LAUNCH(P)                                                                                          \
  (split ? fem_simt_kernel<In, P, true><<<blocks, 128, smem, stream>>>(q, k, v, beta, out, lse, H, T, d, causal)     \
         : fem_simt_kernel<In, P, false><<<blocks, 128, smem, stream>>>(q, k, v, beta, out, lse, H, T, d, causal))
  if (per == 1)
    FEM_SIMT_LAUNCH(1);
  else if (per == 2)
    FEM_SIMT_LAUNCH(2);
  else if (per <= 4)
    FEM_SIMT_LAUNCH(4);
  else
    FEM_SIMT_LAUNCH(8);
#undef FEM_SIMT_LAUNCH
  return cudaGetLastError();
}

// The tiled kernel (fem_f32_tile.cu) takes d up to max_d from 80 keys on, from 48 at d > 32 and from
// 32 with at least 64 (b, h): its time hardly depends on the rows of a tile, this file's grows with
// every row and key.  Measured, this kernel / the tiled one, causal, us: B*H = 1, d = 16: T 32 9.2 /
// 12.5, T 64 13.3 / 12.5, T 96 18.2 / 14; B*H = 1, d = 64: T 32 13.7 / 13.7, T 64 22.2 / 15.9;
// B*H = 16, d = 128: T 64 58.7 / 34.8; B*H = 64, d = 16: T 16 8.5 / 11, T 32 16.9 / 12; B*H = 384,
// d = 64: T 8 14.6 / 36, T 32 103 / 37; B*H = 4, d = 64, T 2048: 2468 / 174.  bf16, B*H = 16, d = 32,
// T 1024: 1271 / 56.
// Before it, fem_row_kernel while all rows' keys and channels (the whole square) are 4 M at most: that
// kernel / the tiled one, us in a graph: B*H = 1 T 80 d 16 4.7 / 13.5, T 80 d 64 9.0 / 18.4; B*H = 4 T 128
// d 16 6.7 / 14.0; B*H = 8 T 100 d 32 10.1 / 12.7; B*H = 16 T 128 d 16 (4.2 M) 13.9 / 13.9; beyond, B*H = 32
// T 64 d 64 21.9 / 17.3, B*H = 16 T 128 d 32 21.3 / 12.9.
constexpr long long kRowWork = 1ll << 22;

static bool use_tile(int B, int H, int T, int d, int max_d) {
  const long long rows = static_cast<long long>(B) * H * T;
  if (row_fits(rows, T, d) && rows * T * d <= kRowWork) return false;
  const bool long_enough = T >= 80 || (T >= 48 && d > 32) || (T >= 32 && static_cast<long long>(B) * H >= 64);
  return d <= max_d && long_enough && T <= kTileMaxT;
}

cudaError_t launch_f32(const float *q, const float *k, const float *v, const float *beta, float *out, float *lse,
                       int B, int H, int T, int d, int causal, cudaStream_t stream) {
  if (use_tile(B, H, T, d, 128)) return launch_tile_f32(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
  return launch_simt<float>(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
}

cudaError_t launch_simt_bf16(const void *q, const void *k, const void *v, const float *beta, float *out, float *lse,
                             int B, int H, int T, int d, int causal, cudaStream_t stream) {
  if (use_tile(B, H, T, d, 32)) return launch_tile_bf16(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
  return launch_simt<__nv_bfloat16>(static_cast<const __nv_bfloat16 *>(q), static_cast<const __nv_bfloat16 *>(k),
                                    static_cast<const __nv_bfloat16 *>(v), beta, out, lse, B, H, T, d, causal, stream);
}

}  // namespace fem
