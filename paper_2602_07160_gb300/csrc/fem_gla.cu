// FEM read over a gated-linear-attention prior (App. "Gated Linear Attention
// (GLA) Prior"): with nonnegative features qf, kf (the caller's
// ReLU(RoPE(.)) + eps) and per-step log-decays g_t <= 0,
//
//   s_t(i) = K_{t,i} <qf_t, kf_i>  (i <= t),  K_{t,i} = exp(g_{i+1} + ... + g_t),
//   p_t = s_t / Z_t,   o_{t,j} = (1/beta_j) log sum_i p_t(i) exp(beta_j v_{i,j}).
//
// The associative form (Eq. "gla-assoc") turns every channel into a linear-
// attention state: o_{t,j} = (1/beta_j) log(<qf_t, S_{t,j}> / <qf_t, S_t>)
// with S_{t,j} = sum_{i<=t} K_{t,i} kf_i exp(beta_j v_{i,j}), and the
// normaliser Z_t = <qf_t, S_t>, S_t = sum_i K_{t,i} kf_i, is the same state for
// a constant channel (the paper's "constant 1 channel").  At beta_j = 0 the
// state carries v itself and o is the ratio (the prior mean).
//
// So is a channel whose beta is below kGlaSmallBeta and whose values stay within kGlaSmallTilt / beta: its
// state carries expm1(beta v) / beta and o is log1p(beta ratio) / beta, since the two logarithms' rounding
// (some 5e-7) over beta would be 0.5 at beta = 1e-6.  Its beta goes negated through the kernels, as the
// first launch that meets it leaves it (above kOwnForm chunks a launch of its own, 2.5 us where no beta is that
// small).
//
// In chunks of 64 steps, with gamma_t the running sum of g in the chunk, three
// launches of fp32 contractions on CUDA cores (a lone chunk needs only the last):
//
//   local  U_j = sum_i kf_i exp(gamma_last - gamma_i + beta v_ij - lam'), the chunk's own state
//   scan   the chunks in turn: start states, S' = exp(mu + gamma_last - mu') S + exp(lam' - mu') U
//   out    in_t = sum_{i <= t} K_{t,i} <qf_t, kf_i> exp(beta v_i - lam), ix_t = <qf_t, S>, and the
//          read of in_t e^lam + ix_t e^{mu + gamma_t} over Z_t, zi_t + exp(gamma_t) zx_t likewise
//
// Scales, so that neither exp(beta v) nor the decay under- or overflows (the per-channel
// stabilisation of App. E): lam is the chunk's largest beta v, lam' its largest
// beta v + gamma_last - gamma_i, and a state's log-scale mu the largest of its terms', decaying with
// the prior; the normaliser's is 0.  lam may belong to a key that a row does not see: where in_t is
// below 2^-90 of the row's in-chunk mass, or both parts together of the row's whole mass (fp32's
// range could then hide terms that count), or not finite, the entry is read again around the largest term
// of the keys the row sees, with the start state (read_again, read_rows).  The decay's sums are taken in float64 and kept as
// two floats, so a difference costs the rounding of its own size (steps of -60 are exact to 1e-7);
// steps below kGlaFloor count as it: their weights are zero either way.
//
// What bounds it: instruction issue around the FMA pipe in out (three 64^3 contractions a chunk and
// 64 channels), latency at the ends of a block.  B4 H4 T2048 m64 d128: local 24, scan 18, out 80 us,
// 121 in all, against 331 for a scan that walked segments of the sequence step by step, four lanes to a
// channel's state (passes of 90 and 229 us, one dependent step at a time); B1 H1 T64 25 against 122,
// B4 H16 T512 m16 d32 62 against 79.  Values of ten times unit spread with beta up to 100 send most
// entries to read_again: 354 us at the first size, 406 for the scan.
#include "fem_common.cuh"
#include "fem_f32.cuh"
#include "fem_launch.h"

namespace fem {
namespace {

constexpr int kSteps = 64, kCh = 64;  // steps of a chunk, channels of a block
constexpr int kThreads = 256;         // thread (ty, tx): four rows (or features) against four keys (or channels)
constexpr int kLd = kSteps + 4;       // leading dimension of the transposed Q and K tiles
constexpr float kGlaGuard = 0x1p-90f;
constexpr float kGlaFloor = -1e6f;
constexpr int kFewFlagged = 24;  // threads of a block with flagged entries up to which rows are read one by one
constexpr float kGlaSmallBeta = 0x1p-5f, kGlaSmallTilt = 0.25f;

// Workspace of a group of heads and a run of chunks; per (head, chunk) unless noted.
struct GlaWs {
  float *u;      // [M][dp]: U, then the start state
  float *z;      // [M]: the constant channel's
  float *lam;    // [dp]: U's log-scale
  float *mu;     // [dp]: the start state's
  float *gl;     // the chunk's summed log-decay
  float *carry;  // per head: [M][dp], [M] and [dp], the state (and mu) behind the run's last chunk
  float *eb;     // per head: [dp], beta as form_beta gives it
};

// gam[t] = g_0 + ... + g_t as a float pair (steps past the end add nothing); by warp 0.
__device__ __forceinline__ void chunk_sums(const float *g, int rows, float2 *gam) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    float a = 2 * lane < rows ? g[2 * lane] : 0.f, b = 2 * lane + 1 < rows ? g[2 * lane + 1] : 0.f;
    a = a < kGlaFloor ? kGlaFloor : a;
    b = b < kGlaFloor ? kGlaFloor : b;
    double s = static_cast<double>(a) + static_cast<double>(b);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, s, off);
      if (lane >= off) s += y;
    }
    const double s0 = s - static_cast<double>(b);
    const float h0 = static_cast<float>(s0), h1 = static_cast<float>(s);
    gam[2 * lane] = make_float2(h0, static_cast<float>(s0 - static_cast<double>(h0)));
    gam[2 * lane + 1] = make_float2(h1, static_cast<float>(s - static_cast<double>(h1)));
  }
}
__device__ __forceinline__ float sum_diff(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }

// The largest of x over the 16 row groups, per channel quad (thread = row group tid / 16, quad tid % 16).
__device__ __forceinline__ float4 max_over_rows(float4 x, float4 (*red)[16]) {
  const int q = threadIdx.x & 15;
  red[threadIdx.x >> 4][q] = x;
  __syncthreads();
  float4 m = red[0][q];
#pragma unroll
  for (int p = 1; p < 16; ++p) {
    const float4 y = red[p][q];
    m = make_float4(fmaxf(m.x, y.x), fmaxf(m.y, y.y), fmaxf(m.z, y.z), fmaxf(m.w, y.w));
  }
  return m;
}
// a shift: 0 in place of -inf (no finite value), and for a linear channel
__device__ __forceinline__ float shift_of(float m, float b) { return b > 0.f && m != -INFINITY ? m : 0.f; }

__device__ __forceinline__ float4 beta4(const float *beta, int h, int d, int j) {
  const float *p = beta + static_cast<size_t>(h) * d;
  return make_float4(j < d ? p[j] : 0.f, j + 1 < d ? p[j + 1] : 0.f, j + 2 < d ? p[j + 2] : 0.f, j + 3 < d ? p[j + 3] : 0.f);
}

// beta of a channel whose largest |v| is top: 0 (the mean), negated for the small-beta form, else itself.
__device__ __forceinline__ float form_beta(float b, float top) {
  if (!(b >= 0x1p-126f)) return b == b ? 0.f : b;  // see normal_beta
  return b < kGlaSmallBeta && b * top <= kGlaSmallTilt ? -b : b;
}
__device__ __forceinline__ bool maybe_small(float4 b) {
  return fminf(fminf(b.x > 0.f ? b.x : 1.f, b.y > 0.f ? b.y : 1.f), fminf(b.z > 0.f ? b.z : 1.f, b.w > 0.f ? b.w : 1.f)) <
         kGlaSmallBeta;
}
__device__ __forceinline__ float4 abs_max(float4 a, float4 x) {
  return make_float4(fmaxf(a.x, fabsf(x.x)), fmaxf(a.y, fabsf(x.y)), fmaxf(a.z, fabsf(x.z)), fmaxf(a.w, fabsf(x.w)));
}
__device__ __forceinline__ float4 form_beta4(float4 b, float4 top) {
  return make_float4(form_beta(b.x, top.x), form_beta(b.y, top.y), form_beta(b.z, top.z), form_beta(b.w, top.w));
}

// A value as a linear channel's state carries it: expm1(beta x) / beta for the small-beta form (x times
// the series of expm1(y) / y, |y| <= 1/4), and the read of such a channel's ratio.
__device__ __forceinline__ float lin_value(float b, float x) {
  const float y = -b * x;
  float p = fmaf(y, 1.f / 720.f, 1.f / 120.f);
  p = fmaf(y, p, 1.f / 24.f);
  p = fmaf(y, p, 1.f / 6.f);
  p = fmaf(y, p, 0.5f);
  p = fmaf(y, p, 1.f);
  return b < 0.f ? x * p : x;
}
__device__ __forceinline__ void lin_values(float4 b, float4 (&x)[4]) {
  if (b.x < 0.f || b.y < 0.f || b.z < 0.f || b.w < 0.f) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      x[u] = make_float4(lin_value(b.x, x[u].x), lin_value(b.y, x[u].y), lin_value(b.z, x[u].z), lin_value(b.w, x[u].w));
  }
}
__device__ __noinline__ float small_read(float b, float ratio) { return log1pf(-b * ratio) / -b; }
__device__ __forceinline__ float lin_read(float b, float ratio) { return b < 0.f ? small_read(b, ratio) : ratio; }

// The forms of a block's 64 channels (all threads; a quad each): the sequence's values are read only where some
// beta is small.
__device__ __forceinline__ float4 sequence_forms(const float *beta, const float *vh, int h, int T, int d, int jq, int vec,
                                                 float4 (*red)[16]) {
  const float4 b = beta4(beta, h, d, jq);
  float4 top = make_float4(0.f, 0.f, 0.f, 0.f);
  if (__syncthreads_or(maybe_small(b))) {
#pragma unroll 4
    for (int r = threadIdx.x >> 4; r < T; r += 16) top = abs_max(top, ld_row4(vh + static_cast<size_t>(r) * d, jq, d, vec));
    top = max_over_rows(top, red);
    __syncthreads();  // red is used again
  }
  return form_beta4(b, top);
}

// ---------------------------------------------------------------------------
// form: block per head and 64 channels, for the longer sequences: up to kOwnForm chunks every block of local
// finds the forms itself, which spares the launch and, with a small beta, reads a sequence's values once a chunk.
// ---------------------------------------------------------------------------
constexpr int kOwnForm = 32;
__global__ void __launch_bounds__(kThreads) gla_form_f32_kernel(const float *__restrict__ v, const float *__restrict__ beta,
                                                                int h0, int H, int T, int d, int dp, int vec, GlaWs w) {
  grid_dep_launch_dependents();
  __shared__ float4 red[16][16];
  const int jq = blockIdx.y * kCh + (threadIdx.x & 15) * 4, hd = blockIdx.x;
  const float4 b = sequence_forms(beta, v + static_cast<size_t>(h0 + hd) * T * d, (h0 + hd) % H, T, d, jq, vec, red);
  if (threadIdx.x < 16) *reinterpret_cast<float4 *>(w.eb + static_cast<size_t>(hd) * dp + jq) = b;
}

// ---------------------------------------------------------------------------
// local: block per chunk and 64 channels.
// ---------------------------------------------------------------------------
template <int M>
__global__ void __launch_bounds__(kThreads, 4) gla_local_f32_kernel(const float *__restrict__ kf, const float *__restrict__ v,
                                                                 const float *__restrict__ logdecay,
                                                                 const float *__restrict__ beta, int h0, int H, int T,
                                                                 int d, int dp, int c0, int nb, int vec, GlaWs w) {
  constexpr int RT = M / 16;  // features of a thread
  __shared__ __align__(16) float sK[kSteps * M], sE[kSteps * kCh];
  __shared__ float4 red[16][16];
  __shared__ float2 gam[kSteps];
  __shared__ float s_dg[kSteps], s_z[4][M];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, hd = blockIdx.z, j0 = blockIdx.y * kCh, jq = j0 + tx * 4;
  const int c = c0 + blockIdx.x, rows = min(kSteps, T - c * kSteps);
  const size_t r0 = static_cast<size_t>(h0 + hd) * T + static_cast<size_t>(c) * kSteps;
  const size_t task = static_cast<size_t>(hd) * nb + blockIdx.x;
  float4 x[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = ty + 16 * u;
    x[u] = r < rows ? ld_row4(v + (r0 + r) * d, jq, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < M / 16; ++u) {
    const int i = tid + u * kThreads;  // the chunk's rows of kf are contiguous
    const float4 y = i * 4 < rows * M ? ld4(kf + r0 * M + i * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(sK + i * 4) = y;
  }
  chunk_sums(logdecay + r0, rows, gam);
  __syncthreads();
  if (tid < kSteps) s_dg[tid] = sum_diff(gam[kSteps - 1], gam[tid]);
  if (tid == 0 && blockIdx.y == 0) w.gl[task] = gam[kSteps - 1].x;
  __syncthreads();
  float4 b;
  if (T > kOwnForm * kSteps) {
    grid_dep_wait();  // a dependent launch on the form kernel, which a block's loads overlap
    b = ld4(w.eb + static_cast<size_t>(hd) * dp + jq);
  } else {
    b = sequence_forms(beta, v + static_cast<size_t>(h0 + hd) * T * d, (h0 + hd) % H, T, d, jq, vec, red);
    if (blockIdx.x == 0 && ty == 0) *reinterpret_cast<float4 *>(w.eb + static_cast<size_t>(hd) * dp + jq) = b;
  }
  lin_values(b, x);
  float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  float4 y[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = ty + 16 * u;
    const float g = s_dg[r];
    y[u] = make_float4(fmaf(b.x, x[u].x, g), fmaf(b.y, x[u].y, g), fmaf(b.z, x[u].z, g), fmaf(b.w, x[u].w, g));
    if (r < rows) m = make_float4(fmaxf(m.x, y[u].x), fmaxf(m.y, y[u].y), fmaxf(m.z, y[u].z), fmaxf(m.w, y[u].w));
  }
  m = max_over_rows(m, red);
  if (ty == 0) *reinterpret_cast<float4 *>(w.lam + task * dp + jq) = m;
  const float4 sh = make_float4(shift_of(m.x, b.x), shift_of(m.y, b.y), shift_of(m.z, b.z), shift_of(m.w, b.w));
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = ty + 16 * u;
    const float dk = expf(s_dg[r]);
    float4 e = make_float4(b.x > 0.f ? expf(y[u].x - sh.x) : x[u].x * dk, b.y > 0.f ? expf(y[u].y - sh.y) : x[u].y * dk,
                           b.z > 0.f ? expf(y[u].z - sh.z) : x[u].z * dk, b.w > 0.f ? expf(y[u].w - sh.w) : x[u].w * dk);
    if (r >= rows) e = make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(sE + r * kCh + tx * 4) = e;
  }
  __syncthreads();
  float2 acc[RT][2];
#pragma unroll
  for (int r = 0; r < RT; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
#pragma unroll 8
  for (int i = 0; i < kSteps; ++i) {
    const float4 e = ld4(sE + i * kCh + tx * 4);
    float a[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r) a[r] = sK[i * M + ty * RT + r];
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      acc[r][0] = __ffma2_rn(make_float2(a[r], a[r]), make_float2(e.x, e.y), acc[r][0]);
      acc[r][1] = __ffma2_rn(make_float2(a[r], a[r]), make_float2(e.z, e.w), acc[r][1]);
    }
  }
#pragma unroll
  for (int r = 0; r < RT; ++r)
    *reinterpret_cast<float4 *>(w.u + (task * M + ty * RT + r) * dp + jq) =
        make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
  if (blockIdx.y == 0) {  // the constant channel, a quarter of the keys a thread
    if (tid < 4 * M) {
      const int f = tid % M, part = tid / M;
      float z = 0.f;
#pragma unroll
      for (int i = 0; i < kSteps / 4; ++i) z = fmaf(sK[(part * (kSteps / 4) + i) * M + f], expf(s_dg[part * (kSteps / 4) + i]), z);
      s_z[part][f] = z;
    }
    __syncthreads();
    if (tid < M) w.z[task * M + tid] = (s_z[0][tid] + s_z[1][tid]) + (s_z[2][tid] + s_z[3][tid]);
  }
}

// ---------------------------------------------------------------------------
// scan: thread per state element (feature, channel; the constant channel's behind them), the run's
// chunks in turn, the start states in U's place.  Bound by the states' bytes (from L2 at moderate
// sizes); kAhead chunks' loads in flight, the scales' chain ahead of the exponentials.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gla_scan_f32_kernel(int d, int dp, int M, int first, int n, int nb, GlaWs w) {
  constexpr int kAhead = 8;
  const int i = blockIdx.x * 256 + threadIdx.x, hd = blockIdx.y;
  if (i >= M * dp + M) return;
  const bool is_z = i >= M * dp;
  const int j = is_z ? 0 : i % dp;
  if (!is_z && j >= d) return;
  const size_t t0 = static_cast<size_t>(hd) * nb, stride = is_z ? M : static_cast<size_t>(M) * dp;
  float *s = is_z ? w.z + t0 * M + (i - M * dp) : w.u + t0 * M * dp + i;
  float *carry = w.carry + static_cast<size_t>(hd) * (M * dp + M + dp);
  const bool scaled = !is_z && w.eb[static_cast<size_t>(hd) * dp + j] > 0.f, wr_mu = !is_z && i < dp;
  float S = first ? 0.f : carry[i], mu = !scaled ? 0.f : first ? -INFINITY : carry[M * dp + M + j];
  for (int c = 0; c < n; c += kAhead) {
    float u[kAhead], lam[kAhead], gl[kAhead], fr[kAhead], fl[kAhead], at[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      const int p = min(c + q, n - 1);
      u[q] = s[p * stride];
      lam[q] = scaled ? w.lam[(t0 + p) * dp + j] : 0.f;
      gl[q] = w.gl[t0 + p];
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      at[q] = mu;
      const float eg = expf(gl[q]);
      fr[q] = eg;
      fl[q] = 1.f;
      if (scaled && c + q < n) {
        const float lo = mu + gl[q], to = fmaxf(lo, lam[q]);
        const bool none = to == -INFINITY;  // no value yet
        // exp(gl) apart, rounded as the constant channel's, unless it could underflow
        fr[q] = none ? 0.f : gl[q] > -60.f ? eg * expf(mu - to) : expf(lo - to);
        fl[q] = lam[q] == -INFINITY ? 0.f : expf(lam[q] - to);
        mu = to;
      }
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      if (c + q >= n) break;
      s[(c + q) * stride] = S;
      if (wr_mu) w.mu[(t0 + c + q) * dp + j] = at[q];
      S = fl[q] == 0.f ? fr[q] * S : fmaf(fr[q], S, fl[q] * u[q]);
    }
  }
  carry[i] = S;
  if (wr_mu) carry[M * dp + M + j] = mu;
}

// ---------------------------------------------------------------------------
// out: block per chunk and 64 channels, about 70 KB of shared memory, three CTAs per SM.  Scores and
// the state's part in one loop over the features; the masked weights take the state's place for the
// in-chunk part, whose loop ends at a warp's last row.
// ---------------------------------------------------------------------------
template <int M>
struct OutF32 {
  static constexpr int kQ = 0, kK = M * kLd, kE = 2 * M * kLd, kS = kE + kSteps * kCh;
  static constexpr int kFloats = kS + kSteps * kSteps;
};

// The read of one entry from its in-chunk sum acc at the shift m (linear: acc alone) and the state's part.
__device__ __forceinline__ float read_entry(float b, float m, float acc, float ix, float mu, float et, float gt, float den,
                                            bool state) {
  if (!(b > 0.f)) return lin_read(b, (state ? fmaf(et, ix, acc) : acc) / den);
  const float la = acc == 0.f ? -INFINITY : m + logf(acc);
  const float lb = ix == 0.f ? -INFINITY : mu + gt + logf(ix);
  const float hi = fmaxf(la, lb), lo = fminf(la, lb);
  const float ln = hi == -INFINITY ? hi : hi + log1pf(expf(lo - hi));
  return ((la != la ? la : lb != lb ? lb : ln) - logf(den)) / b;
}

// The block's flagged entries (s_flag: 64 bits a row) once more, from the keys their rows see and the start
// state: the scores again, then in the warps that have any the largest beta v + decay of the visible keys and
// the sum around it, four rows against four channels a thread as in the sums before.  B4 H4 T2048 m64 d128 with
// values of 10, 30 and 100 times unit spread and beta up to 100, 100 and 200: 354, 354 and 352 us a call; with
// read_rows alone 577, 673, 763.
template <int M>
__device__ __noinline__ void read_again(float *smem, const float2 *gam, const float *s_den, const float *s_b,
                                        const unsigned (*s_flag)[2], const float *v, float *out, int h0, int T, int d,
                                        int dp, int c0, int nb, int vec, const GlaWs &w) {
  using Lay = OutF32<M>;
  // (the block's place again from the launch's parameters: handed over, it stays in registers through the read)
  const int hd = blockIdx.z, j0 = blockIdx.y * kCh, c = c0 + blockIdx.x, rows = min(kSteps, T - c * kSteps);
  const size_t r0 = static_cast<size_t>(h0 + hd) * T + static_cast<size_t>(c) * kSteps;
  const size_t task = static_cast<size_t>(hd) * nb + blockIdx.x;
  const bool state = c > 0;
  v += r0 * d;
  out += r0 * d;
  const float *sQ = smem + Lay::kQ, *sK = smem + Lay::kK;
  float *sV = smem + Lay::kE, *sS = smem + Lay::kS;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, jq = j0 + tx * 4;
  const float4 b = ld4(s_b + tx * 4);
  unsigned flags = 0;  // bit 4 r + q is row 4 ty + r, channel 4 tx + q
#pragma unroll
  for (int r = 0; r < 4; ++r) flags |= ((s_flag[ty * 4 + r][tx >> 3] >> ((tx & 7) * 4)) & 15u) << (4 * r);
  {
    float4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = ty + 16 * u;
      x[u] = r < rows ? ld_row4(v + static_cast<size_t>(r) * d, jq, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    lin_values(b, x);
#pragma unroll
    for (int u = 0; u < 4; ++u) *reinterpret_cast<float4 *>(sV + (ty + 16 * u) * kCh + tx * 4) = x[u];
    float s[4][4];  // [key][row]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int r = 0; r < 4; ++r) s[i][r] = 0.f;
#pragma unroll 4
    for (int f = 0; f < M; ++f) {
      const float4 q4 = ld4(sQ + f * kLd + ty * 4), k4 = ld4(sK + f * kLd + tx * 4);
      const float qr[4] = {q4.x, q4.y, q4.z, q4.w}, kr[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int r = 0; r < 4; ++r) s[i][r] = fmaf(qr[r], kr[i], s[i][r]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<float4 *>(sS + (tx * 4 + i) * kSteps + ((ty ^ tx) << 2)) = make_float4(s[i][0], s[i][1], s[i][2], s[i][3]);
  }
  __syncthreads();
  if (!__any_sync(0xffffffffu, flags != 0u)) return;
  // exponents in units of ln 2; a linear channel's terms are its values times the decays
  const float bj[4] = {b.x, b.y, b.z, b.w};
  float b2[4], m[4][4], acc[4][4];
  float2 g[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    g[r] = gam[ty * 4 + r];
    b2[r] = bj[r] > 0.f ? bj[r] * kLog2e : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      m[r][q] = -INFINITY;
      acc[r][q] = 0.f;
    }
  }
  const int last = min(rows, (tid >> 5) * 8 + 8);  // a warp's rows see no key from here on
  for (int i = 0; i < last; ++i) {
    const float4 x4 = ld4(sV + i * kCh + tx * 4);
    const float x[4] = {x4.x, x4.y, x4.z, x4.w};
    const float2 gi = gam[i];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float dg = i <= ty * 4 + r ? sum_diff(g[r], gi) * kLog2e : -INFINITY;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float y = fmaf(b2[q], x[q], dg);
        m[r][q] = fmaxf(m[r][q], i <= ty * 4 + r ? y : -INFINITY);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (!(bj[q] > 0.f) || m[r][q] == -INFINITY) m[r][q] = 0.f;
  for (int i = 0; i < last; ++i) {
    const float4 x4 = ld4(sV + i * kCh + tx * 4), s4 = ld4(sS + i * kSteps + ((ty ^ (i >> 2)) << 2));
    const float x[4] = {x4.x, x4.y, x4.z, x4.w}, sc[4] = {s4.x, s4.y, s4.z, s4.w};
    const float2 gi = gam[i];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (i > ty * 4 + r) continue;
      const float dg = sum_diff(g[r], gi) * kLog2e;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float y = b2[q] > 0.f ? fmaf(b2[q], x[q], dg) : dg, e = ex2_approx(y - m[r][q]);
        acc[r][q] = fmaf(b2[q] > 0.f ? sc[r] : sc[r] * x[q], e, acc[r][q]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int t = ty * 4 + r;
    const float e0 = expf(g[r].x), et = fmaf(e0, g[r].y, e0), gt = g[r].x + g[r].y;
    float ix[4] = {0.f, 0.f, 0.f, 0.f};
    if (state && ((flags >> (4 * r)) & 15u)) {
#pragma unroll 8
      for (int f = 0; f < M; ++f) {
        const float qr = sQ[f * kLd + t];
        const float4 u4 = ld4(w.u + (task * M + f) * dp + jq);
        ix[0] = fmaf(qr, u4.x, ix[0]);
        ix[1] = fmaf(qr, u4.y, ix[1]);
        ix[2] = fmaf(qr, u4.z, ix[2]);
        ix[3] = fmaf(qr, u4.w, ix[3]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (!((flags >> (4 * r + q)) & 1u)) continue;
      const float mu = state && bj[q] > 0.f ? w.mu[task * dp + jq + q] : 0.f;
      out[static_cast<size_t>(t) * d + jq + q] =
          read_entry(bj[q], m[r][q] * kLn2, acc[r][q], ix[q], mu, et, gt, s_den[t], state);
    }
  }
}

// The same for few flagged entries: a warp per row, its lanes over channels or keys (at kFewFlagged 24 or 40 a
// call at 3 times unit spread 235 or 227 us, at 10 times 333 or 360).
template <int M>
__device__ __noinline__ void read_rows(float *smem, const float2 *gam, const float *s_den, const float *s_b,
                                       const unsigned (*s_flag)[2], const float *v, float *out, int h0, int T, int d,
                                       int dp, int c0, int nb, const GlaWs &w) {
  using Lay = OutF32<M>;
  const int hd = blockIdx.z, j0 = blockIdx.y * kCh, c = c0 + blockIdx.x, rows = min(kSteps, T - c * kSteps);
  const size_t r0 = static_cast<size_t>(h0 + hd) * T + static_cast<size_t>(c) * kSteps;
  const size_t task = static_cast<size_t>(hd) * nb + blockIdx.x;
  const bool state = c > 0;
  v += r0 * d;
  out += r0 * d;
  const float *sQ = smem + Lay::kQ, *sK = smem + Lay::kK;
  float *sP = smem + Lay::kS;
  const int tid = threadIdx.x, lane = tid & 31;
  // the row's scores and decays once (lanes the keys lane and lane + 32 it sees), then for each 32 channels:
  // lane = channel, the keys in turn, where four or more are flagged, else a channel at a time with the lanes
  // over the keys
  float *s_sc = sP + (tid >> 5) * 2 * kSteps, *s_dg = s_sc + kSteps;  // the weights are consumed
  const int t_end = min(rows, (tid >> 5) * 8 + 8);
  for (int t = (tid >> 5) * 8; t < t_end; ++t) {
    if (!(s_flag[t][0] | s_flag[t][1])) continue;
    const float2 g2 = gam[t];
    const float e0 = expf(g2.x), et = fmaf(e0, g2.y, e0), gt = g2.x + g2.y, den = s_den[t];
    float sc[2], dg[2];
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < 2; ++k2) {
      const int i = lane + 32 * k2;
      sc[k2] = 0.f;
      dg[k2] = i <= t ? sum_diff(g2, gam[i]) : -INFINITY;
      if (i <= t)
        for (int f = 0; f < M; ++f) sc[k2] = fmaf(sQ[f * kLd + t], sK[f * kLd + i], sc[k2]);
      s_sc[i] = sc[k2];
      s_dg[i] = dg[k2];
    }
    __syncwarp();
    auto read = [&](float bq, float m, float acc, float ixe, int j) {
      return read_entry(bq, m, acc, ixe, state && bq > 0.f ? w.mu[task * dp + j] : 0.f, et, gt, den, state);
    };
    for (int half = 0; half < 2; ++half) {
      unsigned fm = s_flag[t][half];
      if (__popc(fm) >= 4) {
        const int j = j0 + half * 32 + lane;
        const bool on = (fm >> lane) & 1u;  // below d
        const float bq = on ? s_b[j - j0] : 0.f;
        const float *vc = v + (on ? j : 0);
        float m = -INFINITY, acc = 0.f, ixe = 0.f;
        for (int i = 0; i <= t; ++i) m = fmaxf(m, fmaf(bq, __ldg(vc + static_cast<size_t>(i) * d), s_dg[i]));
        for (int i = 0; i <= t; ++i) {
          const float xv = __ldg(vc + static_cast<size_t>(i) * d), y = fmaf(bq, xv, s_dg[i]);
          const float e = bq > 0.f ? expf(y - m) : expf(s_dg[i]) * lin_value(bq, xv);
          if (!(bq > 0.f) || y != -INFINITY) acc = fmaf(s_sc[i], e, acc);
        }
        if (state && on)
          for (int f = 0; f < M; ++f) ixe = fmaf(sQ[f * kLd + t], w.u[(task * M + f) * dp + j], ixe);
        if (on) out[static_cast<size_t>(t) * d + j] = read(bq, m, acc, ixe, j);
        continue;
      }
      while (fm) {
        const int j = j0 + half * 32 + __ffs(fm) - 1;
        fm &= fm - 1;
        const float bq = s_b[j - j0];
        float y[2], m = -INFINITY, acc = 0.f, ixe = 0.f;
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
          const int i = lane + 32 * k2;
          const float xv = i <= t ? __ldg(v + static_cast<size_t>(i) * d + j) : 0.f;
          y[k2] = i <= t ? fmaf(bq, xv, dg[k2]) : -INFINITY;
          m = fmaxf(m, y[k2]);
          if (!(bq > 0.f) && i <= t) acc = fmaf(sc[k2] * expf(dg[k2]), lin_value(bq, xv), acc);
        }
        if (state)
          for (int f = lane; f < M; f += 32) ixe = fmaf(sQ[f * kLd + t], w.u[(task * M + f) * dp + j], ixe);
#pragma unroll
        for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if (bq > 0.f) {
#pragma unroll
          for (int k2 = 0; k2 < 2; ++k2)
            if (y[k2] != -INFINITY) acc = fmaf(sc[k2], expf(y[k2] - m), acc);
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
          acc += __shfl_xor_sync(0xffffffffu, acc, off);
          ixe += __shfl_xor_sync(0xffffffffu, ixe, off);
        }
        if (lane == 0) out[static_cast<size_t>(t) * d + j] = read(bq, m, acc, ixe, j);
      }
    }
  }
}

// LONE: the sequence is one chunk, so there is no state and the forms are found here.
template <int M, bool LONE>
__global__ void __launch_bounds__(kThreads, 3)
    gla_out_f32_kernel(const float *__restrict__ qf, const float *__restrict__ kf, const float *__restrict__ v,
                       const float *__restrict__ logdecay, const float *__restrict__ beta, float *__restrict__ out,
                       float *__restrict__ logz, int h0, int H, int T, int d, int dp, int c0, int nb, int vec, int vec_o,
                       const __grid_constant__ GlaWs w) {
  using Lay = OutF32<M>;
  extern __shared__ __align__(16) float gla_smem[];
  float *sQ = gla_smem + Lay::kQ, *sK = gla_smem + Lay::kK, *sE = gla_smem + Lay::kE, *sS = gla_smem + Lay::kS, *sP = sS;
  __shared__ float4 red[16][16];
  __shared__ float2 gam[kSteps];
  __shared__ float s_den[kSteps], s_sz[M];
  __shared__ __align__(16) float s_b[kCh];
  __shared__ unsigned s_flag[kSteps][2];
  const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 4, tx = tid & 15, hd = blockIdx.z, j0 = blockIdx.y * kCh, jq = j0 + tx * 4;
  const int c = c0 + blockIdx.x, rows = min(kSteps, T - c * kSteps);
  const size_t r0 = static_cast<size_t>(h0 + hd) * T + static_cast<size_t>(c) * kSteps;
  const size_t task = static_cast<size_t>(hd) * nb + blockIdx.x;
  const bool state = !LONE && c > 0;
  float4 x[4], qx[M / 16], kx[M / 16];
#pragma unroll
  for (int u = 0; u < M / 16; ++u) {  // lanes over rows: the transposed stores hit distinct banks
    const int e = tid + u * kThreads, r = e % kSteps, f = (e / kSteps) * 4;
    qx[u] = r < rows ? ld4(qf + (r0 + r) * M + f) : make_float4(0.f, 0.f, 0.f, 0.f);
    kx[u] = r < rows ? ld4(kf + (r0 + r) * M + f) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = ty + 16 * u;
    x[u] = r < rows ? ld_row4(v + (r0 + r) * d, jq, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (state) {
#pragma unroll
    for (int u = 0; u < M / 16; ++u) {
      const int f = ty + 16 * u;
      *reinterpret_cast<float4 *>(sS + f * kCh + tx * 4) = ld4(w.u + (task * M + f) * dp + jq);
    }
    if (tid < M) s_sz[tid] = w.z[task * M + tid];
  }
  if (tid < 2 * kSteps) s_flag[tid >> 1][tid & 1] = 0u;
  chunk_sums(logdecay + r0, rows, gam);
#pragma unroll
  for (int u = 0; u < M / 16; ++u) {
    const int e = tid + u * kThreads, r = e % kSteps, f = (e / kSteps) * 4;
    sQ[f * kLd + r] = qx[u].x;
    sQ[(f + 1) * kLd + r] = qx[u].y;
    sQ[(f + 2) * kLd + r] = qx[u].z;
    sQ[(f + 3) * kLd + r] = qx[u].w;
    sK[f * kLd + r] = kx[u].x;
    sK[(f + 1) * kLd + r] = kx[u].y;
    sK[(f + 2) * kLd + r] = kx[u].z;
    sK[(f + 3) * kLd + r] = kx[u].w;
  }
  float4 b;
  if constexpr (!LONE) {
    b = ld4(w.eb + static_cast<size_t>(hd) * dp + jq);
  } else {
    b = beta4(beta, (h0 + hd) % H, d, jq);
    float4 top = make_float4(0.f, 0.f, 0.f, 0.f);
    if (__syncthreads_or(maybe_small(b))) {
#pragma unroll
      for (int u = 0; u < 4; ++u) top = abs_max(top, x[u]);
      top = max_over_rows(top, red);
      __syncthreads();  // red is used again
    }
    b = form_beta4(b, top);
  }
  if (ty == 0) *reinterpret_cast<float4 *>(s_b + tx * 4) = b;
  lin_values(b, x);
  float lam[4];
  {
    float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (ty + 16 * u < rows) m = make_float4(fmaxf(m.x, x[u].x), fmaxf(m.y, x[u].y), fmaxf(m.z, x[u].z), fmaxf(m.w, x[u].w));
    m = max_over_rows(m, red);  // also: the tiles are written
    lam[0] = shift_of(b.x * m.x, b.x);
    lam[1] = shift_of(b.y * m.y, b.y);
    lam[2] = shift_of(b.z * m.z, b.z);
    lam[3] = shift_of(b.w * m.w, b.w);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = ty + 16 * u;
    float4 e = make_float4(b.x > 0.f ? expf(fmaf(b.x, x[u].x, -lam[0])) : x[u].x,
                           b.y > 0.f ? expf(fmaf(b.y, x[u].y, -lam[1])) : x[u].y,
                           b.z > 0.f ? expf(fmaf(b.z, x[u].z, -lam[2])) : x[u].z,
                           b.w > 0.f ? expf(fmaf(b.w, x[u].w, -lam[3])) : x[u].w);
    if (r >= rows) e = make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4 *>(sE + r * kCh + tx * 4) = e;
  }
  // ---- scores (rows in packed pairs) and the state's part (channels in packed pairs)
  float2 s[2][4], ix[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    s[0][i] = s[1][i] = make_float2(0.f, 0.f);
    ix[i][0] = ix[i][1] = make_float2(0.f, 0.f);
  }
  const float *qp = sQ + ty * 4, *kp = sK + tx * 4, *sp = sS + tx * 4;
  auto scores = [&](float4 a, float4 k4) {
    const float2 ar[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
    const float kr[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s[0][i] = __ffma2_rn(ar[0], make_float2(kr[i], kr[i]), s[0][i]);
      s[1][i] = __ffma2_rn(ar[1], make_float2(kr[i], kr[i]), s[1][i]);
    }
  };
  auto rows_by_channels = [](float2 (&o)[4][2], float4 a, float4 e) {
    const float ar[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[i][0] = __ffma2_rn(make_float2(ar[i], ar[i]), make_float2(e.x, e.y), o[i][0]);
      o[i][1] = __ffma2_rn(make_float2(ar[i], ar[i]), make_float2(e.z, e.w), o[i][1]);
    }
  };
  if (state) {
#pragma unroll 4
    for (int f = 0; f < M; ++f) {
      const float4 a = ld4(qp + f * kLd);
      scores(a, ld4(kp + f * kLd));
      rows_by_channels(ix, a, ld4(sp + f * kCh));
    }
  } else {
#pragma unroll 8
    for (int f = 0; f < M; ++f) scores(ld4(qp + f * kLd), ld4(kp + f * kLd));
  }
  // ---- the rows' masses (16 lanes share a row) and the masked weights
  float zi[4], zx[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) zi[r] = zx[r] = 0.f;
  if (state) {
    for (int f = tx; f < M; f += 16) {
      const float4 a = ld4(qp + f * kLd);
      const float z = s_sz[f];
      zx[0] = fmaf(a.x, z, zx[0]);
      zx[1] = fmaf(a.y, z, zx[1]);
      zx[2] = fmaf(a.z, z, zx[2]);
      zx[3] = fmaf(a.w, z, zx[3]);
    }
  }
  __syncthreads();  // the state's tile is consumed
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int key = tx * 4 + i;
    const float2 gk = gam[key];
    float p[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float sc = (r & 1) ? s[r >> 1][i].y : s[r >> 1][i].x;
      p[r] = key <= ty * 4 + r ? sc * expf(sum_diff(gam[ty * 4 + r], gk)) : 0.f;
      zi[r] += p[r];
    }
    *reinterpret_cast<float4 *>(sP + key * kSteps + ((ty ^ tx) << 2)) = make_float4(p[0], p[1], p[2], p[3]);
  }
#pragma unroll
  for (int off = 8; off; off >>= 1)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      zi[r] += __shfl_xor_sync(0xffffffffu, zi[r], off);
      zx[r] += __shfl_xor_sync(0xffffffffu, zx[r], off);
    }
  __syncthreads();
  // ---- the in-chunk part
  float2 in[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) in[i][0] = in[i][1] = make_float2(0.f, 0.f);
  const int last = (tid >> 5) * 8 + 8;  // a warp's rows see no key from here on
#pragma unroll 4
  for (int i = 0; i < last; ++i)
    rows_by_channels(in, ld4(sP + i * kSteps + ((ty ^ (i >> 2)) << 2)), ld4(sE + i * kCh + tx * 4));
  // ---- the read
  float mu[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) mu[q] = -INFINITY;
  if (state) {
    const float4 m4 = ld4(w.mu + task * dp + jq);
    mu[0] = m4.x;
    mu[1] = m4.y;
    mu[2] = m4.z;
    mu[3] = m4.w;
  }
  const float bj[4] = {b.x, b.y, b.z, b.w};
  float rb[4], em[4];  // em: the state's scale over the chunk's, infinite where that overflows
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    rb[q] = bj[q] > 0.f ? 1.f / bj[q] : 0.f;
    em[q] = mu[q] - lam[q] < 60.f ? expf(mu[q] - lam[q]) : INFINITY;
  }
  bool any = false;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int t = ty * 4 + r;
    const float2 g2 = gam[t];
    const float e0 = expf(g2.x), et = fmaf(e0, g2.y, e0), gt = g2.x + g2.y;
    const float den = state ? fmaf(et, zx[r], zi[r]) : zi[r];
    const float lo_in = kGlaGuard * zi[r], lo_sum = kGlaGuard * den, rden = 1.f / den;
    unsigned flag = 0;
    float o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = (q & 1) ? in[r][q >> 1].y : in[r][q >> 1].x, y = (q & 1) ? ix[r][q >> 1].y : ix[r][q >> 1].x;
      if (bj[q] > 0.f) {
        // exp(gamma) apart, rounded as in the normaliser, unless it or the scales' ratio leaves fp32's range
        float top = lam[q], sum = state ? fmaf(et * em[q], y, a) : a;
        if (state && !(gt > -60.f && em[q] < INFINITY)) {
          top = fmaxf(lam[q], mu[q] + gt);
          sum = fmaf(a, expf(lam[q] - top), expf((mu[q] + gt) - top) * y);
        }
        flag |= !(a >= lo_in) || !(sum >= lo_sum) ? 1u << q : 0u;
        o[q] = (top + logf(sum * rden)) * rb[q];
      } else {
        flag |= !(fabsf(a) < INFINITY) ? 1u << q : 0u;
        o[q] = (state ? fmaf(et, y, a) : a) * rden;
      }
      if (jq + q >= d) flag &= ~(1u << q);
    }
    if (t < rows) {
      float *orow = out + (r0 + t) * d + jq;
      if (vec_o) {
        if (jq < d) *reinterpret_cast<float4 *>(orow) = make_float4(o[0], o[1], o[2], o[3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (jq + q < d) orow[q] = o[q];
      }
      if (tx == 0) {
        s_den[t] = den;
        if (logz && blockIdx.y == 0) logz[r0 + t] = logf(den);
      }
      if (flag) {
        atomicOr(&s_flag[t][tx >> 3], flag << ((tx & 7) * 4));
        any = true;
      }
    }
  }
  if (b.x < 0.f || b.y < 0.f || b.z < 0.f || b.w < 0.f) {
    // the small-beta channels' ratios, as stored, to their reads (in the loop above this cost 2.5 of 117 us a call)
#pragma unroll 1
    for (int r = 0; r < 4; ++r) {
      float *orow = out + (r0 + ty * 4 + r) * d + jq;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (ty * 4 + r < rows && jq + q < d && bj[q] < 0.f) orow[q] = lin_read(bj[q], orow[q]);
    }
  }
  const int n_flagged = __syncthreads_count(any);  // threads
  if (n_flagged > kFewFlagged)
    read_again<M>(gla_smem, gam, s_den, s_b, s_flag, v, out, h0, T, d, dp, c0, nb, vec, w);
  else if (n_flagged > 0)
    read_rows<M>(gla_smem, gam, s_den, s_b, s_flag, v, out, h0, T, d, dp, c0, nb, w);
}

size_t up64(size_t x) { return (x + 63) & ~size_t(63); }

// Heads of a group, chunks of a run and the workspace's floats for at most `cap` bytes (one head and
// eight chunks at least); none for a lone chunk.
struct GlaPlan {
  int heads, chunks;
  size_t floats;
};
GlaPlan gla_plan(long long BH, int T, int m, int d, size_t cap, float *base, GlaWs *w) {
  const int n_ch = (T + kSteps - 1) / kSteps, dp = (d + kCh - 1) / kCh * kCh;
  if (n_ch == 1) return {static_cast<int>(BH < 65535 ? BH : 65535), 1, 0};
  const size_t per = static_cast<size_t>(m) * dp + m + 2 * dp + 1, head = static_cast<size_t>(m) * dp + m + 2 * dp;
  const size_t room = cap / sizeof(float) / per;
  GlaPlan p;
  if (room >= static_cast<size_t>(n_ch)) {
    p.chunks = n_ch;
    const long long fit = static_cast<long long>(cap / sizeof(float) / (per * n_ch + head));
    p.heads = static_cast<int>(fit < 1 ? 1 : fit > 65535 ? 65535 : fit);
    if (p.heads > BH) p.heads = static_cast<int>(BH);
  } else {
    p.heads = 1;
    p.chunks = room < 8 ? 8 : static_cast<int>(room);
    if (p.chunks > n_ch) p.chunks = n_ch;
  }
  const size_t n = static_cast<size_t>(p.heads) * p.chunks;
  size_t o = 0;
  auto take = [&](size_t count) {
    float *q = base ? base + o : nullptr;
    o += up64(count);
    return q;
  };
  GlaWs l;
  l.u = take(n * m * dp);
  l.z = take(n * m);
  l.lam = take(n * dp);
  l.mu = take(n * dp);
  l.gl = take(n);
  l.eb = take(static_cast<size_t>(p.heads) * dp);
  l.carry = take(static_cast<size_t>(p.heads) * (head - dp));
  p.floats = o;
  if (w) *w = l;
  return p;
}

template <int M>
cudaError_t launch_gla_m(const float *qf, const float *kf, const float *v, const float *logdecay, const float *beta,
                         float *out, float *logz, int BH, int H, int T, int d, size_t cap, void *ws, cudaStream_t stream) {
  constexpr int kBytes = OutF32<M>::kFloats * 4;
  const bool lone = T <= kSteps;
  const auto out_kernel = lone ? gla_out_f32_kernel<M, true> : gla_out_f32_kernel<M, false>;
  cudaError_t e = cudaFuncSetAttribute(out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  if (e != cudaSuccess) return e;
  GlaWs w = {};
  const GlaPlan p = gla_plan(BH, T, M, d, cap, static_cast<float *>(ws), &w);
  const int n_ch = (T + kSteps - 1) / kSteps, groups = (d + kCh - 1) / kCh, dp = groups * kCh;
  const int vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(v) & 15u) == 0;
  const int vec_o = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  for (int h0 = 0; h0 < BH; h0 += p.heads) {
    const int nh = BH - h0 < p.heads ? BH - h0 : p.heads;
    const bool form = n_ch > kOwnForm;
    if (form) gla_form_f32_kernel<<<dim3(nh, groups), kThreads, 0, stream>>>(v, beta, h0, H, T, d, dp, vec, w);
    for (int c0 = 0; c0 < n_ch; c0 += p.chunks) {
      const int n = n_ch - c0 < p.chunks ? n_ch - c0 : p.chunks;
      if (n_ch > 1) {
        // the sequence's last chunk starts no other: what the scan reads in its slot goes nowhere
        const int own = c0 + n == n_ch ? n - 1 : n;
        if (own > 0)
          e = launch_kernel(gla_local_f32_kernel<M>, dim3(own, groups, nh), dim3(kThreads), 0, stream,
                            form && c0 == 0, kf, v, logdecay, beta, h0, H, T, d, dp, c0, p.chunks, vec, w);
        if (e != cudaSuccess) return e;
        gla_scan_f32_kernel<<<dim3((M * dp + M + 255) / 256, nh), 256, 0, stream>>>(d, dp, M, c0 == 0 ? 1 : 0, n,
                                                                                    p.chunks, w);
      }
      out_kernel<<<dim3(n, groups, nh), kThreads, kBytes, stream>>>(qf, kf, v, logdecay, beta, out, logz, h0, H,
                                                                               T, d, dp, c0, p.chunks, vec, vec_o, w);
    }
  }
  return cudaGetLastError();
}

}  // namespace

size_t gla_workspace_bytes(int BH, int T, int m, int d, size_t cap) {
  return gla_plan(BH, T, m, d, cap, nullptr, nullptr).floats * sizeof(float);
}

cudaError_t launch_gla(const float *qf, const float *kf, const float *v, const float *logdecay, const float *beta,
                       float *out, float *logz, int BH, int H, int T, int m, int d, size_t cap, void *ws,
                       cudaStream_t stream) {
  switch (m) {
    case 16: return launch_gla_m<16>(qf, kf, v, logdecay, beta, out, logz, BH, H, T, d, cap, ws, stream);
    case 32: return launch_gla_m<32>(qf, kf, v, logdecay, beta, out, logz, BH, H, T, d, cap, ws, stream);
    case 64: return launch_gla_m<64>(qf, kf, v, logdecay, beta, out, logz, BH, H, T, d, cap, ws, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace fem
