// Gradients of the fp32 read as register-tiled contractions (64 x 64 tiles of
// query rows and keys), instead of two exponentials per (row, key, channel) and
// pass.  With p_ti = exp(s_ti - lse_t), x = beta_j (v_ij - o_tj) and a shift c_j
// per (b, h, channel), x splits into a = beta (v - c) and b = beta (c - o), and
// every sum over pairs becomes a contraction of per-key and per-row factors:
//
//   dS_ti  = sum_j g_tj p expm1(x)/beta = p (sum_j X_ij Z_tj + R_t),   Z = g e^b
//            linear channel:  X = expm1(a)/beta,  R += g expm1(b)/beta
//            shifted channel: X = e^a / beta,     R -= g / beta
//   dq_t   = sum_i dS_ti k_i / sqrt(d),  dk_i = sum_t dS_ti q_t / sqrt(d)
//   dv_ij  = e^a H_ij,  H_ij = sum_t p_ti Z_tj
//   dbeta_j = sum_ti g p phi(x)/beta^2, phi(x) = 1 + (x - 1) e^x, with H2_ij = sum_t p_ti Z_tj (c - o_tj):
//            linear:  sum_i [phi(a)/beta^2 H + expm1(a)/beta H2] + sum_t g phi(b)/beta^2
//            shifted: (sum_i e^a [(a - 1) H + beta H2] + sum_t g) / beta^2       (sum_i p_ti = 1)
//
// A channel is linear when beta times the spread of v is at most 4 (c the mean,
// clamped so that a lies in [-1, 3]): no difference of large terms.  The shifted
// channels' c is the middle of the spread, so e^a and e^b stay within e^+-kWideExp.
// The cotangents enter Z and R over a power of two of their row (its largest, g' in
// [1, 2) there), which comes back at dS; the sums over rows take p times the row's
// power over the head's largest, which comes back at dv and dbeta.  So nothing depends
// on the scale of g, and what fp32's range drops from p e^b (2^-150) stays, times e^a,
// below 2^-40 of the head's largest cotangent.
// All exponents carry their rounding errors (exp_tilt), which keeps the gradients'
// error at that of exp(x) taken directly.  Channels whose spread exceeds that (or is
// not finite) take no part in the contractions; their terms are formed pair by pair
// beside them (wide_terms).  A visible pair whose weight falls below e^-60 marks its
// head (its e^x could leave fp32's range; and where the prior is that peaked, posterior
// and prior differ so little that the factors' differences lose digits: dbeta 4e-4 off
// at scores of deviation 64), as does a head with most channels wide; the kernels of
// fem_bwd.cu, which form every term from its own exponent, take those.
//
// What bounds it: issue around the FMA pipe (3 d multiply-adds per pair in the row
// pass, 5 d in the key pass); fem_bwd.cu's form spends some 50 issue slots a pair and
// channel.  B1 H4 T2048 d64 causal: 185 + 264 us for the two passes against 2233 +
// 1650 us, and a third of the error against 64 bits.  A cluster of CTAs shares one tile's pairs (every size-th tile of the
// other side each) and adds its accumulators through distributed shared memory:
// causal tiles differ by the whole sequence in length.
#include <cooperative_groups.h>

#include "fem_common.cuh"
#include "fem_f32.cuh"
#include "fem_launch.h"

namespace fem {
namespace cg = cooperative_groups;
namespace {

constexpr int kBT = 64;           // rows and keys of a tile (rows of the other side: kRows below)
constexpr int kBLd = 68;          // leading dimension of a transposed 64-row tile
constexpr float kWideExp = 76.f;  // largest |a|, |b| of a factored channel: 2^+-110
constexpr float kPeakLog = -60.f;

// A head's sample of pairs for the mark of peaked priors: warp w takes row T - 1 - w T / 32 and 16 of its keys,
// lanes over channels.  Without it a marked head pays the row pass's first tiles before its own kernels; what
// the sample misses is still found there.  us, plain / peaked heads, without and with: B8 H8 T128 d64 100 / 242,
// 106 / 223, B64 H6 T192 d128 1188 / 2922, 1212 / 2660 (pair by pair alone 2540); below kSampleT it costs the
// plain ones up to 11 % (B64 H6 T64 d16 94, 105).
constexpr int kSampleT = 96, kSampleKeys = 16;
__device__ __forceinline__ bool sample_peaked(const float *q, const float *k, const float *lse, int T, int d, int causal) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = T - 1 - static_cast<int>(static_cast<long long>(warp) * T / 32), n = causal ? t + 1 : T;
  float s[kSampleKeys];
#pragma unroll
  for (int u = 0; u < kSampleKeys; ++u) s[u] = 0.f;
  for (int j = lane; j < d; j += 32) {
    const float a = q[static_cast<size_t>(t) * d + j];
#pragma unroll
    for (int u = 0; u < kSampleKeys; ++u)
      s[u] = fmaf(a, k[static_cast<size_t>(static_cast<long long>(u) * n / kSampleKeys) * d + j], s[u]);
  }
  float least = INFINITY;
#pragma unroll
  for (int u = 0; u < kSampleKeys; ++u) {
#pragma unroll
    for (int off = 16; off; off >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], off);
    least = fminf(least, s[u]);
  }
  return least * rsqrtf(static_cast<float>(d)) - lse[t] < kPeakLog;
}

// Per (b, h, channel): {beta, 1/beta (0 at 0), c, mode}: 1 linear, 0 shifted, 2 wide.  The wide
// channels of a head are also bits of its first four words (in order, so that the sums over them are
// the same from call to call), their dv zeroed for the key pass to add to.  From kSampleT on one more
// block samples the head's weights, and its last word marks a peaked one.
constexpr int kWideWords = 5;
__global__ void __launch_bounds__(1024) bwd_chan_kernel(const float *__restrict__ q, const float *__restrict__ k,
                                                        const float *__restrict__ v, const float *__restrict__ beta,
                                                        const float *__restrict__ lse, int H, int T, int d, int causal,
                                                        float4 *__restrict__ chan, unsigned *__restrict__ wide,
                                                        float *__restrict__ dv) {
  if (blockIdx.y * 32 >= d) {
    const size_t row0 = static_cast<size_t>(blockIdx.x) * T;
    const bool peak = sample_peaked(q + row0 * d, k + row0 * d, lse + row0, T, d, causal);
    if (__syncthreads_or(peak) && threadIdx.x == 0) wide[blockIdx.x * kWideWords + 4] = 1u;
    return;
  }
  __shared__ unsigned s_wide;
  __shared__ float s_mx[32][33], s_mn[32][33], s_sm[32][33];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, bh = blockIdx.x, j = blockIdx.y * 32 + lane;
  const float *vb = v + static_cast<size_t>(bh) * T * d;
  float mx = -INFINITY, mn = INFINITY, sm = 0.f;
  if (j < d) {
#pragma unroll 8
    for (int i = part; i < T; i += 32) {
      const float x = vb[static_cast<size_t>(i) * d + j];
      mx = fmaxf(mx, x);
      mn = fminf(mn, x);
      sm += x;
    }
  }
  s_mx[part][lane] = mx;
  s_mn[part][lane] = mn;
  s_sm[part][lane] = sm;
  __syncthreads();
  if (part == 0) {
    for (int p = 1; p < 32; ++p) {
      mx = fmaxf(mx, s_mx[p][lane]);
      mn = fminf(mn, s_mn[p][lane]);
      sm += s_sm[p][lane];
    }
    const float b = j < d ? beta[(bh % H) * d + j] : 0.f, mean = sm / static_cast<float>(T), lo = mx - 3.f / b, hi = mn + 1.f / b;
    const bool lin = !(b > 0.f) || lo <= hi;
    const float c = lin ? (b > 0.f ? fminf(fmaxf(mean, lo), hi) : mean) : 0.5f * (mx + mn);
    // not finite (also a sum that overflowed), or too wide for the factors (e^a / beta among them)
    const bool wd = j < d && (!(fabsf(sm) < INFINITY) || !(mx - mn < INFINITY) ||
                              !(lin || 0.5f * b * (mx - mn) + fmaxf(-logf(b), 0.f) <= kWideExp));
    const unsigned word = __ballot_sync(0xffffffffu, wd);
    if (lane == 0) s_wide = wide[bh * kWideWords + blockIdx.y] = word;
    if (j < d)
      chan[static_cast<size_t>(bh) * d + j] = make_float4(b, b > 0.f ? 1.f / b : 0.f, c, wd ? 2.f : (lin ? 1.f : 0.f));
  }
  __syncthreads();
  if ((s_wide >> lane) & 1u)
    for (int i = part; i < T; i += 32) dv[(static_cast<size_t>(bh) * T + i) * d + j] = 0.f;
}

// Channel parameters of a quad of channels (zeros past d: every factor and term is then zero).
struct Chan4 {
  float b[4], ib[4], c[4], lin[4];
};
__device__ __forceinline__ Chan4 chan4(const float4 *chan, int j, int d) {
  Chan4 q;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float4 x = j + u < d ? chan[j + u] : make_float4(0.f, 0.f, 0.f, 1.f);
    q.b[u] = x.x;
    q.ib[u] = x.y;
    q.c[u] = x.z;
    q.lin[u] = x.w;
  }
  return q;
}

// expm1(b x)/b (x at b = 0), the exponent's rounding errors carried where they matter.
__device__ __forceinline__ float em1_tilt(float b, float ib, float v, float c) {
  const float x = v - c, y = b * x;
  const float2 r = em1_over_beta2(make_float2(x, x), make_float2(y, y), make_float2(exp_tilt(b, v, c), 1.f),
                                  make_float2(ib, ib));
  return r.x;
}

// phi(x)/b^2 with x = b y, phi(x) = 1 + (x - 1) e^x: y^2 times the series of phi(x)/x^2
// (sum x^n / (n! (n + 2))) for |x| < 1/2, the form itself beyond.
__device__ __forceinline__ float phi_over_b2(float b, float ib, float v, float c) {
  const float y = v - c, x = b * y;
  float p = fmaf(x, 1.f / 45360.f, 1.f / 5760.f);
  p = fmaf(x, p, 1.f / 840.f);
  p = fmaf(x, p, 1.f / 144.f);
  p = fmaf(x, p, 1.f / 30.f);
  p = fmaf(x, p, 0.125f);
  p = fmaf(x, p, 1.f / 3.f);
  p = fmaf(x, p, 0.5f);
  return fabsf(x) < 0.5f ? y * y * p : fmaf(x - 1.f, exp_tilt(b, v, c), 1.f) * ib * ib;
}

// The key factor X and the row factor Z of a channel (zero for a wide one), and a row's term of R.
__device__ __forceinline__ float key_factor(const Chan4 &q, int u, float v) {
  if (q.lin[u] > 1.f) return 0.f;
  return q.lin[u] != 0.f ? em1_tilt(q.b[u], q.ib[u], v, q.c[u]) : exp_tilt(q.b[u], v, q.c[u]) * q.ib[u];
}
__device__ __forceinline__ float row_factor(const Chan4 &q, int u, float o, float g) {
  return q.lin[u] > 1.f ? 0.f : g * exp_tilt(q.b[u], q.c[u], o);
}
__device__ __forceinline__ float row_term(const Chan4 &q, int u, float o, float g) {
  if (q.lin[u] > 1.f) return 0.f;
  return q.lin[u] != 0.f ? g * em1_tilt(q.b[u], q.ib[u], q.c[u], o) : -g * q.ib[u];
}

// The power of two at or below m, the largest finite |g| of a row, where it and its reciprocal are normal.
__device__ __forceinline__ float row_power(float m) {
  return fminf(fmaxf(__int_as_float(__float_as_int(m) & 0x7f800000), 0x1p-126f), 0x1p126f);
}
__device__ __forceinline__ float finite_abs(float x) { return fabsf(x) < INFINITY ? fabsf(x) : 0.f; }

__device__ __forceinline__ int wide_count(const unsigned *wl) {
  return __popc(wl[0]) + __popc(wl[1]) + __popc(wl[2]) + __popc(wl[3]);
}
__device__ __forceinline__ int wide_next(const unsigned *wl, int j) {  // the first wide channel after j; there is one
  int w = ++j >> 5;
  unsigned m = wl[w] & ~0u << (j & 31);
  while (!m) m = wl[++w];
  return w * 32 + __ffs(m) - 1;
}

// One wide channel's terms of a visible pair with log-weight lp, each from its own exponent:
// q = p e^x, p expm1(x)/b and p phi(x)/b^2 with x = b (v - o).
__device__ __forceinline__ void wide_terms(float b, float ib, float v, float o, float lp, float &qv, float &ds,
                                           float &dbt) {
  const float y = v - o, x = b * y, p = expf(lp);
  qv = expf(lp + x);
  const float2 e = em1_over_beta2(make_float2(y, y), make_float2(x, x), make_float2(1.f, 1.f), make_float2(0.f, 0.f));
  ds = fabsf(x) < 0.5f ? p * e.x : (qv - p) * ib;
  dbt = fabsf(x) < 0.5f ? p * phi_over_b2(b, ib, v, o) : fmaf(x - 1.f, qv, p) * ib * ib;
}

__device__ __forceinline__ void st_t4(float *dst, int ld, float4 x) {  // four channels of a row, transposed
  dst[0] = x.x;
  dst[ld] = x.y;
  dst[2 * ld] = x.z;
  dst[3 * ld] = x.w;
}

// acc[i][c] += a (rows in pairs) x b over one step: R/2 pairs by C columns.
template <int P, int C>
__device__ __forceinline__ void outer(float2 (&acc)[P][C], const float2 (&a)[P], const float (&b)[C]) {
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int i = 0; i < P; ++i) acc[i][c] = __ffma2_rn(a[i], make_float2(b[c], b[c]), acc[i][c]);
}

template <int NC>
__device__ __forceinline__ void ld_cols(float (&b)[NC], const float *row, int tx) {  // a thread's NC channels of a row
  if constexpr (NC == 2) {
    const float2 x = *reinterpret_cast<const float2 *>(row + tx * 2);
    b[0] = x.x;
    b[1] = x.y;
  } else {
#pragma unroll
    for (int c = 0; c < NC; c += 4) {
      const float4 x = ld4(row + c * 16 + tx * 4);
      b[c] = x.x;
      b[c + 1] = x.y;
      b[c + 2] = x.z;
      b[c + 3] = x.w;
    }
  }
}
template <int NC>
__device__ __forceinline__ int col_of(int c, int tx) {
  return NC == 2 ? tx * 2 + c : (c >> 2) * 64 + tx * 4 + (c & 3);
}

// The cluster's accumulators added into rank 0's, through distributed shared memory (`buf`: n floats a
// thread, [n][256]); false for the other ranks, which are then done.
template <int N>
__device__ __forceinline__ bool cluster_add(float (&x)[N], float *buf, int tid) {
  cg::cluster_group cl = cg::this_cluster();
  const int size = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
  if (size == 1) return true;
  __syncthreads();  // the space is free
  if (rank > 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) buf[i * 256 + tid] = x[i];
  }
  cl.sync();
  if (rank == 0) {
    for (int r = 1; r < size; ++r) {
      const float *o = cl.map_shared_rank(buf, r);
#pragma unroll
      for (int i = 0; i < N; ++i) x[i] += o[i * 256 + tid];
    }
  }
  cl.sync();  // no block leaves while rank 0 reads it
  return rank == 0;
}

// ---------------------------------------------------------------------------
// Row pass: dq, and the row terms of dbeta.  Thread (ty, tx): rows 4 ty .. + 3
// against keys (or channels) 4 tx .. + 3.
// ---------------------------------------------------------------------------
template <int DP>
struct RowLay {
  static constexpr int kNl = DP + 4;
  static constexpr int kQ = 0, kZ = DP * kBLd, kK = 2 * DP * kBLd, kX = 3 * DP * kBLd, kKn = 4 * DP * kBLd;
  static constexpr int kS = kKn + kBT * kNl;          // dS [key][row], 16-byte chunks swizzled by key
  static constexpr int kR = kS + kBT * kBT;           // R_t: four partials a row
  static constexpr int kDb = kR + 4 * kBT;
  static constexpr int kBytes = (kDb + DP) * 4;
  static_assert(kBytes <= 227 * 1024, "shared memory");
  static_assert(DP / 16 * 4 * 256 <= 2 * DP * kBLd, "the cluster's sums fit the K and X tiles");
};

template <int DP>
__global__ void __launch_bounds__(256, DP <= 64 ? 2 : 1)
    bwd_row_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                   const float *__restrict__ out, const float *__restrict__ lse, const float *__restrict__ dout,
                   const float4 *__restrict__ chan, const unsigned *__restrict__ wide, int *__restrict__ peaked,
                   float *__restrict__ power, float *__restrict__ head_power, float *__restrict__ dbp,
                   float *__restrict__ dq, int T, int d, int causal, int wide_most) {
  using Lay = RowLay<DP>;
  constexpr int NC = DP / 16, CQ = DP / 4, kShare = kBT * CQ / 256;
  extern __shared__ __align__(16) float bwd_smem[];
  float *sQ = bwd_smem + Lay::kQ, *sZ = bwd_smem + Lay::kZ, *sK = bwd_smem + Lay::kK, *sX = bwd_smem + Lay::kX,
        *sKn = bwd_smem + Lay::kKn, *sS = bwd_smem + Lay::kS, *sR = bwd_smem + Lay::kR, *sDb = bwd_smem + Lay::kDb;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, lane = tid & 31;
  const int rank = blockIdx.x, size = gridDim.x, bh = blockIdx.z;
  const unsigned *wl = wide + static_cast<size_t>(bh) * kWideWords;
  const int n_wide = wide_count(wl);
  if (n_wide > wide_most || wl[4]) {  // pair by pair is faster, or needed
    if (tid == 0) peaked[bh] = 1;
    return;
  }
  const int qt = static_cast<int>(gridDim.y) - 1 - static_cast<int>(blockIdx.y), t0 = qt * kBT;  // heaviest first
  const size_t base = static_cast<size_t>(bh) * T * d;
  const float4 *ch = chan + static_cast<size_t>(bh) * d;
  const bool vec = (d & 3) == 0;
  const float inv_sqrt_d = rsqrtf(static_cast<float>(d));
  if (tid < DP) sDb[tid] = 0.f;
  // a pair with a weight below e^-60, here or (thread 0) in another CTA of the head: the head then goes
  // pair by pair, and what the tiles give is dropped
  bool peak = tid == 0 && *reinterpret_cast<volatile int *>(peaked + bh) != 0;
  {
    const int r = tid & 63, t = min(t0 + r, T - 1);
    const bool valid = t0 + r < T;
    // the row's power of two, for the key pass as well (its partial maxima in the space of dS)
    float gm = 0.f;
    for (int jq = tid >> 6; jq < CQ; jq += 4) {
      const float4 g4 = ld_row4(dout + base + static_cast<size_t>(t) * d, jq * 4, d, vec);
      gm = fmaxf(fmaxf(gm, fmaxf(finite_abs(g4.x), finite_abs(g4.y))), fmaxf(finite_abs(g4.z), finite_abs(g4.w)));
    }
    sS[tid] = gm;
    peak = __syncthreads_or(peak);
    if (peak && size == 1) return;
    const float pw = row_power(fmaxf(fmaxf(sS[r], sS[kBT + r]), fmaxf(sS[2 * kBT + r], sS[3 * kBT + r]))), ipw = 1.f / pw;
    if (tid < kBT) {
      sS[4 * kBT + r] = pw;
      if (rank == 0 && valid) {
        power[static_cast<size_t>(bh) * T + t] = pw;
        // positive floats order as their bits
        atomicMax(reinterpret_cast<int *>(head_power) + bh, __float_as_int(pw));
      }
    }
    float R = 0.f;
    for (int jq = tid >> 6; jq < CQ; jq += 4) {
      const int j = jq * 4;
      const Chan4 cp = chan4(ch, j, d);
      const float4 q4 = ld_row4(q + base + static_cast<size_t>(t) * d, j, d, vec),
                   o4 = ld_row4(out + base + static_cast<size_t>(t) * d, j, d, vec),
                   g4 = ld_row4(dout + base + static_cast<size_t>(t) * d, j, d, vec);
      const float ov[4] = {o4.x, o4.y, o4.z, o4.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
      float z[4], db[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float g = valid ? gv[u] : 0.f;
        z[u] = row_factor(cp, u, ov[u], g * ipw);
        R += row_term(cp, u, ov[u], g * ipw);
        db[u] = cp.lin[u] > 1.f ? 0.f
                                : (cp.lin[u] != 0.f ? g * phi_over_b2(cp.b[u], cp.ib[u], cp.c[u], ov[u]) : g * cp.ib[u] * cp.ib[u]);
      }
      st_t4(sQ + j * kBLd + r, kBLd, q4);
      st_t4(sZ + j * kBLd + r, kBLd, make_float4(z[0], z[1], z[2], z[3]));
      if (rank == 0) {
#pragma unroll
        for (int off = 16; off; off >>= 1)
#pragma unroll
          for (int u = 0; u < 4; ++u) db[u] += __shfl_xor_sync(0xffffffffu, db[u], off);
        if (lane == 0)
#pragma unroll
          for (int u = 0; u < 4; ++u) atomicAdd(sDb + j + u, db[u]);
      }
    }
    sR[(tid >> 6) * kBT + r] = R;
  }
  __syncthreads();
  if (rank == 0 && tid < d) atomicAdd(dbp + static_cast<size_t>(bh) * d + tid, sDb[tid]);
  float R[4], ls[4], pw[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = ty * 4 + r;
    pw[r] = sS[4 * kBT + row];
    R[r] = (sR[row] + sR[kBT + row]) + (sR[2 * kBT + row] + sR[3 * kBT + row]);
    ls[r] = lse[static_cast<size_t>(bh) * T + min(t0 + row, T - 1)];
  }
  float2 acc[2][NC];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[i][c] = make_float2(0.f, 0.f);
  const int n_kt = causal ? qt + 1 : (T + kBT - 1) / kBT;
  for (int kt = rank; kt < n_kt; kt += size) {
    const int k0 = kt * kBT, nk = min(kBT, T - k0);
    if (__syncthreads_or(peak)) break;  // also: the previous tile is consumed
#pragma unroll
    for (int u = 0; u < kShare; ++u) {
      const int e = tid + u * 256, r = e & 63, j = (e >> 6) * 4;
      float4 k4 = make_float4(0.f, 0.f, 0.f, 0.f), x4 = k4;
      if (r < nk) {
        k4 = ld_row4(k + base + static_cast<size_t>(k0 + r) * d, j, d, vec);
        const float4 v4 = ld_row4(v + base + static_cast<size_t>(k0 + r) * d, j, d, vec);
        const Chan4 cp = chan4(ch, j, d);
        x4 = make_float4(key_factor(cp, 0, v4.x), key_factor(cp, 1, v4.y), key_factor(cp, 2, v4.z),
                         key_factor(cp, 3, v4.w));
      }
      st_t4(sK + j * kBLd + r, kBLd, k4);
      st_t4(sX + j * kBLd + r, kBLd, x4);
      *reinterpret_cast<float4 *>(sKn + r * Lay::kNl + j) = k4;
    }
    __syncthreads();
    const int others = tid == 0 ? *reinterpret_cast<volatile int *>(peaked + bh) : 0;  // lands under the contractions
    float2 s[2][4], U[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[i][c] = U[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int e = 0; e < DP; ++e) {
      const float4 a = ld4(sQ + e * kBLd + ty * 4), b4 = ld4(sK + e * kBLd + tx * 4), z = ld4(sZ + e * kBLd + ty * 4),
                   x = ld4(sX + e * kBLd + tx * 4);
      const float2 a2[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)}, z2[2] = {make_float2(z.x, z.y), make_float2(z.z, z.w)};
      const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, xx[4] = {x.x, x.y, x.z, x.w};
      outer(s, a2, bb);
      outer(U, z2, xx);
    }
    float ds[4][4], lp[4][4];  // [key][row]; lp -inf where the pair is not visible
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = k0 + tx * 4 + c;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int t = t0 + ty * 4 + r;
        const float sv = (r & 1) ? s[r >> 1][c].y : s[r >> 1][c].x, uv = (r & 1) ? U[r >> 1][c].y : U[r >> 1][c].x;
        const bool vis = i < T && t < T && (!causal || i <= t);
        const float l = fmaf(sv, inv_sqrt_d, -ls[r]);
        peak = peak || (vis && l < kPeakLog);
        lp[c][r] = vis ? l : -INFINITY;
        ds[c][r] = vis ? expf(l) * (uv + R[r]) * pw[r] : 0.f;
      }
    }
    if (peak) peaked[bh] = 1;
    peak = peak || others != 0;
    for (int w = 0, j = -1; w < n_wide; ++w) {
      j = wide_next(wl, j);
      const float b = ch[j].x, ib = ch[j].y;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float vi = v[base + static_cast<size_t>(min(k0 + tx * 4 + c, T - 1)) * d + j];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const size_t o = base + static_cast<size_t>(min(t0 + ty * 4 + r, T - 1)) * d + j;
          float qv, dsw, dbt;
          wide_terms(b, ib, vi, out[o], lp[c][r], qv, dsw, dbt);
          if (lp[c][r] > -INFINITY) ds[c][r] = fmaf(dout[o], dsw, ds[c][r]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      *reinterpret_cast<float4 *>(sS + (tx * 4 + c) * kBT + ((ty ^ tx) << 2)) =
          make_float4(ds[c][0], ds[c][1], ds[c][2], ds[c][3]);
    __syncthreads();
#pragma unroll 4
    for (int k4 = 0; k4 < kBT / 4; ++k4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 a = ld4(sS + (k4 * 4 + u) * kBT + ((ty ^ k4) << 2));
        const float2 a2[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
        float b[NC];
        ld_cols<NC>(b, sKn + (k4 * 4 + u) * Lay::kNl, tx);
        outer(acc, a2, b);
      }
    }
  }
  float x[4 * NC];
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int r = 0; r < 4; ++r) x[c * 4 + r] = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
  if (!cluster_add(x, sK, tid)) return;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int t = t0 + ty * 4 + r;
    if (t >= T) continue;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int j = col_of<NC>(c, tx);
      if (j < d) dq[base + static_cast<size_t>(t) * d + j] = x[c * 4 + r] * inv_sqrt_d;
    }
  }
}

// ---------------------------------------------------------------------------
// Key pass: dk, dv and the pair terms of dbeta.  Scores and dS by thread (ty, tx):
// rows RR ty .. against keys 4 tx .. + 3; the sums over rows by thread (ty, tx):
// keys 4 ty .. + 3 against channels 4 tx .. + 3.
// ---------------------------------------------------------------------------
template <int DP>
struct KeyLay {
  static constexpr int kRows = DP <= 64 ? 64 : 32, RR = kRows / 16, kRl = kRows + 4, kNl = DP + 4;
  static constexpr int kK = 0, kX = DP * kBLd, kQ = 2 * DP * kBLd, kZ = kQ + DP * kRl, kQn = kZ + DP * kRl;
  static constexpr int kZn = kQn + kRows * kNl, kZ2 = kZn + kRows * kNl;
  static constexpr int kP = kZ2 + kRows * kNl, kS = kP + kRows * kBT, kR = kS + kRows * kBT;
  static constexpr int kParts = 256 / kRows, kDb = kR + kParts * kRows;
  static constexpr int kBytes = (kDb + DP) * 4;
  static_assert(kBytes <= 227 * 1024, "shared memory");
  static_assert(DP / 16 * 12 * 256 <= kDb, "the cluster's sums fit the tiles");
};

template <int DP>
__global__ void __launch_bounds__(256, 1)
    bwd_key_kernel(const float *__restrict__ q, const float *__restrict__ k, const float *__restrict__ v,
                   const float *__restrict__ out, const float *__restrict__ lse, const float *__restrict__ dout,
                   const float4 *__restrict__ chan, const unsigned *__restrict__ wide, const int *__restrict__ peaked,
                   const float *__restrict__ power, const float *__restrict__ head_power, float *__restrict__ dbp,
                   float *__restrict__ dk, float *__restrict__ dv, int T, int d, int causal) {
  using Lay = KeyLay<DP>;
  constexpr int NC = DP / 16, CQ = DP / 4, kRows = Lay::kRows, RR = Lay::RR, kRl = Lay::kRl, kNl = Lay::kNl;
  extern __shared__ __align__(16) float bwd_smem[];
  float *sK = bwd_smem + Lay::kK, *sX = bwd_smem + Lay::kX, *sQ = bwd_smem + Lay::kQ, *sZ = bwd_smem + Lay::kZ,
        *sQn = bwd_smem + Lay::kQn, *sZn = bwd_smem + Lay::kZn, *sZ2 = bwd_smem + Lay::kZ2, *sP = bwd_smem + Lay::kP,
        *sS = bwd_smem + Lay::kS, *sR = bwd_smem + Lay::kR, *sDb = bwd_smem + Lay::kDb;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int rank = blockIdx.x, size = gridDim.x, bh = blockIdx.z, k0 = static_cast<int>(blockIdx.y) * kBT;
  if (peaked[bh]) return;  // the head goes pair by pair
  const unsigned *wl = wide + static_cast<size_t>(bh) * kWideWords;
  const int n_wide = wide_count(wl);
  const size_t base = static_cast<size_t>(bh) * T * d;
  const float4 *ch = chan + static_cast<size_t>(bh) * d;
  const bool vec = (d & 3) == 0;
  const float inv_sqrt_d = rsqrtf(static_cast<float>(d)), hpw = head_power[bh], ihpw = 1.f / hpw;
  if (tid < DP) sDb[tid] = 0.f;
  for (int e = tid; e < kBT * CQ; e += 256) {
    const int r = e & 63, j = (e >> 6) * 4;
    float4 k4 = make_float4(0.f, 0.f, 0.f, 0.f), x4 = k4;
    if (k0 + r < T) {
      k4 = ld_row4(k + base + static_cast<size_t>(k0 + r) * d, j, d, vec);
      const float4 v4 = ld_row4(v + base + static_cast<size_t>(k0 + r) * d, j, d, vec);
      const Chan4 cp = chan4(ch, j, d);
      x4 = make_float4(key_factor(cp, 0, v4.x), key_factor(cp, 1, v4.y), key_factor(cp, 2, v4.z), key_factor(cp, 3, v4.w));
    }
    st_t4(sK + j * kBLd + r, kBLd, k4);
    st_t4(sX + j * kBLd + r, kBLd, x4);
  }
  float2 ak[2][NC], ah[2][NC], a2h[2][NC];  // keys 4 ty .. + 3 in pairs: dk, H, H2
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) ak[i][c] = ah[i][c] = a2h[i][c] = make_float2(0.f, 0.f);
  const int first = causal ? k0 / kRows : 0, n_rt = (T + kRows - 1) / kRows;
  for (int rt = first + rank; rt < n_rt; rt += size) {
    const int t0 = rt * kRows;
    __syncthreads();  // the previous tile is consumed
    {
      const int r = tid % kRows, t = min(t0 + r, T - 1);
      const bool valid = t0 + r < T;
      const float ipw = 1.f / power[static_cast<size_t>(bh) * T + t];
      float R = 0.f;
      for (int jq = tid / kRows; jq < CQ; jq += Lay::kParts) {
        const int j = jq * 4;
        const Chan4 cp = chan4(ch, j, d);
        const float4 q4 = ld_row4(q + base + static_cast<size_t>(t) * d, j, d, vec),
                     o4 = ld_row4(out + base + static_cast<size_t>(t) * d, j, d, vec),
                     g4 = ld_row4(dout + base + static_cast<size_t>(t) * d, j, d, vec);
        const float ov[4] = {o4.x, o4.y, o4.z, o4.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
        float z[4], z2[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float g = valid ? gv[u] * ipw : 0.f;
          z[u] = row_factor(cp, u, ov[u], g);
          z2[u] = cp.lin[u] > 1.f ? 0.f : z[u] * (cp.c[u] - ov[u]);
          R += row_term(cp, u, ov[u], g);
        }
        const float4 z4 = make_float4(z[0], z[1], z[2], z[3]);
        st_t4(sQ + j * kRl + r, kRl, q4);
        st_t4(sZ + j * kRl + r, kRl, z4);
        *reinterpret_cast<float4 *>(sQn + r * kNl + j) = q4;
        *reinterpret_cast<float4 *>(sZn + r * kNl + j) = z4;
        *reinterpret_cast<float4 *>(sZ2 + r * kNl + j) = make_float4(z2[0], z2[1], z2[2], z2[3]);
      }
      sR[(tid / kRows) * kRows + r] = R;
    }
    __syncthreads();
    float2 s[RR / 2][4], U[RR / 2][4];
#pragma unroll
    for (int i = 0; i < RR / 2; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[i][c] = U[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int e = 0; e < DP; ++e) {
      float2 a2[RR / 2], z2[RR / 2];
#pragma unroll
      for (int i = 0; i < RR / 2; ++i) {
        a2[i] = *reinterpret_cast<const float2 *>(sQ + e * kRl + ty * RR + 2 * i);
        z2[i] = *reinterpret_cast<const float2 *>(sZ + e * kRl + ty * RR + 2 * i);
      }
      const float4 b4 = ld4(sK + e * kBLd + tx * 4), x = ld4(sX + e * kBLd + tx * 4);
      const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, xx[4] = {x.x, x.y, x.z, x.w};
      outer(s, a2, bb);
      outer(U, z2, xx);
    }
    float ds[RR][4], lp[RR][4];  // [row][key]; lp -inf where the pair is not visible
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int row = ty * RR + r, t = t0 + row;
      float Rt = 0.f;
#pragma unroll
      for (int p = 0; p < Lay::kParts; ++p) Rt += sR[p * kRows + row];
      const float ls = lse[static_cast<size_t>(bh) * T + min(t, T - 1)], pw = power[static_cast<size_t>(bh) * T + min(t, T - 1)];
      const float prel = pw * ihpw;
      float pv[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = k0 + tx * 4 + c;
        const float sv = (r & 1) ? s[r >> 1][c].y : s[r >> 1][c].x, uv = (r & 1) ? U[r >> 1][c].y : U[r >> 1][c].x;
        const bool vis = i < T && t < T && (!causal || i <= t);
        const float l = fmaf(sv, inv_sqrt_d, -ls);
        lp[r][c] = vis ? l : -INFINITY;
        pv[c] = vis ? expf(l) : 0.f;
        ds[r][c] = vis ? pv[c] * (uv + Rt) * pw : 0.f;
      }
      *reinterpret_cast<float4 *>(sP + row * kBT + tx * 4) =
          make_float4(pv[0] * prel, pv[1] * prel, pv[2] * prel, pv[3] * prel);
    }
    for (int w = 0, j = -1; w < n_wide; ++w) {
      j = wide_next(wl, j);
      const float b = ch[j].x, ib = ch[j].y;
      float db = 0.f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = min(k0 + tx * 4 + c, T - 1);
        const float vi = v[base + static_cast<size_t>(i) * d + j];
        float dvi = 0.f;
#pragma unroll
        for (int r = 0; r < RR; ++r) {
          const size_t o = base + static_cast<size_t>(min(t0 + ty * RR + r, T - 1)) * d + j;
          const float g = dout[o];
          float qv, dsw, dbt;
          wide_terms(b, ib, vi, out[o], lp[r][c], qv, dsw, dbt);
          if (lp[r][c] > -INFINITY) {
            ds[r][c] = fmaf(g, dsw, ds[r][c]);
            dvi = fmaf(g, qv, dvi);
            db = fmaf(g, dbt, db);
          }
        }
        dvi += __shfl_xor_sync(0xffffffffu, dvi, 16);  // the warp's two row groups
        if ((tid & 16) == 0 && k0 + tx * 4 + c < T) atomicAdd(dv + base + static_cast<size_t>(i) * d + j, dvi);
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) db += __shfl_xor_sync(0xffffffffu, db, off);
      if ((tid & 31) == 0) atomicAdd(sDb + j, db);
    }
#pragma unroll
    for (int r = 0; r < RR; ++r)
      *reinterpret_cast<float4 *>(sS + (ty * RR + r) * kBT + tx * 4) = make_float4(ds[r][0], ds[r][1], ds[r][2], ds[r][3]);
    __syncthreads();
#pragma unroll 4
    for (int r = 0; r < kRows; ++r) {
      const float4 p4 = ld4(sP + r * kBT + ty * 4), s4 = ld4(sS + r * kBT + ty * 4);
      const float2 p2[2] = {make_float2(p4.x, p4.y), make_float2(p4.z, p4.w)}, s2[2] = {make_float2(s4.x, s4.y), make_float2(s4.z, s4.w)};
      float b[NC];
      ld_cols<NC>(b, sQn + r * kNl, tx);
      outer(ak, s2, b);
      ld_cols<NC>(b, sZn + r * kNl, tx);
      outer(ah, p2, b);
      ld_cols<NC>(b, sZ2 + r * kNl, tx);
      outer(a2h, p2, b);
    }
  }
  float x[12 * NC];
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      x[c * 12 + r] = (r & 1) ? ak[r >> 1][c].y : ak[r >> 1][c].x;
      x[c * 12 + 4 + r] = (r & 1) ? ah[r >> 1][c].y : ah[r >> 1][c].x;
      x[c * 12 + 8 + r] = (r & 1) ? a2h[r >> 1][c].y : a2h[r >> 1][c].x;
    }
  const bool first_rank = cluster_add(x, bwd_smem, tid);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int j = col_of<NC>(c, tx);
    if (j >= d || !first_rank) continue;
    const float4 cp = ch[j];  // {beta, 1/beta, c, mode}
    float db = 0.f;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = k0 + ty * 4 + r;
      if (i >= T) continue;
      const size_t o = base + static_cast<size_t>(i) * d + j;
      const float vi = v[o], h = x[c * 12 + 4 + r], h2 = x[c * 12 + 8 + r], F = exp_tilt(cp.x, vi, cp.z);
      dk[o] = x[c * 12 + r] * inv_sqrt_d;
      if (cp.w > 1.f) continue;
      dv[o] = F * h * hpw;
      if (cp.w != 0.f)
        db += phi_over_b2(cp.x, cp.y, vi, cp.z) * h + em1_tilt(cp.x, cp.y, vi, cp.z) * h2;
      else
        db += F * fmaf(fmaf(cp.x, vi - cp.z, -1.f), h, cp.x * h2) * cp.y * cp.y;
    }
    if (cp.w <= 1.f) atomicAdd(sDb + j, db * hpw);
  }
  __syncthreads();
  if (tid < d) atomicAdd(dbp + static_cast<size_t>(bh) * d + tid, sDb[tid]);
}

// dbeta[h][j]: the (b, h) sums of whichever kernels took the head, over the batch.
__global__ void bwd_dbeta_kernel(const float *__restrict__ tile, const float *__restrict__ pairs,
                                 const int *__restrict__ peaked, int B, int H, int d,
                                 float *__restrict__ dbeta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H * d) return;
  float s = 0.f;
  for (int b = 0; b < B; ++b) {
    const int bh = b * H + i / d;
    s += (peaked[bh] ? pairs : tile)[static_cast<size_t>(bh) * d + i % d];
  }
  dbeta[i] = s;
}

struct BwdWs {
  size_t chan, power, tile, pairs, wide, peaked, head_power, total, zero_from;
};
BwdWs bwd_ws(int BH, int T, int d) {
  BwdWs w;
  const size_t n = static_cast<size_t>(BH) * d;
  w.chan = 0;
  w.power = n * sizeof(float4);  // the rows' powers of two
  w.zero_from = w.tile = w.power + static_cast<size_t>(BH) * T * sizeof(float);
  w.pairs = w.tile + n * sizeof(float);
  w.wide = w.pairs + n * sizeof(float);
  w.peaked = w.wide + static_cast<size_t>(BH) * kWideWords * sizeof(unsigned);
  w.head_power = w.peaked + static_cast<size_t>(BH) * sizeof(int);
  w.total = w.head_power + static_cast<size_t>(BH) * sizeof(float);
  return w;
}

template <typename Kernel, typename... Args>
cudaError_t launch_cluster(Kernel kernel, dim3 grid, int smem, cudaStream_t stream, Args... args) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = grid.x;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int DP>
cudaError_t launch_tile_dp(const float *q, const float *k, const float *v, const float *beta, const float *out,
                           const float *lse, const float *dout, float *dq, float *dk, float *dv, int BH, int H, int T,
                           int d, int causal, uint8_t *ws, const BwdWs &w, int num_sms, cudaStream_t stream) {
  float4 *chan = reinterpret_cast<float4 *>(ws + w.chan);
  float *tile = reinterpret_cast<float *>(ws + w.tile), *power = reinterpret_cast<float *>(ws + w.power),
        *head_power = reinterpret_cast<float *>(ws + w.head_power);
  unsigned *wide = reinterpret_cast<unsigned *>(ws + w.wide);
  int *peaked = reinterpret_cast<int *>(ws + w.peaked);
  const int n_t = (T + kBT - 1) / kBT;
  bwd_chan_kernel<<<dim3(BH, (d + 31) / 32 + (T >= kSampleT ? 1 : 0)), 1024, 0, stream>>>(q, k, v, beta, lse, H, T, d, causal, chan, wide, dv);
  // CTAs sharing a tile: until there are about four per SM, while each has a tile of the other side
  int size = 1;
  while (size < 8 && size * 2 <= n_t && static_cast<long long>(n_t) * BH * size < 3ll * num_sms) size *= 2;
  // Wide channels beyond which a head goes pair by pair, where that is faster: 42 us each at B1 H4 T2048 d64
  // against 2440 pair by pair, 2.4 against 75 at T64, 1.7 against 118 at B1 H1 T96 d128 (and the tiles' 62
  // and 100 are spent besides where other heads stay).
  const int wide_most = T < 256 ? 16 : 3 * d / 4;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = launch_cluster(bwd_row_kernel<DP>, dim3(size, n_t, BH), RowLay<DP>::kBytes, stream, q, k, v, out, lse, dout,
                       static_cast<const float4 *>(chan), static_cast<const unsigned *>(wide), peaked, power, head_power, tile, dq, T, d,
                       causal, wide_most);
  if (e == cudaSuccess)
    e = launch_cluster(bwd_key_kernel<DP>, dim3(size, n_t, BH), KeyLay<DP>::kBytes, stream, q, k, v, out, lse, dout,
                       static_cast<const float4 *>(chan), static_cast<const unsigned *>(wide), static_cast<const int *>(peaked), static_cast<const float *>(power),
                       static_cast<const float *>(head_power), tile, dk, dv, T, d, causal);
  return e;
}

}  // namespace

// Pair by pair / tiled, us, causal, plain heads: B*H = 1: d 16 T 64 64 / 46, d 64 T 64 62 / 63, T 80 76 / 67, T 300
// 254 / 91, d 128 T 96 107 / 103, T 128 138 / 104; B*H = 4 T 2048 d 64 2440 / 478, d 128 4141 / 840; B*H = 384: d 64 T 64
// 235 / 143, T 300 3420 / 1096, d 128 T 96 740 / 592; B*H = 64 d 16 T 1024 4452 / 770.
bool bwd_tile_takes(int B, int H, int T, int d) {
  const bool few = static_cast<long long>(B) * H * T <= kBwdFewRows;
  const int least = d <= 64 ? (d > 32 && few ? 72 : 64) : 96;
  return d <= 128 && T >= least && static_cast<long long>(T) <= 64ll * 65535 && static_cast<long long>(B) * H <= 65535;
}

size_t bwd_workspace_bytes(int B, int H, int T, int d) {
  return bwd_tile_takes(B, H, T, d) ? bwd_ws(B * H, T, d).total : 0;
}

cudaError_t launch_bwd_tile(const float *q, const float *k, const float *v, const float *beta, const float *out,
                            const float *lse, const float *dout, float *dq, float *dk, float *dv, float *dbeta, int B,
                            int H, int T, int d, int causal, void *ws, int num_sms, cudaStream_t stream) {
  const int BH = B * H;
  uint8_t *p = static_cast<uint8_t *>(ws);
  const BwdWs w = bwd_ws(BH, T, d);
  cudaError_t e = cudaMemsetAsync(p + w.zero_from, 0, w.total - w.zero_from, stream);
  if (e != cudaSuccess) return e;
  if (d <= 32)
    e = launch_tile_dp<32>(q, k, v, beta, out, lse, dout, dq, dk, dv, BH, H, T, d, causal, p, w, num_sms, stream);
  else if (d <= 64)
    e = launch_tile_dp<64>(q, k, v, beta, out, lse, dout, dq, dk, dv, BH, H, T, d, causal, p, w, num_sms, stream);
  else
    e = launch_tile_dp<128>(q, k, v, beta, out, lse, dout, dq, dk, dv, BH, H, T, d, causal, p, w, num_sms, stream);
  if (e != cudaSuccess) return e;
  const int *peaked = reinterpret_cast<const int *>(p + w.peaked);
  float *pairs = reinterpret_cast<float *>(p + w.pairs);
  e = launch_bwd_pairs(q, k, v, beta, out, lse, dout, dq, dk, dv, pairs, B, H, T, d, causal, peaked, stream);
  if (e != cudaSuccess) return e;
  bwd_dbeta_kernel<<<(H * d + 255) / 256, 256, 0, stream>>>(reinterpret_cast<const float *>(p + w.tile), pairs, peaked, B, H,
                                                           d, dbeta);
  return cudaGetLastError();
}

}  // namespace fem
