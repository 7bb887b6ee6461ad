// FEM over a gated-linear-attention prior, chunked on the tensor cores
// (App. "Gated Linear Attention (GLA) Prior", Eqs. "gla-score-appendix" and
// "gla-assoc"):
//
//   s_t(i) = K_{t,i} <qf_t, kf_i> (i <= t),  K_{t,i} = exp(g_{i+1} + ... + g_t),
//   p_t = s_t / Z_t,  o_{t,j} = (1/beta_j) log sum_i p_t(i) exp(beta_j v_{i,j}).
//
// In chunks of 128 steps, with gamma_t the running sum of g inside the chunk (so
// K_{t,i} = exp(gamma_t - gamma_i) for i, t in the chunk and exp(gamma_t) from the
// chunk start), a chunk is four contractions on tcgen05 (kind::f16, bf16 operands,
// fp32 accumulation in TMEM):
//
//   S     = Qf Kf^T                                  [128 x 128], K = m
//   intra = (S o decay-mask) E^T                     [128 x 64],  K = 128 keys
//   inter = Qf Shat^T                                [128 x 64],  K = m
//   U     = (Kf o exp(gamma_last - gamma_i))^T E^T   [m x 65],    K = 128 keys
//
// E holds, per channel j and key i, the value bank of the chunk (in U a channel 64
// of ones gives the normaliser Z, "A one-pass implementation appends a constant
// channel to values").  Shat is the state at the chunk's start, sum over earlier
// keys of K_{.,i} kf_i E_ij, kept in fp32 (its bf16 copy only feeds the
// contraction).  Per channel, two forms of the bank, fixed for the sequence:
//
//   beta_j <  1/4: linear, E = expm1(beta (v - c)) / beta with the anchor c the
//     mean of the values so far, at most 1/beta above their minimum; when c moves
//     to c', the state becomes e^{beta (c - c')} Shat_j + expm1(beta (c - c')) / beta
//     Shat_Z, and the read is o = c + log1p(beta num / Z) / beta (c + num / Z at
//     beta = 0);
//   beta_j >= 1/4: shifted, E = exp(beta v - lambda) with lambda the chunk's
//     largest beta v, the state carried as e^{mu} Shat with mu the log of its
//     scale, and the read o = (log num - log Z) / beta with log num the
//     log-sum-exp of the chunk's and the state's parts.
//
// The recurrence over chunks is linear in the state, so the chunks run in parallel
// (a CTA pair per head that walked its 64 chunks in turn, operand preparation,
// mask, read-out and state update one behind the other, took 1.08 ms at B4 H16 T8192,
// 14.5 us a chunk on 128 of 152 SMs):
//
//   stats   the values' extremes and sums per chunk, the summed log-decay
//   anchor  per channel, the chunks' shifts c or lambda and the scan's factors
//   local   per chunk: E and Kf as bf16 operand images, and U
//   scan    per state element, the chunks in turn: the start states
//   out     per chunk: S, mask, intra, inter and the read
//
// B4 H16 T8192: 23 + 10 + 102 + 34 + 171 us, 356 in all (the inputs and outputs once are 80).
// local and scan run at 4.7 and 4 TB/s; out is bound by its phases' latencies (2 us of loads, then scores,
// mask, sums and read behind one another, two chunks an SM at a time: TMEM holds no more).  All five run
// over groups of heads (gla_par_group).
//
// The bf16 operands' relative error (2^-9) reaches o as about 2^-9 |v - c| (linear)
// or 2^-9 / beta (shifted), the same order as the bf16 softmax read's.  The mask's
// rounded weights are the ones summed into Z.  A shifted channel's in-chunk sum for
// row t uses the chunk's largest value as its shift, which may come after t; when
// that sum falls below 2^-100 of the row's in-chunk prior mass (terms under fp32's
// range could then carry it) the entry is recomputed exactly, from the scores of
// the bf16 operands in fp32, with the running maximum of the row's visible keys as the shift.
#include "fem_common.cuh"
#include "fem_gla_tc.cuh"
#include "fem_launch.h"

namespace fem {
namespace {

constexpr int kGD = 64;    // value channels
constexpr int kGN = 80;    // U's columns: the channels, the constant one, zero padding to a multiple of 16
constexpr int kSt = (kGD + 1) * kGM;  // floats of a state: channel rows of 64 features, Z's last
constexpr uint32_t kImg = 16384;  // a 128 x 64 bf16 operand image

// Workspace of a group of heads; per (head, chunk) unless noted.
struct GlaTcWs {
  float4 *stat;   // [64]: the chunk's max, min and sum of v
  float *shift;   // [64]: c (linear) or lambda (shifted)
  float *mu;      // [64]: the log-scale of the start state (shifted)
  float4 *fac;    // [64]: the scan's factors {e, w, fr, fl}
  float *glast;   // the chunk's summed log-decay
  uint8_t *k16;   // Kf, 128-byte-swizzled rows of 64 features
  uint8_t *e16;   // E, two boxes of 64 channels x 64 keys, likewise
  float *u;       // [65][64]
  float *s;       // [65][64]
};

__device__ __forceinline__ float2 unpack_bf16x2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// 8 consecutive fp32 as bf16 into a 16-byte chunk of a 128-byte-swizzled row.
__device__ __forceinline__ void st_bf16x8(uint8_t *dst, float4 a, float4 b) {
  *reinterpret_cast<uint4 *>(dst) =
      make_uint4(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w), pack_bf16x2(b.x, b.y), pack_bf16x2(b.z, b.w));
}

// gam[t] = g_0 + ... + g_t over the chunk (steps past the end add nothing); 128 threads or more, `tot` 4 floats.
__device__ __forceinline__ void chunk_decay(const float *g, int rows, float *gam, float *tot) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float x = 0.f;
  if (tid < kGC) {
    x = tid < rows ? g[tid] : 0.f;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= off) x += y;
    }
    if (lane == 31) tot[warp] = x;
  }
  __syncthreads();
  if (tid < kGC) {
    float add = 0.f;
    for (int w = 0; w < warp; ++w) add += tot[w];
    gam[tid] = x + add;
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// stats: block per chunk; thread = four channels of 16 rows.  The sums' order is the walking kernel's, here
// and in the anchors and scales: their last bits decide roundings of the bank and the state to bf16.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) gla_stats_kernel(const float *__restrict__ v, const float *__restrict__ logdecay,
                                                        int T, int n_ch, float4 *__restrict__ stat,
                                                        float *__restrict__ glast) {
  __shared__ float4 s_mx[8][16], s_mn[8][16], s_sm[8][16];
  __shared__ float gam[kGC], tot[4];
  const int c = blockIdx.x, hd = blockIdx.y, q = threadIdx.x & 15, part = threadIdx.x >> 4;
  const int rows = min(kGC, T - c * kGC);
  const size_t r0 = static_cast<size_t>(hd) * T + static_cast<size_t>(c) * kGC;
  const float4 *src = reinterpret_cast<const float4 *>(v + r0 * kGD);
  float4 x[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) x[u] = part * 16 + u < rows ? src[(part * 16 + u) * 16 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
  chunk_decay(logdecay + r0, rows, gam, tot);
  if (threadIdx.x == 0) glast[static_cast<size_t>(hd) * n_ch + c] = gam[kGC - 1];
  float4 mx = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), mn = make_float4(INFINITY, INFINITY, INFINITY, INFINITY),
         sm = make_float4(0.f, 0.f, 0.f, 0.f);
  auto fold = [&](float4 a, float4 b, float4 s) {
    mx = make_float4(fmaxf(mx.x, a.x), fmaxf(mx.y, a.y), fmaxf(mx.z, a.z), fmaxf(mx.w, a.w));
    mn = make_float4(fminf(mn.x, b.x), fminf(mn.y, b.y), fminf(mn.z, b.z), fminf(mn.w, b.w));
    sm = make_float4(sm.x + s.x, sm.y + s.y, sm.z + s.z, sm.w + s.w);
  };
#pragma unroll
  for (int u = 0; u < 16; ++u)
    if (part * 16 + u < rows) fold(x[u], x[u], x[u]);
  s_mx[part][q] = mx;
  s_mn[part][q] = mn;
  s_sm[part][q] = sm;
  __syncthreads();
  if (part == 0) {
    for (int p = 1; p < 8; ++p) fold(s_mx[p][q], s_mn[p][q], s_sm[p][q]);
    float4 *o = stat + (static_cast<size_t>(hd) * n_ch + c) * kGD + q * 4;
    o[0] = make_float4(mx.x, mn.x, sm.x, 0.f);
    o[1] = make_float4(mx.y, mn.y, sm.y, 0.f);
    o[2] = make_float4(mx.z, mn.z, sm.z, 0.f);
    o[3] = make_float4(mx.w, mn.w, sm.w, 0.f);
  }
}

// ---------------------------------------------------------------------------
// anchor: warp per channel, lane = chunk; the running sum and scale over 32 chunks at a time, in order, from
// shuffles that don't wait for the chain (a thread per channel walking the chunks took 21 us at 64 of them).  The state element S of a channel (Z its
// feature's in the normaliser's state) goes from chunk to chunk as
//   start = e S + w Z     (linear: the move with the anchor; shifted: e = 1, w = 0)
//   S     = fr start + fl U
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gla_anchor_kernel(const float *__restrict__ beta, int h0, int H, int T, int n_ch,
                                                         GlaTcWs w) {
  const int lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5), hd = blockIdx.y;
  const float b = normal_beta(beta[((h0 + hd) % H) * kGD + j]);
  const bool shifted = b >= kGlaLinBeta;
  const size_t t0 = static_cast<size_t>(hd) * n_ch;
  float rmin = INFINITY, rsum = 0.f, c_old = INFINITY, mu = -INFINITY;  // carried over the groups of 32 chunks
  for (int c0 = 0; c0 < n_ch; c0 += 32) {
    const int c = c0 + lane;
    const bool in = c < n_ch;
    const size_t o = (t0 + (in ? c : 0)) * kGD + j;
    const float4 x = w.stat[o];
    const float gl = in ? w.glast[t0 + c] : 0.f;
    if (shifted) {
      const float lam = in ? b * x.x : -INFINITY;
      float after = mu, before = mu;  // the log-scales after and before this chunk
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const float gk = __shfl_sync(0xffffffffu, gl, k), lk = __shfl_sync(0xffffffffu, lam, k);
        if (lane == k) before = mu;
        mu = fmaxf(mu + gk, lk);
        if (lane == k) after = mu;
      }
      if (in) {
        w.shift[o] = lam;
        w.mu[o] = before;
        w.fac[o] = make_float4(1.f, 0.f, __expf(before + gl - after), __expf(lam - after));
      }
    } else {
      // the anchor: the mean of the values so far, at most 1/beta above their minimum (so that
      // 1 + beta num / Z >= 1/e); the state moves with it (either way)
      float mn = in ? x.y : INFINITY, sm = 0.f;
      const float own = in ? x.z : 0.f;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const float pm = __shfl_up_sync(0xffffffffu, mn, off);
        if (lane >= off) mn = fminf(mn, pm);
      }
      mn = fminf(mn, rmin);
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        rsum += __shfl_sync(0xffffffffu, own, k);
        if (lane == k) sm = rsum;
      }
      const float mean = sm / static_cast<float>(min(T, (c + 1) * kGC));
      const float cn = b > 0.f ? fminf(mean, mn + 1.f / b) : mean;
      float co = __shfl_up_sync(0xffffffffu, cn, 1);
      if (lane == 0) co = c_old;
      const bool mv = c > 0 && cn != co;
      const float d = co - cn;
      if (in) {
        w.shift[o] = cn;
        w.fac[o] = make_float4(mv ? expf(b * d) : 1.f, mv ? (b != 0.f ? expm1f(b * d) / b : d) : 0.f, __expf(gl), 1.f);
      }
      rmin = __shfl_sync(0xffffffffu, mn, 31);
      c_old = __shfl_sync(0xffffffffu, cn, 31);
    }
  }
}

// ---------------------------------------------------------------------------
// local: per chunk, E and Kf as operand images, U.  Bound by the inputs' loads (K
// and V once); about 70 KB of shared memory, three CTAs per SM.
// ---------------------------------------------------------------------------
struct LocLay {
  static constexpr uint32_t kE16 = 0;                        // two boxes of kGN channels x 64 keys
  static constexpr uint32_t kEBox = kGN * 128;
  static constexpr uint32_t kKT16 = 2 * kEBox;               // two boxes of 128 rows (64 features) x 64 keys;
  static constexpr uint32_t kK16 = kKT16 + kImg + 8192;      // rows 64..127 are not written nor their results read
  static constexpr uint32_t kGam = kK16 + kImg;
  static constexpr uint32_t kDk = kGam + 512;
  static constexpr uint32_t kTot = kDk + 512;
  static constexpr uint32_t kBar = kTot + 64;
  static constexpr uint32_t kTmemSlot = kBar + 16;
  static constexpr uint32_t kBytes = kTmemSlot + 16;
  static constexpr uint32_t kAlloc = kBytes + 1024;
  static_assert(kEBox % 1024 == 0 && kKT16 % 1024 == 0 && kK16 % 1024 == 0, "swizzled operands on 1024-byte boundaries");
};

__global__ void __launch_bounds__(256, 3) gla_local_kernel(const float *__restrict__ kf, const float *__restrict__ v,
                                                        const float *__restrict__ logdecay,
                                                        const float *__restrict__ beta, int h0, int H, int T, int n_ch,
                                                        GlaTcWs w, unsigned *__restrict__ err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem), bar = sbase + LocLay::kBar;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int c = blockIdx.x, hd = blockIdx.y, rows = min(kGC, T - c * kGC);
  const size_t r0 = static_cast<size_t>(hd) * T + static_cast<size_t>(c) * kGC, task = static_cast<size_t>(hd) * n_ch + c;
  float *gam = reinterpret_cast<float *>(smem + LocLay::kGam), *dk = reinterpret_cast<float *>(smem + LocLay::kDk);
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(sbase + LocLay::kTmemSlot, 128);
    tmem_relinquish();
  }
  // channel (or feature) j, 32 keys of it: lanes over channels, 32 loads in flight
  const int j = tid & 63, grp = tid >> 6;
  float x[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) x[u] = grp * 32 + u < rows ? __ldg(v + (r0 + grp * 32 + u) * kGD + j) : 0.f;
  chunk_decay(logdecay + r0, rows, gam, reinterpret_cast<float *>(smem + LocLay::kTot));
  const float glast = gam[kGC - 1];
  if (tid < kGC) dk[tid] = expf(glast - gam[tid]);
  __syncthreads();
  {
    // the bank: 8 keys' entries to a 16-byte chunk
    const float b = normal_beta(beta[((h0 + hd) % H) * kGD + j]), sh = w.shift[task * kGD + j], rb = b != 0.f ? 1.f / b : 0.f;
    const bool lin = b < kGlaLinBeta;
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
      float e[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float xv = x[kc * 8 + u];
        const float val = lin ? em1_beta_fast(xv - sh, b * (xv - sh), rb) : __expf(b * xv - sh);
        e[u] = grp * 32 + kc * 8 + u < rows ? val : 0.f;
      }
      const int kq = grp * 4 + kc;  // the row's 16-byte chunk over both boxes
      *reinterpret_cast<uint4 *>(smem + LocLay::kE16 + (kq >> 3) * LocLay::kEBox + sw128_offset(j, kq & 7)) =
          make_uint4(pack_bf16x2(e[0], e[1]), pack_bf16x2(e[2], e[3]), pack_bf16x2(e[4], e[5]), pack_bf16x2(e[6], e[7]));
    }
  }
  // the constant channel and the padding
  for (int i = tid; i < 2 * (kGN - kGD) * 8; i += 256) {
    const int bx = i / ((kGN - kGD) * 8), r = kGD + (i >> 3) % (kGN - kGD), chk = i & 7;
    const uint32_t one = r == kGD ? pack_bf16x2(1.f, 1.f) : 0u;
    *reinterpret_cast<uint4 *>(smem + LocLay::kE16 + bx * LocLay::kEBox + sw128_offset(r, chk)) = make_uint4(one, one, one, one);
  }
  {
#pragma unroll
    for (int u = 0; u < 32; ++u) x[u] = grp * 32 + u < rows ? __ldg(kf + (r0 + grp * 32 + u) * kGM + j) : 0.f;
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
      const int kq = grp * 4 + kc;
      float t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = x[kc * 8 + u] * dk[kq * 8 + u];
      *reinterpret_cast<uint4 *>(smem + LocLay::kKT16 + (kq >> 3) * kImg + sw128_offset(j, kq & 7)) =
          make_uint4(pack_bf16x2(t[0], t[1]), pack_bf16x2(t[2], t[3]), pack_bf16x2(t[4], t[5]), pack_bf16x2(t[6], t[7]));
    }
  }
  // Kf by rows (the same lines, from L1 or L2)
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = tid + u * 256, rr = i >> 3, chk = i & 7;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (rr < rows) {
      const float4 *src = reinterpret_cast<const float4 *>(kf + (r0 + rr) * kGM + chk * 8);
      a = __ldg(src);
      b = __ldg(src + 1);
    }
    st_bf16x8(smem + LocLay::kK16 + sw128_offset(rr, chk), a, b);
  }
  fence_proxy_async_smem();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + LocLay::kTmemSlot);
  if (warp == 1) {
    const uint32_t lead = lane == 0 ? 1u : 0u;
    constexpr uint32_t id_n = idesc_f16(128, kGN, true, false);
#pragma unroll
    for (int kk = 0; kk < kGC / 16; ++kk)
      mma_f16_ss(lead, tmem, smem_desc_sw128(sbase + LocLay::kKT16 + (kk >> 2) * kImg + (kk & 3) * 32, 16, 1024),
                 smem_desc_sw128(sbase + LocLay::kE16 + (kk >> 2) * LocLay::kEBox + (kk & 3) * 32, 16, 1024), id_n,
                 kk > 0 ? 1u : 0u);
    mma_commit(lead, bar);
  } else if (tid == 64) {
    bulk_store(w.k16 + task * kImg, sbase + LocLay::kK16, kImg);
    bulk_store(w.e16 + task * kImg, sbase + LocLay::kE16, kGD * 128);
    bulk_store(w.e16 + task * kImg + kGD * 128, sbase + LocLay::kE16 + LocLay::kEBox, kGD * 128);
    bulk_commit_group();
    bulk_wait_group_read0();
  }
  const bool ok = __all_sync(0xffffffffu, mbar_wait(bar, 0, err, kErrWaitMma));
  if (ok && warp < 2) {
    tc_fence_after_sync();
    // thread = feature (TMEM lane); a channel's 64 features are consecutive
    float *u = w.u + task * kSt + tid;
    const uint32_t lo = static_cast<uint32_t>(warp * 32) << 16;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t x[32];
      tmem_ld32(tmem + lo + q * 32, x);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 32; ++i) u[(q * 32 + i) * kGM] = __uint_as_float(x[i]);
    }
    const uint32_t z = tmem_ld1(tmem + lo + kGD);
    tmem_ld_wait();
    u[kGD * kGM] = __uint_as_float(z);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 128);
  }
}

// ---------------------------------------------------------------------------
// scan: thread per state element (channel, feature), the chunks in turn; block = four
// channels of a head, the last block the normaliser's.  Bound by U's and the start states'
// bytes; kAhead chunks' loads in flight (with the factors formed here the chain of
// exponentials took 88 us at B4 H16 T8192).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gla_scan_kernel(int n_ch, GlaTcWs w) {
  constexpr int kAhead = 8;
  const int f = threadIdx.x & 63, j = blockIdx.x * 4 + (threadIdx.x >> 6), hd = blockIdx.y;
  if (j > kGD) return;
  const bool is_z = j == kGD;
  const size_t t0 = static_cast<size_t>(hd) * n_ch;
  const float *uj = w.u + t0 * kSt + j * kGM + f, *uz = w.u + t0 * kSt + kGD * kGM + f;
  const float4 *fj = w.fac + t0 * kGD + j;
  float *sj = w.s + t0 * kSt + j * kGM + f;
  float S = 0.f, Z = 0.f;
  for (int c0 = 0; c0 < n_ch; c0 += kAhead) {
    float nu[kAhead], nz[kAhead], eg[kAhead];
    float4 fc[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      const size_t p = c0 + q;
      if (c0 + q < n_ch) {
        nu[q] = uj[p * kSt];
        nz[q] = is_z ? 0.f : uz[p * kSt];
        eg[q] = w.glast[t0 + p];
        fc[q] = is_z ? make_float4(1.f, 0.f, 0.f, 1.f) : fj[p * kGD];
      }
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      const size_t p = c0 + q;
      if (c0 + q >= n_ch) break;
      const float g = __expf(eg[q]), start = fmaf(fc[q].x, S, fc[q].y * Z);
      sj[p * kSt] = start;
      S = fmaf(is_z ? g : fc[q].z, start, fc[q].w * nu[q]);
      Z = fmaf(g, Z, nz[q]);
    }
  }
}

// ---------------------------------------------------------------------------
// out: per chunk, the scores, the mask, both parts of every channel's sum and the read.
// 256 threads, half of TMEM and about 94 KB of shared memory: two CTAs per SM.
// ---------------------------------------------------------------------------
struct OutLay {
  static constexpr uint32_t kQ16 = 0, kK16 = kImg;
  static constexpr uint32_t kE16 = 2 * kImg;        // two boxes of 64 channels x 64 keys
  static constexpr uint32_t kS16 = 3 * kImg;        // 64 channels x 64 features
  static constexpr uint32_t kOut = kS16 + 8192;     // the outputs, 128 rows of kOutLd fp32
  static constexpr int kOutLd = kGD + 4;            // a thread per row: 16-byte stores over all banks
  static constexpr uint32_t kSz = kOut + kGC * kOutLd * 4;  // Z's state, rounded to bf16, as fp32 [64]
  static constexpr uint32_t kGam = kSz + 256;
  static constexpr uint32_t kZ = kGam + 512;         // per row: in-chunk mass by halves of the keys, then the state's
  // per channel: linear {beta, 1/beta, c, -}, shifted {beta, ln 2 / beta, lambda log2 e, mu log2 e}
  static constexpr uint32_t kPar = kZ + 3 * 512;
  static constexpr uint32_t kTot = kPar + 64 * 16;
  static constexpr uint32_t kBar = kTot + 64;       // inputs, scores, sums
  static constexpr uint32_t kTmemSlot = kBar + 32;
  static constexpr uint32_t kBytes = kTmemSlot + 32;
  static constexpr uint32_t kAlloc = kBytes + 1024;
  static_assert(kAlloc <= 113 * 1024, "two CTAs per SM");
};
// TMEM columns: the scores (then, over their first 64, the masked bf16 weights), intra, inter
constexpr uint32_t kColS = 0, kColIntra = 128, kColInter = 192;

__global__ void __launch_bounds__(256, 2) gla_out_kernel(const float *__restrict__ qf, const float *__restrict__ v,
                                                         const float *__restrict__ logdecay,
                                                         const float *__restrict__ beta, float *__restrict__ out,
                                                         float *__restrict__ logz, int h0, int H, int T, int n_ch, GlaTcWs w,
                                                         unsigned *__restrict__ err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem), bar_in = sbase + OutLay::kBar, bar_s = bar_in + 8, bar_a = bar_in + 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int c = blockIdx.x, hd = blockIdx.y, rows = min(kGC, T - c * kGC);
  const size_t r0 = static_cast<size_t>(hd) * T + static_cast<size_t>(c) * kGC, task = static_cast<size_t>(hd) * n_ch + c;
  float *gam = reinterpret_cast<float *>(smem + OutLay::kGam), *s_z = reinterpret_cast<float *>(smem + OutLay::kZ),
        *s_sz = reinterpret_cast<float *>(smem + OutLay::kSz);
  float4 *par = reinterpret_cast<float4 *>(smem + OutLay::kPar);
  if (tid == 0) {
    mbar_init(bar_in, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_a, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar_in, 2 * kImg);
    bulk_load(sbase + OutLay::kK16, w.k16 + task * kImg, kImg, bar_in);
    bulk_load(sbase + OutLay::kE16, w.e16 + task * kImg, kImg, bar_in);
  }
  if (warp == 1) {
    tmem_alloc(sbase + OutLay::kTmemSlot, 256);
    tmem_relinquish();
  }
  // Qf and the start state as bf16 (K-major, 128-byte swizzle); all loads in flight
  {
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = tid + u * 256, rr = i >> 3, chk = i & 7;
      a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (rr < rows) {
        const float4 *src = reinterpret_cast<const float4 *>(qf + (r0 + rr) * kGM + chk * 8);
        a[u] = __ldg(src);
        b[u] = __ldg(src + 1);
      }
    }
    float4 sa[2], sb[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float4 *src = reinterpret_cast<const float4 *>(w.s + task * kSt) + (tid + u * 256) * 2;
      sa[u] = src[0];
      sb[u] = src[1];
    }
    const float sz = tid < kGM ? w.s[task * kSt + kGD * kGM + tid] : 0.f;
    if (tid < kGD) {
      const float bj = normal_beta(beta[((h0 + hd) % H) * kGD + tid]), sh = w.shift[task * kGD + tid];
      par[tid] = bj >= kGlaLinBeta ? make_float4(bj, kLn2 / bj, sh * kLog2e, w.mu[task * kGD + tid] * kLog2e)
                                   : make_float4(bj, bj != 0.f ? 1.f / bj : 0.f, sh, 0.f);
    }
    chunk_decay(logdecay + r0, rows, gam, reinterpret_cast<float *>(smem + OutLay::kTot));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = tid + u * 256;
      st_bf16x8(smem + OutLay::kQ16 + sw128_offset(i >> 3, i & 7), a[u], b[u]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int i = tid + u * 256;
      st_bf16x8(smem + OutLay::kS16 + sw128_offset(i >> 3, i & 7), sa[u], sb[u]);
    }
    if (tid < kGM) s_sz[tid] = __bfloat162float(__float2bfloat16_rn(sz));
  }
  fence_proxy_async_smem();
  tc_fence_before_sync();
  bool ok = __syncthreads_and(mbar_wait(bar_in, 0, err, kErrWaitTma));
  tc_fence_after_sync();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + OutLay::kTmemSlot);
  const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const uint32_t lead = lane == 0 ? 1u : 0u;
  const int t = (warp & 3) * 32 + lane, half = warp >> 2;  // row; half of the keys, then of the channels
  if (ok) {
    if (warp == 0) {
      constexpr uint32_t id_s = idesc_f16(128, 128, true, false), id_n = idesc_f16(128, kGD, true, false);
#pragma unroll
      for (int kk = 0; kk < kGM / 16; ++kk)
        mma_f16_ss(lead, tmem + kColS, smem_desc_sw128(sbase + OutLay::kQ16 + kk * 32, 16, 1024),
                   smem_desc_sw128(sbase + OutLay::kK16 + kk * 32, 16, 1024), id_s, kk > 0 ? 1u : 0u);
#pragma unroll
      for (int kk = 0; kk < kGM / 16; ++kk)
        mma_f16_ss(lead, tmem + kColInter, smem_desc_sw128(sbase + OutLay::kQ16 + kk * 32, 16, 1024),
                   smem_desc_sw128(sbase + OutLay::kS16 + kk * 32, 16, 1024), id_n, kk > 0 ? 1u : 0u);
      mma_commit(lead, bar_s);
    }
    // meanwhile the state's mass of row tid: the rounded operands of a contraction with Z's state
    if (tid >= 128) {
      const int rr = tid - 128;
      float z0 = 0.f, z1 = 0.f;
#pragma unroll
      for (int chk = 0; chk < 8; ++chk) {
        const uint4 q4 = *reinterpret_cast<const uint4 *>(smem + OutLay::kQ16 + sw128_offset(rr, chk));
        const uint32_t qw[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float2 q2 = unpack_bf16x2(qw[u]);
          z0 = fmaf(q2.x, s_sz[chk * 8 + 2 * u], z0);
          z1 = fmaf(q2.y, s_sz[chk * 8 + 2 * u + 1], z1);
        }
      }
      s_z[2 * kGC + rr] = z0 + z1;
    }
    // ---- S o decay mask, as bf16 over the scores' first 64 columns, and the rounded weights' row sum
    ok = __all_sync(0xffffffffu, mbar_wait(bar_s, 0, err, kErrWaitMma));
  }
  uint32_t p[32];
  if (ok) {
    tc_fence_after_sync();
    uint32_t s[2][32];
#pragma unroll
    for (int q = 0; q < 2; ++q) tmem_ld32(tmem + kColS + lane_off + (half * 2 + q) * 32, s[q]);
    tmem_ld_wait();
    // by 32 x 32 blocks, a warp's rows against two of them; those after the diagonal are zero
    const float gt = gam[t];
    float z0 = 0.f, z1 = 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int kb = half * 2 + q, rb = warp & 3;
      if (kb > rb) {
#pragma unroll
        for (int i2 = 0; i2 < 16; ++i2) p[q * 16 + i2] = 0u;
        continue;
      }
#pragma unroll
      for (int i2 = 0; i2 < 16; ++i2) {
        const int i = kb * 32 + 2 * i2;
        const float2 gi = *reinterpret_cast<const float2 *>(gam + i);
        const float d0 = i <= t ? __expf(gt - gi.x) : 0.f, d1 = i + 1 <= t ? __expf(gt - gi.y) : 0.f;
        p[q * 16 + i2] = pack_bf16x2(__uint_as_float(s[q][2 * i2]) * d0, __uint_as_float(s[q][2 * i2 + 1]) * d1);
        const float2 r2 = unpack_bf16x2(p[q * 16 + i2]);
        z0 += r2.x;
        z1 += r2.y;
      }
    }
    s_z[half * kGC + t] = z0 + z1;
  }
  tc_fence_before_sync();
  ok = __syncthreads_and(ok);  // both halves have read the scores
  if (ok) {
    tc_fence_after_sync();
    tmem_st32(tmem + kColS + lane_off + half * 32, p);
    tmem_st_wait();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (ok) {
    if (warp == 0) {
      tc_fence_after_sync();
      constexpr uint32_t id_n = idesc_f16(128, kGD, true, false);
#pragma unroll
      for (int kk = 0; kk < kGC / 16; ++kk)
        mma_f16_ts(lead, tmem + kColIntra, tmem + kColS + kk * 8,
                   smem_desc_sw128(sbase + OutLay::kE16 + (kk >> 2) * 8192 + (kk & 3) * 32, 16, 1024), id_n, kk > 0 ? 1u : 0u);
      mma_commit(lead, bar_a);
    }
    ok = __all_sync(0xffffffffu, mbar_wait(bar_a, 0, err, kErrWaitMma));
  }
  ok = __syncthreads_and(ok);  // also: the operands in shared memory are consumed
  // ---- the read: thread = row, half of the channels, eight at a time; outputs staged by row
  float *so = reinterpret_cast<float *>(smem + OutLay::kOut);
  if (ok) {
    tc_fence_after_sync();
    const float gt = gam[t], gt2 = gt * kLog2e, et = __expf(gt), zi = s_z[t] + s_z[kGC + t];
    const float Z = fmaf(et, s_z[2 * kGC + t], zi), lz2 = lg2_approx(Z), lz = lz2 * kLn2, rZ = 1.f / Z, zmin = 0x1p-100f * zi;
    if (half == 0 && t < rows && logz) logz[r0 + t] = lz;
    // shifted channels whose in-chunk sum fell below 2^-100 of the row's in-chunk prior mass:
    // the chunk's shift may lie far above every key the row sees (the largest value came
    // later in the chunk), so terms under fp32's range may carry the sum; recomputed below
    unsigned flag = 0;
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      const int j0 = half * 32 + q * 8;
      uint32_t ai[8], ax[8];
      tmem_ld8(tmem + kColIntra + lane_off + j0, ai);
      tmem_ld8(tmem + kColInter + lane_off + j0, ax);
      tmem_ld_wait();
      float o[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float4 pj = par[j0 + u];  // beta, 1/beta, c or lambda, mu
        const float in = __uint_as_float(ai[u]), ix = __uint_as_float(ax[u]);
        if (pj.x < kGlaLinBeta) {  // the form is the channel's: no divergence
          const float num = fmaf(et, ix, in);
          o[u] = pj.x != 0.f ? fmaf(log1p_fast(pj.x * num * rZ), pj.y, pj.z) : fmaf(num, rZ, pj.z);
        } else {
          const float lb = pj.w + gt2, dl = pj.z - lb, ed = ex2_approx(-fabsf(dl));
          const float sum = dl >= 0.f ? fmaf(ix, ed, in) : fmaf(in, ed, ix);
          flag |= !(in >= zmin) ? 1u << (q * 8 + u) : 0u;
          o[u] = ((fmaxf(pj.z, lb) - lz2) + lg2_approx(sum)) * pj.y;
          // the larger scale's part too small to be the shift (or none, for features that meet no key of the chunk)
          if (!(sum > 0x1p-100f) && (in > 0.f || ix > 0.f)) {
            const float la2 = in > 0.f ? pj.z + lg2_approx(in) : -INFINITY,
                        lb2 = ix > 0.f ? lb + lg2_approx(ix) : -INFINITY;
            o[u] = ((fmaxf(la2, lb2) - lz2) + lg2_approx(1.f + ex2_approx(-fabsf(la2 - lb2)))) * pj.y;
          }
        }
      }
      float4 *orow = reinterpret_cast<float4 *>(so + t * OutLay::kOutLd + j0);
      orow[0] = make_float4(o[0], o[1], o[2], o[3]);
      orow[1] = make_float4(o[4], o[5], o[6], o[7]);
    }
    // the flagged entries exactly, one at a time by the warp: lanes take every 32nd key, scores from the
    // operands in shared memory, the visible keys' largest beta v as the shift
    unsigned who = __ballot_sync(0xffffffffu, flag != 0u && t < rows);
    while (who) {
      const int src = __ffs(who) - 1;
      who &= who - 1;
      unsigned fm = __shfl_sync(0xffffffffu, flag, src);
      const int te = __shfl_sync(0xffffffffu, t, src);
      const float ge = gam[te], lze = __shfl_sync(0xffffffffu, lz, src);
      const float *qrow = qf + (r0 + te) * kGM;
      float a[4];  // the row's weights on the lane's keys
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) {
        const int i = lane + 32 * k2;
        float d = 0.f;
        if (i <= te) {
#pragma unroll
          for (int chk = 0; chk < 8; ++chk) {
            const uint4 q4 = *reinterpret_cast<const uint4 *>(smem + OutLay::kQ16 + sw128_offset(te, chk)),
                        k4 = *reinterpret_cast<const uint4 *>(smem + OutLay::kK16 + sw128_offset(i, chk));
            const uint32_t qw[4] = {q4.x, q4.y, q4.z, q4.w}, kw[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float2 q2 = unpack_bf16x2(qw[u]), k2v = unpack_bf16x2(kw[u]);
              d = fmaf(q2.x, k2v.x, d);
              d = fmaf(q2.y, k2v.y, d);
            }
          }
          d *= expf(ge - gam[i]);
        }
        a[k2] = d;
      }
      while (fm) {
        const int jj = half * 32 + __ffs(fm) - 1;
        fm &= fm - 1;
        const float4 pj = par[jj];
        float x[4], m = -INFINITY;
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
          const int i = lane + 32 * k2;
          x[k2] = i <= te ? pj.x * __ldg(v + (r0 + i) * kGD + jj) : -INFINITY;
          m = fmaxf(m, x[k2]);
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        float acc = 0.f, ix = fmaf(__ldg(qrow + lane), w.s[task * kSt + jj * kGM + lane],
                                   __ldg(qrow + 32 + lane) * w.s[task * kSt + jj * kGM + 32 + lane]);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) acc = x[k2] > -INFINITY ? fmaf(a[k2], expf(x[k2] - m), acc) : acc;
#pragma unroll
        for (int off = 16; off; off >>= 1) {
          acc += __shfl_xor_sync(0xffffffffu, acc, off);
          ix += __shfl_xor_sync(0xffffffffu, ix, off);
        }
        const float la = acc > 0.f ? m + logf(acc) : -INFINITY;
        const float lb = ix > 0.f ? w.mu[task * kGD + jj] + ge + logf(ix) : -INFINITY;
        const float hi = fmaxf(la, lb), lo = fminf(la, lb);
        const float ln = hi == -INFINITY ? -INFINITY : hi + log1pf(expf(lo - hi));
        __syncwarp();
        if (lane == 0) so[te * OutLay::kOutLd + jj] = (ln - lze) / pj.x;
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (ok) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = tid + u * 256, rr = i >> 4, cc = (i & 15) * 4;
      if (rr < rows)
        __stcs(reinterpret_cast<float4 *>(out + (r0 + rr) * kGD + cc),
               *reinterpret_cast<const float4 *>(so + rr * OutLay::kOutLd + cc));
    }
  }
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 256);
  }
}

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

// Layout of a group of `heads` heads; returns its bytes.
size_t gla_par_layout(int heads, int n_ch, uint8_t *p, GlaTcWs *w) {
  const size_t n = static_cast<size_t>(heads) * n_ch;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    uint8_t *q = p + off;
    off += up256(bytes);
    return q;
  };
  uint8_t *k16 = take(n * kImg), *e16 = take(n * kImg), *u = take(n * kSt * 4), *s = take(n * kSt * 4);
  uint8_t *stat = take(n * kGD * sizeof(float4)), *shift = take(n * kGD * 4), *mu = take(n * kGD * 4), *gl = take(n * 4),
          *fac = take(n * kGD * sizeof(float4));
  if (w)
    *w = GlaTcWs{reinterpret_cast<float4 *>(stat), reinterpret_cast<float *>(shift), reinterpret_cast<float *>(mu),
                 reinterpret_cast<float4 *>(fac), reinterpret_cast<float *>(gl), k16, e16, reinterpret_cast<float *>(u), reinterpret_cast<float *>(s)};
  return off;
}

// Heads per group: as many as keep the group's workspace below 320 MB (4.3 MB a head at T = 8192), at
// least one; groups of equal size.  Fewer launches and fuller waves outweigh what smaller groups keep in
// L2: 64 heads of T = 8192 in groups of 13, 22 or all: 452, 412, 348 us.
int gla_par_group(int BH, int n_ch) {
  const size_t fit = (size_t{320} << 20) / gla_par_layout(1, n_ch, nullptr, nullptr);
  const size_t cap = fit < 1 ? 1 : (fit > 16384 ? 16384 : fit);
  const int n = static_cast<int>((static_cast<size_t>(BH) + cap - 1) / cap);
  return (BH + n - 1) / n;
}

}  // namespace

size_t gla_par_workspace_bytes(int BH, int T) {
  const int n_ch = (T + kGC - 1) / kGC;
  if (n_ch < kGlaParMinChunks) return 0;
  return gla_par_layout(gla_par_group(BH, n_ch), n_ch, nullptr, nullptr);
}

cudaError_t launch_gla_par(const float *qf, const float *kf, const float *v, const float *logdecay, const float *beta,
                          float *out, float *logz, int B, int H, int T, void *ws, unsigned *err, cudaStream_t stream) {
  const int BH = B * H, n_ch = (T + kGC - 1) / kGC, grp = gla_par_group(BH, n_ch);
  GlaTcWs w;
  gla_par_layout(grp, n_ch, static_cast<uint8_t *>(ws), &w);
  cudaError_t e = cudaFuncSetAttribute(gla_local_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LocLay::kAlloc);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gla_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OutLay::kAlloc);
  for (int h0 = 0; h0 < BH && e == cudaSuccess; h0 += grp) {
    const int n = BH - h0 < grp ? BH - h0 : grp;
    const size_t r = static_cast<size_t>(h0) * T;
    const dim3 grid(n_ch, n);
    gla_stats_kernel<<<grid, 128, 0, stream>>>(v + r * kGD, logdecay + r, T, n_ch, w.stat, w.glast);
    gla_anchor_kernel<<<dim3(kGD / 8, n), 256, 0, stream>>>(beta, h0, H, T, n_ch, w);
    gla_local_kernel<<<grid, 256, LocLay::kAlloc, stream>>>(kf + r * kGM, v + r * kGD, logdecay + r, beta, h0, H, T, n_ch,
                                                            w, err);
    gla_scan_kernel<<<dim3((kGD + 4) / 4, n), 256, 0, stream>>>(n_ch, w);
    gla_out_kernel<<<grid, 256, OutLay::kAlloc, stream>>>(qf + r * kGM, v + r * kGD, logdecay + r, beta, out + r * kGD,
                                                          logz ? logz + r : nullptr, h0, H, T, n_ch, w, err);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace fem
