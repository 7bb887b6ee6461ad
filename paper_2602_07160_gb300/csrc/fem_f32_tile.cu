// The FEM read on CUDA cores for longer sequences: 64-row query tiles against
// 64-key tiles as two register-tiled fp32 contractions (S = Q K^T, then the
// prior weights against a value bank), instead of one exponential per (row,
// key, channel).
//
// What bounds it: instruction issue around the FMA pipe (2 d multiply-adds per
// visible pair); the exponentials are one per (row, key) and one per (key,
// channel) of a tile.  B1 H4 T2048 d64 causal: 174 us against 2468 us for the
// warp-per-row form of fem_simt.cu, whose every (row, key) is an exponential
// pair per channel behind a butterfly sum; full prior 175 against 3873 us (the
// heaviest tile sets both), d 128 causal 316 against 4386 us.  use_tile in
// fem_simt.cu has both sides around the rule.
//
// The bank of a query tile is fixed before its first key: one pass over the
// values of the keys the tile sees gives every channel's extremes and mean.
//   linear channel (beta times the spread of v at most 1 + kLinTop):
//     D_ij = expm1(beta (v_ij - c)) / beta, c the mean clamped to [max v - kLinTop / beta,
//     min v + 1 / beta], read as c + log1p(beta W / L) / beta, W = sum_i P_i D_ij
//   shifted channel: E_ij = exp(beta (v_ij - c)), read as c + log(A / L) / beta.  c is the largest
//     value among the keys every row of the tile sees, raised to at most kTopExp / beta under the
//     largest of all, so E neither overflows on the keys only later rows see nor leaves an earlier
//     row without a term until a channel spans some 90 nats.
// The weights carry a factor 2^40, which spends fp32's range on both sides of the product: weights
// reach 2^52 (with the row maximum's lag), bank entries 2^52, their sums 2^119 at 2^15 keys, and
// what the range can drop from a sum (2^-126 of either's largest) stays below 2^-24 of an A / L of
// kTileGuard.  An entry whose A / L is not finite or lies below that (peaked priors, wide spans,
// infinities among the values of keys the row does not see) is summed again around its own largest
// s_i + beta v_i, the key tiles once more (sweep_again), or by itself (read_exact) where a warp has few;
// likewise one of a linear channel, which only values that are not finite can reject.  Every product and sum is fp32, as in fem_simt.cu.
//
// Layout: two groups of 256 threads take the key tiles in turn, each with its own K, bank and P
// tiles in shared memory and its own accumulators (the heaviest block's chain is half as long, and
// one group's staging runs beside the other's contractions); the first merges them.  Thread
// (ty, tx) holds rows 4 ty .. 4 ty + 3 against keys (or channels) 4 tx .. 4 tx + 3, rows in packed
// pairs: four warps per scheduler (eight rows a thread, with half the warps, left the FMA pipe at
// 31 %: a warp waits out every dependent pair).  K and Q lie transposed ([channel][row]); P's
// 16-byte chunks are swizzled by key so its transposed stores spread over the banks.  Up to 64
// channels the next tile's K and V rows are loaded into registers ahead of the contractions.
#include <type_traits>

#include "fem_common.cuh"
#include "fem_f32.cuh"
#include "fem_launch.h"

namespace fem {
namespace {

constexpr int kTR = 64, kTK = 64;     // query rows and keys of a tile
constexpr int kTLd = 68;              // leading dimension of the transposed Q and K tiles
constexpr int kGroups = 2, kGT = 256;  // thread groups sharing a query tile's keys, threads of a group
constexpr float kLinTop = 3.f;
constexpr float kTopExp = 36.f;       // largest exponent of a shifted bank
constexpr float kWeightScale = 0x1p40f;
constexpr float kTileGuard = 0x1p-84f;
// What a warp evaluates one by one: its rejected entries, each counted as often as its row has 64 keys.  An
// entry takes some 500 us at 2048 keys of 64 channels, a sweep 350 there; in a sequence's first rows a few
// entries are common (B9 H6 T71 d64: 20.6 us, with a sweep for any 30.8).
constexpr unsigned kFewRejected = 4;
constexpr float kTileLag = 8.f;       // the row maximum moves when it grows by more (nats)

template <int DP>
struct TileLay {
  static constexpr int kEl = DP + 4;                         // leading dimension of the bank tile
  static constexpr int kGroupFloats = DP * kTLd + kTK * kEl + kTK * kTR;
  static constexpr int kPar = DP * kTLd + kGroups * kGroupFloats;  // per channel: beta, 1/beta, c, linear
  static constexpr int kRed = kPar + 4 * DP;                 // the groups' m and L for the merge
  static constexpr int kAny = kRed + kGroups * kTR * 2;      // per thread of a group: entries to sum again
  static constexpr int kFloats = kAny + kGT;
  static constexpr int kBytes = kFloats * 4;
  static_assert(kBytes <= 227 * 1024, "shared memory");
  static_assert(2 * kTR * DP <= kGroupFloats, "a group's state of the second sweep fits its tiles");
  static_assert(4 * (kGroups * kGT / (DP / 4)) * DP <= kGroups * kGroupFloats, "statistics' partials fit the tiles");
};

// Row t against keys 0 .. n - 1 for channel j, key by key: the warp's lanes take every 32nd key.
// Joint maximum of s + beta v for the tilted sum; expm1 sums where the read lies near c.
template <typename In>
__device__ __noinline__ float read_exact(const In *qr, const In *kb, const In *vb, int n, int d, int j, float b,
                                         float inv_sqrt_d, int lane) {
  float m = -INFINITY, c = -INFINITY, top = -INFINITY;
  for (int i = lane; i < n; i += 32) {
    float s = 0.f;
    for (int e = 0; e < d; ++e) s = fmaf(ld1(qr + e), ld1(kb + static_cast<size_t>(i) * d + e), s);
    s *= inv_sqrt_d;
    const float x = ld1(vb + static_cast<size_t>(i) * d + j);
    m = fmaxf(m, s);
    c = fmaxf(c, x);
    top = fmaxf(top, fmaf(b, x, s));
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, off));
    top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, off));
  }
  float L = 0.f, A = 0.f, W = 0.f;
  for (int i = lane; i < n; i += 32) {
    float s = 0.f;
    for (int e = 0; e < d; ++e) s = fmaf(ld1(qr + e), ld1(kb + static_cast<size_t>(i) * d + e), s);
    s *= inv_sqrt_d;
    const float x = ld1(vb + static_cast<size_t>(i) * d + j), p = expf(s - m);
    L += p;
    A += expf(fmaf(b, x, s) - top);
    W += p * (b != 0.f ? expm1f(b * (x - c)) / b : x - c);
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    L += __shfl_xor_sync(0xffffffffu, L, off);
    A += __shfl_xor_sync(0xffffffffu, A, off);
    W += __shfl_xor_sync(0xffffffffu, W, off);
  }
  if (b == 0.f) return c + W / L;
  const float z = b * W / L;
  return z > -0.5f ? c + log1pf(z) / b : ((top - m) + (logf(A) - logf(L))) / b;
}

// The block's key tiles once more for the rejected entries of shifted channels (Lay::kAny: bit 4 c + r of a
// thread's word is row 4 ty + r, channel chan(c)): scores as before, then in warps that have any the largest
// s_i + beta v_i of the tile and the sum around the running one.  What bounds it is the issue of the tile's
// (row, key, channel) terms and their exponentials.  Entry by entry, scores and all, a warp spends some 500 us on each at
// T2048 d64 and peaked priors reject most of them: B1 H4 T2048 d64 causal, scores of deviation 16, beta 10 to
// 100 73.5 ms (the warp-per-row form 2.5, with -inf for many); now 0.53 ms.
template <typename In, int DP>
__device__ __noinline__ void sweep_again(float *smem, const In *kb, const In *vb, float *ob, int T, int d, int t0,
                                         int n_keys, int causal) {
  using Lay = TileLay<DP>;
  constexpr int NC = DP / 16, kEl = Lay::kEl, CQ = DP / 4;
  const int tid = threadIdx.x, g = tid / kGT, gt = tid % kGT, ty = gt >> 4, tx = gt & 15;
  float *sQ = smem, *sK = smem + DP * kTLd + g * Lay::kGroupFloats, *sV = sK + DP * kTLd, *sS = sV + kTK * kEl;
  const float *pB = smem + Lay::kPar, *sRed = smem + Lay::kRed;
  const unsigned mask = reinterpret_cast<const unsigned *>(smem + Lay::kAny)[gt];
  const bool any = __any_sync(0xffffffffu, mask != 0u);
  const bool vec = (d & 3) == 0;
  const float scale = kLog2e * rsqrtf(static_cast<float>(d));
  auto chan = [&](int c) { return NC == 2 ? tx * 2 + c : (c >> 2) * 64 + tx * 4 + (c & 3); };
  float b[NC];
  float2 top[2][NC], A[2][NC];  // rows 2 u, 2 u + 1 of the thread's four; exponents in units of ln 2
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    b[c] = pB[chan(c)] * kLog2e;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      top[u][c] = make_float2(-INFINITY, -INFINITY);
      A[u][c] = make_float2(0.f, 0.f);
    }
  }
  const int n_kt = (n_keys + kTK - 1) / kTK;
  for (int kt = g; kt < n_kt; kt += kGroups) {
    const int k0 = kt * kTK, nk = min(kTK, n_keys - k0);
    bar_sync(1 + g, kGT);  // the previous tile is consumed
#pragma unroll 4
    for (int e = gt; e < kTK * CQ; e += kGT) {
      const int r = e % kTK, j = (e / kTK) * 4;
      const float4 k4 = r < nk ? ld_row4(kb + static_cast<size_t>(k0 + r) * d, j, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      sK[j * kTLd + r] = k4.x;
      sK[(j + 1) * kTLd + r] = k4.y;
      sK[(j + 2) * kTLd + r] = k4.z;
      sK[(j + 3) * kTLd + r] = k4.w;
      const int rv = e / CQ, jv = (e % CQ) * 4;
      *reinterpret_cast<float4 *>(sV + rv * kEl + jv) =
          rv < nk ? ld_row4(vb + static_cast<size_t>(k0 + rv) * d, jv, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    bar_sync(1 + g, kGT);
    float2 s[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[i][c] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int e = 0; e < DP; ++e) {
      const float4 a = ld4(sQ + e * kTLd + ty * 4), k4 = ld4(sK + e * kTLd + tx * 4);
      const float2 ar[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
      const float kr[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 2; ++i) s[i][c] = __ffma2_rn(ar[i], make_float2(kr[c], kr[c]), s[i][c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float x[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int lim = causal ? min(nk, t0 + ty * 4 + r + 1 - k0) : nk;
        x[r] = ((r & 1) ? s[r >> 1][c].y : s[r >> 1][c].x) * scale;
        if (tx * 4 + c >= lim) x[r] = -INFINITY;
      }
      *reinterpret_cast<float4 *>(sS + (tx * 4 + c) * kTR + ((ty ^ tx) << 2)) = make_float4(x[0], x[1], x[2], x[3]);
    }
    bar_sync(1 + g, kGT);
    if (!any) continue;
    float2 was[2][NC];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < NC; ++c) was[i][c] = top[i][c];
    // s_i + beta v_i of key i; masked: -inf whatever the value, which may not be finite
    auto terms = [&](int i, float2 (&y)[2][NC], bool masked) {
      const float4 a = ld4(sS + i * kTR + ((ty ^ (i >> 2)) << 2));
      const float2 sr[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float v = sV[i * kEl + chan(c)];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          y[u][c] = __ffma2_rn(make_float2(b[c], b[c]), make_float2(v, v), sr[u]);
          if (masked) {
            if (sr[u].x == -INFINITY) y[u][c].x = -INFINITY;
            if (sr[u].y == -INFINITY) y[u][c].y = -INFINITY;
          }
        }
      }
    };
    auto sweep = [&](auto ragged) {
      constexpr bool kMasked = decltype(ragged)::value;
#pragma unroll 2
      for (int i = 0; i < nk; ++i) {
        float2 y[2][NC];
        terms(i, y, kMasked);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int c = 0; c < NC; ++c)
            top[u][c] = make_float2(fmaxf(top[u][c].x, y[u][c].x), fmaxf(top[u][c].y, y[u][c].y));
      }
      float2 neg[2][NC];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float2 t = top[u][c], w = was[u][c];
          A[u][c] = make_float2(t.x > w.x ? A[u][c].x * ex2_approx(w.x - t.x) : A[u][c].x,
                                t.y > w.y ? A[u][c].y * ex2_approx(w.y - t.y) : A[u][c].y);
          // no finite term yet: every exponential below is that of -inf
          neg[u][c] = make_float2(t.x == -INFINITY ? 0.f : -t.x, t.y == -INFINITY ? 0.f : -t.y);
        }
#pragma unroll 2
      for (int i = 0; i < nk; ++i) {
        float2 y[2][NC];
        terms(i, y, kMasked);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const float2 x = __fadd2_rn(y[u][c], neg[u][c]);
            A[u][c] = __fadd2_rn(A[u][c], make_float2(ex2_approx(x.x), ex2_approx(x.y)));
          }
      }
    };
    if (causal && k0 + kTK > t0 + 1)
      sweep(std::true_type());
    else
      sweep(std::false_type());
  }
  // the groups' states merged by the first
  bar_sync(1 + g, kGT);
  float *st = smem + DP * kTLd + Lay::kGroupFloats;  // the second group's tiles: [64][DP] top, then A
  auto of_row = [](const float2 (&x)[2][NC], int r, int c) { return (r & 1) ? x[r >> 1][c].y : x[r >> 1][c].x; };
  if (g > 0 && any) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        st[(ty * 4 + r) * DP + chan(c)] = of_row(top, r, c);
        st[(kTR + ty * 4 + r) * DP + chan(c)] = of_row(A, r, c);
      }
  }
  __syncthreads();
  if (g > 0 || !mask) return;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = ty * 4 + r;
    const float m = sRed[row * 2], ll = logf(sRed[row * 2 + 1]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (!((mask >> (4 * c + r)) & 1u)) continue;
      const float t1 = of_row(top, r, c), t2 = st[row * DP + chan(c)], tn = fmaxf(t1, t2);
      const float sum = (t1 == -INFINITY ? 0.f : of_row(A, r, c) * ex2_approx(t1 - tn)) +
                        (t2 == -INFINITY ? 0.f : st[(kTR + row) * DP + chan(c)] * ex2_approx(t2 - tn));
      ob[static_cast<size_t>(t0 + row) * d + chan(c)] = (fmaf(tn, kLn2, -m) + (logf(sum) - ll)) / pB[chan(c)];
    }
  }
}

template <typename In, int DP>
__global__ void __launch_bounds__(kGroups * kGT, 1)
    fem_tile_kernel(const In *__restrict__ q, const In *__restrict__ k, const In *__restrict__ v,
                    const float *__restrict__ beta, float *__restrict__ out, float *__restrict__ lse, int H, int T,
                    int d, int causal) {
  using Lay = TileLay<DP>;
  constexpr int NC = DP / 16, kEl = Lay::kEl;  // channels of a thread
  constexpr int kThreads = kGroups * kGT;
  extern __shared__ __align__(16) float tile_smem[];
  const int tid = threadIdx.x, g = tid / kGT, gt = tid % kGT, ty = gt >> 4, tx = gt & 15, lane = tid & 31;
  float *sQ = tile_smem, *sK = tile_smem + DP * kTLd + g * Lay::kGroupFloats, *sE = sK + DP * kTLd, *sP = sE + kTK * kEl;
  float *pB = tile_smem + Lay::kPar, *pI = pB + DP, *pC = pI + DP, *pL = pC + DP, *sRed = tile_smem + Lay::kRed;
  const int n_qt = (T + kTR - 1) / kTR;
  const long long bh = blockIdx.x;
  const int qt = n_qt - 1 - static_cast<int>(blockIdx.y), t0 = qt * kTR;  // heaviest causal tiles first
  const int h = static_cast<int>(bh % H);
  const int n_keys = causal ? min(T, t0 + kTR) : T;  // keys any row of the tile sees
  const int n_all = causal ? t0 + 1 : T;             // keys every row of it sees
  const bool vec = (d & 3) == 0;
  const In *qb = q + bh * T * d, *kb = k + bh * T * d, *vb = v + bh * T * d;
  const float inv_sqrt_d = rsqrtf(static_cast<float>(d));

  // ---- Q transposed, and the channels' statistics over the keys
  for (int e = tid; e < kTR * (DP / 4); e += kThreads) {
    const int r = e % kTR, j = (e / kTR) * 4;
    const float4 x = ld_row4(qb + static_cast<size_t>(min(t0 + r, T - 1)) * d, j, d, vec);
    sQ[j * kTLd + r] = x.x;
    sQ[(j + 1) * kTLd + r] = x.y;
    sQ[(j + 2) * kTLd + r] = x.z;
    sQ[(j + 3) * kTLd + r] = x.w;
  }
  {
    constexpr int CQ = DP / 4, PARTS = kThreads / CQ;  // four channels a thread, every PARTS-th key
    float *sStat = tile_smem + DP * kTLd;              // the tiles' space, not yet in use
    const int cq = tid % CQ, part = tid / CQ;
    float mx[4], ma[4], mn[4], sm[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      mx[u] = ma[u] = -INFINITY;
      mn[u] = INFINITY;
      sm[u] = 0.f;
    }
    constexpr int kAhead = 8;
    for (int i0 = part; i0 < n_keys; i0 += kAhead * PARTS) {
      float4 x[kAhead];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int i = i0 + u * PARTS;
        x[u] = i < n_keys ? ld_row4(vb + static_cast<size_t>(i) * d, cq * 4, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int i = i0 + u * PARTS;
        if (i >= n_keys) break;
        const float xv[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          mx[c] = fmaxf(mx[c], xv[c]);
          if (i < n_all) ma[c] = fmaxf(ma[c], xv[c]);
          mn[c] = fminf(mn[c], xv[c]);
          sm[c] += xv[c];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float *r = sStat + (part * DP + cq * 4 + c) * 4;
      r[0] = mx[c];
      r[1] = ma[c];
      r[2] = mn[c];
      r[3] = sm[c];
    }
    __syncthreads();
    for (int j = tid; j < DP; j += kThreads) {
      float gx = -INFINITY, ga = -INFINITY, gn = INFINITY, gs = 0.f;
      for (int p = 0; p < PARTS; ++p) {
        const float *r = sStat + (p * DP + j) * 4;
        gx = fmaxf(gx, r[0]);
        ga = fmaxf(ga, r[1]);
        gn = fminf(gn, r[2]);
        gs += r[3];
      }
      const float b = j < d ? normal_beta(beta[h * d + j]) : 0.f, mean = gs / static_cast<float>(n_keys);
      bool lin = true;
      float c = mean;
      if (b > 0.f) {
        const float lo = gx - kLinTop / b, hi = gn + 1.f / b;
        lin = lo <= hi;
        c = lin ? fminf(fmaxf(mean, lo), hi) : fmaxf(ga, gx - kTopExp / b);
      }
      pB[j] = b;
      pI[j] = b > 0.f ? 1.f / b : 0.f;
      pC[j] = c;
      pL[j] = lin ? 1.f : 0.f;
    }
  }
  __syncthreads();

  float2 acc[2][NC];  // rows 2 i, 2 i + 1 of the thread's four, per channel
  float m[4], l[4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
  }

  // the thread's share of a tile: K chunks (lanes over keys: the transposed stores hit distinct
  // banks) and V chunks (lanes over channels, one channel quad a thread)
  constexpr int CQ = DP / 4, kShare = kTK * CQ / kGT;
  constexpr bool kAheadLoads = DP <= 64;
  const int n_kt = (n_keys + kTK - 1) / kTK, vj = (gt % CQ) * 4;
  float4 nk4[kShare], nv4[kShare];
  auto load_tile = [&](int kt) {
    const int k0 = kt * kTK, nk = min(kTK, n_keys - k0);
#pragma unroll
    for (int u = 0; u < kShare; ++u) {
      const int e = gt + u * kGT, r = e % kTK, j = (e / kTK) * 4, rv = gt / CQ + u * (kGT / CQ);
      nk4[u] = r < nk ? ld_row4(kb + static_cast<size_t>(k0 + r) * d, j, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
      nv4[u] = rv < nk ? ld_row4(vb + static_cast<size_t>(k0 + rv) * d, vj, d, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  const float4 vB = ld4(pB + vj), vI = ld4(pI + vj), vC = ld4(pC + vj), vL = ld4(pL + vj);
  const bool any_lin = vL.x != 0.f || vL.y != 0.f || vL.z != 0.f || vL.w != 0.f;
  if (kAheadLoads && g < n_kt) load_tile(g);
  for (int kt = g; kt < n_kt; kt += kGroups) {
    const int k0 = kt * kTK, nk = min(kTK, n_keys - k0);
    if (!kAheadLoads) load_tile(kt);
    bar_sync(1 + g, kGT);  // the previous tile is consumed
#pragma unroll
    for (int u = 0; u < kShare; ++u) {
      const int e = gt + u * kGT, r = e % kTK, j = (e / kTK) * 4;
      sK[j * kTLd + r] = nk4[u].x;
      sK[(j + 1) * kTLd + r] = nk4[u].y;
      sK[(j + 2) * kTLd + r] = nk4[u].z;
      sK[(j + 3) * kTLd + r] = nk4[u].w;
    }
#pragma unroll
    for (int u = 0; u < kShare; ++u) {
      const int r = gt / CQ + u * (kGT / CQ);
      const float2 x0 = make_float2(nv4[u].x - vC.x, nv4[u].y - vC.y), x1 = make_float2(nv4[u].z - vC.z, nv4[u].w - vC.w);
      const float2 y0 = __fmul2_rn(x0, make_float2(vB.x, vB.y)), y1 = __fmul2_rn(x1, make_float2(vB.z, vB.w));
      float4 e = make_float4(exp_tilt(vB.x, nv4[u].x, vC.x), exp_tilt(vB.y, nv4[u].y, vC.y),
                             exp_tilt(vB.z, nv4[u].z, vC.z), exp_tilt(vB.w, nv4[u].w, vC.w));
      if (any_lin) {
        const float2 d0 = em1_over_beta2(x0, y0, make_float2(e.x, e.y), make_float2(vI.x, vI.y));
        const float2 d1 = em1_over_beta2(x1, y1, make_float2(e.z, e.w), make_float2(vI.z, vI.w));
        e = make_float4(vL.x != 0.f ? d0.x : e.x, vL.y != 0.f ? d0.y : e.y, vL.z != 0.f ? d1.x : e.z,
                        vL.w != 0.f ? d1.y : e.w);
      }
      if (r >= nk) e = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4 *>(sE + r * kEl + vj) = e;
    }
    bar_sync(1 + g, kGT);
    if (kAheadLoads && kt + kGroups < n_kt) load_tile(kt + kGroups);
    // ---- S = Q K^T
    float2 s[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[i][c] = make_float2(0.f, 0.f);
    const float *qp = sQ + ty * 4, *kp = sK + tx * 4;
#pragma unroll 8
    for (int e = 0; e < DP; ++e) {
      const float4 a = ld4(qp + e * kTLd), bk = ld4(kp + e * kTLd);
      const float2 ar[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
      const float br[4] = {bk.x, bk.y, bk.z, bk.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 2; ++i) s[i][c] = __ffma2_rn(ar[i], make_float2(br[c], br[c]), s[i][c]);
    }
    // ---- the rows' maxima over the tile (16 lanes share a row), then P and its sums
    const bool ragged = nk < kTK || (causal && k0 + kTK > t0 + 1);
    float mx[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      mx[r] = -INFINITY;
      const int lim = causal ? min(nk, t0 + ty * 4 + r + 1 - k0) : nk;  // keys k0 .. k0 + lim - 1 are visible
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float &x = (r & 1) ? s[r >> 1][c].y : s[r >> 1][c].x;
        x *= inv_sqrt_d;
        if (ragged && tx * 4 + c >= lim) x = -INFINITY;
        mx[r] = fmaxf(mx[r], x);
      }
    }
#pragma unroll
    for (int off = 8; off; off >>= 1)
#pragma unroll
      for (int r = 0; r < 4; ++r) mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], off));
    bool moved = false;
#pragma unroll
    for (int r = 0; r < 4; ++r) moved = moved || mx[r] > m[r] + kTileLag;
    if (moved) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (mx[r] > m[r] + kTileLag) {
          const float alpha = expf(m[r] - mx[r]);  // 0 from an empty state
          l[r] *= alpha;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            float &a = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
            a *= alpha;
          }
          m[r] = mx[r];
        }
      }
    }
    float m0[4];  // the row's shift, 0 while no score of the row is above -inf (its weights are then 0)
#pragma unroll
    for (int r = 0; r < 4; ++r) m0[r] = m[r] == -INFINITY ? 0.f : m[r];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float p[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float x = (r & 1) ? s[r >> 1][c].y : s[r >> 1][c].x;
        const float tm = x - m0[r];
        p[r] = tm < -60.f ? expf(tm + 40.f * kLn2) : expf(tm) * kWeightScale;
        l[r] += p[r];
      }
      *reinterpret_cast<float4 *>(sP + (tx * 4 + c) * kTR + ((ty ^ tx) << 2)) = make_float4(p[0], p[1], p[2], p[3]);
    }
    bar_sync(1 + g, kGT);
    // ---- acc += P bank
#pragma unroll 4
    for (int k4 = 0; k4 < kTK / 4; ++k4) {
      const float *pp = sP + k4 * 4 * kTR + ((ty ^ k4) << 2);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 a = ld4(pp + u * kTR);
        const float2 ar[2] = {make_float2(a.x, a.y), make_float2(a.z, a.w)};
        const float *ep = sE + (k4 * 4 + u) * kEl;
        float br[NC];
        if constexpr (NC == 2) {
          const float2 e2 = *reinterpret_cast<const float2 *>(ep + tx * 2);
          br[0] = e2.x;
          br[1] = e2.y;
        } else {
#pragma unroll
          for (int c4 = 0; c4 < NC / 4; ++c4) {
            const float4 e4 = ld4(ep + c4 * 64 + tx * 4);
            br[4 * c4] = e4.x;
            br[4 * c4 + 1] = e4.y;
            br[4 * c4 + 2] = e4.z;
            br[4 * c4 + 3] = e4.w;
          }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int i = 0; i < 2; ++i) acc[i][c] = __ffma2_rn(ar[i], make_float2(br[c], br[c]), acc[i][c]);
      }
    }
  }
#pragma unroll
  for (int off = 8; off; off >>= 1)
#pragma unroll
    for (int r = 0; r < 4; ++r) l[r] += __shfl_xor_sync(0xffffffffu, l[r], off);
  // ---- the groups' states merged by the first (the others' K and bank tiles are free)
  auto chan = [&](int c) { return NC == 2 ? tx * 2 + c : (c >> 2) * 64 + tx * 4 + (c & 3); };
  bar_sync(1 + g, kGT);
  if (g > 0) {
    float *st = sK;  // [64][DP], then m and L
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        st[(ty * 4 + r) * DP + chan(c)] = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
    if (tx == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        sRed[(g * kTR + ty * 4 + r) * 2] = m[r];
        sRed[(g * kTR + ty * 4 + r) * 2 + 1] = l[r];
      }
    }
  }
  __syncthreads();
  unsigned rejected = 0, linear = 0;  // entries to evaluate again, those of linear channels: bit 4 c + r
  if (g == 0) {
    for (int og = 1; og < kGroups; ++og) {
      const float *st = tile_smem + DP * kTLd + og * Lay::kGroupFloats;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float m2 = sRed[(og * kTR + ty * 4 + r) * 2], l2 = sRed[(og * kTR + ty * 4 + r) * 2 + 1];
        const float mn = fmaxf(m[r], m2);
        const float a1 = m[r] == -INFINITY ? 0.f : expf(m[r] - mn), a2 = m2 == -INFINITY ? 0.f : expf(m2 - mn);
        l[r] = l[r] * a1 + l2 * a2;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          float &a = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
          a = a * a1 + st[(ty * 4 + r) * DP + chan(c)] * a2;
        }
        m[r] = mn;
      }
    }
    // ---- the read
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int j = chan(c);
      const float b = pB[j], ib = pI[j], cc = pC[j];
      const bool lin = pL[j] != 0.f;
      const float ib_lo = b > 0.f ? fmaf(-b, ib, 1.f) * ib : 0.f;  // 1 / b is ib + ib_lo
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float &a = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
        const float x = a / l[r];
        const bool bad = lin ? !(b * x > -0.9f && fabsf(x) < INFINITY) : !(x > kTileGuard && x < INFINITY);
        if (bad && j < d && t0 + ty * 4 + r < T) {
          rejected |= 1u << (4 * c + r);
          if (lin) linear |= 1u << (4 * c + r);
        }
        if (b > 0.f) {
          // log1p(b x) or log(x), the latter as n ln 2 + log(mantissa) with ln 2 in two parts (Cody and Waite),
          // over b and onto c with the rounding errors of both steps carried: |c - o| may be several times |o|
          float hi, lo = 0.f;
          if (lin) {
            hi = log1pf(b * x);
          } else {
            const int n = ((__float_as_int(x) - 0x3f400000) >> 23);  // the mantissa in [3/4, 3/2)
            const float f = static_cast<float>(n), lm = logf(__int_as_float(__float_as_int(x) - (n << 23)));
            hi = f * 0x1.62e4p-1f;  // ln 2 to 16 bits: exact
            lo = fmaf(f, 0x1.7f7d1cp-20f, lm);
          }
          const float t = hi + lo, tlo = lo - (t - hi), qv = t * ib, qlo = fmaf(t, ib, -qv) + fmaf(tlo, ib, t * ib_lo);
          const float o = cc + qv, z = o - cc;
          a = o + (((cc - (o - z)) + (qv - z)) + qlo);
        } else {
          a = cc + x;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int t = t0 + ty * 4 + r;
      if (t >= T) continue;
      float *o = out + (bh * T + t) * d;
      if (lse && tx == 0) lse[bh * T + t] = m[r] + logf(l[r] * (1.f / kWeightScale));
      if constexpr (NC == 2) {
#pragma unroll
        for (int c = 0; c < 2; ++c)
          if (chan(c) < d) o[chan(c)] = (r & 1) ? acc[r >> 1][c].y : acc[r >> 1][c].x;
      } else {
#pragma unroll
        for (int c = 0; c < NC; c += 4) {
          float x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = (r & 1) ? acc[r >> 1][c + u].y : acc[r >> 1][c + u].x;
          if (vec && chan(c) < d) *reinterpret_cast<float4 *>(o + chan(c)) = make_float4(x[0], x[1], x[2], x[3]);
          if (!vec)
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (chan(c + u) < d) o[chan(c + u)] = x[u];
        }
      }
    }
    if (tx == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        sRed[(ty * 4 + r) * 2] = m[r];
        sRed[(ty * 4 + r) * 2 + 1] = l[r] * (1.f / kWeightScale);
      }
    }
    reinterpret_cast<unsigned *>(tile_smem + Lay::kAny)[gt] = rejected & ~linear;
  }
  unsigned cost = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    cost += __popc(rejected & ~linear & (0x11111111u << r)) * static_cast<unsigned>(((causal ? t0 + ty * 4 + r : T - 1) >> 6) + 1);
  const bool many = __reduce_add_sync(0xffffffffu, cost) > kFewRejected;
  const bool sweep = __syncthreads_or(many);  // also: the rejected values are stored
  // ---- a linear channel's entries, and others where they are few, one at a time by the whole warp
  unsigned mine = sweep ? rejected & linear : rejected;
  unsigned who = __ballot_sync(0xffffffffu, mine != 0u);
  while (who) {
    const int src = __ffs(who) - 1, sx = (src & 15) * (NC == 2 ? 2 : 4), ry = __shfl_sync(0xffffffffu, ty, src);
    who &= who - 1;
    unsigned bits = __shfl_sync(0xffffffffu, mine, src);
    while (bits) {
      const int e = __ffs(bits) - 1, c = e >> 2, t = t0 + ry * 4 + (e & 3);
      bits &= bits - 1;
      const int j = NC == 2 ? sx + c : (c >> 2) * 64 + sx + (c & 3);
      const float o = read_exact(qb + static_cast<size_t>(t) * d, kb, vb, causal ? t + 1 : T, d, j, pB[j], inv_sqrt_d, lane);
      if (lane == 0) out[(bh * T + t) * d + j] = o;
    }
  }
  if (sweep) sweep_again<In, DP>(tile_smem, kb, vb, out + bh * T * d, T, d, t0, n_keys, causal);
}

template <typename In, int DP>
cudaError_t launch_tile_dp(const In *q, const In *k, const In *v, const float *beta, float *out, float *lse, int B,
                           int H, int T, int d, int causal, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(fem_tile_kernel<In, DP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       TileLay<DP>::kBytes);
  if (e != cudaSuccess) return e;
  fem_tile_kernel<In, DP><<<dim3(B * H, (T + kTR - 1) / kTR), kGroups * kGT, TileLay<DP>::kBytes, stream>>>(
      q, k, v, beta, out, lse, H, T, d, causal);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tile_f32(const float *q, const float *k, const float *v, const float *beta, float *out, float *lse,
                            int B, int H, int T, int d, int causal, cudaStream_t stream) {
  if (d <= 32) return launch_tile_dp<float, 32>(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
  if (d <= 64) return launch_tile_dp<float, 64>(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
  if (d <= 128) return launch_tile_dp<float, 128>(q, k, v, beta, out, lse, B, H, T, d, causal, stream);
  return cudaErrorInvalidValue;
}

cudaError_t launch_tile_bf16(const void *q, const void *k, const void *v, const float *beta, float *out, float *lse,
                             int B, int H, int T, int d, int causal, cudaStream_t stream) {
  using In = __nv_bfloat16;
  if (d > 32) return cudaErrorInvalidValue;
  return launch_tile_dp<In, 32>(static_cast<const In *>(q), static_cast<const In *>(k), static_cast<const In *>(v),
                                beta, out, lse, B, H, T, d, causal, stream);
}

}  // namespace fem
