// Tensor-core read at d = 64 with two CTAs per SM (sm_103a, tcgen05): the read
// of fem_tc.cu (same operands, softmax, rescale, guard and entry list, the same
// results up to the order of a rescale's two factors) in a CTA of half an SM's tensor memory, shared memory and
// registers.
//
// What bounded the one-CTA form: a CTA holds the SM while it fills its pipeline
// and runs its epilogue (7.4 us a CTA, nothing beside it), more than half of the
// time of 16 key tiles and nearly all of that of two.  Two independent CTAs
// overlap one's fill, softmax chain and epilogue with the other's, without any
// synchronisation between them.  Kernel times, one CTA / two CTAs per SM:
// B64 H6 T197 full prior 43.6 / 29.3 us, B8 H12 T2048 causal 130.8 / 112.6 us,
// B4 H16 T8192 causal 762 / 668 us, B2 H16 T13768 full prior 1784 / 1618 us.  What
// bounds it now: the softmax warps' issue (two per scheduler, each waiting out
// its dependent pairs; the tensor pipe is a quarter busy).  With a CTA to itself
// per SM the one-CTA form is faster (B1 H1 T2048: 20.1 / 26.1 us, its rescale runs
// in warps of its own), and at d = 128, where only one K and one bank tile would
// fit beside Q, it stays faster as well (910 against 1067 us at B4 H16 T8192); see
// launch_tc.
//
//   warps 0-3   softmax, rescale and epilogue (thread = row = TMEM lane)
//   warp 4      TMEM allocation; S = Q K^T; TMA of Q, K tiles (with their side
//               data) and bank tiles
//   warp 5      acc += P E
//
// TMEM (256 of the SM's 512 columns): scores [0, 128), P [128, 192), acc [192,
// 256): the scores' buffer is free for the next tile's contraction as soon as the
// softmax has read it.  Shared memory (about 107 KB a CTA): Q, two K stages,
// three bank slots, barriers and per-channel state.
//
// Causal diagonal tile (with earlier tiles): the softmax warps move acc to the
// idle Q and K space before the tile's P E starts acc afresh, and the epilogue
// adds the two, keeping the state before the diagonal tile for the fix-up as
// fem_tc.cu does.
#include "fem_common.cuh"
#include "fem_launch.h"
#include "fem_order.h"

namespace fem {
namespace {

// Whether the phase has completed, without suspending the thread.
__device__ __forceinline__ int mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return static_cast<int>(done);
}

constexpr int D = 64;

struct HalfLayout {
  static constexpr uint32_t kTile = D * 128 * 2;
  static constexpr int kStagesK = 2, kSlotsE = 3;
  static constexpr uint32_t kQ = 0;
  static constexpr uint32_t kK = kTile;
  static constexpr uint32_t kE = kK + kStagesK * kTile;
  static constexpr uint32_t kBox = kQ;  // epilogue staging, 128 x D fp32 over Q and the first K stage
  static constexpr uint32_t kBar = kE + kSlotsE * kTile;
  static constexpr uint32_t kTmemSlot = kBar + 256;
  static constexpr uint32_t kAbort = kTmemSlot + 4;
  static constexpr uint32_t kChan = kBar + 512;  // per channel: {anchor, mode, beta, last shift}, then the epilogue's coefficients
  // side ring: per key tile its rescale factors [D], the bank's column sums [D] and the moved-channel
  // mask [4].  Slot kt % 4 was last read before PFull(kt - 4); K tile kt's load follows SFree(kt - 2).
  static constexpr int kSideStages = 4;
  static constexpr uint32_t kSideMask = 2 * D * 4;
  static constexpr uint32_t kSideStride = kSideMask + 128;
  static constexpr uint32_t kSide = kChan + D * 16;
  static constexpr uint32_t kGco = kSide + kSideStages * kSideStride;  // guard coefficients, as fem_tc.cu
  static constexpr uint32_t kThr = kGco + D * 16;
  static constexpr uint32_t kFlag = kThr + D * 8;   // per row and 32-channel group: entries the guard rejects
  static constexpr uint32_t kInvLT = kFlag + 128 * 16;  // 1/L of row 4 k + q at [32 q + k]
  static constexpr uint32_t kMisc = kInvLT + 128 * 4;
  static constexpr uint32_t kBytes = kMisc + 128;
  static constexpr uint32_t kAlloc = kBytes + 1024;
  static constexpr uint32_t kColP = 128, kColAcc = 192;
  static_assert(D / 32 * 16384 <= kTile + kStagesK * kTile, "epilogue staging fits Q and the K stages");
  static_assert(kAlloc <= 113 * 1024, "two CTAs per SM");
};

// mbarrier indices; S, P and acc have one buffer each, so their barriers complete once per key tile
enum : int {
  kHQ = 0,
  kHKFull = 1,    // + stage (2)
  kHEFull = 3,    // + slot (3)
  kHEEmpty = 6,   // + slot (3)
  kHSide = 9,     // + slot (4)
  kHSFull = 13,   // S_k complete
  kHSFree = 14,   // the softmax has read S_k (128 arrivals)
  kHPFull = 15,   // P_k written and acc rescaled (128 arrivals)
  kHPvDone = 16,  // P_k E_k complete
  kHAll = 17,     // everything the two issuers started is complete (2 arrivals)
  kHCount = 18
};

__global__ void __launch_bounds__(192, 2)
    fem_tc_half_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                       const __grid_constant__ CUtensorMap tmap_e, float *__restrict__ out,
                       const float *__restrict__ beta, const BankWorkspace w, float *__restrict__ lse, int H, int T,
                       int causal, unsigned *__restrict__ err) {
  using Lay = HalfLayout;
  constexpr int kStagesK = Lay::kStagesK, kSlotsE = Lay::kSlotsE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + Lay::kAbort);
  float4 *c_coef = reinterpret_cast<float4 *>(smem + Lay::kChan);
  const uint32_t bars = sbase + Lay::kBar;
#define FEM_BAR(i) (bars + 8u * static_cast<uint32_t>(i))

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // provably warp-uniform
  const int n_qt = (T + kBlockQ - 1) / kBlockQ;
  const int n_kt_all = (T + kBlockK - 1) / kBlockK;
  const int rank = static_cast<int>(blockIdx.y * gridDim.x + blockIdx.x), BH = static_cast<int>(gridDim.y);
  int bh, qt;
  tc_tile_of_rank(rank, BH, n_qt, causal, bh, qt);
  const int h = bh % H;
  const int nk = causal ? qt + 1 : n_kt_all;  // key tiles this query tile reads
  const bool split = causal && nk > 1;        // the diagonal tile's P E apart from the earlier tiles'

  auto load_k = [&](int kt) {
    const int st = kt % kStagesK, ss = kt % Lay::kSideStages;
    mbar_arrive_expect_tx(FEM_BAR(kHKFull + st), Lay::kTile);
    for (int b = 0; b < D / 64; ++b)
      tma_load_3d(sbase + Lay::kK + st * Lay::kTile + b * 16384, &tmap_k, FEM_BAR(kHKFull + st), b * 64,
                  kt * kBlockK, bh);
    const size_t row = static_cast<size_t>(bh) * n_kt_all + kt;
    const uint32_t slot = sbase + Lay::kSide + ss * Lay::kSideStride;
    mbar_arrive_expect_tx(FEM_BAR(kHSide + ss), Lay::kSideMask + 16);
    bulk_load(slot, w.rfac + row * D, D * 4, FEM_BAR(kHSide + ss));
    bulk_load(slot + D * 4, w.colsum + row * D, D * 4, FEM_BAR(kHSide + ss));
    bulk_load(slot + Lay::kSideMask, w.colmask + row * 4, 16, FEM_BAR(kHSide + ss));
  };
  auto load_e = [&](int kt) {
    const int st = kt % kSlotsE;
    mbar_arrive_expect_tx(FEM_BAR(kHEFull + st), Lay::kTile);
    for (int b = 0; b < D / 64; ++b)
      tma_load_3d(sbase + Lay::kE + st * Lay::kTile + b * 16384, &tmap_e, FEM_BAR(kHEFull + st), b * 64,
                  kt * kBlockK, bh);
  };

  grid_dep_launch_dependents();
  if (warp == 4) {
    tmem_alloc(sbase + Lay::kTmemSlot, 256);
    tmem_relinquish();
  }
  grid_dep_wait();  // the value bank, its plan and column sums; the fix-up list's counters
  if (tid == 0) {
    for (int i = 0; i < kHCount; ++i) mbar_init(FEM_BAR(i), i == kHSFree || i == kHPFull ? 128 : (i == kHAll ? 2 : 1));
    fence_mbar_init();
    *abort_flag = 0;
    // the first loads leave before the rest of the prologue
    mbar_arrive_expect_tx(FEM_BAR(kHQ), Lay::kTile);
    for (int b = 0; b < D / 64; ++b)
      tma_load_3d(sbase + Lay::kQ + b * 16384, &tmap_q, FEM_BAR(kHQ), b * 64, qt * kBlockQ, bh);
    for (int kt = 0; kt < min(nk, kStagesK); ++kt) load_k(kt);
    for (int kt = 0; kt < min(nk, kSlotsE); ++kt) load_e(kt);
  }
  // rows with listed entries [16..19], rows with candidate entries [20..23]
  if (tid < 8) reinterpret_cast<unsigned *>(smem + Lay::kMisc)[16 + tid] = 0u;
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(smem + Lay::kTmemSlot);

  // The issuing warps run converged, lane 0 issuing.
  const uint32_t lead = lane == 0 ? 1u : 0u;
  auto wait = [&](int bar, int parity, unsigned code) {
    return __all_sync(0xffffffffu, wait_or_abort(FEM_BAR(bar), parity, err, code, abort_flag)) != 0;
  };
  if (warp == 4) {
    // ---------------------------------------------------------------- S_k = Q K_k^T once the softmax has
    // read S_(k-1), and the loads.  S_(k-1) is then complete, so K_(k+1) may take its stage at once; the
    // bank tile k+1 takes the slot that P E of tile k-2 left.
    constexpr uint32_t idesc_qk = idesc_f16(128, 128, true, false);
    bool ok = wait(kHQ, 0, kErrWaitTma);
    for (int kt = 0; ok && kt < nk; ++kt) {
      const int ks = kt % kStagesK;
      if (!(ok = wait(kHKFull + ks, (kt / kStagesK) & 1, kErrWaitTma))) break;
      if (kt > 0 && !(ok = wait(kHSFree, (kt - 1) & 1, kErrWaitMma))) break;
      tc_fence_after_sync();
      const uint32_t sK = sbase + Lay::kK + ks * Lay::kTile;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t off = (kk >> 2) * 16384 + (kk & 3) * 32;
        mma_f16_ss(lead, tmem, smem_desc_sw128(sbase + Lay::kQ + off, 16, 1024), smem_desc_sw128(sK + off, 16, 1024),
                   idesc_qk, kk > 0 ? 1u : 0u);
      }
      mma_commit(lead, FEM_BAR(kHSFull));
      if (kt > 0 && kt + 1 < nk) {
        if (lane == 0) load_k(kt + 1);
        if (kt + 1 >= kSlotsE) {
          if (!(ok = wait(kHEEmpty + (kt + 1) % kSlotsE, ((kt + 1) / kSlotsE - 1) & 1, kErrWaitMma))) break;
          if (lane == 0) load_e(kt + 1);
        }
      }
      __syncwarp();
    }
    mma_commit(lead, FEM_BAR(kHAll));
    // no contraction may be in flight when the TMEM allocation is released: both issuers commit this
    // barrier on every exit path
    if (lane == 0) mbar_wait(FEM_BAR(kHAll), 0, err, kErrWaitMma);
    __syncwarp();
  } else if (warp == 5) {
    // ---------------------------------------------------------------- acc += P_k E_k
    constexpr uint32_t idesc_pv = idesc_f16(128, D, false, true);
    bool ok = true;
    for (int kt = 0; ok && kt < nk; ++kt) {
      const int st = kt % kSlotsE;
      if (!(ok = wait(kHEFull + st, (kt / kSlotsE) & 1, kErrWaitTma))) break;
      if (!(ok = wait(kHPFull, kt & 1, kErrWaitMma))) break;
      tc_fence_after_sync();
      const uint32_t sE = sbase + Lay::kE + st * Lay::kTile;
      const bool afresh = kt == 0 || (split && kt == nk - 1);  // acc starts from this tile
#pragma unroll
      for (int kk = 0; kk < kBlockK / 16; ++kk)
        mma_f16_ts(lead, tmem + Lay::kColAcc, tmem + Lay::kColP + kk * 8, smem_desc_sw128(sE + kk * 2048, 16384, 1024),
                   idesc_pv, (!afresh || kk > 0) ? 1u : 0u);
      mma_commit(lead, FEM_BAR(kHPvDone));
      mma_commit(lead, FEM_BAR(kHEEmpty + st));
    }
    mma_commit(lead, FEM_BAR(kHAll));  // completes once everything this warp issued is done
  } else {
    // ---------------------------------------------------------------- softmax and rescale
    const int r = tid;  // row within the tile
    const int t_row = qt * kBlockQ + r;
    const uint32_t lane_off = static_cast<uint32_t>(warp * 32) << 16;
    const uint32_t tS = tmem + lane_off, tP = tmem + Lay::kColP + lane_off, tAcc = tmem + Lay::kColAcc + lane_off;
    float4 *s_gco = reinterpret_cast<float4 *>(smem + Lay::kGco);
    unsigned *s_flag = reinterpret_cast<unsigned *>(smem + Lay::kFlag);  // [128][4]
    int *s_misc = reinterpret_cast<int *>(smem + Lay::kMisc);
    float m_row = -INFINITY, L_row = 0.f, alpha_last = 1.f;
    float2 pre = make_float2(-INFINITY, 0.f);  // (m, L) before the last key tile
    float ecol = 0.f, ecol_pre = 0.f;          // thread j < D: channel j's sum of |bank|, in the current shift's units
    bool ok = true;
    if (r < D) {
      const ChanInfo ci = w.chan[bh * D + r];
      c_coef[r] = make_float4(ci.c_lin, ci.linear, beta[h * D + r],
                              w.shift[(static_cast<size_t>(bh) * n_kt_all + nk - 1) * D + r]);
    }
    const float qk_scale = kLog2e * rsqrtf(static_cast<float>(D));
    // Barriers are tested ahead of the exponentials and voted on after them, so that a phase that has
    // completed by then (nearly always) costs no round trip on the row's chain: 1 done, 0 to be waited for.
    int s_done = 0, side_done = 0;
    auto settle = [&](int done, int bar, int parity, unsigned code) {
      return __all_sync(0xffffffffu, done != 0) ||
             __all_sync(0xffffffffu, wait_or_abort(FEM_BAR(bar), parity, err, code, abort_flag));
    };
    for (int kt = 0; kt < nk; ++kt) {
      // every lane takes the same branch: the waits' outcomes are made warp-uniform
      const int ss = kt % Lay::kSideStages;
      ok = settle(side_done, kHSide + ss, (kt / Lay::kSideStages) & 1, kErrWaitTma) &&
           settle(s_done, kHSFull, kt & 1, kErrWaitMma);
      if (!ok) break;
      tc_fence_after_sync();
      const bool last_split = split && kt == nk - 1;
      // this tile's rescale factors exp(beta_j (c_old - c_new)), 1 for unmoved channels, its column
      // sums and its moved-channel mask
      const float *rf = reinterpret_cast<const float *>(smem + Lay::kSide + ss * Lay::kSideStride);
      const uint4 m4 = *reinterpret_cast<const uint4 *>(rf + Lay::kSideMask / 4);
      float alpha = 1.f;
      {
        // the whole 128-column score row: four loads in flight, one wait
        uint32_t sr[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[c * 32]));
        if (last_split) ecol_pre = ecol;
        if (r < D) ecol = fmaf(ecol, rf[r], rf[D + r]);
        tmem_ld_wait();
        tc_fence_before_sync();
        mbar_arrive(FEM_BAR(kHSFree));
        float *s = reinterpret_cast<float *>(sr);
        const int k0 = kt * kBlockK;
        if ((causal && kt == qt) || k0 + kBlockK > T) {
          // keys k0 + n are visible for n < lim (key < T, and key <= row when causal)
          const int lim = min(T, causal ? t_row + 1 : T) - k0;
#pragma unroll
          for (int n = 0; n < 128; ++n) s[n] = n < lim ? s[n] : -INFINITY;
        }
        float mx[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) mx[u] = fmax3(s[u], s[u + 8], s[u + 16]);
#pragma unroll
        for (int n = 24; n < 120; n += 16)
#pragma unroll
          for (int u = 0; u < 8; ++u) mx[u] = fmax3(mx[u], s[n + u], s[n + 8 + u]);
#pragma unroll
        for (int u = 0; u < 8; ++u) mx[u] = fmaxf(mx[u], s[120 + u]);
        float tmax = fmax3(fmax3(mx[0], mx[1], mx[2]), fmax3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]));
        tmax *= qk_scale;  // log2-domain row maximum of this tile
        if (kt == nk - 1) pre = make_float2(m_row, L_row);
        if (tmax > m_row + kRowMaxLag) {
          alpha = ex2_approx(m_row - tmax);  // 0 on the first tile
          m_row = tmax;
        }
        int pv_done = 1;
        if (kt > 0) pv_done = mbar_test_wait(FEM_BAR(kHPvDone), (kt - 1) & 1);
        side_done = s_done = 0;
        if (kt + 1 < nk) {
          side_done = mbar_test_wait(FEM_BAR(kHSide + (kt + 1) % Lay::kSideStages), ((kt + 1) / Lay::kSideStages) & 1);
          s_done = mbar_test_wait(FEM_BAR(kHSFull), (kt + 1) & 1);
        }
        // P = exp2(s * scale - m) as fp16, kept in registers until P_(k-1) has been read; L from the fp32
        // values
        const float2 scale2 = make_float2(qk_scale, qk_scale), negm2 = make_float2(-m_row, -m_row);
        float2 ls[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) ls[u] = make_float2(0.f, 0.f);
        uint32_t p[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) {
          const float2 x = __ffma2_rn(make_float2(s[2 * i], s[2 * i + 1]), scale2, negm2);
          const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
          ls[i & 3] = __fadd2_rn(ls[i & 3], e);
          p[i] = pack_half2(e.x, e.y);
        }
        // P_(k-1) is read and acc final for tile k-1 once its P E completed
        if (kt > 0) {
          ok = settle(pv_done, kHPvDone, (kt - 1) & 1, kErrWaitMma);
          if (!ok) break;
          tc_fence_after_sync();
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_st16(tP + c * 16, *reinterpret_cast<const uint32_t(*)[16]>(&p[c * 16]));
        const float lsum = (ls[0].x + ls[0].y) + (ls[1].x + ls[1].y) + (ls[2].x + ls[2].y) + (ls[3].x + ls[3].y);
        L_row = L_row * alpha + lsum;
      }
      if (last_split) {
        // acc leaves for shared memory (every score contraction is complete: Q and K are idle)
        alpha_last = alpha;
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v[32];
          tmem_ld32(tAcc + c * 32, v);
          tmem_ld_wait();
          uint8_t *box = smem + Lay::kBox + c * 16384;  // 128 rows x 32 fp32, 128-byte swizzle
#pragma unroll
          for (int i4 = 0; i4 < 8; ++i4)
            *reinterpret_cast<uint4 *>(box + sw128_offset(r, i4)) =
                make_uint4(v[4 * i4], v[4 * i4 + 1], v[4 * i4 + 2], v[4 * i4 + 3]);
        }
      } else if (kt > 0) {
        // the joint rescale of acc: every column when a row maximum of the warp moved, the 32-column
        // groups holding a moved channel otherwise
        const bool rowmv = __any_sync(0xffffffffu, alpha != 1.f);
        const unsigned gm = (m4.x ? 1u : 0u) | (m4.y ? 2u : 0u) | (m4.z ? 4u : 0u) | (m4.w ? 8u : 0u);
        if (rowmv || gm != 0u) {
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            const bool mv = (gm >> c) & 1u;
            if (!rowmv && !mv) continue;
            uint32_t v[32];
            tmem_ld32(tAcc + c * 32, v);
            float f[32];
#pragma unroll
            for (int i4 = 0; i4 < 8; ++i4) {
              const float4 f4 = *reinterpret_cast<const float4 *>(rf + c * 32 + i4 * 4);  // exactly 1 where unmoved
              f[4 * i4] = f4.x * alpha;
              f[4 * i4 + 1] = f4.y * alpha;
              f[4 * i4 + 2] = f4.z * alpha;
              f[4 * i4 + 3] = f4.w * alpha;
            }
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * f[i]);
            tmem_st32(tAcc + c * 32, v);
          }
        }
      }
      tmem_st_wait();
      tc_fence_before_sync();
      mbar_arrive(FEM_BAR(kHPFull));
    }
    // the guard's coefficients of channel j: an entry is rejected when
    //   X a + Z / L < Y          (final state, a = acc / L)
    //   X a_pre + Zp < Y L_pre   (state before the diagonal tile)
    // with X = tau beta, Z = -2^-25 Ecol, Zp = -2^-25 Ecol_pre and Y = 2^-25
    // (shifted bank) or -tau (linear bank); see kGuardTau
    if (r < D) {
      const float4 raw = c_coef[r];
      const bool lin = raw.y != 0.f;
      const float beta_r = raw.z;
      c_coef[r] = lin ? make_float4(beta_r, raw.x, beta_r != 0.f ? kLn2 / beta_r : 0.f, 0.f)
                      : make_float4(0.f, raw.w - kBankOffset / beta_r, kLn2 / beta_r, 1.f);
      const float4 g = make_float4(kGuardTau * beta_r, -kGuardUlp * ecol, lin ? -kGuardTau : kGuardUlp, -kGuardUlp * ecol_pre);
      s_gco[r] = g;
      // the same test on the final state as a < A + B / L: A = Y / X, B = -Z / X for
      // X > 0; at beta = 0 (X = 0, linear) it holds for no L >= 1 unless -Z > tau,
      // in which case every entry of the channel goes to the exact test
      reinterpret_cast<float2 *>(smem + Lay::kThr)[r] =
          g.x > 0.f ? make_float2(g.z / g.x, -g.y / g.x) : make_float2(-g.y > kGuardTau ? INFINITY : -INFINITY, 0.f);
    }
    // ---- epilogue.  acc / L is staged in shared memory (Q and K are idle) as 32-column boxes, row r
    // by thread r; the transform then runs column-parallel and writes each row's 32 columns of a box
    // as one coalesced 128-byte store.
    if (ok)
      ok = __all_sync(0xffffffffu, wait_or_abort(FEM_BAR(kHPvDone), (nk - 1) & 1, err, kErrWaitMma, abort_flag));
    ok = bar_and(4, 128, ok);
    if (ok) {
      tc_fence_after_sync();
      const float invL = 1.f / L_row;
      reinterpret_cast<float *>(smem + Lay::kInvLT)[(r & 3) * 32 + (r >> 2)] = invL;
      if (lse && t_row < T) lse[static_cast<size_t>(bh) * T + t_row] = (m_row + lg2_approx(L_row)) * kLn2;
      const float *rf_last =
          reinterpret_cast<const float *>(smem + Lay::kSide + ((nk - 1) % Lay::kSideStages) * Lay::kSideStride);
      unsigned bad = 0;  // a rejected entry whose state before the diagonal tile is rejected too
      const float2 *s_ab = reinterpret_cast<const float2 *>(smem + Lay::kThr);
      // chunk by chunk: acc before the diagonal tile (split) times the diagonal tile's factors, alpha
      // of the row and exp(beta (c_old - c_new)) of the channel, plus the diagonal tile's P E, over L,
      // staged; the state before goes back to acc's columns for the exact test below
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        uint32_t v[32];
        tmem_ld32(tAcc + c * 32, v);
        uint8_t *box = smem + Lay::kBox + c * 16384;
        if (split) {
          uint32_t vp[32];
#pragma unroll
          for (int i4 = 0; i4 < 8; ++i4) {
            const uint4 q4 = *reinterpret_cast<const uint4 *>(box + sw128_offset(r, i4));
            vp[4 * i4] = q4.x;
            vp[4 * i4 + 1] = q4.y;
            vp[4 * i4 + 2] = q4.z;
            vp[4 * i4 + 3] = q4.w;
          }
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i)
            v[i] = __float_as_uint(
                fmaf(__uint_as_float(vp[i]), alpha_last * rf_last[c * 32 + i], __uint_as_float(v[i])));
          tmem_st32(tAcc + c * 32, vp);
        } else {
          tmem_ld_wait();
        }
#pragma unroll
        for (int i4 = 0; i4 < 8; ++i4)
          *reinterpret_cast<float4 *>(box + sw128_offset(r, i4)) =
              make_float4(__uint_as_float(v[4 * i4]) * invL, __uint_as_float(v[4 * i4 + 1]) * invL,
                          __uint_as_float(v[4 * i4 + 2]) * invL, __uint_as_float(v[4 * i4 + 3]) * invL);
      }
      tmem_st_wait();
      bar_sync(4, 128);  // every box is staged
      // Thread r takes column r % 32 of a chunk and rows r / 32 + 4k, so its
      // channel's coefficients stay in registers, each warp access is one
      // 128-byte row of the box, and 8 loads at a time are in flight before the math.
      //   shifted bank: c + (log a - kappa)/beta = lg2(a) ln2/beta + (c - kappa/beta)
      //   linear bank:  c + log1p(x)/beta with x = beta a, as lg2(1 + x) ln2/beta + c,
      //                 or, for |x| < 2^-6 (also beta = 0), as c + a times the
      //                 series of log1p(x)/x
      // The underflow guard's test a < A + B / L runs here too, thread per channel
      // with A, B in registers; rows with a candidate entry are marked for the
      // exact test after the transform.
      const int col = r & 31, row0 = r >> 5;
      const int rows_left = T - qt * kBlockQ;
      const size_t tile_off = (static_cast<size_t>(bh) * T + static_cast<size_t>(qt) * kBlockQ) * D + col;
      float *out_tile = out + tile_off;
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        const float4 cf = c_coef[c * 32 + col];
        const float2 thr = s_ab[c * 32 + col];
        const bool lin = cf.w == 0.f;
        // pairs of rows go through the packed fp32x2 pipe; the lg2 argument is
        // a (shifted) or 1 + beta a (linear)
        const float2 bx2 = make_float2(cf.x, cf.x), y2 = make_float2(cf.y, cf.y), z2 = make_float2(cf.z, cf.z);
        const float2 s12 = lin ? bx2 : make_float2(1.f, 1.f), s02 = make_float2(lin ? 1.f : 0.f, lin ? 1.f : 0.f);
        const uint8_t *box = smem + Lay::kBox + c * 16384 + ((col & 3) << 2);
#pragma unroll 1
        for (int k0 = 0; k0 < 32; k0 += 8) {
          float a[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            a[k] = *reinterpret_cast<const float *>(box + sw128_offset(row0 + 4 * (k0 + k), col >> 2));
          // the guard's quick test on the 8 rows (row0 + 4 (k0 + k) lies in word k0 / 8, bit row0 + 4 k)
          {
            const float4 il0 = *reinterpret_cast<const float4 *>(smem + Lay::kInvLT + (row0 * 32 + k0) * 4);
            const float4 il1 = *reinterpret_cast<const float4 *>(smem + Lay::kInvLT + (row0 * 32 + k0 + 4) * 4);
            const float il[8] = {il0.x, il0.y, il0.z, il0.w, il1.x, il1.y, il1.z, il1.w};
            // two rows per packed fma; the rows' own marks only when some entry of the batch is a candidate
            bool anyc = false;
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
              const float2 t2 = __ffma2_rn(make_float2(thr.y, thr.y), make_float2(il[k], il[k + 1]),
                                           make_float2(thr.x, thr.x));
              anyc = anyc || a[k] < t2.x || a[k + 1] < t2.y;
            }
            if (__any_sync(0xffffffffu, anyc)) {
              unsigned cm = 0;
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const bool cnd = a[k] < fmaf(thr.y, il[k], thr.x);
                cm |= (cnd && row0 + 4 * (k0 + k) < rows_left) ? 1u << (row0 + 4 * k) : 0u;
              }
              cm = __reduce_or_sync(0xffffffffu, cm);
              if (cm && lane == 0) atomicOr(reinterpret_cast<unsigned *>(smem + Lay::kMisc) + 20 + (k0 >> 3), cm);
            }
          }
          float o[8];
#pragma unroll
          for (int k = 0; k < 8; k += 2) {
            const float2 a2 = make_float2(a[k], a[k + 1]);
            const float2 x2 = __fmul2_rn(bx2, a2);
            const float2 g2 = __ffma2_rn(a2, s12, s02);
            const float2 lg = __ffma2_rn(make_float2(lg2_approx(g2.x), lg2_approx(g2.y)), z2, y2);
            float2 q = __ffma2_rn(x2, make_float2(0.2f, 0.2f), make_float2(-0.25f, -0.25f));
            q = __ffma2_rn(x2, q, make_float2(1.f / 3.f, 1.f / 3.f));
            q = __ffma2_rn(x2, q, make_float2(-0.5f, -0.5f));
            q = __ffma2_rn(x2, q, make_float2(1.f, 1.f));
            const float2 se = __ffma2_rn(a2, q, y2);
            o[k] = (lin && fabsf(x2.x) < 0.015625f) ? se.x : lg.x;
            o[k + 1] = (lin && fabsf(x2.y) < 0.015625f) ? se.y : lg.y;
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int row = row0 + 4 * (k0 + k);
            if (row < rows_left) __stcs(out_tile + static_cast<size_t>(row) * D + c * 32, o[k]);
          }
        }
      }
      // ---- the exact guard on the marked rows, row r by thread r: a rejected
      // entry's accumulator before the diagonal tile replaces its output (the
      // fix-up's starting state), and whether that state passes the guard too
      // decides where the fix-up starts
      bar_sync(4, 128);  // the transform's stores and marks are complete
      const unsigned *rowcand = reinterpret_cast<const unsigned *>(smem + Lay::kMisc) + 20;
      if ((rowcand[0] | rowcand[1] | rowcand[2] | rowcand[3]) != 0u) {
        const bool cand = (rowcand[r >> 5] >> (r & 31)) & 1u;
        if (__any_sync(0xffffffffu, cand)) {
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            uint32_t vp[32];
            tmem_ld32(tAcc + c * 32, vp);
            tmem_ld_wait();
            unsigned fm = 0;
            if (cand) {
              const uint8_t *box = smem + Lay::kBox + c * 16384;
              const float4 *gco = s_gco + c * 32;
              const size_t orow = (static_cast<size_t>(bh) * T + t_row) * D + c * 32;
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                const float cell = *(reinterpret_cast<const float *>(box + sw128_offset(r, i >> 2)) + (i & 3));
                const float4 g = gco[i];
                const float2 t = s_ab[c * 32 + i];
                if (!(cell < fmaf(t.y, invL, t.x))) continue;
                fm |= 1u << i;
                const float a_pre = split ? __uint_as_float(vp[i]) : 0.f;
                if (split && fmaf(g.x, a_pre, g.w) < g.z * pre.y) bad = 1;
                out[orow + i] = a_pre;
              }
            }
            s_flag[r * 4 + c] = fm;
            if (fm) atomicOr(reinterpret_cast<unsigned *>(smem + Lay::kMisc) + 16 + (r >> 5), 1u << (r & 31));
          }
        } else {
#pragma unroll
          for (int c = 0; c < D / 32; ++c) s_flag[r * 4 + c] = 0u;
        }
        bar_sync(4, 128);
      }
      // ---- list the rejected rows: one block of entries that restart from the
      // diagonal tile, one of entries recomputed over every key tile, each padded
      // to a multiple of kFixChunk rows (rows -1) for the fix-up's chunks
      const unsigned *rowflags = reinterpret_cast<const unsigned *>(smem + Lay::kMisc) + 16;
      const bool any_listed = (rowflags[0] | rowflags[1] | rowflags[2] | rowflags[3]) != 0u;
      int base = 0;  // thread 0: the first reserved slot
      if (any_listed) {
        const bool listed = (rowflags[r >> 5] >> (r & 31)) & 1u;
        const bool diag = listed && split && bad == 0u;
        const unsigned bd = __ballot_sync(0xffffffffu, diag), bf = __ballot_sync(0xffffffffu, listed && !diag);
        if (lane == 0) {
          s_misc[8 + warp] = __popc(bd);
          s_misc[12 + warp] = __popc(bf);
        }
        bar_sync(4, 128);
        if (r == 0) {
          int nd = 0, nf = 0;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            nd += s_misc[8 + q];
            nf += s_misc[12 + q];
          }
          base = atomicAdd(w.fixup_count, pad_chunk(nd) + pad_chunk(nf));
          atomicAdd(w.fixup_rows, nd + nf);
        }
      }
      // ---- the listed rows' entries, in the reserved slots
      if (any_listed) {
        if (r == 0) s_misc[0] = base;
        bar_sync(4, 128);
        const int b0 = s_misc[0], wq = warp & 3;
        int nd = 0, nf = 0, pd = 0, pf = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int a = s_misc[8 + q], b = s_misc[12 + q];
          nd += a;
          nf += b;
          pd += q < wq ? a : 0;
          pf += q < wq ? b : 0;
        }
        const int sd = pad_chunk(nd), sf = pad_chunk(nf);
        const bool listed = (rowflags[r >> 5] >> (r & 31)) & 1u;
        const bool diag = listed && split && bad == 0u;
        const unsigned bd = __ballot_sync(0xffffffffu, diag), bf = __ballot_sync(0xffffffffu, listed && !diag);
        const unsigned below = (1u << lane) - 1u;
        if (listed) {
          FixupEntry e;
          e.row = bh * T + t_row;
#pragma unroll
          for (int g = 0; g < 4; ++g) e.mask[g] = g < D / 32 ? s_flag[r * 4 + g] : 0u;
          e.m_pre = pre.x;
          e.l_pre = pre.y;
          e.kt0 = diag ? nk - 1 : 0;
          if (!diag) e.l_pre = 0.f;
          w.fixups[diag ? b0 + pd + __popc(bd & below) : b0 + sd + pf + __popc(bf & below)] = e;
        }
        FixupEntry padding;
        padding.row = -1;
        padding.mask[0] = padding.mask[1] = padding.mask[2] = padding.mask[3] = 0u;
        padding.m_pre = -INFINITY;
        padding.l_pre = 0.f;
        if (r < sd - nd) {
          padding.kt0 = nk - 1;
          w.fixups[b0 + nd + r] = padding;
        }
        if (r < sf - nf) {
          padding.kt0 = 0;
          w.fixups[b0 + sd + nf + r] = padding;
        }
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 4) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 256);
  }
#undef FEM_BAR
}

}  // namespace

cudaError_t launch_tc_half(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &te, float *out,
                           const float *beta, const BankWorkspace &w, float *lse, int BH, int H, int T, int causal,
                           unsigned *err, cudaStream_t stream, bool pdl) {
  const int n_qt = (T + kBlockQ - 1) / kBlockQ;
  if (T > kMaxSeqLen || BH > 65535) return cudaErrorInvalidValue;
  cudaError_t e =
      cudaFuncSetAttribute(fem_tc_half_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, HalfLayout::kAlloc);
  if (e != cudaSuccess) return e;
  e = launch_kernel(fem_tc_half_kernel, dim3(n_qt, BH), dim3(192), HalfLayout::kAlloc, stream, pdl, tq, tk, te, out,
                    beta, w, lse, H, T, causal, err);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace fem
