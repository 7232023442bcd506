// nbm_tc_fwd.cu -- forward passes of the mixed-precision NBM step on the tensor
// cores (arXiv 2210.14907 Sec. 3 / Fig. 2): the residual of uncut points
// (MODE_RESIDUAL) and the networks at cut cells (MODE_CUT_FWD).
//
// The half-tiles (8 points x 8 stencil columns), images and arithmetic of the
// training kernel (nbm_tc.cu).  Without a backward a half-tile needs one operand
// image and no weight-gradient columns, so each of the CTA's two groups of 8
// warps keeps kX = 3 half-tiles in flight (an image of 16 KB and 64 TMEM
// accumulator columns each), and the 128 columns left hold the first two hidden
// layers' weights as the GEMMs' A operand.  A warp that has written its part of a
// half-tile's image arrives on that half-tile's `ready` barrier and goes on to the
// next one; a warp per group (the 17th and 18th) waits for the 8 arrivals, issues
// the GEMM and fetches the next half-tiles' records.  So one half-tile's GEMM latency
// is covered by the other two's epilogues, and the warps of a group meet once per
// three half-tiles, before the rows.
// The training kernel ran these passes with one half-tile per group in flight and
// every GEMM exposed to its group: a residual call of 50,001 points, 3 -> 128 x 3 -> 1,
// over four spacings took 874 us and takes 636 with this kernel.
#include "nbm_device.cuh"
#include "nbm_tc_layer.cuh"
#include "nbm_tc_ptx.cuh"

namespace nbm {

using namespace tc;

namespace {

constexpr int kX = 3;          // half-tiles in flight per group
constexpr int kFwdT = 576;     // 16 compute warps, 2 issuing warps
constexpr int kGroupT = 288;   // a group's threads with its issuing warp
// byte offsets in the miscellaneous block
constexpr int kBarMma = 8, kBarRdy = kBarMma + 16 * kX, kBarP = kBarRdy + 16 * kX;
constexpr int kSlot = kBarP + 16, kAbort = kSlot + 4, kLossRed = 128;
constexpr int kRed = kLossRed + 128, kPbuf = kRed + 2 * kX * 4 * 64 * 4;
constexpr int kMiscF = kPbuf + 2 * 2 * kX * kHP * (int)sizeof(PRec);
static_assert(kAbort + 4 <= kLossRed, "barriers overlap the loss partials");

size_t fwd_smem_bytes(int L) { return (size_t)(L - 1) * kImg + 2 * kX * kImgH + kMiscF + 1024; }

template <int L, bool FAST>
__global__ void __launch_bounds__(kFwdT, 1) k_fwd_tc(ProbDev P, StepArgs a) {
  pdl_enter();
  constexpr int H = 128, NG = L - 1, kPPT = 4;
  constexpr uint32_t NCOLS = 512, kWCol = 2 * kX * 64;  // TMEM columns; the first past the D's
  constexpr int kWT = NG < 2 ? NG : 2;                  // layers with their weights in TMEM
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = align1024(smem_raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const bool issuer = w >= 16;
  const int grp = issuer ? w - 16 : tid >> 8, gtid = tid & 255;
  const int q = w & 3, cgl = (w >> 2) & 1, u = 32 * q + lane, col0 = 32 * cgl;
  const uint32_t gbar = 1u + (uint32_t)grp;
  unsigned char* Wimg = sm;                                // [NG][32 KB]
  unsigned char* Aimg = sm + NG * kImg + grp * kX * kImgH;  // this group's [kX][16 KB]
  unsigned char* misc = sm + NG * kImg + 2 * kX * kImgH;
  uint64_t* bar_w = (uint64_t*)misc;
  uint64_t* bar_mma = (uint64_t*)(misc + kBarMma) + kX * grp;
  uint64_t* bar_rdy = (uint64_t*)(misc + kBarRdy) + kX * grp;
  uint64_t* bar_p = (uint64_t*)(misc + kBarP) + grp;
  uint32_t* tslot = (uint32_t*)(misc + kSlot);
  volatile int* abort_f = (volatile int*)(misc + kAbort);
  double* loss_red = (double*)(misc + kLossRed);                 // [16]
  float* red = (float*)(misc + kRed) + grp * kX * 4 * 64;        // [kX][4][64]
  PRec* pbuf = (PRec*)(misc + kPbuf) + grp * 2 * kX * kHP;       // [2][kX][8]
  // (point chunk j of this thread's row: the swizzled 16-byte chunks differ by an xor)
  const uint32_t off0 = (uint32_t)((u >> 3) * 1024 + (u & 7) * 128 + ((((cgl << 2) ^ u) & 7) << 4));
  auto poff = [&](int j) -> uint32_t { return off0 ^ (uint32_t)(j << 4); };
  const uint32_t idf = idesc_f16_n(true, false, true, kHP * 8);

  if (tid == 0) {
    mbar_init(smem_u32(bar_w), 1);
    for (int b = 0; b < 2 * kX; ++b) {
      mbar_init(smem_u32((uint64_t*)(misc + kBarMma) + b), 1);
      mbar_init(smem_u32((uint64_t*)(misc + kBarRdy) + b), 8);  // one arrival per warp
    }
    mbar_init(smem_u32((uint64_t*)(misc + kBarP)), 1);
    mbar_init(smem_u32((uint64_t*)(misc + kBarP) + 1), 1);
    *abort_f = 0;
    fence_mbar_init();
  }
  if (w == 0) tmem_alloc(smem_u32(tslot), NCOLS);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t d_tm = tmem + (uint32_t)(kX * 64 * grp);  // half-tile X: d_tm + 64 X
  const uint32_t lane_base = (uint32_t)(32 * q) << 16;
  // per-half-tile state as bit X: barrier phase (MMA; in the issuing warps: ready),
  // and a GEMM not yet waited for
  uint32_t ph_w = 0, ph_bits = 0, pending_bits = 0, ph_p = 0;
  bool aborted = false;

  const int nm = a.counters[0], np = a.counters[1], nc = a.counters[2];
  const bool cutfwd = a.mode == MODE_CUT_FWD;
  const int T0 = cutfwd ? (nc + kHP - 1) / kHP : (nm + kHP - 1) / kHP;
  const int T = cutfwd ? 2 * T0 : T0 + (np + kHP - 1) / kHP;
  const int tb = (int)((int64_t)blockIdx.x * T / gridDim.x);
  const int te = (int)((int64_t)(blockIdx.x + 1) * T / gridDim.x);

  // records of the half-tiles t, t + 2, .. (kX at most, below s1) into record buffer b
  // (one lane of the issuing warp; one bulk copy each)
  auto fetch = [&](int t, int s1, int b) {
    const int cnt = s1 <= t ? 0 : (s1 - t + 1) / 2 < kX ? (s1 - t + 1) / 2 : kX;
    if (!cnt) return;
    fence_proxy_async();
    mbar_expect_tx(smem_u32(bar_p), (uint32_t)(cnt * kHP * sizeof(PRec)));
    for (int X = 0; X < cnt; ++X) {
      const int tau = t + 2 * X;
      // the record lists are padded to 16 per list; net 1 starts after net 0's padding
      const PRec* src = cutfwd ? a.rec_cut + (int64_t)kHP * (tau < T0 ? tau : tau - T0)
                      : tau < T0 ? a.rec + (int64_t)kHP * tau
                                 : a.rec + 16 * (int64_t)((nm + 15) / 16) + (int64_t)kHP * (tau - T0);
      bulk_g2s(smem_u32(pbuf + (b * kX + X) * kHP), src, kHP * sizeof(PRec), smem_u32(bar_p));
    }
  };
  // the layer-g GEMM of half-tile X once the 8 warps have written its image (a wait
  // that gave up wakes the waiters without a GEMM)
  auto issue = [&](int X, int g) -> bool {
    const bool ok = mbar_wait_bounded(smem_u32(bar_rdy + X), (ph_bits >> X) & 1u);
    ph_bits ^= 1u << X;
    fence_after_sync();
    if (lane == 0) {
      if (!ok) {
        atomicOr(a.status, 2);
        *abort_f = 1;
        mbar_arrive(smem_u32(bar_mma + X));
      } else {
        const uint32_t ab = smem_u32(Aimg + X * kImgH);
        if (g < kWT) {
          const uint32_t wt = tmem + kWCol + 64u * (uint32_t)g;
#pragma unroll
          for (int k = 0; k < 8; ++k)
            mma_f16_ta(d_tm + 64 * X, wt + 8u * (uint32_t)k, desc_mnmajor(ab) + kstep_mnmajor(k), idf,
                       k > 0);
        } else {
          const uint32_t wa = smem_u32(Wimg + g * kImg);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            mma_f16(d_tm + 64 * X, desc_kmajor(wa) + kstep_kmajor(k),
                    desc_mnmajor(ab) + kstep_mnmajor(k), idf, k > 0);
        }
        mma_commit(smem_u32(bar_mma + X));
      }
    }
    __syncwarp();
    return ok;
  };
  // this warp's part of half-tile X's image is written (and its accumulators are read)
  auto ready = [&](int X) {
    fence_proxy_async();
    fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(bar_rdy + X));
    pending_bits |= 1u << X;
  };
  // bounded wait for half-tile X's GEMM; false if it gave up
  auto wait_mma = [&](int X) -> bool {
    const bool ok = mbar_wait_bounded(smem_u32(bar_mma + X), (ph_bits >> X) & 1u);
    if (ok) {  // a wait that gave up leaves the GEMM pending for the exit path
      ph_bits ^= 1u << X;
      pending_bits &= ~(1u << X);
    }
    fence_after_sync();
    return ok;
  };
  // the group's barrier at the end of a set; it agrees on an abort.  False: abort.
  auto end_set = [&](bool ok) -> bool {
    const bool bad = named_sync_or(gbar, kGroupT, !ok || *abort_f != 0);
    if (bad && lane == 0) {
      if (!ok) atomicOr(a.status, 2);
      *abort_f = 1;
    }
    return !bad;
  };

  float loss_acc = 0.f;     // FP32 rows
  double loss_acc_d = 0.0;  // FP64 rows
  int set = 0;              // sets of this group so far (record buffer parity)
#pragma unroll 1
  for (int net = 0; net < 2; ++net) {
    const int s0 = net == 0 ? tb : (tb > T0 ? tb : T0);
    const int s1 = net == 0 ? (te < T0 ? te : T0) : te;
    if (s0 >= s1) continue;  // the same in every thread of the CTA
    if (tid == 0) {
      const unsigned char* src = (const unsigned char*)a.wtc + (int64_t)net * NG * kImg;
      mbar_expect_tx(smem_u32(bar_w), NG * kImg);
      for (int g = 0; g < NG; ++g)
        bulk_g2s(smem_u32(Wimg + g * kImg), src + (int64_t)g * kImg, kImg, smem_u32(bar_w));
    }
    if (issuer && lane == 0) fetch(s0 + grp, s1, set & 1);
    const float* th = a.params + net * P.p_net;
    const int64_t oo = 4 * H + (int64_t)NG * (H * H + H);
    const float w1[3] = {th[3 * u], th[3 * u + 1], th[3 * u + 2]}, b1 = th[3 * H + u];
    const float wo = th[oo + u], bo = th[oo + H];
    float Td[3];
    bool sd1;
    layer1_increments<FAST>(w1, P.hf, Td, sd1);
    {
      const bool ok = mbar_wait_bounded(smem_u32(bar_w), ph_w);
      if (ok) ph_w ^= 1u;
      if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(a.status, 2);
        aborted = true;
        break;
      }
    }
    // the first kWT layers' weights into TMEM (the previous network's GEMMs have
    // all completed)
    if (w < 4) stage_weights_tmem(Wimg, kImg, tmem + ((uint32_t)(32 * w) << 16) + kWCol, u, kWT);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();

#pragma unroll 1
    for (int t = s0 + grp; t < s1; t += 2 * kX, ++set) {
      const int cnt = (s1 - t + 1) / 2 < kX ? (s1 - t + 1) / 2 : kX;  // half-tiles of this set
      if (issuer) {
        bool ok = true;
#pragma unroll 1
        for (int g = 0; g < NG; ++g)
#pragma unroll 1
          for (int X = 0; X < cnt; ++X) {
            ok = issue(X, g) && ok;
            // (the 8 warps are past the previous set's rows: its records are free)
            if (g == 0 && X == 0 && lane == 0) fetch(t + 2 * kX, s1, (set + 1) & 1);
          }
        if (!end_set(ok)) {
          aborted = true;
          break;
        }
        continue;
      }
      bool ok_all = mbar_wait_bounded(smem_u32(bar_p), ph_p);
      if (ok_all) ph_p ^= 1u;
      const PRec* pr = pbuf + (set & 1) * kX * kHP;  // [kX][8]
      // ---- layer 1 (3 -> H) in FP32
#pragma unroll 1
      for (int X = 0; X < cnt; ++X) {
#pragma unroll
        for (int pp = 0; pp < kPPT; pp += 2) {
          const PRec& pa = pr[X * kHP + 4 * cgl + pp];
          F2 o[8];
          layer1_pair<FAST>(w1, b1, Td, sd1, pa, (&pa)[1], o);
          store_pair(Aimg + X * kImgH, poff(pp), poff(pp + 1), o);
        }
        ready(X);
      }
      // ---- hidden layers; the last one feeds the output layer (H -> 1) in FP32:
      // the sum over the warp's 32 units, then over the four lane quadrants
#pragma unroll 1
      for (int g = 1; g <= NG; ++g) {
        const float bb = th[4 * H + (g - 1) * (H * H + H) + H * H + u];
#pragma unroll 1
        for (int X = 0; X < cnt; ++X) {
          const PRec* px = pr + X * kHP + 4 * cgl;
          ok_all = wait_mma(X) && ok_all;
          float acc[32];
          tmem_ld32(d_tm + 64 * X + lane_base + col0, acc);
#pragma unroll
          for (int jp = 0; jp < kPPT; jp += 2) {
            F2 o[8];
            hidden_pair<FAST>(acc + 8 * jp, bb, px + jp, px + jp + 1, o);
            if (g < NG) {
              store_pair(Aimg + X * kImgH, poff(jp), poff(jp + 1), o);
            } else {
#pragma unroll
              for (int c = 0; c < 8; ++c) f2get(o[c], acc[8 * jp + 2 * c], acc[8 * jp + 2 * c + 1]);
            }
          }
          if (g < NG) {
            ready(X);
          } else {
            float s;
            warp_transpose_reduce32(acc, wo, lane, s);  // lane l: column col0 + l
            red[(X * 4 + q) * 64 + col0 + lane] = s;
          }
        }
      }
      fence_before_sync();
      if (!end_set(ok_all)) {
        aborted = true;
        break;
      }
      // ---- output columns and residual rows: 8 lanes per point, lane c column c
      if (gtid < 64 * cnt) {
        const int X = gtid >> 6, p = (gtid >> 3) & 7, c = gtid & 7;
        const unsigned gmask = 0xFFu << (gtid & 24);
        const float* rx = red + X * 256 + pair_col(p, c);
        float oc = rx[0];
#pragma unroll
        for (int qq = 1; qq < 4; ++qq) oc += rx[64 * qq];
        if (c == 0 || c == 7) oc += bo;
        // the scaled convention of the rows: U, Mt_i = M_i/h^2, Dt_i = D_i/h
        oc *= (c >= 1 && c <= 3) ? P.inv_h2f : (c >= 4 && c <= 6) ? P.inv_hf : 1.f;
        const float Uc = __shfl_sync(gmask, oc, 0, 8);
        const float Mtc = __shfl_sync(gmask, oc, 1 + (c >> 1), 8);
        const float Dtc = __shfl_sync(gmask, oc, 4 + (c >> 1), 8);
        const PRec pi = pr[X * kHP + p];
        if (cutfwd) {
          if (pi.pt >= 0) a.cut_out[(int64_t)(pi.cutj >> 1) * 16 + net * 8 + c] = oc;
        } else if (pi.pt >= 0 && pi.cutj < 0) {
          float sdc, r2;
          bool rows64 = false;
          if constexpr (!FAST) rows64 = P.fp64;
          if (rows64) {
            const double r2d = uncut_residual_lanes<double>(P, net, pi.x, pi.y, pi.z,
                                                            (double)pi.gx + (double)pi.gy, Uc, Mtc,
                                                            Dtc, (double)a.scale, c, gmask, sdc);
            if (c == 0) loss_acc_d += r2d;
            r2 = (float)r2d;
          } else {
            r2 = uncut_residual_lanes<float>(P, net, pi.x, pi.y, pi.z, pi.gx, Uc, Mtc, Dtc, a.scale,
                                             c, gmask, sdc);
            if (c == 0) loss_acc += r2;
          }
          if (c == 0 && a.r2_out) a.r2_out[pi.pt] = (P.level ? a.r2_out[pi.pt] : 0.f) + r2;
        }
      }
      // no barrier here: red is next written after GEMMs of the next set, which wait
      // for every warp's arrival past these reads
    }
    // both groups are done with this network before its weights are replaced
    if (__syncthreads_or(aborted)) {
      aborted = true;
      break;
    }
    fence_after_sync();
  }

  double lsum = (double)loss_acc + loss_acc_d;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0 && !issuer) loss_red[w] = lsum;
  fence_before_sync();
  __syncthreads();
  if (tid == 0 && !cutfwd) {
    double s = 0.0;
    for (int ww = 0; ww < 16; ++ww) s += loss_red[ww];
    a.loss_part[blockIdx.x] = s;
  }
  if (aborted) {
    // a GEMM, a record copy or a weight copy may still be in flight: a short bounded
    // wait (about 1 ms) each before TMEM and shared memory are released
    if (!issuer) {
      for (int X = 0; X < kX; ++X)
        if ((pending_bits >> X) & 1u)
          (void)mbar_wait_bounded(smem_u32(bar_mma + X), (ph_bits >> X) & 1u, 2000000LL);
      (void)mbar_wait_bounded(smem_u32(bar_p), ph_p, 2000000LL);
    }
    (void)mbar_wait_bounded(smem_u32(bar_w), ph_w, 2000000LL);
    fence_before_sync();
    __syncthreads();
  }
  fence_after_sync();
  if (w == 0) tmem_dealloc(tmem, NCOLS);
}

template <int L, bool FAST>
cudaError_t launch_fwd_t(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  const size_t smem = fwd_smem_bytes(L);
  cudaError_t e = cudaFuncSetAttribute(k_fwd_tc<L, FAST>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_fwd_tc<L, FAST>, dim3(grid), dim3(kFwdT), smem, st, P, a);
}

}  // namespace

// MODE_RESIDUAL and MODE_CUT_FWD on BF16 operands; FP64 rows take the accurate
// tanh and reciprocal, as in the training kernel.
cudaError_t launch_fwd_tc(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  if (P.L == 2) return P.fp64 ? launch_fwd_t<2, false>(P, a, grid, st) : launch_fwd_t<2, true>(P, a, grid, st);
  if (P.L == 3) return P.fp64 ? launch_fwd_t<3, false>(P, a, grid, st) : launch_fwd_t<3, true>(P, a, grid, st);
  if (P.L == 4) return P.fp64 ? launch_fwd_t<4, false>(P, a, grid, st) : launch_fwd_t<4, true>(P, a, grid, st);
  return cudaErrorInvalidValue;
}

}  // namespace nbm
