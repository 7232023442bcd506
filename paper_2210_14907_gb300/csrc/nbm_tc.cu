// nbm_tc.cu -- the mixed-precision fused NBM training step on the 5th-generation
// tensor cores (tcgen05, TMEM accumulators), arXiv 2210.14907 Sec. 3 / Fig. 2.
// (The forward-only passes are nbm_tc_fwd.cu's.)
//
// One persistent CTA per SM, 16 warps in two groups of 8.  Each group owns a
// half-tile: 8 collocation points x 8 columns (centre value, symmetric and
// antisymmetric stencil increments of the three axes in difference form, and
// the interface-point value of cut cells), i.e. 64 GEMM columns, with its own
// operand images and its own 64 TMEM accumulator columns.  The groups run
// independently, so that one group's epilogue (CUDA cores) overlaps the other
// group's GEMMs (tensor pipe).  Every hidden layer is one 128 x 64 x 128
// product D[unit][col] = W[unit][k] A[k][col] with BF16 operands and FP32
// accumulation in TMEM; warp w reads TMEM lanes 32(w%4).. (one unit per
// thread) for 32 columns (4 points).  The epilogue applies the tanh stencil
// layer in FP32 and writes the next BF16 operand image to shared memory.
// The first layer (K = 3), the output layer (H -> 1, a warp
// transpose-reduction), the residual rows and the seeds stay FP32 (FP64 rows
// on request).  The epilogues' FP32 arithmetic runs on packed pairs
// (add/mul/fma .f32x2: two points per instruction, each rounded as its scalar
// form).  The backward reuses the stored images: per hidden layer one
// input-gradient MMA (W^T gz, into the group's D columns) and one
// weight-gradient MMA (gz A^T, K = 64) accumulated across all half-tiles of
// the CTA in shared TMEM columns, in a fixed order of the half-tiles, so the
// weight gradient never leaves the SM until the CTA's partial is written once
// per network and is bitwise reproducible.
//
// Bound: instruction issue in the epilogues and the GEMM latency of a group's
// phases that the other group does not fill.  262,144 points, 3 -> 128 x 3 -> 1: a step
// took 1.080 ms with 601 M warp instructions and takes 0.932 with 462 M (issue slots
// busy 46 %, tensor pipe 20 %); what was taken out were the moves that put points'
// columns together into pairs (they are interleaved in the images now), generic
// addresses, votes per point and the descriptors' arithmetic.  Two groups of 8 warps
// are what 120 registers a thread leave room for.
//
// Shared memory: (L-1) weight images of 32 KB + 2 x L operand images of 16 KB.
// TMEM: 2 x 64 columns for D + 128 per hidden layer for the weight gradient.
// Every wait is bounded.  The group barrier that ends each phase agrees on an
// abort; an aborted CTA gives its MMAs and copies in flight a short bounded
// wait before it frees TMEM.
#include "nbm_device.cuh"
#include "nbm_f32x2.cuh"
#include "nbm_tc_layer.cuh"
#include "nbm_tc_ptx.cuh"

namespace nbm {

using namespace tc;

namespace {

constexpr int kMisc = 2048;
constexpr int kPrefetchT = 224;  // rank in the group of the thread that fetches tile records

// Two points' adjoint of one stencil axis (unscaled columns): the arithmetic of
// tanh_stencil_bwd on packed pairs.
__device__ __forceinline__ F2 tanh_stencil_bwd_pair(F2 T, F2 S0, F2 MO, F2 DO, F2 GM, F2 GD,
                                                    F2& gmu, F2& gdel) {
  const F2 P = mul2(fma2(mul2(T, f2s(2.0f)), MO, fma2(MO, MO, mul2(DO, DO))), f2s(-1.0f));
  const F2 Q = mul2(mul2(DO, f2s(-2.0f)), add2(T, MO));
  const F2 S = add2(S0, P);
  const F2 qgd = mul2(Q, GD);
  gmu = fma2(S, GM, qgd);
  gdel = fma2(Q, GM, mul2(S, GD));
  return fma2(P, GM, qgd);
}

}  // namespace

size_t tc_smem_bytes(int L) { return (size_t)(2 * L - 1) * kImg + 1024 + kMisc; }
int tc_supported(int H, int L) { return H == 128 && L >= 2 && L <= 4; }

// Column convention: the difference columns hold mu and del themselves (BF16 has
// the exponent range of FP32); the output stage converts to the scaled convention
// of the residual rows (mu/h^2, del/h).
template <int L, bool FAST>
__global__ void __launch_bounds__(512, 1) k_step_tc(ProbDev P, StepArgs a) {
  pdl_enter();
  constexpr int H = 128;
  constexpr int NG = L - 1;  // hidden GEMM layers
  constexpr int kPPT = 4;    // points per thread (8 warps = 4 lane quadrants x 2 column groups)
  constexpr uint32_t NCOLS = (NG + 1) * 128 <= 256 ? 256 : 512;
  // Two hidden GEMMs use 384 of the 512 columns: the forward GEMMs then take
  // their weights (the A operand) from the last 128, which spares each of them
  // the 32 KB weight read from shared memory.
  constexpr bool kWTmem = NG == 2;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = align1024(smem_raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int grp = tid >> 8, gtid = tid & 255;  // warp group and rank in it
  const int q = w & 3, cgl = (w >> 2) & 1;     // TMEM lane quadrant, column group
  const int u = 32 * q + lane;                 // unit (TMEM lane) of this thread
  const int col0 = 32 * cgl;                   // first of its 32 columns (points 4cgl .. 4cgl+3)
  const uint32_t gbar = 1u + (uint32_t)grp;    // named barrier of the group
  unsigned char* Wimg = sm;                                   // [NG][32 KB]
  unsigned char* Aimg = sm + NG * kImg + grp * L * kImgH;     // this group's [L][16 KB]
  unsigned char* misc = sm + NG * kImg + 2 * L * kImgH;
  uint64_t* bar_w = (uint64_t*)misc;
  uint64_t* bar_mma = (uint64_t*)(misc + 8 + 8 * grp);
  uint64_t* bar_p = (uint64_t*)(misc + 24 + 8 * grp);
  uint32_t* tslot = (uint32_t*)(misc + 40);
  int* done_cnt = (int*)(misc + 44);               // [2] backward MMA phases completed
  volatile int* abort_f = (volatile int*)(misc + 52);
  float* gbo_red = (float*)(misc + 56);            // [2]
  PRec* pbuf = (PRec*)(misc + 64 + grp * 512);     // this group's [2][8] tile records
  float* seeds = (float*)(misc + 1088 + grp * 256);  // this group's 64 seeds
  double* loss_red = (double*)(misc + 1600);         // 16 doubles
  float* red = (float*)(Aimg + (L - 1) * kImgH);     // [4][64] scratch (forward end only)

  // image byte offset of (unit u, point 4cgl + j): the row part is fixed per
  // thread, the 16-byte chunk is (4cgl + j) xor u, mod 8 (the
  // chunks of j = 0 .. 3 differ by an xor)
  const uint32_t off0 = (uint32_t)((u >> 3) * 1024 + (u & 7) * 128 + ((((cgl << 2) ^ u) & 7) << 4));
  auto poff = [&](int j) -> uint32_t { return off0 ^ (uint32_t)(j << 4); };
  const uint32_t id_fwd = idesc_f16_n(true, false, true, kHP * 8);
  const uint32_t id_dgr = idesc_f16_n(true, true, true, kHP * 8);
  const uint32_t id_wgr = idesc_f16_n(true, false, false, 128);

  if (tid == 0) {
    mbar_init(smem_u32(bar_w), 1);
    mbar_init(smem_u32((uint64_t*)(misc + 8)), 1);
    mbar_init(smem_u32((uint64_t*)(misc + 16)), 1);
    mbar_init(smem_u32((uint64_t*)(misc + 24)), 1);
    mbar_init(smem_u32((uint64_t*)(misc + 32)), 1);
    *abort_f = 0;
    fence_mbar_init();
  }
  if (w == 0) tmem_alloc(smem_u32(tslot), NCOLS);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  const uint32_t d_tm = tmem + 64u * (uint32_t)grp;  // this group's D: 64 columns
  const uint32_t lane_base = (uint32_t)(32 * q) << 16;
  uint32_t ph_w = 0, ph_mma = 0, ph_p = 0;
  bool aborted = false;

  // half-tiles of 8 points: net 0, then net 1
  const int nm = a.counters[0], np = a.counters[1];
  const int T0 = (nm + kHP - 1) / kHP, T = T0 + (np + kHP - 1) / kHP;
  const int tb = (int)((int64_t)blockIdx.x * T / gridDim.x);
  const int te = (int)((int64_t)(blockIdx.x + 1) * T / gridDim.x);

  // tile records: one 256-byte bulk copy per half-tile, fetched a tile ahead
  auto prefetch = [&](int tau, int buf) {
    // the record lists are padded to 16 per list; net 1 starts after net 0's padding
    const PRec* src = tau < T0 ? a.rec + (int64_t)kHP * tau
                               : a.rec + 16 * (int64_t)((nm + 15) / 16) + (int64_t)kHP * (tau - T0);
    fence_proxy_async();
    mbar_expect_tx(smem_u32(bar_p), kHP * sizeof(PRec));
    bulk_g2s(smem_u32(pbuf + kHP * buf), src, kHP * sizeof(PRec), smem_u32(bar_p));
  };

  // per-net constants of this thread's unit
  // (first-layer weights and hidden biases are read where they are used, from
  // the L1-resident parameter vector: registers are short at the output stage)
  float wo = 0.f, bo = 0.f;
  const float* th = a.params;
  // gradient accumulators of the small parameters
  float gW1[3] = {0.f, 0.f, 0.f}, gb1 = 0.f, gbh[NG], gwo = 0.f, gbo = 0.f;
#pragma unroll
  for (int g = 0; g < NG; ++g) gbh[g] = 0.f;
  float loss_acc = 0.f;     // per-thread FP32 sum of r^2 (FP32 rows)
  double loss_acc_d = 0.0;  // per-thread FP64 sum of r^2 (FP64 rows)
  int wrote0 = 0, wrote1 = 0;

  // Completion of this group's MMA phase; false (and the CTA-wide abort flag
  // set) if the wait ran out or either group gave up.
  // Bounded wait for the group's MMA phase (no group barrier: the one that ends
  // the phase's epilogue agrees on an abort; until then a thread whose wait
  // gave up only computes on undefined accumulator values).
  auto wait_mma = [&]() -> bool {
    const bool ok = mbar_wait_bounded(smem_u32(bar_mma), ph_mma);
    if (ok) ph_mma ^= 1u;  // a wait that gave up leaves the phase for the exit drain
    fence_after_sync();
    return ok;
  };
  // The group barrier that ends an MMA phase's epilogue.  It orders the
  // epilogue's shared-memory images before the next MMA, keeps every thread
  // within one phase of bar_mma, and agrees on an abort (a wait that gave up,
  // or the abort flag).  False: abort.
  auto end_phase = [&](bool ok) -> bool {
    fence_before_sync();
    fence_proxy_async();
    const bool bad = named_sync_or(gbar, 256, !ok || *abort_f != 0);
    if (bad && gtid == 0) {
      if (!ok) atomicOr(a.status, 2);
      *abort_f = 1;
    }
    return !bad;
  };
  // Gate of one MMA phase, run by the group's first thread before it issues.
  // `order` > 0: wait until the other group has completed that many backward
  // phases first (the weight-gradient accumulators are shared, and a fixed
  // accumulation order keeps the result bitwise reproducible).  Returns false
  // when it gives up; the thread then arrives on the barrier itself, so that
  // its group wakes up and sees the abort flag.
  auto gate = [&](int order) -> bool {
    bool ok = true;
    if (order > 0) {
      const int* other = done_cnt + (grp ^ 1);
      if (ld_acquire_s32(other) < order) {
        const long long t0 = clock64();
        while (ld_acquire_s32(other) < order) {
          if (*abort_f) { ok = false; break; }
          if (clock64() - t0 > 4000000000LL) {
            atomicOr(a.status, 2);
            ok = false;
            break;
          }
          __nanosleep(20);
        }
      }
    }
    if (!ok || *abort_f) {
      *abort_f = 1;
      mbar_arrive(smem_u32(bar_mma));
      return false;
    }
    fence_after_sync();
    return true;
  };

  auto flush = [&](int net) {
    // weight gradients of the hidden layers straight from TMEM: warp w reads
    // lanes 32(w%4).. and columns 32(w/4)..
    const int cgf = w >> 2;
    float* gp = a.gpart + ((int64_t)blockIdx.x * 2 + net) * P.gstride;
#pragma unroll 1
    for (int g = 1; g <= NG; ++g) {
      float* dst = gp + 4 * H + (int64_t)(g - 1) * (H * H + H) + (int64_t)u * H + 32 * cgf;
      float v[32];
      tmem_ld32(tmem + 128u * g + lane_base + 32u * cgf, v);
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
    // small parameters: the four column groups of a unit are combined in smem
    float* stage = (float*)(sm + NG * kImg);  // [4 column groups][128 units][8]
    if (gtid == 0) gbo_red[grp] = gbo;
    fence_before_sync();
    __syncthreads();
    {
      float* s = stage + (cgf * 128 + u) * 8;
      s[0] = gW1[0]; s[1] = gW1[1]; s[2] = gW1[2]; s[3] = gb1; s[4] = gwo;
#pragma unroll
      for (int g = 0; g < NG; ++g) s[5 + g] = gbh[g];
    }
    __syncthreads();
    if (cgf == 0) {
      float t[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) t[k] = stage[u * 8 + k];
#pragma unroll
      for (int c2 = 1; c2 < 4; ++c2)
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k] += stage[(c2 * 128 + u) * 8 + k];
      gp[3 * u] = t[0];
      gp[3 * u + 1] = t[1];
      gp[3 * u + 2] = t[2];
      gp[3 * H + u] = t[3];
#pragma unroll
      for (int g = 0; g < NG; ++g) gp[4 * H + (int64_t)g * (H * H + H) + (int64_t)H * H + u] = t[5 + g];
      const int64_t oo = 4 * H + (int64_t)NG * (H * H + H);
      gp[oo + u] = t[4];
      if (tid == 0) gp[oo + H] = gbo_red[0] + gbo_red[1];
    }
    gW1[0] = gW1[1] = gW1[2] = gb1 = gwo = gbo = 0.f;
#pragma unroll
    for (int g = 0; g < NG; ++g) gbh[g] = 0.f;
    if (net) wrote1 = 1; else wrote0 = 1;
    __syncthreads();
  };

  int kk = 0;  // half-tiles of this group so far (record buffer parity)
#pragma unroll 1
  for (int net = 0; net < 2; ++net) {
    const int s0 = net == 0 ? tb : (tb > T0 ? tb : T0);
    const int s1 = net == 0 ? (te < T0 ? te : T0) : te;
    if (s0 >= s1) continue;  // the same in every thread of the CTA
    // stage this network's hidden weights (bulk copy engine); the two groups
    // take the segment's half-tiles alternately, group 0 the first
    if (tid == 0) {
      done_cnt[0] = 0;
      done_cnt[1] = 0;
      const unsigned char* src = (const unsigned char*)a.wtc + (int64_t)net * NG * kImg;
      mbar_expect_tx(smem_u32(bar_w), NG * kImg);
      for (int g = 0; g < NG; ++g)
        bulk_g2s(smem_u32(Wimg + g * kImg), src + (int64_t)g * kImg, kImg, smem_u32(bar_w));
    }
    if (gtid == kPrefetchT && s0 + grp < s1) prefetch(s0 + grp, kk & 1);
    {
      th = a.params + net * P.p_net;
      const int64_t oo = 4 * H + (int64_t)NG * (H * H + H);
      wo = th[oo + u];
      bo = th[oo + H];
    }
    {
      const bool ok = mbar_wait_bounded(smem_u32(bar_w), ph_w);
      if (ok) ph_w ^= 1u;
      if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(a.status, 2);
        aborted = true;
        break;
      }
    }
    if constexpr (kWTmem) {
      // this network's forward weights into TMEM: layer g in columns 384 +
      // 64 (g-1) .., unit u (row of W) in lane u, W[u][2c] and W[u][2c+1] in
      // column c; the previous segment's GEMMs have all completed
      if (w < 4) stage_weights_tmem(Wimg, kImg, tmem + ((uint32_t)(32 * w) << 16) + 384u, u, NG);
      fence_before_sync();
      __syncthreads();
      fence_after_sync();
    }

    int tile_i = 0;  // index of the half-tile among this group's tiles of the segment
#pragma unroll 1
    for (int tau = s0 + grp; tau < s1; tau += 2, ++tile_i, ++kk) {
      // layer-1 weights of this thread's unit, loaded while the records arrive
      const float w1[3] = {th[3 * u], th[3 * u + 1], th[3 * u + 2]};
      const float b1 = th[3 * H + u];
      // ---- tile records (prefetched during the previous tile)
      {
        const bool ok = mbar_wait_bounded(smem_u32(bar_p), ph_p);
        if (ok) ph_p ^= 1u;
        if (named_sync_or(gbar, 256, !ok || *abort_f != 0)) {
          if (gtid == 0) {
            if (!ok) atomicOr(a.status, 2);
            *abort_f = 1;
          }
          aborted = true;
          break;
        }
        if (gtid == kPrefetchT && tau + 2 < s1) prefetch(tau + 2, (kk + 1) & 1);
      }
      const PRec* pr = pbuf + kHP * (kk & 1);
      // seeds of cut points (from the cut-row kernel): copied into the seed
      // buffer now (asynchronously), used after the forward
      if (gtid < 8 * kHP) {
        const PRec& pc = pr[gtid >> 3];
        if (pc.pt >= 0 && pc.cutj >= 0)
          cp_async4(smem_u32(seeds + pair_col(gtid >> 3, gtid & 7)),
                    a.cut_seed + (int64_t)(pc.cutj >> 1) * 16 + net * 8 + (gtid & 7));
      }

      // ---- layer 1 (3 -> H) in FP32, two points per packed FP32 instruction
      {
        float Td[3];
        bool sd1;
        layer1_increments<FAST>(w1, P.hf, Td, sd1);
#pragma unroll
        for (int pp = 0; pp < kPPT; pp += 2) {
          const PRec pa = pr[4 * cgl + pp], pb = pr[4 * cgl + pp + 1];
          F2 o[8];
          layer1_pair<FAST>(w1, b1, Td, sd1, pa, pb, o);
          store_pair(Aimg, poff(pp), poff(pp + 1), o);
        }
      }
      fence_proxy_async();
      named_sync(gbar, 256);

      // ---- hidden layers on the tensor cores: D[unit][col] = W[unit][k] A[k][col]
      float last[32];
#pragma unroll 1
      for (int g = 1; g <= NG; ++g) {
        // the layer's bias, loaded while the GEMM runs
        const float bb = th[4 * H + (g - 1) * (H * H + H) + H * H + u];
        if (gtid == 0 && gate(0)) {
          const uint32_t ab = smem_u32(Aimg + (g - 1) * kImgH);
          if constexpr (kWTmem) {
            const uint32_t wt = tmem + 384u + 64u * (uint32_t)(g - 1);
#pragma unroll
            for (int k = 0; k < 8; ++k)
              mma_f16_ta(d_tm, wt + 8u * (uint32_t)k, desc_mnmajor(ab) + kstep_mnmajor(k), id_fwd,
                         k > 0);
          } else {
            const uint32_t wa = smem_u32(Wimg + (g - 1) * kImg);
#pragma unroll
            for (int k = 0; k < 8; ++k)
              mma_f16(d_tm, desc_kmajor(wa) + kstep_kmajor(k), desc_mnmajor(ab) + kstep_mnmajor(k),
                      id_fwd, k > 0);
          }
          mma_commit(smem_u32(bar_mma));
        }
        const bool ok_w = wait_mma();
        float acc[32];
        tmem_ld32(d_tm + lane_base + col0, acc);
#pragma unroll
        for (int jp = 0; jp < kPPT; jp += 2) {
          F2 o[8];
          hidden_pair<FAST>(acc + 8 * jp, bb, pr + 4 * cgl + jp, pr + 4 * cgl + jp + 1, o);
          if (g < NG) {
            store_pair(Aimg + g * kImgH, poff(jp), poff(jp + 1), o);
          } else {
#pragma unroll
            for (int c2 = 0; c2 < 8; ++c2) f2get(o[c2], last[8 * jp + 2 * c2], last[8 * jp + 2 * c2 + 1]);
          }
        }
        if (!end_phase(ok_w)) {
          aborted = true;
          break;
        }
      }
      if (aborted) break;

      // ---- output layer (H -> 1) in FP32: sum over the 32 units of the warp,
      // then over the four lane quadrants
      {
        float s;
        warp_transpose_reduce32(last, wo, lane, s);  // lane l: column col0 + l
        red[q * 64 + col0 + lane] = s;
      }
      if (gtid < 8 * kHP) cp_async_wait_all();
      named_sync(gbar, 256);
      // ---- output columns and residual rows: lane c of the 8 lanes
      // gtid = 8 p + c of the group's first two warps takes column c of point
      // p, and the point's row is spread over its 8 lanes
      // (uncut_residual_lanes: one face per lane, sums by shuffles), so the
      // row's dependency chain runs on 8 lanes instead of 1.  FP64 rows only
      // occur in the accurate (!FAST) instances.
      if (gtid < 8 * kHP) {
        const int p = gtid >> 3, c = gtid & 7;
        const unsigned gmask = 0xFFu << (gtid & 24);
        const int pc = pair_col(p, c);
        float oc = red[pc];
#pragma unroll
        for (int qq = 1; qq < 4; ++qq) oc += red[64 * qq + pc];
        if (c == 0 || c == 7) oc += bo;
        const float csc = (c >= 1 && c <= 3) ? P.inv_h2f : (c >= 4 && c <= 6) ? P.inv_hf : 1.f;
        oc *= csc;  // the scaled convention of the rows: U, Mt_i = M_i/h^2, Dt_i = D_i/h
        // U and the Mt, Dt columns of this lane's face axis (c / 2)
        const float Uc = __shfl_sync(gmask, oc, 0, 8);
        const float Mtc = __shfl_sync(gmask, oc, 1 + (c >> 1), 8);
        const float Dtc = __shfl_sync(gmask, oc, 4 + (c >> 1), 8);
        const PRec pi = pr[p];
        const bool valid = pi.pt >= 0, is_cut = pi.cutj >= 0;
        float& sdp = seeds[pc];
        if (valid && !is_cut) {
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
            r2 = uncut_residual_lanes<float>(P, net, pi.x, pi.y, pi.z, pi.gx, Uc, Mtc, Dtc,
                                             a.scale, c, gmask, sdc);
            if (c == 0) loss_acc += r2;
          }
          sdp = sdc * csc;  // seeds in this kernel's column convention
        } else if (valid) {
          sdp *= csc;  // cut point: the seeds copied at the start of the tile, rescaled
        } else {
          sdp = 0.f;
        }
      }
      named_sync(gbar, 256);
      // ---- backward: adjoint of the last tanh layer (FP32 state in registers)
      {
        // two points per packed FP32 instruction
#pragma unroll
        for (int pp = 0; pp < kPPT; pp += 2) {
          F2 sd[8], st[8], gz[8];
          {
            const float4* s4 = reinterpret_cast<const float4*>(seeds + 8 * (4 * cgl + pp));
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float4 v = s4[c];
              sd[2 * c] = f2(v.x, v.y);
              sd[2 * c + 1] = f2(v.z, v.w);
            }
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) st[c] = f2(last[8 * pp + 2 * c], last[8 * pp + 2 * c + 1]);
          F2 sw = mul2(sd[0], st[0]);
#pragma unroll
          for (int c = 1; c < 8; ++c) sw = fma2(sd[c], st[c], sw);
          {
            float x, y;
            f2get(sw, x, y);
            gwo += x;
            gwo += y;
          }
          const F2 WO = f2s(wo);
          const F2 T = st[0];
          const F2 S0 = fma2(mul2(T, f2s(-1.0f)), T, f2s(1.0f));
          F2 gzc = mul2(S0, mul2(WO, sd[0]));
#pragma unroll
          for (int i = 0; i < 3; ++i)
            gzc = add2(gzc, tanh_stencil_bwd_pair(T, S0, st[1 + i], st[4 + i], mul2(WO, sd[1 + i]),
                                                  mul2(WO, sd[4 + i]), gz[1 + i], gz[4 + i]));
          gz[0] = gzc;
          gz[7] = mul2(fma2(mul2(st[7], f2s(-1.0f)), st[7], f2s(1.0f)), mul2(WO, sd[7]));
          {
            float x, y;
            f2get(add2(gz[0], gz[7]), x, y);
            gbh[NG - 1] += x;
            gbh[NG - 1] += y;
          }
          store_pair(Aimg + (L - 1) * kImgH, poff(pp), poff(pp + 1), gz);
        }
      }
      if (gtid == 0) {
        float s = 0.f;
        for (int p = 0; p < kHP; ++p) s += seeds[pair_col(p, 0)] + seeds[pair_col(p, 7)];
        gbo += s;
      }
      fence_proxy_async();
      named_sync(gbar, 256);

      // ---- backward through the hidden GEMMs g = NG .. 1.  Phase n of this
      // group's tile i is n = i NG + (NG - g); group 0 issues it after group 1
      // completed its phase n - NG (tile i-1), group 1 after group 0 completed
      // phase n (tile i): the shared weight-gradient accumulators receive the
      // half-tiles in segment order.
#pragma unroll 1
      for (int g = NG; g >= 1; --g) {
        const int nph = tile_i * NG + (NG - g);
        const int order = grp == 0 ? nph - NG + 1 : nph + 1;
        const uint32_t acc_w = (grp == 0 && tile_i == 0) ? 0u : 1u;
        if (gtid == 0 && gate(order)) {
          const uint32_t wa = smem_u32(Wimg + (g - 1) * kImg);
          const uint32_t gzb = smem_u32(Aimg + g * kImgH);        // gz of act[g]
          const uint32_t ain = smem_u32(Aimg + (g - 1) * kImgH);  // act[g-1]
#pragma unroll
          for (int k = 0; k < 8; ++k)  // input gradient: D = W^T gz
            mma_f16(d_tm, desc_mnmajor(wa) + kstep_mnmajor(k), desc_mnmajor(gzb) + kstep_mnmajor(k),
                    id_dgr, k > 0);
#pragma unroll
          for (int k = 0; k < kHP / 2; ++k)  // weight gradient: Wacc += gz act^T (K = 8 kHP)
            mma_f16(tmem + 128u * g, desc_kmajor(gzb) + kstep_kmajor(k),
                    desc_kmajor(ain) + kstep_kmajor(k), id_wgr,
                    (k > 0 || acc_w) ? 1u : 0u);
          mma_commit(smem_u32(bar_mma));
        }
        const bool ok_w = wait_mma();
        if (gtid == 0 && ok_w) st_release_s32(done_cnt + grp, nph + 1);
        unsigned char* img = Aimg + (g - 1) * kImgH;  // state of act[g-1]
#pragma unroll
        for (int j = 0; j < kPPT; j += 2) {  // two points at a time: registers are short here
          float G[16];
          tmem_ld16(d_tm + lane_base + col0 + 8 * j, G);
          F2 st[8], gz[8];
          load_pair(img, poff(j), poff(j + 1), st);
          const F2 T = st[0];
          const F2 S0 = fma2(mul2(T, f2s(-1.0f)), T, f2s(1.0f));
          F2 gzc = mul2(S0, f2(G[0], G[1]));
#pragma unroll
          for (int i = 0; i < 3; ++i)
            gzc = add2(gzc, tanh_stencil_bwd_pair(T, S0, st[1 + i], st[4 + i],
                                                  f2(G[2 + 2 * i], G[3 + 2 * i]),
                                                  f2(G[8 + 2 * i], G[9 + 2 * i]), gz[1 + i],
                                                  gz[4 + i]));
          gz[0] = gzc;
          gz[7] = mul2(fma2(mul2(st[7], f2s(-1.0f)), st[7], f2s(1.0f)), f2(G[14], G[15]));
          float gsA, gsB;
          f2get(add2(gz[0], gz[7]), gsA, gsB);
          if (g > 1) {
#pragma unroll
            for (int i = 0; i < NG; ++i) {
              gbh[i] += (g - 2 == i) ? gsA : 0.f;
              gbh[i] += (g - 2 == i) ? gsB : 0.f;
            }
            store_pair(img, poff(j), poff(j + 1), gz);
          } else {
            // d del_i / d W1[u][i] = h
            const PRec &pa = pr[4 * cgl + j], &pb = pr[4 * cgl + j + 1];
            const F2 dd = f2s(P.hf);
            float x, y;
            f2get(fma2(gz[0], f2(pa.x, pb.x), fma2(gz[7], f2(pa.gx, pb.gx), mul2(gz[4], dd))), x, y);
            gW1[0] += x;
            gW1[0] += y;
            f2get(fma2(gz[0], f2(pa.y, pb.y), fma2(gz[7], f2(pa.gy, pb.gy), mul2(gz[5], dd))), x, y);
            gW1[1] += x;
            gW1[1] += y;
            f2get(fma2(gz[0], f2(pa.z, pb.z), fma2(gz[7], f2(pa.gz, pb.gz), mul2(gz[6], dd))), x, y);
            gW1[2] += x;
            gW1[2] += y;
            gb1 += gsA;
            gb1 += gsB;
          }
        }
        if (!end_phase(ok_w)) {
          aborted = true;
          break;
        }
      }
      if (aborted) break;
    }
    // ---- end of the segment: both groups are done with this network
    if (__syncthreads_or(aborted)) {
      aborted = true;
      break;
    }
    fence_after_sync();
    flush(net);
  }

  double lsum = (double)loss_acc + loss_acc_d;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0) loss_red[w] = lsum;
  fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int ww = 0; ww < 16; ++ww) s += loss_red[ww];
    a.loss_part[blockIdx.x] = s;
    a.gpart_flag[2 * blockIdx.x] = aborted ? 0 : wrote0;
    a.gpart_flag[2 * blockIdx.x + 1] = aborted ? 0 : wrote1;
  }
  if (aborted) {
    // an MMA or record copy of this group may still be in flight: give it a
    // short bounded wait (about 1 ms) before TMEM and shared memory are released
    (void)mbar_wait_bounded(smem_u32(bar_mma), ph_mma, 2000000LL);
    (void)mbar_wait_bounded(smem_u32(bar_p), ph_p, 2000000LL);
    (void)mbar_wait_bounded(smem_u32(bar_w), ph_w, 2000000LL);
    fence_before_sync();
    __syncthreads();
  }
  fence_after_sync();
  if (w == 0) tmem_dealloc(tmem, NCOLS);
}

// Diagnostics: one warp waits, with the bounded wait every kernel of the
// library uses, on a barrier that nothing completes.  Every thread's wait must
// give up after about `budget` clock cycles; *out = 2 (the status bit of a
// wait that ran out) if all gave up, 0 if the barrier completed.
__global__ void k_selftest_wait(long long budget, int* out) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
  }
  __syncthreads();
  const bool ok = mbar_wait_bounded(smem_u32(&bar), 0, budget);
  const bool any = __syncthreads_or(ok);
  if (threadIdx.x == 0) *out = any ? 0 : 2;
}

cudaError_t launch_selftest_wait(long long budget, int* out, cudaStream_t st) {
  k_selftest_wait<<<1, 32, 0, st>>>(budget, out);
  return cudaGetLastError();
}

template <int L, bool FAST>
static cudaError_t launch_tc_t(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  const size_t smem = tc_smem_bytes(L);
  cudaError_t e = cudaFuncSetAttribute(k_step_tc<L, FAST>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_step_tc<L, FAST>, dim3(grid), dim3(512), smem, st, P, a);
}

cudaError_t launch_step_tc(const ProbDev& P, const StepArgs& a, int grid, int prec, cudaStream_t st) {
  if (P.H != 128 || prec != NBM_PREC_BF16) return cudaErrorInvalidValue;
  if (a.mode != MODE_TRAIN) return launch_fwd_tc(P, a, grid, st);
  // The tanh/reciprocal of the epilogue run on the SFU (tanh.approx, rcp.approx,
  // relative error ~2^-11): every value they produce is rounded to BF16
  // (2^-9) before the next GEMM, so they do not add an error class.  The
  // fine-h mode (FP64 rows) keeps the accurate functions: there the BF16
  // rounding alone already uses most of the gradient tolerance.
  if (P.L == 2) return P.fp64 ? launch_tc_t<2, false>(P, a, grid, st) : launch_tc_t<2, true>(P, a, grid, st);
  if (P.L == 3) return P.fp64 ? launch_tc_t<3, false>(P, a, grid, st) : launch_tc_t<3, true>(P, a, grid, st);
  if (P.L == 4) return P.fp64 ? launch_tc_t<4, false>(P, a, grid, st) : launch_tc_t<4, true>(P, a, grid, st);
  return cudaErrorInvalidValue;
}


}  // namespace nbm
