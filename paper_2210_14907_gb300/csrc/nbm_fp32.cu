// nbm_fp32.cu -- the plain FP32 fused NBM step (arXiv 2210.14907, Sec. 3,
// Fig. 2): hidden-layer GEMMs in FP32 FFMA on the SIMT pipes.
//
// One persistent CTA of 512 threads per SM, tiles of 16 collocation points.
// Each point carries 8 columns through the network: the centre value, the
// symmetric and antisymmetric stencil increments of the three axes
// (difference form, see nbm_device.cuh) and the value at the interface point of
// a cut cell; a tile's layer is one [H x H] x [H x 128] product.  A thread
// computes H/32 units x the 8 columns of one point, so that its column sums
// feed its own tanh stencil layer without an exchange.  A warp takes 4 points
// x 8 unit groups with the lane bits dealt so that neighbouring lanes (x ^ 1,
// x ^ 2) share one of the two operands: a 16-byte shared load then takes two
// wavefronts instead of four (as 8 neighbouring unit groups it took four, and
// the shared pipe was 74 % busy instead of 49 %).
//
// The weights stream through a ring of three 16-row chunks (cp.async, two
// chunks ahead and across the GEMM and tile boundaries), so that every weight
// is read from L2 once per tile of 16 points; with one warp per point, each
// reading all weights through L1, the kernel was bound by that traffic.  Shared
// memory holds the tile's columns of every layer for the backward.  The
// weight gradient of a hidden layer is one [H x 128] x [128 x H] product per
// tile, added to this CTA's slice of the partial-gradient buffer by
// fire-and-forget reductions: each element belongs to one thread, so they
// apply in tile order (no atomics across threads: the final reduction over
// CTAs runs in a fixed order).  (A load, a sum and a store in their place read the slice
// through L2: 200,003 points at 128 x 3 7.93 ms against 7.27.)
//
// Bound: the FFMA pipe (21 H^2 FMA per point and hidden layer; 24 with the
// interface column).  200,003
// points, 3 -> 128 x 3 -> 1: 17.4 -> 7.1 ms per launch (49 % of the 80.5 TFLOP/s
// FFMA peak, pipe 61 % busy; in its GEMM loops 55-62 %, the rest in the chunk
// barriers and the issue of packed-pair operands); 4096 points, 64 x 2: a
// step of 107 -> 82 us.
#include "nbm_device.cuh"
#include "nbm_f32x2.cuh"
#include "nbm_host.h"
#include "nbm_tc_ptx.cuh"

namespace nbm {

namespace {

constexpr int kPT = 16;  // points per tile
constexpr int kNT = 512;
constexpr int kKC = 16;  // contraction rows per weight chunk
constexpr int kStages = 3;

template <int H, int L>
struct Fp32Cfg {
  static constexpr int TU = H / 32;  // units per thread
  // activation slots: act[0..L-2] and the last layer's adjoint.  Three fit at
  // H = 128; four layers then put that adjoint in slot 0 and evaluate the (cheap,
  // K = 3) first layer again for the backward.
  static constexpr int S = H == 128 && L == 4 ? 3 : L;
  static constexpr bool kRecompute = S < L;
  static constexpr int PS = H * 8 + 8;  // floats per point: the pad puts 4 points on distinct banks
  static constexpr int SLOT = kPT * PS;
  static constexpr int kW = S * SLOT;                   // weight ring
  static constexpr int kRed = kW + kStages * kKC * H;   // [4 unit quarters][16][8] output partials
  static constexpr int kSeed = kRed + 4 * kPT * 8;      // [16][8]
  static constexpr int kGwo = kSeed + kPT * 8;          // [4 point groups][H] output weights
  static constexpr int kGb = kGwo + 4 * H;              // [4 point groups][H] biases
  static constexpr int kRec = kGb + 4 * H;              // [2][16] point records
  static constexpr size_t bytes = (size_t)(kRec + 2 * kPT * 8) * sizeof(float);
};

__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// reduction without a return value: the calling thread's additions to one
// address apply in program order.  It takes subnormal operands and results as 0, so
// only values of at least kRedMin go through it: there a subnormal in memory is below
// half a unit of the sum's last place, and a sum of opposite signs is 0 or normal.
constexpr float kRedMin = 0x1p-101f;
__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

// offset of the 4-column half `hf` of unit u of a point (floats): the halves of
// every other group of 4 units are swapped, so that 8 consecutive units' (or 8
// unit groups') same halves lie in distinct banks
__device__ __forceinline__ int col_off(int u, int hf) { return u * 8 + ((hf ^ ((u >> 2) & 1)) << 2); }

__device__ __forceinline__ void ld_cols(const float* pt, int u, float (&v)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(pt + col_off(u, 0));
  const float4 b = *reinterpret_cast<const float4*>(pt + col_off(u, 1));
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st_cols(float* pt, int u, const float (&v)[8]) {
  *reinterpret_cast<float4*>(pt + col_off(u, 0)) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(pt + col_off(u, 1)) = make_float4(v[4], v[5], v[6], v[7]);
}

struct TileRec {  // one point of a tile
  float x, y, z;
  float gx, gy, gz;  // cut cell: interface point.  Uncut point: gx (FP64 rows: gx + gy) = f^s(p)
  int pt;    // -1: padding
  int cutj;  // -1: uncut, else 2 cut_id + has_jump
};
static_assert(sizeof(TileRec) == 32, "eight words");

}  // namespace

template <int H, int L>
__global__ void __launch_bounds__(kNT, 1) k_step_fp32(ProbDev P, StepArgs a) {
  pdl_enter();
  using C = Fp32Cfg<H, L>;
  constexpr int TU = C::TU, PS = C::PS, NCH = H / kKC;
  extern __shared__ __align__(16) float sm[];
  __shared__ double loss_red[kPT];
  __shared__ float gbo_red[kPT];
  float* wbuf = sm + C::kW;
  float* red = sm + C::kRed;
  float* seeds = sm + C::kSeed;
  float* gwos = sm + C::kGwo;
  float* gbs = sm + C::kGb;
  TileRec* recs = reinterpret_cast<TileRec*>(sm + C::kRec);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // a warp takes 4 points x 8 unit groups: lane bits 0 and 3 pick the point, 1, 2
  // and 4 the unit group, so that neighbouring lanes (x ^ 1, x ^ 2) share one of
  // the operands
  const int ugl = ((lane >> 1) & 3) | ((lane >> 4) << 2), ug = (w >> 2) * 8 + ugl;  // of 32
  const int pg = w & 3, pl = 4 * pg + (lane & 1) + ((lane >> 3) & 1) * 2;
  auto unit = [&](int i) { return TU * ug + i; };

  const int nm = a.counters[0], np = a.counters[1], nc = a.counters[2];
  const bool cutfwd = a.mode == MODE_CUT_FWD, train = a.mode == MODE_TRAIN;
  const int T0 = ((cutfwd ? nc : nm) + kPT - 1) / kPT;
  const int T = cutfwd ? 2 * T0 : T0 + (np + kPT - 1) / kPT;
  const int tb = (int)((int64_t)blockIdx.x * T / gridDim.x);
  const int te = (int)((int64_t)(blockIdx.x + 1) * T / gridDim.x);
  const float hf = P.hf, h2f = P.h2f, ihf = P.inv_hf, ih2f = P.inv_h2f;

  // record q of tile tau into buffer b: two or three dependent loads and the
  // source term, so one warp that has no rows does it during the previous tile's
  auto fetch = [&](int tau, int b, int q) {
    const int net = tau < T0 ? 0 : 1, slot = (tau - (net ? T0 : 0)) * kPT + q;
    TileRec r;
    r.x = r.y = r.z = r.gx = r.gy = r.gz = 0.f;
    r.pt = -1;
    r.cutj = -1;
    int cut_id = -1;
    if (cutfwd) {
      if (slot < nc) cut_id = slot;
    } else if (slot < (net ? np : nm)) {
      const int e = a.list[net][slot];
      if (e < 0) cut_id = -e - 1;
      else r.pt = e;
    }
    if (cut_id >= 0) {
      const CutRec& c = a.cut[cut_id];
      r.pt = c.point;
      r.cutj = 2 * cut_id + (c.has_jump ? 1 : 0);
      r.gx = (float)c.xg[0];
      r.gy = (float)c.xg[1];
      r.gz = (float)c.xg[2];
    }
    if (r.pt >= 0) {
      r.x = a.x[r.pt];
      r.y = a.y[r.pt];
      r.z = a.z[r.pt];
      if (cut_id < 0) {
        if (P.fp64) {
          const double f = rhs_f<double>(P, net, r.x, r.y, r.z);
          r.gx = (float)f;
          r.gy = (float)(f - (double)r.gx);
        } else {
          r.gx = rhs_f<float>(P, net, r.x, r.y, r.z);
        }
      }
    }
    recs[b * kPT + q] = r;
  };

  // ---- weight stream: chunk ch (16 rows of H) of a matrix into the ring.  The
  // transposed workspace copy (forward) is 16-byte aligned; the parameter
  // vector (input gradient) only 4-byte aligned.
  int wst = 0, rst = 0;  // ring positions: next chunk to write, to read
  auto wsrc = [&](int net, int g, bool fwd) -> const float* {
    return fwd ? a.wt + ((int64_t)net * (L - 1) + (g - 1)) * H * H
               : a.params + net * P.p_net + 4 * H + (int64_t)(g - 1) * (H * H + H);
  };
  auto issue = [&](const float* src, bool fwd, int ch) {
    if (src) {
      const float* s = src + ch * (kKC * H);
      const uint32_t d = tc::smem_u32(wbuf + wst * (kKC * H));
      if (fwd) {
        if (tid < kKC * H / 4) cp_async16(d + 16u * (uint32_t)tid, s + 4 * tid);
      } else {
#pragma unroll
        for (int i = 0; i < kKC * H / kNT; ++i)
          tc::cp_async4(d + 4u * (uint32_t)(tid + i * kNT), s + tid + i * kNT);
      }
    }
    cp_async_commit();
    wst = wst == kStages - 1 ? 0 : wst + 1;
  };
  // acc[i][.] += sum_k M[k][unit i] x columns of row k of this thread's point;
  // the chunks of (src, fwd) are in flight from chunk 0, and those of the next
  // matrix are requested in the last two steps
  auto gemm = [&](F2 (&acc)[TU][4], const float* pt, const float* src, bool fwd, const float* nsrc,
                  bool nfwd) {
#pragma unroll 1
    for (int ch = 0; ch < NCH; ++ch) {
      cp_async_wait<1>();
      __syncthreads();  // the chunk has landed, and every warp is done with the one before
      if (ch + 2 < NCH) issue(src, fwd, ch + 2);
      else issue(nsrc, nfwd, ch + 2 - NCH);
      const float* wr = wbuf + rst * (kKC * H) + TU * ug;
      const float* ar = pt + ch * (kKC * 8);
      rst = rst == kStages - 1 ? 0 : rst + 1;
#pragma unroll 8
      for (int k = 0; k < kKC; ++k) {
        const float4 c0 = *reinterpret_cast<const float4*>(ar + col_off(k, 0));
        const float4 c1 = *reinterpret_cast<const float4*>(ar + col_off(k, 1));
        const F2 a0 = f2(c0.x, c0.y), a1 = f2(c0.z, c0.w), a2 = f2(c1.x, c1.y), a3 = f2(c1.z, c1.w);
        float wj[TU];
        if constexpr (TU == 4) {
          const float4 wv = *reinterpret_cast<const float4*>(wr + k * H);
          wj[0] = wv.x; wj[1] = wv.y; wj[2] = wv.z; wj[3] = wv.w;
        } else {
          const float2 wv = *reinterpret_cast<const float2*>(wr + k * H);
          wj[0] = wv.x; wj[1] = wv.y;
        }
#pragma unroll
        for (int j = 0; j < TU; ++j) {
          const F2 ww = f2s(wj[j]);
          acc[j][0] = fma2(ww, a0, acc[j][0]);
          acc[j][1] = fma2(ww, a1, acc[j][1]);
          acc[j][2] = fma2(ww, a2, acc[j][2]);
          acc[j][3] = fma2(ww, a3, acc[j][3]);
        }
      }
    }
  };

  // gradient accumulators: thread u < H owns unit u's small parameters
  float gW1[3] = {0.f, 0.f, 0.f}, gb1 = 0.f, gwo = 0.f, gbh[L - 1], gbo = 0.f;
#pragma unroll
  for (int g = 0; g < L - 1; ++g) gbh[g] = 0.f;
  double loss_acc = 0.0;
  int wrote0 = 0, wrote1 = 0;
  bool first_tile = true;

  auto flush = [&](int net) {
    float* gp = a.gpart + ((int64_t)blockIdx.x * 2 + net) * P.gstride;
    const int64_t oo = 4 * H + (int64_t)(L - 1) * (H * H + H);
    if ((tid & 7) == 0 && tid < 8 * kPT) gbo_red[tid >> 3] = gbo;
    __syncthreads();
    if (tid < H) {
      gp[3 * tid] = gW1[0];
      gp[3 * tid + 1] = gW1[1];
      gp[3 * tid + 2] = gW1[2];
      gp[3 * H + tid] = gb1;
#pragma unroll
      for (int g = 0; g < L - 1; ++g) gp[4 * H + (int64_t)g * (H * H + H) + H * H + tid] = gbh[g];
      gp[oo + tid] = gwo;
    }
    if (tid == 0) {
      float s = 0.f;
      for (int q = 0; q < kPT; ++q) s += gbo_red[q];
      gp[oo + H] = s;
    }
    gW1[0] = gW1[1] = gW1[2] = gb1 = gwo = gbo = 0.f;
#pragma unroll
    for (int g = 0; g < L - 1; ++g) gbh[g] = 0.f;
    if (net) wrote1 = 1; else wrote0 = 1;
  };

  if (tb < te) {
    if (tid < kPT) fetch(tb, 0, tid);
    const float* s0 = wsrc(tb < T0 ? 0 : 1, 1, true);
    issue(s0, true, 0);
    issue(s0, true, 1);
  }
#pragma unroll 1
  for (int tau = tb; tau < te; ++tau) {
    const int net = tau < T0 ? 0 : 1, buf = (tau - tb) & 1;
    __syncthreads();  // the tile's records; the previous tile's buffers are free
    const float* nxt = tau + 1 < te ? wsrc(tau + 1 < T0 ? 0 : 1, 1, true) : nullptr;
    const TileRec& rp = recs[buf * kPT + pl];
    const bool jump = rp.cutj >= 0 && (rp.cutj & 1);
    const float jx = jump ? rp.gx : 0.f, jy = jump ? rp.gy : 0.f, jz = jump ? rp.gz : 0.f;
    const float* th = a.params + net * P.p_net;
    const float* wo = th + 4 * H + (int64_t)(L - 1) * (H * H + H);
    float* mypt = sm + pl * PS;  // this thread's point in slot 0

    // ---- layer 1 (3 -> H), FP32, stencil increments exact: mt = 0, dt_i = W1[u][i]
    auto layer1 = [&]() {
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        const int u = unit(i);
        const float w1[3] = {th[3 * u], th[3 * u + 1], th[3 * u + 2]}, bb = th[3 * H + u];
        const float t = act_tanh<false>(fmaf(w1[0], rp.x, fmaf(w1[1], rp.y, fmaf(w1[2], rp.z, bb))));
        float o[8];
        o[0] = t;
        const float md = fmaxf(fabsf(w1[0]), fmaxf(fabsf(w1[1]), fabsf(w1[2]))) * hf;
        const bool sm_de = __all_sync(0xffffffffu, md <= kSmallDelAccurate);
#pragma unroll
        for (int q = 0; q < 3; ++q)
          tanh_stencil_fwd0<false>(t, w1[q], hf, ihf, ih2f, o[1 + q], o[4 + q], sm_de);
        o[7] = jump ? act_tanh<false>(fmaf(w1[0], jx, fmaf(w1[1], jy, fmaf(w1[2], jz, bb))))
                    : 0.f;
        st_cols(mypt, u, o);
      }
    };
    layer1();

    // ---- hidden layers (H -> H), FP32 FFMA
    F2 acc[TU][4];
    float last[TU][8];
#pragma unroll 1
    for (int g = 1; g < L; ++g) {
      const float* bg = th + 4 * H + (int64_t)(g - 1) * (H * H + H) + (int64_t)H * H;
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        const float bb = bg[unit(i)];
        acc[i][0] = f2(bb, 0.f);
        acc[i][1] = acc[i][2] = f2(0.f, 0.f);
        acc[i][3] = f2(0.f, bb);
      }
      const float* nsrc = g < L - 1 ? wsrc(net, g + 1, true) : train ? wsrc(net, L - 1, false) : nxt;
      gemm(acc, mypt + (g - 1) * C::SLOT, wsrc(net, g, true), true, nsrc, g < L - 1 || !train);
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        float z[8], (&o)[8] = last[i];
#pragma unroll
        for (int c = 0; c < 4; ++c) f2get(acc[i][c], z[2 * c], z[2 * c + 1]);
        const float t = act_tanh<false>(z[0]);
        o[0] = t;
        // small increments in every lane: their series (see tanh_stencil_fwd)
        const float mm = fmaxf(fabsf(z[1]), fmaxf(fabsf(z[2]), fabsf(z[3]))) * h2f;
        const float md = fmaxf(fabsf(z[4]), fmaxf(fabsf(z[5]), fabsf(z[6]))) * hf;
        const bool sm_mu = __all_sync(0xffffffffu, mm <= kSmallMuAccurate);
        const bool sm_de = __all_sync(0xffffffffu, md <= kSmallDelAccurate);
#pragma unroll
        for (int q = 0; q < 3; ++q)
          tanh_stencil_fwd<false>(t, z[1 + q], z[4 + q], hf, h2f, ihf, ih2f, o[1 + q], o[4 + q],
                                  sm_mu, sm_de);
        // the interface column only matters to a jump row (its seeds are 0 elsewhere)
        o[7] = jump ? act_tanh<false>(z[7]) : 0.f;
        if (g < L - 1) st_cols(mypt + g * C::SLOT, unit(i), o);
      }
    }

    // ---- output layer (H -> 1): this thread's units, then the 8 unit groups of
    // the warp by recursive halving (lane ugl ends with column ugl)
    float wov[TU];
    {
      float s[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) s[c] = 0.f;
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        wov[i] = wo[unit(i)];
#pragma unroll
        for (int c = 0; c < 8; ++c) s[c] = fmaf(wov[i], last[i][c], s[c]);
      }
#pragma unroll
      for (int m = 4; m > 0; m >>= 1) {
        const bool hi = ugl & m;
        const int x = m == 4 ? 16 : 2 * m;  // the lane bit of unit-group bit m
#pragma unroll
        for (int c = 0; c < m; ++c) {
          const float keep = hi ? s[m + c] : s[c], send = hi ? s[c] : s[m + c];
          s[c] = keep + __shfl_xor_sync(0xffffffffu, send, x);
        }
      }
      red[((w >> 2) * kPT + pl) * 8 + ugl] = s[0];
    }
    __syncthreads();

    // ---- residual rows and seeds: 8 lanes per point (one face per lane)
    if (tid < 8 * kPT) {
      const int q = tid >> 3, c = tid & 7;
      const unsigned gmask = 0xFFu << (tid & 24);
      const TileRec& r = recs[buf * kPT + q];
      float oc = red[q * 8 + c];
#pragma unroll
      for (int uq = 1; uq < 4; ++uq) oc += red[(uq * kPT + q) * 8 + c];
      if (c == 0 || c == 7) oc += wo[H];
      const float Uc = __shfl_sync(gmask, oc, 0, 8);
      const float Mtc = __shfl_sync(gmask, oc, 1 + (c >> 1), 8);
      const float Dtc = __shfl_sync(gmask, oc, 4 + (c >> 1), 8);
      if (cutfwd) {
        if (r.pt >= 0) a.cut_out[(int64_t)(r.cutj >> 1) * 16 + net * 8 + c] = oc;
      } else {
        float sd = 0.f;
        if (r.pt >= 0 && r.cutj < 0) {
          double r2;
          if (P.fp64) {
            r2 = uncut_residual_lanes<double>(P, net, r.x, r.y, r.z, (double)r.gx + (double)r.gy,
                                              Uc, Mtc, Dtc, (double)a.scale, c, gmask, sd);
          } else {
            r2 = uncut_residual_lanes<float, true>(P, net, r.x, r.y, r.z, r.gx, Uc, Mtc, Dtc,
                                                   a.scale, c, gmask, sd);
          }
          if (c == 0) {
            loss_acc += r2;
            if (a.r2_out) a.r2_out[r.pt] = (P.level ? a.r2_out[r.pt] : 0.f) + (float)r2;
          }
        } else if (r.pt >= 0 && train) {
          sd = a.cut_seed[(int64_t)(r.cutj >> 1) * 16 + net * 8 + c];
        }
        seeds[tid] = sd;
        const float sd7 = __shfl_sync(gmask, sd, 7, 8);
        if (c == 0) gbo += sd + sd7;
      }
    } else if (tid >= kNT - 32 && tid < kNT - 32 + kPT && tau + 1 < te) {
      fetch(tau + 1, buf ^ 1, tid - (kNT - 32));
    }
    if (!train) continue;
    __syncthreads();

    // ---- backward: the output layer and the adjoint of the last tanh layer.  The
    // small parameters' sums over the tile's points: the warp's 4 points by
    // shuffles, then thread u adds the 4 point groups' partials
    auto sum4 = [](float v) {
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      return v + __shfl_xor_sync(0xffffffffu, v, 8);
    };
    auto groups = [&](const float* p) {
      return (p[tid] + p[H + tid]) + (p[2 * H + tid] + p[3 * H + tid]);
    };
    {
      float sd[8];
      {
        const float4 lo = *reinterpret_cast<const float4*>(seeds + 8 * pl);
        const float4 hi = *reinterpret_cast<const float4*>(seeds + 8 * pl + 4);
        sd[0] = lo.x; sd[1] = lo.y; sd[2] = lo.z; sd[3] = lo.w;
        sd[4] = hi.x; sd[5] = hi.y; sd[6] = hi.z; sd[7] = hi.w;
      }
      float* dst = mypt + (C::kRecompute ? 0 : L - 1) * C::SLOT;
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        const float(&st)[8] = last[i];
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) s = fmaf(sd[c], st[c], s);
        s = sum4(s);
        if ((lane & 9) == 0) gwos[pg * H + unit(i)] = s;
        const float t = st[0], s0 = fmaf(-t, t, 1.f);
        float gz[8];
        float gzc = s0 * (wov[i] * sd[0]);
#pragma unroll
        for (int q = 0; q < 3; ++q)
          gzc += tanh_stencil_bwd(t, s0, st[1 + q], st[4 + q], wov[i] * sd[1 + q],
                                  wov[i] * sd[4 + q], hf, h2f, ihf, ih2f, gz[1 + q], gz[4 + q]);
        gz[0] = gzc;
        gz[7] = fmaf(-st[7], st[7], 1.f) * (wov[i] * sd[7]);
        const float b = sum4(gz[0] + gz[7]);
        if ((lane & 9) == 0) gbs[pg * H + unit(i)] = b;
        st_cols(dst, unit(i), gz);
      }
    }

    // ---- backward through the hidden layers g = L-1 .. 1
#pragma unroll 1
    for (int g = L - 1; g >= 1; --g) {
      const float* gz = sm + (C::kRecompute && g == L - 1 ? 0 : g) * C::SLOT;
      float* ain = sm + (g - 1) * C::SLOT;
      if (C::kRecompute && g == 1) layer1();  // slot 0 held the last layer's adjoint
      __syncthreads();
      if (tid < H) {
        const float sb = groups(gbs);
#pragma unroll
        for (int i = 0; i < L - 1; ++i) gbh[i] += (g - 1 == i) ? sb : 0.f;
        if (g == L - 1) gwo += groups(gwos);
      }
      // weight gradient: dW[u][k] += sum over the tile's 128 columns of
      // gz[u][col] act[k][col]; units u = ub + 16 i and k = kb + 32 j, 4 ub x 8 kb
      // per warp; the even and the odd columns add up
      // apart (packed pairs) and meet at the end
      {
        const int ub = (w >> 2) * 4 + ((lane >> 1) & 1) + ((lane >> 4) << 1);
        const int kb = (w & 3) * 8 + (lane & 1) + ((lane >> 2) & 3) * 2;
        float* gp = a.gpart + ((int64_t)blockIdx.x * 2 + net) * P.gstride + 4 * H +
                    (int64_t)(g - 1) * (H * H + H) + ub * H + kb;
        constexpr int NU = H / 16, NK = H / 32;
        F2 c[NU][NK];
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
          for (int j = 0; j < NK; ++j) c[i][j] = f2(0.f, 0.f);
        // the four half-columns (swapped halves included) of the point in the loop
        const float* gq = gz + col_off(ub, 0);
        const float* aq = ain + col_off(kb, 0);
        const int gx = col_off(ub, 1) - col_off(ub, 0), ax = col_off(kb, 1) - col_off(kb, 0);
#pragma unroll 1
        for (int q = 0; q < 2 * kPT; ++q) {
          float4 av[NK];
#pragma unroll
          for (int j = 0; j < NK; ++j) av[j] = *reinterpret_cast<const float4*>(aq + 256 * j);
#pragma unroll
          for (int i = 0; i < NU; ++i) {
            const float4 gv = *reinterpret_cast<const float4*>(gq + 128 * i);
#pragma unroll
            for (int j = 0; j < NK; ++j) c[i][j] = fma2(f2(gv.x, gv.y), f2(av[j].x, av[j].y), c[i][j]);
#pragma unroll
            for (int j = 0; j < NK; ++j) c[i][j] = fma2(f2(gv.z, gv.w), f2(av[j].z, av[j].w), c[i][j]);
          }
          gq += q & 1 ? PS - gx : gx;
          aq += q & 1 ? PS - ax : ax;
        }
        bool tiny = false;
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
          for (int j = 0; j < NK; ++j) {
            float ev, od;
            f2get(c[i][j], ev, od);
            const float v = ev + od;
            float* dst = gp + 16 * i * H + 32 * j;
            if (first_tile) *dst = v;
            else if (fabsf(v) >= kRedMin) red_add(dst, v);
            else tiny |= v != 0.f;  // (NaN included)
          }
        if (tiny) {
#pragma unroll
          for (int i = 0; i < NU; ++i)
#pragma unroll
            for (int j = 0; j < NK; ++j) {
              float ev, od;
              f2get(c[i][j], ev, od);
              const float v = ev + od;
              float* dst = gp + 16 * i * H + 32 * j;
              if (!(fabsf(v) >= kRedMin) && v != 0.f) __stcg(dst, __ldcg(dst) + v);
            }
        }
      }
      // input gradient: G[k][c] = sum_u W_g[u][k] gz[u][c]
#pragma unroll
      for (int i = 0; i < TU; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = f2(0.f, 0.f);
      gemm(acc, gz + pl * PS, wsrc(net, g, false), false, g > 1 ? wsrc(net, g - 1, false) : nxt,
           g == 1);
      // adjoint of the tanh layer that produced act[g-1], in place (every
      // weight-gradient read of it came before the GEMM's barriers)
#pragma unroll
      for (int i = 0; i < TU; ++i) {
        float st[8], G[8], gzv[8];
        ld_cols(ain + pl * PS, unit(i), st);
#pragma unroll
        for (int c = 0; c < 4; ++c) f2get(acc[i][c], G[2 * c], G[2 * c + 1]);
        const float t = st[0], s0 = fmaf(-t, t, 1.f);
        float gzc = s0 * G[0];
#pragma unroll
        for (int q = 0; q < 3; ++q)
          gzc += tanh_stencil_bwd(t, s0, st[1 + q], st[4 + q], G[1 + q], G[4 + q], hf, h2f, ihf,
                                  ih2f, gzv[1 + q], gzv[4 + q]);
        gzv[0] = gzc;
        gzv[7] = fmaf(-st[7], st[7], 1.f) * G[7];
        const float sb = sum4(gzv[0] + gzv[7]);
        if (g > 1) {
          if ((lane & 9) == 0) gbs[pg * H + unit(i)] = sb;
          st_cols(ain + pl * PS, unit(i), gzv);
        } else {
          // layer 1: the (3 -> H) gradient; the partials replace the first point's
          // columns, which this lane has read
          const float s0v = sum4(fmaf(gzv[0], rp.x, fmaf(gzv[7], jx, gzv[4])));
          const float s1v = sum4(fmaf(gzv[0], rp.y, fmaf(gzv[7], jy, gzv[5])));
          const float s2v = sum4(fmaf(gzv[0], rp.z, fmaf(gzv[7], jz, gzv[6])));
          if ((lane & 9) == 0)
            *reinterpret_cast<float4*>(mypt + col_off(unit(i), 0)) = make_float4(s0v, s1v, s2v, sb);
        }
      }
    }
    __syncthreads();
    if (tid < H) {
#pragma unroll
      for (int q = 0; q < kPT; q += 4) {
        const float4 v = *reinterpret_cast<const float4*>(sm + q * PS + col_off(tid, 0));
        gW1[0] += v.x;
        gW1[1] += v.y;
        gW1[2] += v.z;
        gb1 += v.w;
      }
    }
    first_tile = false;
    // the last tile of this network: write its partial
    if (tau + 1 == te || (tau + 1 < T0 ? 0 : 1) != net) {
      flush(net);
      first_tile = true;
    }
  }
  cp_async_wait<0>();
  // loss partial of this CTA (fixed order)
  if ((tid & 7) == 0 && tid < 8 * kPT) loss_red[tid >> 3] = loss_acc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int q = 0; q < kPT; ++q) s += loss_red[q];
    if (!cutfwd) a.loss_part[blockIdx.x] = s;
    if (train) {
      a.gpart_flag[2 * blockIdx.x] = wrote0;
      a.gpart_flag[2 * blockIdx.x + 1] = wrote1;
    }
  }
}

template <int H, int L>
static cudaError_t launch_fp32_t(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  constexpr size_t smem = Fp32Cfg<H, L>::bytes;
  cudaError_t e = cudaFuncSetAttribute(k_step_fp32<H, L>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_step_fp32<H, L>, dim3(grid), dim3(kNT), smem, st, P, a);
}

cudaError_t launch_step_fp32(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  if (P.H <= 32) return launch_step_small(P, a, grid, st);  // narrow networks (nbm_small.cu)
#define NBM_FP32_CASE(HH, LL) \
  if (P.H == HH && P.L == LL) return launch_fp32_t<HH, LL>(P, a, grid, st);
  NBM_FP32_CASE(64, 2)
  NBM_FP32_CASE(64, 3)
  NBM_FP32_CASE(64, 4)
  NBM_FP32_CASE(128, 2)
  NBM_FP32_CASE(128, 3)
  NBM_FP32_CASE(128, 4)
#undef NBM_FP32_CASE
  return cudaErrorInvalidValue;
}

}  // namespace nbm
