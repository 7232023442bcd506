// nbm_small.cu -- the FP32 fused NBM step for narrow networks (width <= 32, up
// to five tanh or sine layers): the sine-activated 5 x 10 networks of the
// convergence study (arXiv 2210.14907, Sec. 4.1).
//
// Every point carries 8 difference-form stencil columns (centre value,
// symmetric and antisymmetric increments of the three axes, value at the
// interface point of a cut cell).  A warp takes as many points as its lanes
// hold (32 / H, at most 4; three at H = 10), one lane per point and unit, and
// runs them through forward, rows and backward by itself: each layer's
// pre-activation columns (the sine adjoint needs z, mu, del) and output
// columns are in the warp's own shared memory, and the weight gradient of a
// lane's unit stays in its registers over all of the warp's tiles.  So no
// barrier wider than the warp occurs in a tile, and the warps of an SM fill
// each other's latencies.  With one point per warp (10 of 32 lanes busy),
// block barriers in every layer and the weight gradient summed in global
// memory tile by tile, a step of 16,384 points through 5 x 10 sine networks took
// 222 us in this kernel (the step 270; 72 and 116 now); the
// bound now is the warps' dependency chains.
// At the end of a network the lanes' sums are added over the warps in a fixed
// order (deterministic).
#include <climits>

#include "nbm_device.cuh"
#include "nbm_f32x2.cuh"
#include "nbm_host.h"

namespace nbm {

namespace {

constexpr int kLM = 5;     // maximum number of activation layers
constexpr int kMaxPt = 4;  // points per warp (8 lanes each for the rows)

template <int ACT>
__device__ __forceinline__ float act_f(float z) {
  if constexpr (ACT == NBM_ACT_SIN) return sincos_full(z).x;
  else return act_tanh<false>(z);
}

// whether the stencil increments of every lane allow their series
template <int ACT>
__device__ __forceinline__ void small_increments(const float zc[8], float h, float h2, bool& sm_mu,
                                                 bool& sm_de) {
  const float mm = fmaxf(fabsf(zc[1]), fmaxf(fabsf(zc[2]), fabsf(zc[3]))) * h2;
  const float md = fmaxf(fabsf(zc[4]), fmaxf(fabsf(zc[5]), fabsf(zc[6]))) * h;
  if constexpr (ACT == NBM_ACT_SIN) {
    sm_mu = sm_de = __all_sync(0xffffffffu, 0.5f * fmaxf(mm, md) <= kSmallHalf);
  } else {
    sm_mu = __all_sync(0xffffffffu, mm <= kSmallMuAccurate);
    sm_de = __all_sync(0xffffffffu, md <= kSmallDelAccurate);
  }
}

// outputs of one unit's activation layer from its pre-activation columns
// zc[8] (scaled convention); o[8] receives the output columns
template <int ACT>
__device__ __forceinline__ void layer_fwd(const float zc[8], bool jump, float h, float h2,
                                          float ih, float ih2, float o[8]) {
  bool sm_mu, sm_de;
  small_increments<ACT>(zc, h, h2, sm_mu, sm_de);
  if constexpr (ACT == NBM_ACT_SIN) {
    const float2 sc = sincos_full(zc[0]);
    const float sz = sc.x, cz = sc.y;
    o[0] = sz;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      sin_stencil_fwd(sz, cz, zc[1 + i], zc[4 + i], h, h2, ih, ih2, o[1 + i], o[4 + i], sm_mu);
  } else {
    const float t = act_tanh<false>(zc[0]);
    o[0] = t;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      tanh_stencil_fwd<false>(t, zc[1 + i], zc[4 + i], h, h2, ih, ih2, o[1 + i], o[4 + i], sm_mu,
                              sm_de);
  }
  o[7] = jump ? act_f<ACT>(zc[7]) : 0.f;
}

// adjoint of one unit's activation layer: upstream gradients G[8] with respect
// to the output columns, gz[8] receives the gradients with respect to the
// pre-activation columns
template <int ACT>
__device__ __forceinline__ void layer_bwd(const float zc[8], const float oc[8], const float G[8],
                                          bool jump, float h, float h2, float ih, float ih2,
                                          float gz[8]) {
  if constexpr (ACT == NBM_ACT_SIN) {
    bool small, unused;
    small_increments<ACT>(zc, h, h2, small, unused);
    const float2 sc = sincos_full(zc[0]);
    const float sz = sc.x, cz = sc.y;
    float gzc = cz * G[0];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      gzc += sin_stencil_bwd(sz, cz, zc[1 + i], zc[4 + i], G[1 + i], G[4 + i], h, h2, ih, ih2,
                             gz[1 + i], gz[4 + i], small);
    gz[0] = gzc;
    gz[7] = jump ? sincos_full(zc[7]).y * G[7] : 0.f;
  } else {
    const float t = oc[0], s0 = fmaf(-t, t, 1.f);
    float gzc = s0 * G[0];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      gzc += tanh_stencil_bwd(t, s0, oc[1 + i], oc[4 + i], G[1 + i], G[4 + i], h, h2, ih, ih2,
                              gz[1 + i], gz[4 + i]);
    gz[0] = gzc;
    gz[7] = fmaf(-oc[7], oc[7], 1.f) * G[7];
  }
}

// 8 columns of lane `ln`: the two 16-byte halves swapped for every other group of
// 4 lanes, so that 8 neighbouring lanes' same halves lie in distinct banks
__device__ __forceinline__ int half_off(int ln, int hf) { return ln * 8 + ((hf ^ ((ln >> 2) & 1)) << 2); }
__device__ __forceinline__ void ld8(const float* p, int ln, float v[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p + half_off(ln, 0));
  const float4 b = *reinterpret_cast<const float4*>(p + half_off(ln, 1));
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st8(float* p, int ln, const float v[8]) {
  *reinterpret_cast<float4*>(p + half_off(ln, 0)) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + half_off(ln, 1)) = make_float4(v[4], v[5], v[6], v[7]);
}

struct SmallRec {  // one point of a warp's tile
  float x, y, z;
  float gx, gy, gz;  // cut cell: interface point
  int pt;            // -1: padding
  int cutj;          // -1: uncut, else 2 cut_id + has_jump
};
static_assert(sizeof(SmallRec) == 32, "eight words");

// Threads of a CTA: at H <= 16 a lane holds at most 4 x 16 weight-gradient sums,
// and 16 warps fit the register file; at H <= 32 twice as many, and 8 do.
constexpr int small_threads(int HM) { return HM <= 16 ? 512 : 256; }
// floats of a warp's shared memory: columns, seeds, two sets of records
constexpr int small_warp_floats(int L) { return 2 * L * 256 + kMaxPt * 8 + 2 * kMaxPt * 8; }
size_t small_smem_bytes(int H, int L, int HM) {
  return ((size_t)(small_threads(HM) / 32) * small_warp_floats(L) + 2 * (size_t)(L - 1) * H * H) *
         sizeof(float);
}

}  // namespace

template <int ACT, int HM>
__global__ void __launch_bounds__(small_threads(HM), 1) k_step_small(ProbDev P, StepArgs a) {
  pdl_enter();
  constexpr int NT = small_threads(HM), NW = NT / 32;
  extern __shared__ __align__(16) float sbuf[];
  __shared__ double loss_red[NW];
  __shared__ float gbo_red[NW];
  const int H = P.H, L = P.L;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
  const int ppw = 32 / H < kMaxPt ? 32 / H : kMaxPt;  // points per warp
  const bool own = lane < ppw * H;                    // lane pq H + u: unit u of point pq
  const int pq = own ? lane / H : 0, u = own ? lane - pq * H : 0, pbase = pq * H;
  // A lane without a unit repeats lane 0's (it stores nothing): it reads that lane's
  // columns and not its own, which nothing wrote, since its vote on the series
  // (small_increments) counts like the others'.
  const int ln = pbase + u;
  float* wsm = sbuf + w * small_warp_floats(L);
  float* Zb = wsm;                    // [L][32][8] pre-activations, then their gradients
  float* Ab = wsm + L * 256;          // [L][32][8] outputs
  float* seeds_s = wsm + 2 * L * 256;  // [4][8]
  SmallRec* recs = reinterpret_cast<SmallRec*>(seeds_s + kMaxPt * 8);  // [2][4]
  float* Wf = sbuf + NW * small_warp_floats(L);  // [L-1][k][u] hidden weights, transposed
  float* Wb = Wf + (L - 1) * H * H;              // [L-1][u][k]

  const int nm = a.counters[0], np = a.counters[1], nc = a.counters[2];
  const bool cutfwd = a.mode == MODE_CUT_FWD, train = a.mode == MODE_TRAIN;
  const int64_t T0 = ((cutfwd ? nc : nm) + ppw - 1) / ppw;
  const int64_t T = cutfwd ? 2 * T0 : T0 + (np + ppw - 1) / ppw;
  // The CTAs are dealt to the networks (the one with fewer tiles gets its share rounded
  // up), so that none does two networks' weights, tiles and sums one after the other:
  // a step of 2,293 points 89 -> 74 us, of 16,384 132 -> 123.
  const int64_t ng = gridDim.x, T1 = T - T0, Ts = T0 < T1 ? T0 : T1;
  const int64_t gs = Ts > 0 && ng > 1 ? (ng * Ts + T - 1) / T : 0;  // CTAs of that one
  const int64_t g0 = gs == 0 ? ng : T0 < T1 ? gs : ng - gs;         // CTAs of the first
  const bool first = blockIdx.x < g0;
  const int64_t base = first || gs == 0 ? 0 : T0, span = gs == 0 ? T : first ? T0 : T1;
  const int64_t bi = first ? blockIdx.x : blockIdx.x - g0, bn = first ? g0 : ng - g0;
  const int64_t tb = base + bi * span / bn, te = base + (bi + 1) * span / bn;
  const float hf = P.hf, h2f = P.h2f, ihf = P.inv_hf, ih2f = P.inv_h2f;

  // gradient sums of this lane's unit (its point slot's share of the current net)
  float gW1[3] = {0.f, 0.f, 0.f}, gb1 = 0.f, gwo = 0.f, gbo = 0.f;
  float gbh[kLM - 1], gW[kLM - 1][HM];
#pragma unroll
  for (int g = 0; g < kLM - 1; ++g) {
    gbh[g] = 0.f;
#pragma unroll
    for (int k = 0; k < HM; ++k) gW[g][k] = 0.f;
  }
  double loss_acc = 0.0;
  int wrote0 = 0, wrote1 = 0;

  // this CTA's partial of net `net`: the lanes' sums staged in each warp's column
  // memory, added over the `used` warps that had tiles and their point slots in a
  // fixed order.  At H <= 16 the sums of all layers fit at once (32 (H + 1) (L - 1) +
  // 160 floats of 512 L + 96), else layer by layer.  Layer by layer and over all 16
  // warps, a step of 2,293 points took 116 us (89 so), of 16,384 145 (132 so).
  auto flush = [&](int net, int used) {
    float* gp = a.gpart + ((int64_t)blockIdx.x * 2 + net) * P.gstride;
    const int wf = small_warp_floats(L), hh = H * H;
    const int64_t oo = 4 * H + (int64_t)(L - 1) * (hh + H);
    constexpr bool kAll = HM <= 16;
    const int hid = kAll ? (L - 1) * (hh + H) : 0, per = hid + 5 * H;  // last staging, per point slot
    // sum over the warps and their point slots (stride `st` floats) of staged element i:
    // a warp's slots first, then the warps in four chains.  (One chain over all 48 at H = 10
    // rounds more: the gradient of 16,384 points 7.3e-8 off against 5.3e-8, and 0.7 us longer.)
    auto warps = [&](int i, int st) {
      float t[4] = {0.f, 0.f, 0.f, 0.f};
      for (int ww = 0; ww < used; ww += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (ww + k < used) {
            const float* e = sbuf + (ww + k) * wf + i;
            float s = e[0];
            for (int q = 1; q < ppw; ++q) s += e[q * st];
            t[k] += s;
          }
      return (t[0] + t[1]) + (t[2] + t[3]);
    };
    float go = gbo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) go += __shfl_xor_sync(0xffffffffu, go, o);
    if (lane == 0) gbo_red[w] = go;
#pragma unroll
    for (int g = 0; g < kLM - 1; ++g) {
      if (g >= L - 1) break;
      // (a warp's staging memory is its own: with all layers at once nobody waits here, and
      // warps without tiles have fetched this code when the others come to it: a step of
      // 600 points 73.8 -> 73.2 us)
      if (!kAll) __syncthreads();
      else if (g == 0) __syncwarp();
      if (own) {
        float* st = kAll ? wsm + pq * per + g * (hh + H) : wsm + pq * (hh + H);
#pragma unroll
        for (int k = 0; k < HM; ++k)
          if (k < H) st[u * H + k] = gW[g][k];
        st[hh + u] = gbh[g];
      }
      if constexpr (!kAll) {
        __syncthreads();
        for (int i = tid; i < hh + H; i += NT) {
          gp[4 * H + (int64_t)g * (hh + H) + i] = warps(i, hh + H);  // weights, then biases
        }
      }
    }
    if constexpr (!kAll) __syncthreads();
    if (own) {
      float* st = wsm + pq * per + hid;
      st[3 * u] = gW1[0];
      st[3 * u + 1] = gW1[1];
      st[3 * u + 2] = gW1[2];
      st[3 * H + u] = gb1;
      st[4 * H + u] = gwo;
    }
    __syncthreads();
    for (int i = tid; i < per; i += NT) {
      const float s = warps(i, per);
      const int r = i - hid;  // hidden layers' weights and biases, then layer 1 and the output
      gp[r < 0 ? 4 * H + i : r < 4 * H ? r : oo + r - 4 * H] = s;
    }
    if (tid == NT - 1) {
      float s = 0.f;
      for (int ww = 0; ww < used; ++ww) s += gbo_red[ww];
      gp[oo + H] = s;
    }
    gW1[0] = gW1[1] = gW1[2] = gb1 = gwo = gbo = 0.f;
#pragma unroll
    for (int g = 0; g < kLM - 1; ++g) {
      gbh[g] = 0.f;
#pragma unroll
      for (int k = 0; k < HM; ++k) gW[g][k] = 0.f;
    }
    if (net) wrote1 = 1; else wrote0 = 1;
    __syncthreads();
  };

#pragma unroll 1
  for (int net = 0; net < 2; ++net) {
    const int64_t s0 = net == 0 ? tb : (tb > T0 ? tb : T0);
    const int64_t s1 = net == 0 ? (te < T0 ? te : T0) : te;
    if (s0 >= s1) continue;  // the same in every thread
    const float* th = a.params + net * P.p_net;
    const float* wo = th + 4 * H + (int64_t)(L - 1) * (H * H + H);
    for (int i = tid; i < (L - 1) * H * H; i += NT) {
      const int g = i / (H * H), r = i - g * H * H;
      const float v = th[4 * H + (int64_t)g * (H * H + H) + r];
      Wb[i] = v;
      Wf[g * H * H + (r % H) * H + r / H] = v;
    }
    // record of point q < ppw of tile tau: the list entry, then what it points to
    auto entry = [&](int64_t tau) -> int {
      const int64_t slot = (tau - (net ? T0 : 0)) * ppw + lane;
      if (tau >= s1 || lane >= ppw) return INT_MIN;  // no point
      if (cutfwd) return slot < nc ? -(int)slot - 1 : INT_MIN;
      return slot < (net ? np : nm) ? a.list[net][slot] : INT_MIN;
    };
    auto fill = [&](int e, int b) {
      if (lane >= ppw) return;
      SmallRec r;
      r.x = r.y = r.z = r.gx = r.gy = r.gz = 0.f;
      r.pt = -1;
      r.cutj = -1;
      if (e != INT_MIN) {
        r.pt = e;
        if (e < 0) {
          const CutRec& c = a.cut[-e - 1];
          r.pt = c.point;
          r.cutj = 2 * (-e - 1) + (c.has_jump ? 1 : 0);
          r.gx = (float)c.xg[0];
          r.gy = (float)c.xg[1];
          r.gz = (float)c.xg[2];
        }
        r.x = a.x[r.pt];
        r.y = a.y[r.pt];
        r.z = a.z[r.pt];
      }
      recs[b * kMaxPt + lane] = r;
    };
    if (s0 + w < s1) fill(entry(s0 + w), 0);
    __syncthreads();  // the weights

    int buf = 0;
#pragma unroll 1
    for (int64_t tau = s0 + w; tau < s1; tau += NW, buf ^= 1) {
      __syncwarp();
      const int e_next = entry(tau + NW);  // loaded while this tile computes
      const SmallRec& r = recs[buf * kMaxPt + pq];
      const bool jump = r.cutj >= 0 && (r.cutj & 1);

      // ---- layer 1 (3 -> H): exact increments mu = 0, del_i = h W1[u][i]
      {
        const float w0 = th[3 * u], w1 = th[3 * u + 1], w2 = th[3 * u + 2], bb = th[3 * H + u];
        const float zc[8] = {fmaf(w0, r.x, fmaf(w1, r.y, fmaf(w2, r.z, bb))), 0.f, 0.f, 0.f, w0, w1,
                             w2, jump ? fmaf(w0, r.gx, fmaf(w1, r.gy, fmaf(w2, r.gz, bb))) : 0.f};
        float o[8];
        layer_fwd<ACT>(zc, jump, hf, h2f, ihf, ih2f, o);
        if (own) {
          if constexpr (ACT == NBM_ACT_SIN) st8(Zb, lane, zc);
          st8(Ab, lane, o);
        }
      }
      __syncwarp();

      // ---- hidden layers (H -> H), FP32 FFMA.  (Five terms at a time: with two, the
      // shared-memory latency of every pair showed: 2 x 16,384 points 294 -> 290 us, a
      // residual of 877 points on three spacings 214 -> 211.)
#pragma unroll 1
      for (int g = 1; g < L; ++g) {
        const float* Wg = Wf + (g - 1) * H * H + u;
        const float* ap = Ab + (g - 1) * 256;
        const float bb = th[4 * H + (int64_t)(g - 1) * (H * H + H) + H * H + u];
        F2 acc[4] = {f2(bb, 0.f), f2(0.f, 0.f), f2(0.f, 0.f), f2(0.f, bb)};
#pragma unroll 5
        for (int k = 0; k < H; ++k) {
          float av[8];
          ld8(ap, pbase + k, av);
          const F2 wv = f2s(Wg[k * H]);
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[c] = fma2(wv, f2(av[2 * c], av[2 * c + 1]), acc[c]);
        }
        float zc[8], o[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) f2get(acc[c], zc[2 * c], zc[2 * c + 1]);
        layer_fwd<ACT>(zc, jump, hf, h2f, ihf, ih2f, o);
        if (own) {
          if constexpr (ACT == NBM_ACT_SIN) st8(Zb + g * 256, lane, zc);
          st8(Ab + g * 256, lane, o);
        }
        __syncwarp();
      }

      // ---- output layer and residual rows: 8 lanes per point, lane 8 q + c sums
      // column c of point q and takes one face of its row
      {
        const int q = lane >> 3, c = lane & 7;
        const unsigned gmask = 0xFFu << (lane & 24);
        if (q < ppw) {
          const SmallRec& rq = recs[buf * kMaxPt + q];
          const float* ap = Ab + (L - 1) * 256;
          float oc = (c == 0 || c == 7) ? wo[H] : 0.f;
#pragma unroll 5
          for (int k = 0; k < H; ++k)
            oc = fmaf(wo[k], ap[half_off(q * H + k, c >> 2) + (c & 3)], oc);
          const float Uc = __shfl_sync(gmask, oc, 0, 8);
          const float Mtc = __shfl_sync(gmask, oc, 1 + (c >> 1), 8);
          const float Dtc = __shfl_sync(gmask, oc, 4 + (c >> 1), 8);
          float sd = 0.f;
          if (cutfwd) {
            if (rq.pt >= 0) a.cut_out[(int64_t)(rq.cutj >> 1) * 16 + net * 8 + c] = oc;
          } else if (rq.pt >= 0 && rq.cutj < 0) {
            double r2;
            if (P.fp64) {
              const double f = c == 6 ? rhs_f<double>(P, net, rq.x, rq.y, rq.z) : 0.0;
              r2 = uncut_residual_lanes<double>(P, net, rq.x, rq.y, rq.z, f, Uc, Mtc, Dtc,
                                                (double)a.scale, c, gmask, sd);
            } else {
              const float f = c == 6 ? rhs_f<float>(P, net, rq.x, rq.y, rq.z) : 0.f;
              r2 = uncut_residual_lanes<float, true>(P, net, rq.x, rq.y, rq.z, f, Uc, Mtc, Dtc,
                                                     a.scale, c, gmask, sd);
            }
            if (c == 0) {
              loss_acc += r2;
              if (a.r2_out) a.r2_out[rq.pt] = (P.level ? a.r2_out[rq.pt] : 0.f) + (float)r2;
            }
          } else if (rq.pt >= 0 && train) {
            sd = a.cut_seed[(int64_t)(rq.cutj >> 1) * 16 + net * 8 + c];
          }
          seeds_s[lane] = sd;
          if (c == 0 || c == 7) gbo += sd;
        }
      }
      fill(e_next, buf ^ 1);
      if (!train) continue;
      __syncwarp();

      // ---- backward: output layer
      float G[8];
      {
        const float4 lo = *reinterpret_cast<const float4*>(seeds_s + 8 * pq);
        const float4 hi = *reinterpret_cast<const float4*>(seeds_s + 8 * pq + 4);
        const float sd[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        float oc[8];
        ld8(Ab + (L - 1) * 256, ln, oc);
        const float wv = wo[u];
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          s = fmaf(sd[c], oc[c], s);
          G[c] = wv * sd[c];
        }
        gwo += s;
      }

      // ---- backward through the hidden layers g = L-1 .. 1: the adjoint of the
      // activation layer, then the weight gradient dW[u][k] += gz[u] . act[k] of
      // this lane's unit and point, and G[u] = sum_k W[k][u] gz[k].  (Not unrolled:
      // the layer's sums are picked by a predicate, four copies of this body
      // would not fit the instruction cache.)
#pragma unroll 1
      for (int g = L - 1; g >= 1; --g) {
        float zc[8], oc[8], gzv[8];
        if constexpr (ACT == NBM_ACT_SIN) ld8(Zb + g * 256, ln, zc);
        ld8(Ab + g * 256, ln, oc);
        layer_bwd<ACT>(zc, oc, G, jump, hf, h2f, ihf, ih2f, gzv);
#pragma unroll
        for (int i = 0; i < kLM - 1; ++i) gbh[i] += (g - 1 == i) ? gzv[0] + gzv[7] : 0.f;
        if (own) st8(Zb + g * 256, lane, gzv);
        __syncwarp();
        const float* ap = Ab + (g - 1) * 256;
        const float* zp = Zb + g * 256;
        const float* Wg = Wb + (g - 1) * H * H + u;
        F2 gg[4], acc[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          gg[c] = f2(gzv[2 * c], gzv[2 * c + 1]);
          acc[c] = f2(0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < HM; ++k) {
          if (k < H) {
            float av[8], gv[8];
            ld8(ap, pbase + k, av);
            ld8(zp, pbase + k, gv);
            F2 d = mul2(gg[0], f2(av[0], av[1]));
#pragma unroll
            for (int c = 1; c < 4; ++c) d = fma2(gg[c], f2(av[2 * c], av[2 * c + 1]), d);
            float ev, od;
            f2get(d, ev, od);
            const float dw = ev + od;
#pragma unroll
            for (int i = 0; i < kLM - 1; ++i)
              if (g - 1 == i) gW[i][k] += dw;
            const F2 wv = f2s(Wg[k * H]);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] = fma2(wv, f2(gv[2 * c], gv[2 * c + 1]), acc[c]);
          }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) f2get(acc[c], G[2 * c], G[2 * c + 1]);
      }

      // ---- adjoint of layer 1 and its (3 -> H) parameter gradient; the
      // increments del_i = h W1[u][i] give d(dt_i)/dW1[u][i] = 1 (scaled columns)
      {
        float zc[8], oc[8], gzv[8];
        if constexpr (ACT == NBM_ACT_SIN) ld8(Zb, ln, zc);
        ld8(Ab, ln, oc);
        layer_bwd<ACT>(zc, oc, G, jump, hf, h2f, ihf, ih2f, gzv);
        gW1[0] += fmaf(gzv[0], r.x, fmaf(gzv[7], r.gx, gzv[4]));
        gW1[1] += fmaf(gzv[0], r.y, fmaf(gzv[7], r.gy, gzv[5]));
        gW1[2] += fmaf(gzv[0], r.z, fmaf(gzv[7], r.gz, gzv[6]));
        gb1 += gzv[0] + gzv[7];
      }
    }
    if (train) flush(net, (int)(s1 - s0 < NW ? s1 - s0 : NW));
    else __syncthreads();  // before the next network's weights
  }
  // loss partial of this CTA (fixed order)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
  if (lane == 0) loss_red[w] = loss_acc;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int ww = 0; ww < NW; ++ww) s += loss_red[ww];
    if (!cutfwd) a.loss_part[blockIdx.x] = s;
    if (train) {
      a.gpart_flag[2 * blockIdx.x] = wrote0;
      a.gpart_flag[2 * blockIdx.x + 1] = wrote1;
    }
  }
}

template <int ACT, int HM>
static cudaError_t launch_small_t(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  const size_t smem = small_smem_bytes(P.H, P.L, HM);
  cudaError_t e = cudaFuncSetAttribute(k_step_small<ACT, HM>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_step_small<ACT, HM>, dim3(grid), dim3(small_threads(HM)), smem, st, P, a);
}

cudaError_t launch_step_small(const ProbDev& P, const StepArgs& a, int grid, cudaStream_t st) {
  if (P.H < 1 || P.H > 32 || P.L < 2 || P.L > kLM) return cudaErrorInvalidValue;
  const bool sine = P.activation == NBM_ACT_SIN;
  if (P.H <= 16) return sine ? launch_small_t<NBM_ACT_SIN, 16>(P, a, grid, st)
                             : launch_small_t<NBM_ACT_TANH, 16>(P, a, grid, st);
  return sine ? launch_small_t<NBM_ACT_SIN, 32>(P, a, grid, st)
              : launch_small_t<NBM_ACT_TANH, 32>(P, a, grid, st);
}

}  // namespace nbm
