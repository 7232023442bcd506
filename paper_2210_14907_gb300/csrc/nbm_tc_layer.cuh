// nbm_tc_layer.cuh -- the pieces that the tensor-core step kernels share: 16-bit
// operand images, the output layer's warp reduction, and the forward tanh stencil
// layers of two points on packed FP32 pairs (unscaled difference columns).
#pragma once

#include <cuda_bf16.h>

#include "nbm_device.cuh"
#include "nbm_f32x2.cuh"
#include "nbm_tc_ptx.cuh"

namespace nbm {

constexpr int kHP = 8;        // points per half-tile (one warp group)
constexpr int kImg = 32768;   // 128 x 128 16-bit weight image
constexpr int kImgH = 16384;  // 128 x 64 16-bit operand image of a half-tile

// Column order of an operand image.  The 16 columns of two neighbouring points A, B
// are interleaved: column 16 P + 2 c + s is column c of point 2 P + s.  A thread's
// accumulator registers 2 c and 2 c + 1 are then the pair (A, B) that the packed FP32
// instructions take, and a 32-bit word of the image holds the same pair in BF16, so
// neither needs moves to be put together or taken apart.
__device__ __forceinline__ int pair_col(int p, int c) { return (p >> 1) * 16 + 2 * c + (p & 1); }

__device__ __forceinline__ uint32_t pack_bf2(F2 v) {
  float a, b;
  f2get(v, a, b);
  const __nv_bfloat162 w = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&w);
}
__device__ __forceinline__ F2 unpack_bf2(uint32_t u) {
  return f2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
// the pair's 16 columns: 16-byte chunks at off0 (c = 0..3) and off1 (c = 4..7)
__device__ __forceinline__ void store_pair(unsigned char* img, uint32_t off0, uint32_t off1,
                                           const F2 (&o)[8]) {
  *reinterpret_cast<uint4*>(img + off0) =
      make_uint4(pack_bf2(o[0]), pack_bf2(o[1]), pack_bf2(o[2]), pack_bf2(o[3]));
  *reinterpret_cast<uint4*>(img + off1) =
      make_uint4(pack_bf2(o[4]), pack_bf2(o[5]), pack_bf2(o[6]), pack_bf2(o[7]));
}
__device__ __forceinline__ void load_pair(const unsigned char* img, uint32_t off0, uint32_t off1,
                                          F2 (&o)[8]) {
  const uint4 a = *reinterpret_cast<const uint4*>(img + off0);
  const uint4 b = *reinterpret_cast<const uint4*>(img + off1);
  o[0] = unpack_bf2(a.x); o[1] = unpack_bf2(a.y); o[2] = unpack_bf2(a.z); o[3] = unpack_bf2(a.w);
  o[4] = unpack_bf2(b.x); o[5] = unpack_bf2(b.y); o[6] = unpack_bf2(b.z); o[7] = unpack_bf2(b.w);
}

// Sum of wo * x[0..31] over the 32 lanes of the warp: on return lane l holds
// the sum of column l (recursive halving, one exchange per value; the scaling
// is folded into the first halving so that x stays intact for the backward).
__device__ __forceinline__ void warp_transpose_reduce32(const float (&x)[32], float wo, int lane,
                                                        float& s) {
  float v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const bool hi = lane & 16;
    const float keep = wo * (hi ? x[16 + i] : x[i]), send = wo * (hi ? x[i] : x[16 + i]);
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool hi = lane & 8;
    const float keep = hi ? v[8 + i] : v[i], send = hi ? v[i] : v[8 + i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool hi = lane & 4;
    const float keep = hi ? v[4 + i] : v[i], send = hi ? v[i] : v[4 + i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool hi = lane & 2;
    const float keep = hi ? v[2 + i] : v[i], send = hi ? v[i] : v[2 + i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  {
    const bool hi = lane & 1;
    const float keep = hi ? v[1] : v[0], send = hi ? v[0] : v[1];
    s = keep + __shfl_xor_sync(0xffffffffu, send, 1);
  }
}

// Two points' tanh stencil layer on packed FP32 pairs (unscaled columns, every
// lane's symmetric increments small): the arithmetic of tanh_stencil_fwd's
// series path.
template <bool FAST>
__device__ __forceinline__ void tanh_stencil_fwd_pair(F2 T, F2 NT, F2 S0, F2 MU, F2 DE, F2& M,
                                                      F2& D, bool small_de = false) {
  const bool sde = !FAST && small_de;  // the series of tanh d and 1/(1-x) (accurate path)
  F2 TD;
  if (sde) {
    const F2 d2 = mul2(DE, DE);
    TD = mul2(DE, fma2(d2, fma2(d2, f2s(2.0f / 15.0f), f2s(-1.0f / 3.0f)), f2s(1.0f)));
  } else {
    float dA, dB;
    f2get(DE, dA, dB);
    TD = f2(act_tanh<FAST>(dA), act_tanh<FAST>(dB));
  }
  const F2 poly = fma2(fma2(T, T, f2s(-1.0f / 3.0f)), mul2(MU, MU), fma2(NT, MU, f2s(1.0f)));
  const F2 dm = mul2(mul2(S0, MU), poly);
  const F2 tw = add2(T, dm);
  const F2 ntw = mul2(tw, f2s(-1.0f));
  const F2 sw = fma2(ntw, tw, f2s(1.0f));
  const F2 td2 = mul2(TD, TD);
  const F2 ntd = mul2(ntw, td2);
  F2 r2;
  if (sde) {
    const F2 x = mul2(mul2(tw, tw), td2);  // 1/(1-x) = 1 + x (1 + x (1 + x))
    r2 = fma2(x, fma2(x, add2(x, f2s(1.0f)), f2s(1.0f)), f2s(1.0f));
  } else {
    float eA, eB;
    f2get(fma2(ntd, tw, f2s(1.0f)), eA, eB);  // 1 - tw^2 Td^2
    r2 = f2(rcp<FAST>(eA), rcp<FAST>(eB));
  }
  const F2 k = mul2(sw, r2);
  M = fma2(ntd, k, dm);
  D = mul2(k, TD);
}

// Layer 1 (3 -> H) of two points in one unit: exact increments mu = 0, del_i = h
// W1[u][i]; Td[i] = tanh(del_i), sd1: the series of 1/(1-x) (accurate path).
template <bool FAST>
__device__ __forceinline__ void layer1_pair(const float (&w1)[3], float b1, const float (&Td)[3],
                                            bool sd1, const PRec& pa, const PRec& pb,
                                            F2 (&o)[8]) {
  const F2 W0 = f2s(w1[0]), W1 = f2s(w1[1]), W2 = f2s(w1[2]), B1 = f2s(b1);
  float zA, zB;
  f2get(fma2(W0, f2(pa.x, pb.x), fma2(W1, f2(pa.y, pb.y), fma2(W2, f2(pa.z, pb.z), B1))), zA, zB);
  const F2 T = f2(act_tanh<FAST>(zA), act_tanh<FAST>(zB));
  const F2 NT = mul2(T, f2s(-1.0f));
  const F2 SW = fma2(NT, T, f2s(1.0f));
  const F2 NTT = mul2(NT, T);
  const F2 NTS = mul2(NT, SW);
  o[0] = T;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const F2 TD = f2s(Td[i]), TD2 = mul2(TD, TD);
    F2 R2;
    if (sd1) {  // 1 / (1 - t^2 Td^2) by its series
      const F2 x = mul2(mul2(T, T), TD2);
      R2 = fma2(x, fma2(x, add2(x, f2s(1.0f)), f2s(1.0f)), f2s(1.0f));
    } else {
      float eA, eB;
      f2get(fma2(NTT, TD2, f2s(1.0f)), eA, eB);
      R2 = f2(rcp<FAST>(eA), rcp<FAST>(eB));
    }
    o[1 + i] = mul2(mul2(NTS, TD2), R2);
    o[4 + i] = mul2(mul2(SW, TD), R2);
  }
  const bool ja = pa.cutj >= 0 && (pa.cutj & 1), jb = pb.cutj >= 0 && (pb.cutj & 1);
  o[7] = f2(ja ? act_tanh<FAST>(fmaf(w1[0], pa.gx, fmaf(w1[1], pa.gy, fmaf(w1[2], pa.gz, b1)))) : 0.f,
            jb ? act_tanh<FAST>(fmaf(w1[0], pb.gx, fmaf(w1[1], pb.gy, fmaf(w1[2], pb.gz, b1)))) : 0.f);
}

// tanh(h W1[u][i]) of the first layer (it depends on the unit only); sd1: every
// lane's increments are small and their series serves (accurate path)
template <bool FAST>
__device__ __forceinline__ void layer1_increments(const float (&w1)[3], float h, float (&Td)[3],
                                                  bool& sd1) {
  const float d[3] = {w1[0] * h, w1[1] * h, w1[2] * h};
  sd1 = false;
  if constexpr (!FAST)
    sd1 = __all_sync(0xffffffffu,
                     fmaxf(fabsf(d[0]), fmaxf(fabsf(d[1]), fabsf(d[2]))) <= kSmallDelAccurate);
#pragma unroll
  for (int i = 0; i < 3; ++i) Td[i] = sd1 ? tanh_small(d[i]) : act_tanh<FAST>(d[i]);
}

// A hidden layer's outputs of two points in one unit from the GEMM's 16 columns z
// and the bias.  Column 7 (the interface point) only matters for cut cells with a
// jump row; elsewhere its seeds are 0.  The accurate path skips its tanh there (0,
// as layer 1 leaves it); in the SFU path the test cost more than it saved (C2 6 %
// slower), so that path keeps computing it.
template <bool FAST>
__device__ __forceinline__ void hidden_pair(const float* z, float bb, const PRec* pa,
                                            const PRec* pb, F2 (&o)[8]) {
  constexpr float kSmall = FAST ? kSmallMu : kSmallMuAccurate;
  const F2 BB = f2s(bb);
  float zA, zB;
  f2get(add2(f2(z[0], z[1]), BB), zA, zB);
  const float tA = act_tanh<FAST>(zA), tB = act_tanh<FAST>(zB);
  const F2 T = f2(tA, tB);
  o[0] = T;
  // small increments of both points in every lane: the series (symmetric; accurate
  // path: antisymmetric too)
  const float mA = fmaxf(fabsf(z[2]), fmaxf(fabsf(z[4]), fabsf(z[6])));
  const float mB = fmaxf(fabsf(z[3]), fmaxf(fabsf(z[5]), fabsf(z[7])));
  const bool sm = __all_sync(0xffffffffu, fmaxf(mA, mB) <= kSmall);
  float dA = 0.f, dB = 0.f;
  bool sd = false;
  if constexpr (!FAST) {
    dA = fmaxf(fabsf(z[8]), fmaxf(fabsf(z[10]), fabsf(z[12])));
    dB = fmaxf(fabsf(z[9]), fmaxf(fabsf(z[11]), fabsf(z[13])));
    sd = __all_sync(0xffffffffu, fmaxf(dA, dB) <= kSmallDelAccurate);
  }
  if (sm) {
    const F2 NT = mul2(T, f2s(-1.0f));
    const F2 S0 = fma2(NT, T, f2s(1.0f));
#pragma unroll
    for (int i = 0; i < 3; ++i)
      tanh_stencil_fwd_pair<FAST>(T, NT, S0, f2(z[2 + 2 * i], z[3 + 2 * i]),
                                  f2(z[8 + 2 * i], z[9 + 2 * i]), o[1 + i], o[4 + i], sd);
  } else {
    const bool smA = __all_sync(0xffffffffu, mA <= kSmall);
    const bool smB = __all_sync(0xffffffffu, mB <= kSmall);
    const bool sdA = !FAST && __all_sync(0xffffffffu, dA <= kSmallDelAccurate);
    const bool sdB = !FAST && __all_sync(0xffffffffu, dB <= kSmallDelAccurate);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      float m0, d0, m1, d1;
      tanh_stencil_fwd<FAST>(tA, z[2 + 2 * i], z[8 + 2 * i], 1.f, 1.f, 1.f, 1.f, m0, d0, smA, sdA);
      tanh_stencil_fwd<FAST>(tB, z[3 + 2 * i], z[9 + 2 * i], 1.f, 1.f, 1.f, 1.f, m1, d1, smB, sdB);
      o[1 + i] = f2(m0, m1);
      o[4 + i] = f2(d0, d1);
    }
  }
  float gA, gB;
  f2get(add2(f2(z[14], z[15]), BB), gA, gB);
  if constexpr (FAST) {
    o[7] = f2(act_tanh<FAST>(gA), act_tanh<FAST>(gB));
  } else {
    o[7] = f2((pa->cutj >= 0 && (pa->cutj & 1)) ? act_tanh<FAST>(gA) : 0.f,
              (pb->cutj >= 0 && (pb->cutj & 1)) ? act_tanh<FAST>(gB) : 0.f);
  }
}

}  // namespace nbm
