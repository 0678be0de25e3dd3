// Balanced base-2^7 digits of scaled FP64 values in shared-memory operands, the schedule of
// their products on tcgen05 and the exact read-out of the level accumulators: shared by the
// fused transforms (kernels_oztf.cu) and the chained contractions (kernels_chain.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>

#include "oz.h"
#include "ozaki.h"
#include "umma.h"

namespace gw {

namespace {

using namespace umma;

constexpr uint32_t kTfPlane = 128 * 16 * 2;        // one digit plane of a 128 x 16 K step
// 64 in every base-2^7 position below the top one: m + kTfBias has non-negative 7-bit
// fields u_s, and m = t_0 2^49 + sum_{s>=1} (u_s - 64) 2^(49 - 7 s) with balanced digits.
constexpr long long kTfBias = 64ll * ((1ll << 42) + (1ll << 35) + (1ll << 28) + (1ll << 21) + (1ll << 14) +
                                      (1ll << 7) + 1ll);

// Tensor-memory accumulators: one per level up to nslot - 1, the last one takes the rest.
__host__ __device__ constexpr int tf_nslot(int NT) { return 512 / NT >= 8 ? 8 : 512 / NT; }

// BF16 bits (upper half of the FP32 word) of balanced digit s of a scaled value, from
// M = m + kTfBias: s = 0 gives t_0 = floor(M / 2^49) (|t_0| <= 128), s >= 1 gives
// (u_s - 64) 2^-7s with u_s the 7-bit field of M at bit 49 - 7 s.  Every digit has at most
// 8 significant bits, so its FP32 form has a zero low half and the top half is exact BF16.
template <int s>
__device__ __forceinline__ uint32_t tf_digit(long long M) {
  if (s == 0) return __float_as_uint(__int_as_float(0x4B400000 + (int)(M >> 49)) - 12582912.0f);  // 1.5 2^23 + t0
  const uint32_t u = (uint32_t)((unsigned long long)M >> (49 - 7 * s)) & 127u;
  const float sc = __int_as_float((127 - 7 * s) << 23);  // 2^-7s
  // (2^23 + u) 2^-7s - (2^23 + 64) 2^-7s = (u - 64) 2^-7s, exact in one FMA
  return __float_as_uint(fmaf(__int_as_float(0x4B000000 | u), sc, -8388672.0f * sc));
}

// The 16-byte core-matrix row of digit plane s for 8 consecutive values.
template <int s>
__device__ __forceinline__ uint4 tf_plane_row(const long long* M) {
  return make_uint4(__byte_perm(tf_digit<s>(M[0]), tf_digit<s>(M[1]), 0x7632),
                    __byte_perm(tf_digit<s>(M[2]), tf_digit<s>(M[3]), 0x7632),
                    __byte_perm(tf_digit<s>(M[4]), tf_digit<s>(M[5]), 0x7632),
                    __byte_perm(tf_digit<s>(M[6]), tf_digit<s>(M[7]), 0x7632));
}

// The digit products of one K step for columns NT wide, as a schedule fixed at compile
// time: digit s of the rows against digits t .. t + cnt - 1 of the columns (consecutive
// planes, one MMA cnt NT wide) into accumulators slot .. slot + cnt - 1; `init`: the MMA
// writes (does not add to) its accumulators in the first K step of a tile.
struct TfMma {
  int s, t, cnt, slot, init;
};
template <int NT>
struct TfSchedule {
  TfMma m[kOzDigits * kOzDigits];
  int n;
  constexpr TfSchedule() : m(), n(0) {
    const int nslot = tf_nslot(NT);
    unsigned inited = 0;
    for (int s = 0; s < kOzDigits; ++s)
      for (int t = 0; t <= kOzLmax - s;) {
        const int slot = s + t < nslot - 1 ? s + t : nslot - 1;
        int cnt = 1;
        while (t + cnt <= kOzLmax - s && (s + t + cnt < nslot - 1 ? s + t + cnt : nslot - 1) == slot + cnt &&
               (cnt + 1) * NT <= 256)
          ++cnt;
        m[n].s = s;
        m[n].t = t;
        m[n].cnt = cnt;
        m[n].slot = slot;
        m[n].init = ((inited >> slot) & 1u) ? 0 : 1;
        inited |= ((1u << cnt) - 1u) << slot;
        ++n;
        t += cnt;
      }
  }
};

// Issues the digit products of one K step: dA, dB the descriptors of the step's first row
// and column digit planes (planes kTfPlane and NT x 32 bytes apart: the descriptor's address
// field counts 16-byte units); idesc_bits: further bits of the instruction descriptor.
template <int NT>
__device__ __forceinline__ void tf_issue_step(uint32_t tm, uint64_t dA, uint64_t dB, bool first, uint32_t idesc_bits = 0u) {
  constexpr TfSchedule<NT> S{};
#pragma unroll
  for (int i = 0; i < S.n; ++i) {
    const TfMma m = S.m[i];
    mma_bf16(tm + (uint32_t)(m.slot * NT), dA + (uint64_t)(m.s * (kTfPlane >> 4)),
             dB + (uint64_t)(m.t * (NT * 32 / 16)), idesc_bf16_f32(128, m.cnt * NT) | idesc_bits,
             (first && m.init) ? 0u : 1u);
  }
}
__device__ __forceinline__ void tf_issue(int NT, uint32_t tm, uint64_t dA, uint64_t dB, bool first) {
  switch (NT) {
    case 16: tf_issue_step<16>(tm, dA, dB, first); break;
    case 32: tf_issue_step<32>(tm, dA, dB, first); break;
    case 48: tf_issue_step<48>(tm, dA, dB, first); break;
    case 64: tf_issue_step<64>(tm, dA, dB, first); break;
    default: tf_issue_step<80>(tm, dA, dB, first); break;
  }
}

// Exact integer of a single level's accumulator value v 2^7l (|.| <= 2^22, or < 2^24 WIDE).
template <bool WIDE>
__device__ __forceinline__ int tf_level_int(float v, float sc) {
  if (!WIDE) return __float_as_int(fmaf(v, sc, 12582912.0f)) - 0x4B400000;
  const float x = v * sc;
  const float y = x + 50331648.0f;
  return 4 * (__float_as_int(y) - 0x4C400000) + (__float_as_int((x - (y - 50331648.0f)) + 12582912.0f) - 0x4B400000);
}

// Adds the single levels l and l + 1 (two accumulators read together) to the 64-bit sums:
// I_l 2^7 + I_{l+1} is a 32-bit integer, shifted once into units of 2^-52 (levels 6 and 7:
// rounded, half up, at 2^-52).
template <bool WIDE>
__device__ __forceinline__ void tf_add_pair(long long* S, const float* v, int l) {
  const float s0 = __int_as_float((127 + 7 * l) << 23), s1 = __int_as_float((127 + 7 * (l + 1)) << 23);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int P = tf_level_int<WIDE>(v[j], s0) * 128 + tf_level_int<WIDE>(v[16 + j], s1);
    if (l + 1 <= 5) S[j] += (long long)P << (38 - 7 * (l + 1));
    else S[j] += (long long)((P + 1024) >> 11);  // l = 6: I_6 2^-4 + I_7 2^-11
  }
}

// BF16 bits of the balanced digits of one scaled value, as tf_digit on the device.
inline void host_tf_digits(long long m, uint16_t* out) {
  const long long M = m + kTfBias;
  const long long t0 = M >= 0 ? (M >> 49) : -((-M + (1ll << 49) - 1) >> 49);  // floor(M / 2^49)
  auto bits = [](float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    return (uint16_t)(u >> 16);
  };
  out[0] = bits((float)t0);
  for (int s = 1; s < kOzDigits; ++s) {
    const int u = (int)((unsigned long long)M >> (49 - 7 * s)) & 127;
    out[s] = bits(std::ldexp((float)(u - 64), -7 * s));
  }
}

}  // namespace

}  // namespace gw
