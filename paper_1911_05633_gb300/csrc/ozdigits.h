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
// Tensor-memory accumulators: one per level up to nslot - 1, the last one takes the rest.
__host__ __device__ constexpr int tf_nslot(int NT) { return 512 / NT >= 8 ? 8 : 512 / NT; }

// The eight balanced digits d_s 2^-7s of a scaled value m = sum_s d_s 2^(49 - 7s), |m| <= 2^56, as
// FP32 words whose upper halves are exact BF16: |d_0| <= 128, |d_s| <= 64 after it.  m falls
// into fields of 21, 21 and 14 bits around zero; each becomes a float of the right scale by
// setting its bits under an exponent, and the digits come off by adding 1.5 2^k and taking it
// away again.  The cut is bound by the integer pipe (half the rate of the FP32 one): this
// takes 7 integer and 18 FP32 operations per value, a shift and a mask per digit 20 and 7.  With
// tf_i2d: transforms of the 72-atom cell 20.5 -> 19.3 ms, k_chain of 9024 units 0.73 -> 0.69 ms,
// lattice transforms 1.16 -> 0.99 ms.
__device__ __forceinline__ void tf_digits(long long m, uint32_t* d) {
  const long long M = m + (1ll << 34) + (1ll << 13);
  auto bits = [](float f) { return __float_as_uint(f); };
  {
    const float f = __uint_as_float(0x44400000u + (uint32_t)(int)(M >> 35)) - 768.0f;  // 2^-14 of |.| <= 2^21
    const float d0 = (f + 12582912.0f) - 12582912.0f, r = f - d0;
    const float d1 = (r + 98304.0f) - 98304.0f;
    d[0] = bits(d0);
    d[1] = bits(d1);
    d[2] = bits(r - d1);
  }
  {
    const float f = __uint_as_float(0x39800000u | ((uint32_t)(M >> 14) & 0x1FFFFFu)) - (0x1p-12f + 0x1p-15f);  // 2^-35
    const float d3 = (f + 6.0f) - 6.0f, r = f - d3;
    const float d4 = (r + 0x1.8p-5f) - 0x1.8p-5f;
    d[3] = bits(d3);
    d[4] = bits(d4);
    d[5] = bits(r - d4);
  }
  {
    const float f = __uint_as_float(0x32800000u | ((uint32_t)M & 0x3FFFu)) - (0x1p-26f + 0x1p-36f);  // 2^-49
    const float d6 = (f + 0x1.8p-19f) - 0x1.8p-19f;
    d[6] = bits(d6);
    d[7] = bits(f - d6);
  }
}

// The digits of 8 consecutive scaled values: one 16-byte core-matrix row in each of the eight
// planes, kTfPlane apart, from A on.
__device__ __forceinline__ void tf_cut8(const long long* m, unsigned char* A) {
  uint32_t w[kOzDigits][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t a[kOzDigits], b[kOzDigits];
    tf_digits(m[2 * q], a);
    tf_digits(m[2 * q + 1], b);
#pragma unroll
    for (int s = 0; s < kOzDigits; ++s) w[s][q] = __byte_perm(a[s], b[s], 0x7632);
  }
#pragma unroll
  for (int s = 0; s < kOzDigits; ++s)
    *reinterpret_cast<uint4*>(A + s * kTfPlane) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// S 2^e as a double, rounded once: the conversion runs on the FP64 pipe, which these kernels
// leave idle (i2d_scaled does it in about 28 operations of the integer pipe that bounds them).
// The result has to be a normal double, as there.
__device__ __forceinline__ double tf_i2d(long long S, int e) {
  const double d = __ll2double_rn(S);
  const int hi = __double2hiint(d);
  return __hiloint2double(S ? hi + (e << 20) : 0, __double2loint(d));
}

// Scale exponent of a row that holds an infinity or a NaN (its digits are zero): what is
// computed from it is NaN.
constexpr int kOzNaN = 1 << 20;
__device__ __forceinline__ int tf_row_scale(int m) { return m == 2047 ? kOzNaN : m > 0 ? m - 1022 : 0; }
// tf_i2d for any exponent: subnormal, zero or infinite where the result is.
__device__ __forceinline__ double tf_i2d_any(long long S, int e) {
  return e > kOzNaN / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(__ll2double_rn(S), e);
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

// I_l 2^7 + I_{l+1} of two single levels; the two offsets of the reads go out in one subtraction.
template <bool WIDE>
__device__ __forceinline__ int tf_pair_int(float v0, float s0, float v1, float s1) {
  if (WIDE) return tf_level_int<true>(v0, s0) * 128 + tf_level_int<true>(v1, s1);
  return (int)(__float_as_uint(fmaf(v0, s0, 12582912.0f)) * 128u +
               (__float_as_uint(fmaf(v1, s1, 12582912.0f)) - 129u * 0x4B400000u));
}

// Adds the single levels l and l + 1 (two accumulators read together) to the 64-bit sums:
// I_l 2^7 + I_{l+1} is a 32-bit integer, shifted once into units of 2^-52 (levels 6 and 7:
// rounded, half up, at 2^-52).
template <bool WIDE>
__device__ __forceinline__ void tf_add_pair(long long* S, const float* v, int l) {
  const float s0 = __int_as_float((127 + 7 * l) << 23), s1 = __int_as_float((127 + 7 * (l + 1)) << 23);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int P = tf_pair_int<WIDE>(v[j], s0, v[16 + j], s1);
    if (l + 1 <= 5) S[j] += (long long)P << (38 - 7 * (l + 1));
    else S[j] += (long long)((P + 1024) >> 11);  // l = 6: I_6 2^-4 + I_7 2^-11
  }
}

// 64 in every base-2^7 position below the top one: m + kHostBias has non-negative 7-bit
// fields u_s, and m = t_0 2^49 + sum_{s>=1} (u_s - 64) 2^(49 - 7 s) with balanced digits.
constexpr long long kHostBias = 64ll * ((1ll << 42) + (1ll << 35) + (1ll << 28) + (1ll << 21) + (1ll << 14) +
                                      (1ll << 7) + 1ll);

// BF16 bits of balanced digits of one scaled value (another choice than tf_digits where a
// digit is +-64: the values are the same).
inline void host_tf_digits(long long m, uint16_t* out) {
  const long long M = m + kHostBias;
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
