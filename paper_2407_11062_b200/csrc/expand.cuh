// Packed weights as the GEMM kernels read them: the device-side view of a packed
// matrix, the fetch of its codes and group parameters, and the expansion of
// codes to bf16 operand rows.
#pragma once
#include <stdint.h>

#include "common.cuh"
#include "ptx.cuh"

namespace eqat {

// A packed weight matrix with its step sizes and zero points.
struct PackedWeight {
  const uint8_t* Wq;         // [out, in*bits/8]
  const eqat_fp16* s16;      // [out, in/group]
  const void* zq;            // [out, in/group]: uint8, or fp16 when z_fp16
  int z_fp16;
  int out_features, in_features;
  int group_shift;           // log2(group) for groups of 32..256 (31 for one group per row: every index shifts to 0)
  int groups_per_row;
  int wq_sectors;            // Wq is 32-byte aligned: a thread may fetch a whole 32-byte sector with one load
};

inline int log2_exact(int v) {
  int s = 0;
  while ((1 << s) < v) ++s;
  return s;
}

inline void set_weight(PackedWeight& p, const eqat_desc& d, const uint8_t* Wq, const eqat_fp16* s16, const void* zq) {
  p.Wq = Wq; p.s16 = s16; p.zq = zq;
  p.z_fp16 = d.zero_point_format == EQAT_ZP_FP16 ? 1 : 0;
  p.out_features = d.out_features;
  p.in_features = d.in_features;
  const bool whole_row = d.group == d.in_features && d.group > 256;
  p.group_shift = whole_row ? 31 : log2_exact(d.group);
  p.groups_per_row = d.in_features / d.group;
  p.wq_sectors = (reinterpret_cast<uintptr_t>(Wq) & 31u) == 0 ? 1 : 0;
}

// ------------------------------------------------------------------ expansion of packed codes
// 64 consecutive codes of one weight row become one 128-byte swizzled shared-memory row: element e of the row
// goes to 16-byte chunk (e/8) ^ rx.  `row_sx` is the shared-memory address of the row XOR (rx << 4): the row is
// 128-byte aligned, so chunk c lies at row_sx ^ (c << 4), one logic operation per store.
//
// 3- and 4-bit codes: a code q is dropped into bits 16..23 of the float 0x4B000000 (= 2^23), giving
// x = 2^23 + 65536*q exactly, and fma(x, s/65536, -(128 + z)*s) = (q - z)*s.  With an integer zero point both
// constants are exact in fp32 (s is an fp16 value, 11 significant bits) and so is the result: the only rounding
// is the final one to bf16.  With a real-valued (fp16) zero point the constant (128 + z)*s is rounded to fp32
// first, an error of at most 2^-17 s.  4-bit codes reach byte positions with one shift+mask per 4 codes and one
// byte permute each; 3-bit codes sit at other positions (below).
// 2-bit codes: the four possible values of a group are built once as bf16 ((q - z)*s in fp32, rounded once) and
// each code is looked up with a byte permute: lut01 = (v0, v1), lut23 = (v2, v3); value q occupies bytes 2q, 2q+1
// of the 8-byte pair, so the selector byte of a code is 0x10 + 0x22*q.
template <int BITS>
struct GroupValues {
  float sp, cz;
  __device__ __forceinline__ GroupValues() : sp(0.0f), cz(0.0f) {}
  __device__ __forceinline__ GroupValues(float s, float z) : sp(s * (1.0f / 65536.0f)), cz(-(128.0f + z) * s) {}
  __device__ __forceinline__ float operator()(uint32_t xbits) const { return fmaf(__uint_as_float(xbits), sp, cz); }
};
// 3-bit codes are not byte-aligned, and a shift per code costs as much as the multiply-add that follows it.  A
// code may instead sit at any mantissa position p as long as the constants follow it: with x = 2^23 + 2^p * q,
// fma(x, s / 2^p, -(2^(23-p) + z) * s) = (q - z) * s, exact while (2^(23-p) + z) * s is (p >= 11 for 11-bit s and
// z < 8).  Three consecutive codes of the stream land on p = 12, 15, 18 with ONE shift of the word (or of two
// words, for a code that straddles them), so a triple costs one shift instead of three.
template <>
struct GroupValues<3> {
  float sp[3], cz[3];
  __device__ __forceinline__ GroupValues() : sp{0.0f, 0.0f, 0.0f}, cz{0.0f, 0.0f, 0.0f} {}
  __device__ __forceinline__ GroupValues(float s, float z) {
    sp[0] = s * (1.0f / 4096.0f);   cz[0] = -(2048.0f + z) * s;
    sp[1] = s * (1.0f / 32768.0f);  cz[1] = -(256.0f + z) * s;
    sp[2] = s * (1.0f / 262144.0f); cz[2] = -(32.0f + z) * s;
  }
  // code of slot k (0..2) of a triple, still at bits [12 + 3k, 15 + 3k) of `win`
  __device__ __forceinline__ float at(int k, uint32_t win) const {
    return fmaf(__uint_as_float((win & (7u << (12 + 3 * k))) | 0x4B000000u), sp[k], cz[k]);
  }
};

template <>
struct GroupValues<2> {
  uint32_t lut01, lut23;
  __device__ __forceinline__ GroupValues() : lut01(0u), lut23(0u) {}
  __device__ __forceinline__ GroupValues(float s, float z) {
    const float zs = z * s;                              // exact: 11 x 11 significant bits
    lut01 = pack_bf16x2(-zs, s - zs);
    lut23 = pack_bf16x2(fmaf(2.0f, s, -zs), fmaf(3.0f, s, -zs));
  }
};

// 32 consecutive codes as 16 registers of bf16 pairs, (q - z) * s rounded once, in the order of the stream.
template <int BITS>
__device__ __forceinline__ void values32(const uint32_t* w, const GroupValues<BITS>& f, uint32_t* o) {
  constexpr uint32_t kMagic = 0x4B000000u;
  if constexpr (BITS == 2) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {                       // word i: codes 16i .. 16i+15
      uint32_t sel[4];                                  // byte b of sel[r] = selector byte of code 4b + r
#pragma unroll
      for (int r = 0; r < 4; ++r) sel[r] = ((w[i] >> (2 * r)) & 0x03030303u) * 0x22u + 0x10101010u;
#pragma unroll
      for (int pr = 0; pr < 8; ++pr) {
        const uint32_t b = (uint32_t)(pr >> 1), r = (uint32_t)((2 * pr) & 3);   // even code 2pr = 4b + r, r in {0, 2}
        o[8 * i + pr] = __byte_perm(f.lut01, f.lut23, __byte_perm(sel[r], sel[r + 1], b | ((4u + b) << 4)));
      }
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {                       // word i: codes 8i .. 8i+7
      const uint32_t m0 = w[i] & 0x0F0F0F0Fu, m1 = (w[i] >> 4) & 0x0F0F0F0Fu;   // byte b = code 2b (+1)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        o[4 * i + b] = pack_bf16x2(f(__byte_perm(m0, kMagic, 0x7044u | ((uint32_t)b << 8))),
                                   f(__byte_perm(m1, kMagic, 0x7044u | ((uint32_t)b << 8))));
    }
  } else {
    // 32 codes = 3 words = 96 bits, code j at bit 3j.  Triple m (codes 3m .. 3m+2) is brought to bits 12..20 of a
    // register by one shift of the stream: the 32-bit window that starts at bit 9m - 12.
    float v[33];
#pragma unroll
    for (int m = 0; m < 11; ++m) {
      const int start = 9 * m - 12;
      uint32_t win;
      if (start < 0) {
        win = w[0] << (-start);
      } else {
        const int word = start >> 5, sh = start & 31;
        const uint32_t hi = word + 1 < 3 ? w[word + 1 < 3 ? word + 1 : 2] : 0u;
        win = sh == 0 ? w[word] : __funnelshift_r(w[word], hi, sh);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (3 * m + k < 32) v[3 * m + k] = f.at(k, win);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
  }
}

// Expands 32 consecutive codes (half h of a 64-code row) into chunks 4h .. 4h+3.
template <int BITS>
__device__ __forceinline__ void dequant_half32(const uint32_t (&w)[BITS], const GroupValues<BITS>& f, uint32_t row_sx, int h) {
  uint32_t o[16];
  values32<BITS>(w, f, o);
#pragma unroll
  for (int c = 0; c < 4; ++c)
    ptx::sts_128(row_sx ^ ((uint32_t)(4 * h + c) << 4), o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
}

// 64 codes = 2*BITS consecutive 32-bit words, at a multiple of 8*BITS bytes.
template <int BITS>
__device__ __forceinline__ void load_codes64(const uint8_t* p, uint32_t (&w)[2 * BITS]) {
  if constexpr (BITS == 2) {
    const uint4 t = ptx::ld_global(reinterpret_cast<const uint4*>(p));
    w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
  } else if constexpr (BITS == 3) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const uint2 t = ptx::ld_global(reinterpret_cast<const uint2*>(p) + i);
      w[2 * i] = t.x; w[2 * i + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint4 t = ptx::ld_global(reinterpret_cast<const uint4*>(p) + i);
      w[4 * i] = t.x; w[4 * i + 1] = t.y; w[4 * i + 2] = t.z; w[4 * i + 3] = t.w;
    }
  }
}

// Step sizes and zero points of up to four consecutive groups of one weight row, as fetched: fp16 step sizes in
// s, zero points in z either as bytes (z.x) or as fp16 values.  `count` (1, 2 or 4) consecutive groups starting
// at group index gi, which is a multiple of count; in_features is a multiple of 128, so the vector loads below
// are aligned.
struct GroupParamsRaw {
  uint2 s, z;
};
__device__ __forceinline__ void load_group_params(const PackedWeight& p, size_t gi, int count, GroupParamsRaw& r) {
  const eqat_fp16* sp = p.s16 + gi;
  if (count == 1) {
    r.s.x = ptx::ld_global(sp);
  } else if (count == 2) {
    r.s.x = ptx::ld_global(reinterpret_cast<const uint32_t*>(sp));
  } else {
    r.s = ptx::ld_global(reinterpret_cast<const uint2*>(sp));
  }
  if (p.z_fp16) {
    const eqat_fp16* zp = static_cast<const eqat_fp16*>(p.zq) + gi;
    if (count == 1) {
      r.z.x = ptx::ld_global(zp);
    } else if (count == 2) {
      r.z.x = ptx::ld_global(reinterpret_cast<const uint32_t*>(zp));
    } else {
      r.z = ptx::ld_global(reinterpret_cast<const uint2*>(zp));
    }
  } else {
    const uint8_t* zp = static_cast<const uint8_t*>(p.zq) + gi;
    if (count == 1) {
      r.z.x = ptx::ld_global(zp);
    } else if (count == 2) {
      r.z.x = ptx::ld_global(reinterpret_cast<const unsigned short*>(zp));
    } else {
      r.z.x = ptx::ld_global(reinterpret_cast<const uint32_t*>(zp));
    }
  }
}
__device__ __forceinline__ float half_at(const uint2& v, int i) {
  const uint32_t w = (i & 2) ? v.y : v.x;
  return __half2float(__ushort_as_half((unsigned short)((i & 1) ? (w >> 16) : (w & 0xFFFFu))));
}
__device__ __forceinline__ float step_size_at(const GroupParamsRaw& r, int i) { return half_at(r.s, i); }
__device__ __forceinline__ float zero_point_at(const GroupParamsRaw& r, int i, int z_fp16) {
  return z_fp16 ? half_at(r.z, i) : (float)((r.z.x >> (8 * i)) & 0xFFu);
}
}  // namespace eqat
