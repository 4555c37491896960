// Staging of sparse codes in shared memory, shared by the decode and the
// splatting preprocess.
#pragma once

#include <stdint.h>

namespace dlsh {

// Whether a code array can be read in groups of four slots: rows of a multiple
// of four slots, and arrays aligned to a group (four 8- or 16-bit indices, four
// 16- or 32-bit coefficients).
template <bool U8, bool F16>
__device__ __forceinline__ bool codes_in_quads(const void* idx, const void* coef, int s) {
  return (s & 3) == 0 && (reinterpret_cast<uintptr_t>(idx) & (U8 ? 3u : 7u)) == 0 &&
         (reinterpret_cast<uintptr_t>(coef) & (F16 ? 7u : 15u)) == 0;
}

// One warp stages n consecutive code slots from element e0 on (whole rows of s
// slots, e0 a multiple of s) as (index, coefficient bits) pairs, row g's slot t
// at cpk[g * sp + t], sp even: a group of four slots per lane and step, so that
// the division by s, the address and the bounds are taken once for four (one
// slot at a time took about 14 instructions a slot, this 7).  SCALE multiplies
// the index.  An index of K or more counts as a zero entry; returns whether
// there was one.
template <bool U8, bool F16, int SCALE = 1>
__device__ __forceinline__ bool stage_quads(const void* __restrict__ idx, const void* __restrict__ coef, int64_t e0,
                                            int n, int s, int sp, uint32_t sdiv, uint32_t K, uint2* cpk) {
  constexpr int U = 2;  // groups in flight per lane
  const int lane = threadIdx.x & 31;
  bool bad = false;
  for (int q0 = lane; 4 * q0 < n; q0 += 32 * U) {
    uint32_t j[U][4], a[U][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int q = q0 + 32 * u;
      const bool on = 4 * q < n;
      const int64_t e = on ? e0 / 4 + q : 0;  // in groups
      if constexpr (U8) {
        const uint32_t w = on ? __ldg(static_cast<const uint32_t*>(idx) + e) : 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) j[u][i] = (w >> (8 * i)) & 255u;
      } else {
        const uint2 w = on ? __ldg(static_cast<const uint2*>(idx) + e) : make_uint2(0u, 0u);
        j[u][0] = w.x & 0xffffu;
        j[u][1] = w.x >> 16;
        j[u][2] = w.y & 0xffffu;
        j[u][3] = w.y >> 16;
      }
      if constexpr (F16) {
        const uint2 w = on ? __ldg(static_cast<const uint2*>(coef) + e) : make_uint2(0u, 0u);
        a[u][0] = w.x & 0xffffu;
        a[u][1] = w.x >> 16;
        a[u][2] = w.y & 0xffffu;
        a[u][3] = w.y >> 16;
      } else {
        const uint4 w = on ? __ldg(static_cast<const uint4*>(coef) + e) : make_uint4(0u, 0u, 0u, 0u);
        a[u][0] = w.x;
        a[u][1] = w.y;
        a[u][2] = w.z;
        a[u][3] = w.w;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int f = 4 * (q0 + 32 * u);
      if (f < n) {
        const int g = static_cast<int>(__umulhi(static_cast<uint32_t>(f), sdiv));
        uint4* d = reinterpret_cast<uint4*>(cpk + g * sp + (f - g * s));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool ok = j[u][i] < K;
          bad |= !ok;
          j[u][i] = ok ? j[u][i] * SCALE : 0u;
          a[u][i] = ok ? a[u][i] : 0u;
        }
        d[0] = make_uint4(j[u][0], a[u][0], j[u][1], a[u][1]);
        d[1] = make_uint4(j[u][2], a[u][2], j[u][3], a[u][3]);
      }
    }
  }
  return bad;
}

}  // namespace dlsh
