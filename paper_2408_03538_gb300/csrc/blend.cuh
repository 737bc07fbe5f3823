// Sums of the composite that do not depend on the kernel around them (also compiled for the host by the tests).
#pragma once

namespace prtgs {

// Floats of k colour sets, on a 16-byte boundary.
__host__ __device__ constexpr int color_floats(int kg) { return (3 * kg + 3) / 4 * 4; }

// acc[e] += w row[e] over the 3 KG channels of a group of KG colour sets; row: color_floats(KG) floats, read in
// 16-byte words, of which the last may hold up to three floats that belong to no channel.
template <int KG>
__host__ __device__ __forceinline__ void blend_row(float (&acc)[3 * KG], const float* row, float w) {
#pragma unroll
  for (int e = 0; e < 3 * KG; e += 4) {
    const float4 c = *reinterpret_cast<const float4*>(row + e);
    acc[e] = fmaf(c.x, w, acc[e]);
    if (e + 1 < 3 * KG) acc[e + 1] = fmaf(c.y, w, acc[e + 1]);
    if (e + 2 < 3 * KG) acc[e + 2] = fmaf(c.z, w, acc[e + 2]);
    if (e + 3 < 3 * KG) acc[e + 3] = fmaf(c.w, w, acc[e + 3]);
  }
}

}  // namespace prtgs
