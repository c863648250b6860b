// Reads of RGB8 textures (the environment map and the planes' textures), for
// host and device, so that a CPU test can hold every read to the texture's own
// bytes.
#pragma once

#include <cstddef>
#include <cstdint>

#ifndef HH_HD
#ifdef __CUDACC__
#define HH_HD __host__ __device__ __forceinline__
#else
#define HH_HD inline
#endif
#endif

namespace hh {

// Two neighbouring texels, six bytes from p on, to lo (the first four) and hi, by
// Load: the four that begin at an even address as two halves, the other two, one
// at each end or both at the last, by bytes. Four loads for six, at any address,
// of the texels' bytes alone. (Whole 32-bit words, 2 or 3 loads, hold up to three
// bytes of what lies beside the texture; with the first and the last texels read
// by bytes in a branch of their own, eight 720p views on FP16 storage take 1208
// us, so 1201, with words everywhere 1199.)
template <class Load>
HH_HD void texel_pair(const uint8_t* p, Load load, uint32_t& lo, uint32_t& hi) {
    const unsigned odd = static_cast<unsigned>(reinterpret_cast<uintptr_t>(p)) & 1u;
    const uint16_t* q = reinterpret_cast<const uint16_t*>(p + odd);
    const uint32_t h0 = load(q), h1 = load(q + 1), a = load(odd ? p : p + 4), b = load(p + 5);
    const uint32_t mid = h0 | h1 << 16;
    lo = odd ? (mid << 8 | a) : mid;
    hi = odd ? (mid >> 24 | b << 8) : (a | b << 8);
}

// The pairs at texels (i0, j0) and (i0, j0 + 1), i0 <= W - 2, j0 <= H - 2, of a
// texture W wide.
template <class Load>
HH_HD void texel_square(const uint8_t* tex, int W, int i0, int j0, Load load, uint32_t& lo0,
                        uint32_t& hi0, uint32_t& lo1, uint32_t& hi1) {
    const uint8_t* p = tex + (static_cast<size_t>(j0) * W + i0) * 3;
    texel_pair(p, load, lo0, hi0);
    texel_pair(p + static_cast<size_t>(W) * 3, load, lo1, hi1);
}

}  // namespace hh
