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

// Bytes s / 8 to s / 8 + 3 of the eight of lo, then hi (s < 32).
HH_HD uint32_t shift_pair(uint32_t lo, uint32_t hi, unsigned s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return static_cast<uint32_t>((static_cast<uint64_t>(hi) << 32 | lo) >> s);
#endif
}

// Two neighbouring texels, six bytes from p on, to lo (the first four) and hi, by
// Load: from the aligned 32-bit words that hold them, two, or three where p is
// the last byte of a word, instead of six loads.
template <class Load>
HH_HD void texel_words(const uint8_t* p, Load load, uint32_t& lo, uint32_t& hi) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(p);
    const uint32_t* w = reinterpret_cast<const uint32_t*>(at & ~uintptr_t(3));
    const unsigned byte = static_cast<unsigned>(at) & 3u;
    const uint32_t w0 = load(w), w1 = load(w + 1), w2 = byte == 3u ? load(w + 2) : 0u;
    lo = shift_pair(w0, w1, 8u * byte);
    hi = shift_pair(w1, w2, 8u * byte);
}
template <class Load>
HH_HD void texel_bytes(const uint8_t* p, Load load, uint32_t& lo, uint32_t& hi) {
    lo = load(p) | load(p + 1) << 8 | load(p + 2) << 16 | load(p + 3) << 24;
    hi = load(p + 4) | load(p + 5) << 8;
}

// The pairs at texels (i0, j0) and (i0, j0 + 1), i0 <= W - 2, j0 <= H - 2, of a W x
// H texture at any address. The words around a pair have up to three bytes
// before and behind it. They are the texture's own except before its first pair
// and behind its last, and the squares that have one of these are read by bytes
// (one branch for both pairs, so that their loads still go out together).
template <class Load>
HH_HD void texel_square(const uint8_t* tex, int W, int H, int i0, int j0, Load load, uint32_t& lo0,
                        uint32_t& hi0, uint32_t& lo1, uint32_t& hi1) {
    const uint8_t* p0 = tex + (static_cast<size_t>(j0) * W + i0) * 3;
    const uint8_t* p1 = p0 + static_cast<size_t>(W) * 3;
    if ((i0 == 0 && j0 == 0) || (i0 == W - 2 && j0 == H - 2)) {
        texel_bytes(p0, load, lo0, hi0);
        texel_bytes(p1, load, lo1, hi1);
    } else {
        texel_words(p0, load, lo0, hi0);
        texel_words(p1, load, lo1, hi1);
    }
}

}  // namespace hh
