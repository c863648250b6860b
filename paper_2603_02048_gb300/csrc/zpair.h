// The ZPAIR volume layout (hh_internal.h says what it is for): which grids an
// entry point takes, the layout's strides, and the addresses of a cell's eight
// corners. Plain arithmetic for host and device, so that a CPU test can hold
// it, at the limits of the grids, to 64-bit element numbers.
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define HH_HD __host__ __device__ __forceinline__
#else
#define HH_HD inline
#endif

namespace hh {

// Largest grid axis and number of stored voxels (grid and halo, every axis
// padded to even) that the entry points take. A ZPAIR volume pads its rows
// further: 256^3 by 0.4 % on FP32 storage and 1.6 % on FP16, long narrow grids to
// 1.76 times the stored voxels, one of 2x2x2 voxels to 2.06 times. Its element
// numbers fit 32 bits; byte offsets do not.
constexpr int kMaxAxis = 1 << 14;
constexpr size_t kMaxStored = size_t(1) << 31;

inline size_t stored_voxels(int nx, int ny, int nz) {
    return static_cast<size_t>((nx + 3) / 2) * ((ny + 3) / 2) * ((nz + 3) / 2) * 8;
}

// Strides in elements: of a row, and of a pair of slices (voxel_bytes: 16 for
// FP32 storage, 8 for FP16).
inline unsigned zpair_row(int nx, unsigned voxel_bytes) {
    const unsigned n = 2u * (static_cast<unsigned>(nx) + 2u);
    return voxel_bytes == 16u ? (n + 1u) / 8u * 8u + 6u : (n + 3u) / 16u * 16u + 12u;
}
inline unsigned zpair_pair(unsigned row, int ny) {
    return (row * (static_cast<unsigned>(ny) + 2u) + 13u) / 16u * 16u + 2u;
}
inline size_t zpair_elements(unsigned pair, int nz) {
    return static_cast<size_t>(pair) * ((static_cast<size_t>(nz) + 3) / 2);
}

// How a kernel addresses the volume. Below 4 GiB, as 32-bit byte offsets from
// base addresses that the whole grid shares, which cost a load no address
// arithmetic (ADDR_BASE; FP16 384^3 4K view: 1733 against 1657 us), or, for a
// volume of a pointer of its own (the serving worker's jobs), as 64-bit addresses
// with 32-bit byte steps (ADDR_PTR); ADDR_ANY, for any size, multiplies the step
// out in 64 bits (six requests of three views on a 384^3 FP16 volume: 10.41 ms
// with ADDR_PTR, 10.58 so).
enum { ADDR_BASE = 0, ADDR_ANY = 1, ADDR_PTR = 2 };

// Strides of the march: a row, half of a pair of slices, and in bytes a row and
// the step from an odd slice to the next, less one element. A pair of slices can
// take 4 GiB and more, so up_bytes, which wraps there, is not for ADDR_ANY.
struct ZPairStrides {
    unsigned row, half_pair;  // elements
    unsigned row_bytes, up_bytes;
};
inline ZPairStrides zpair_strides(unsigned row, unsigned pair, unsigned voxel_bytes) {
    return {row, pair / 2, row * voxel_bytes, (pair - 2u) * voxel_bytes};
}

// Element of padded (ix, iy, iz), odd = iz & 1: (iz >> 1) pair + iy row + 2 ix +
// odd, the pair's half taken out by the parity.
HH_HD unsigned zpair_element(const ZPairStrides& Z, int ix, int iy, int iz, unsigned odd) {
    return static_cast<unsigned>(iz) * Z.half_pair + static_cast<unsigned>(iy) * Z.row +
           2u * static_cast<unsigned>(ix) - odd * (Z.half_pair - 1u);
}

// Addresses of corners (ix, iy + 0 or 1, iz + 0 or 1) of the cell whose first
// corner is element b of the volume at `base`: the next column is 2 elements on
// (not asked for here), the next row `row`, the next slice 1 from an even slice
// (odd = 0), else pair - 1.
template <int ADDR, typename V>
HH_HD void zpair_corners(const ZPairStrides& Z, const char* base, unsigned b, unsigned odd,
                         const V*& c00, const V*& c10, const V*& c01, const V*& c11) {
    constexpr unsigned size = sizeof(V);
    const unsigned up = odd * Z.up_bytes + size;
    if (ADDR == ADDR_BASE) {
        const char* next = base + Z.row_bytes;
        const unsigned at = b * size, above = at + up;
        c00 = reinterpret_cast<const V*>(base + at);
        c10 = reinterpret_cast<const V*>(next + at);
        c01 = reinterpret_cast<const V*>(base + above);
        c11 = reinterpret_cast<const V*>(next + above);
    } else {
        c00 = reinterpret_cast<const V*>(base) + b;
        c01 = ADDR == ADDR_PTR
                  ? reinterpret_cast<const V*>(reinterpret_cast<const char*>(c00) + up)
                  : c00 + (odd * (2u * Z.half_pair - 2u) + 1u);
        c10 = reinterpret_cast<const V*>(reinterpret_cast<const char*>(c00) + Z.row_bytes);
        c11 = reinterpret_cast<const V*>(reinterpret_cast<const char*>(c01) + Z.row_bytes);
    }
}

}  // namespace hh
