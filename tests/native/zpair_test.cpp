// CPU test of the stored volume's arithmetic (paper_2603_02048_gb300/csrc/
// zpair.h) at the limits of the grids an entry point takes: element numbers fit
// 32 bits, and the addresses that the march forms for a cell's corners, with
// 32-bit offsets below 4 GiB and with 64-bit ones on any volume, are those of
// the layout's definition in 64-bit integers, inside the volume.
#include <cstdio>
#include <set>
#include <vector>

#include "zpair.h"

#define CHECK(c)                                                                   \
    do {                                                                           \
        if (!(c)) {                                                                \
            std::printf("FAIL line %d: %s (%d x %d x %d, %u B)\n", __LINE__, #c, g.nx, g.ny, \
                        g.nz, size);                                               \
            return 1;                                                              \
        }                                                                          \
    } while (0)

struct Grid {
    int nx, ny, nz;
};
template <unsigned N>
struct Voxel {
    unsigned char b[N];
};

static bool accepted(const Grid& g) {
    return g.nx >= 2 && g.ny >= 2 && g.nz >= 2 && g.nx <= hh::kMaxAxis && g.ny <= hh::kMaxAxis &&
           g.nz <= hh::kMaxAxis && hh::stored_voxels(g.nx, g.ny, g.nz) <= hh::kMaxStored;
}

// Largest nz accepted with these axes (0: none).
static int deepest(int nx, int ny) {
    const size_t plane = static_cast<size_t>((nx + 3) / 2) * ((ny + 3) / 2) * 4;
    const size_t pairs = hh::kMaxStored / (2 * plane);  // of slices, halo included
    if (pairs < 2) return 0;
    return static_cast<int>(pairs * 2 - 2 < static_cast<size_t>(hh::kMaxAxis) ? pairs * 2 - 2
                                                                              : hh::kMaxAxis);
}

template <unsigned N>
static int corners(const Grid& g) {
    const unsigned size = N;
    const unsigned row = hh::zpair_row(g.nx, size), pair = hh::zpair_pair(row, g.ny);
    const hh::ZPairStrides Z = hh::zpair_strides(row, pair, size);
    const uint64_t bytes = hh::zpair_elements(pair, g.nz) * size;
    const uint64_t origin = uint64_t(1) << 44;
    const char* base = reinterpret_cast<const char*>(origin);
    auto at = [&](const Voxel<N>* p) { return reinterpret_cast<uint64_t>(p) - origin; };
    auto want = [&](uint64_t I, uint64_t J, uint64_t K) {
        return ((K >> 1) * pair + J * row + 2 * I + (K & 1)) * size;
    };
    auto picks = [](int n) {  // first corners along an axis: padded 0 to n
        std::set<int> s = {0, 1, 2, 3, n / 2, n / 2 + 1, n - 2, n - 1, n};
        std::vector<int> v;
        for (int i : s)
            if (i >= 0 && i <= n) v.push_back(i);
        return v;
    };
    for (int iz : picks(g.nz))
        for (int iy : picks(g.ny))
            for (int ix : picks(g.nx)) {
                const unsigned odd = static_cast<unsigned>(iz) & 1u;
                const unsigned b = hh::zpair_element(Z, ix, iy, iz, odd);
                CHECK(static_cast<uint64_t>(b) * size == want(ix, iy, iz));
                const Voxel<N>*c00, *c10, *c01, *c11;
                for (int mode : {hh::ADDR_ANY, hh::ADDR_BASE, hh::ADDR_PTR}) {
                    if (mode == hh::ADDR_ANY)
                        hh::zpair_corners<hh::ADDR_ANY>(Z, base, b, odd, c00, c10, c01, c11);
                    else if (bytes >= (uint64_t(1) << 32))
                        continue;
                    else if (mode == hh::ADDR_BASE)
                        hh::zpair_corners<hh::ADDR_BASE>(Z, base, b, odd, c00, c10, c01, c11);
                    else
                        hh::zpair_corners<hh::ADDR_PTR>(Z, base, b, odd, c00, c10, c01, c11);
                    CHECK(at(c00) == want(ix, iy, iz));
                    CHECK(at(c10) == want(ix, iy + 1, iz));
                    CHECK(at(c01) == want(ix, iy, iz + 1));
                    CHECK(at(c11) == want(ix, iy + 1, iz + 1));
                    CHECK(at(c11 + 2) + size <= bytes);
                }
            }
    return 0;
}

int main() {
    // every plane, as deep as it is accepted (the element number grows with nz)
    for (unsigned size : {16u, 8u})
        for (int nx = 2; nx <= hh::kMaxAxis; ++nx) {
            const unsigned row = hh::zpair_row(nx, size);
            for (int ny = 2; ny <= hh::kMaxAxis; ny += ny < 64 ? 1 : 61) {
                const Grid g = {nx, ny, deepest(nx, ny)};
                if (g.nz < 2) continue;
                CHECK(accepted(g));
                CHECK(g.nz == hh::kMaxAxis || !accepted({nx, ny, g.nz + 2}));
                const uint64_t pair = (static_cast<uint64_t>(row) * (ny + 2u) + 13u) / 16u * 16u + 2u;
                CHECK(pair == hh::zpair_pair(row, ny));
                CHECK(hh::zpair_elements(hh::zpair_pair(row, ny), g.nz) < (uint64_t(1) << 32));
            }
        }
    // corners: small, odd and ragged grids, and the limits; a pair of slices of
    // the first three (FP32) and the fourth (FP16) takes 4 GiB and more
    std::vector<Grid> grids = {{16384, 8192, 2}, {11600, 11600, 8}, {16384, 8192, 12},
                               {16384, 16384, 4}, {11580, 11580, 8}, {8, 4400, 4400},
                               {2, 2, 2}, {2, 16384, 16384}, {16384, 2, 16384},
                               {16384, 16384, 2}, {5, 16384, 16384}, {1290, 1290, 1286}};
    for (int nx : {2, 3, 5, 6, 7, 31, 33, 65, 256, 4097, 16383, 16384})
        for (int ny : {2, 3, 6, 33, 1024, 16383, 16384})
            for (int nz : {2, 3, 4, 65, deepest(nx, ny)}) grids.push_back({nx, ny, nz});
    int wide = 0;
    for (const Grid& g : grids) {
        if (!accepted(g)) continue;
        if (corners<16>(g) || corners<8>(g)) return 1;
        for (unsigned size : {16u, 8u})
            wide += uint64_t(hh::zpair_pair(hh::zpair_row(g.nx, size), g.ny)) * size >>
                    32 != 0;
    }
    const Grid g = {0, 0, wide};
    const unsigned size = 0;
    CHECK(wide >= 8);
    std::printf("zpair ok\n");
    return 0;
}
