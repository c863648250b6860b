// CPU test of the texture reads (paper_2603_02048_gb300/csrc/texels.h): every pair
// of texels of small textures at every byte offset, with the values that are
// there and no read outside the texture's own bytes.
#include <cstdio>
#include <cstring>
#include <vector>

#include "texels.h"

static const uint8_t* g_begin;
static const uint8_t* g_end;
static int g_outside;

struct Load {
    static void check(const void* p, size_t n) {
        const uint8_t* b = static_cast<const uint8_t*>(p);
        if (b < g_begin || b + n > g_end) ++g_outside;
    }
    uint32_t operator()(const uint8_t* p) const {
        check(p, 1);
        return *p;
    }
    uint32_t operator()(const uint16_t* p) const {
        check(p, 2);
        if (reinterpret_cast<uintptr_t>(p) % 2) ++g_outside;  // misaligned
        uint16_t v;
        std::memcpy(&v, p, 2);
        return v;
    }
    uint32_t operator()(const uint32_t* p) const {
        check(p, 4);
        uint32_t v;
        std::memcpy(&v, p, 4);
        return v;
    }
};

int main() {
    for (int W = 2; W <= 9; ++W)
        for (int H = 2; H <= 5; ++H)
            for (int offset = 0; offset < 8; ++offset) {
                std::vector<uint64_t> store((W * H * 3 + offset + 16) / 8 + 2);
                uint8_t* tex = reinterpret_cast<uint8_t*>(store.data() + 1) + offset;
                for (int i = 0; i < W * H * 3; ++i) tex[i] = static_cast<uint8_t>(37 * i + 11);
                g_begin = tex;
                g_end = tex + W * H * 3;
                for (int j = 0; j <= H - 2; ++j)
                    for (int i = 0; i <= W - 2; ++i) {
                        uint32_t w[2][2];
                        g_outside = 0;
                        hh::texel_square(tex, W, i, j, Load(), w[0][0], w[0][1], w[1][0], w[1][1]);
                        bool ok = g_outside == 0;
                        for (int r = 0; r < 2; ++r)
                            for (int b = 0; b < 6; ++b)
                                ok = ok && ((w[r][b / 4] >> (8 * (b % 4))) & 0xFFu) ==
                                               tex[((j + r) * W + i) * 3 + b];
                        if (!ok) {
                            std::printf("FAIL: %d x %d at offset %d, texel %d, %d: %d reads outside\n",
                                        W, H, offset, i, j, g_outside);
                            return 1;
                        }
                    }
            }
    std::printf("texels ok\n");
    return 0;
}
