// Shared memory of the three-dimensional slab kernels: two blocks per SM for
// the tile with compiled copies (their speed rests on 16 resident warps per SM),
// and every tile that dust_create accepts in mixed precision, up to the 254 zones
// a side that the bulk copy takes, within a block's limit.  Host code only: no kernel is instantiated and no CUDA call is made.
#include <cstdio>

#include "dust_slab.cuh"

int main()
{
    using namespace dust;
    // GB300: 228 KB of shared memory per SM, 1 KB of it reserved per block
    const size_t per_sm = 228 * 1024, reserved = 1024;
    auto bytes = [](int a, int b, int c) {
        GridDev g{};
        const int T[3] = {a, b, c};
        for (int d = 0; d < 3; ++d) {
            g.T[d] = T[d];
            g.n[d] = 2 * T[d];
        }
        g.tvol = a * b * c;
        return cube_smem_bytes(g);
    };
    if (2 * (bytes(8, 8, 8) + reserved) > per_sm) {
        std::printf("8^3 tile: %zu bytes per block, two blocks do not fit\n", bytes(8, 8, 8));
        return 1;
    }
    // the limit of dust_create: 48 bytes per zone of the box with its halo and
    // the records of 256 grains
    long tiles = 0;
    for (int a = 1; a <= 254; ++a)
        for (int b = 1; b <= 254; ++b)
            for (int c = 1; c <= 254; ++c) {
                const size_t box = (size_t)(a + 2) * (b + 2) * (c + 2);
                if (box * 48 + 256 * (8 + 13 * 4 + 64) + 16 > 220 * 1024) break;
                ++tiles;
                if (bytes(a, b, c) + reserved > per_sm) {
                    std::printf("tile %dx%dx%d: %zu bytes do not fit\n", a, b, c, bytes(a, b, c));
                    return 1;
                }
            }
    std::printf(tiles > 1000 ? "ok\n" : "too few tiles\n");
    return 0;
}
