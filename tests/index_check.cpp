// Host check of the window index arithmetic that wraps modulo 2^32: the offset
// of a cell in its window from whole parts that carry kSplitBias.  Built so that
// signed overflow traps.  Prints the number of offsets compared.
#include <cstdio>
#include <cstring>

#include "mboit_device.cuh"

using namespace mb;

static uint32_t carried(int n) {   // as split2: the bits of 2^23 + n
    const float m = 8388608.0f + (float)n;
    uint32_t b;
    std::memcpy(&b, &m, sizeof b);
    return b;
}

int main() {
    long offsets = 0;
    // window shapes: (row pitch, plane) of the scalar, vector and TMA windows
    const int shapes[][2] = {{9, 72}, {12, 100}, {16, 132}, {12, 132}, {16, 128}};
    const int origins[] = {0, 1, 4, 511, 65535, 4194299};
    for (const auto& s : shapes)
        for (int lx : origins)
            for (int ly : origins)
                for (int lz : origins) {
                    const uint32_t base = window_offset((uint32_t)lx + kSplitBias, (uint32_t)ly + kSplitBias,
                                                        (uint32_t)lz + kSplitBias, (uint32_t)s[0], (uint32_t)s[1]);
                    for (int k = 0; k < 8 * 8 * 8; ++k, ++offsets) {
                        const int x = k & 7, y = k >> 3 & 7, z = k >> 6;
                        const int got = (int)(window_offset(carried(lx + x), carried(ly + y), carried(lz + z),
                                                            (uint32_t)s[0], (uint32_t)s[1]) - base);
                        if (got != z * s[1] + y * s[0] + x) return 1;
                    }
                }
    std::printf("%ld\n", offsets);
    return 0;
}
