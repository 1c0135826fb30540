// Host check of ghost_shift_x (compiled and run by tests/test_ghost_shift_host.py): in
// every box at least 16 nodes wide, and in one whose interleaved row is longer than 2^31
// elements, the distance is the one between the two positions, and columns without a
// copy have none.
#include <cstdio>

#include "layout.cuh"

using namespace llb;

template <class S>
static int check(int nx, int align) {
    const Layout L = make_layout(nx, 2, 1, true, 1, align);
    int bad = 0;
    for (int i = 0; i < 32; ++i) {
        const int x = i < 16 ? i : nx - 32 + i;  // both ends
        if (x < 0 || x >= nx) continue;
        const int copy = x < kGhostX ? x + nx : x >= nx - kGhostX ? x - nx : x;
        for (int y = 0; y < 2; ++y)
            for (int f = 0; f < 10; ++f) {
                const size_t from = FieldMap<S, 10>::at(L.at(x, y, 0), f, L.fs);
                const size_t want = FieldMap<S, 10>::at(L.at(copy, y, 0), f, L.fs);
                const size_t got = from + (size_t)ghost_shift_x<S, 10>(L, x);
                if (got != want || got >= 10 * L.fs) ++bad;
            }
    }
    if (bad) std::printf("FAIL nx %d: %d wrong distances\n", nx, bad);
    return bad;
}

int main() {
    static_assert(sizeof(ghost_shift_x<float, 10>(Layout{}, 0)) == 8, "64-bit distance");
    int bad = 0;
    for (int nx : {16, 17, 31, 32, 40, 1000, 214748364, 220000000, 2000000000}) {
        bad += check<float>(nx, 32);   // interleaved
        bad += check<double>(nx, 8);   // field-major
        bad += check<short>(nx, 8);
    }
    std::printf(bad ? "ghost shift check failed\n" : "ghost shift check ok\n");
    return bad ? 1 : 0;
}
