// Which launches take a companion, worked out on the host as the launch does: split trajectories of up to 18 actions do but for
// few large tiles, a launch whose groups have a tile each does not, and large ones up to where their companion's requests hold
// up their own.
#include <stdio.h>

#include "impact_categorical.cuh"

using namespace impact;

static int bad = 0;
static void expect(bool want, long long B, long long T, int A, size_t in, size_t out, int groups, bool split) {
    DeviceInfo di;
    di.sm_count = 148;
    di.max_smem_optin = 227 * 1024;
    BatchGeometry g = {};
    g.B = B;
    g.T = T;
    LaunchShape ls;
    bool got = !want;
    if (launch_shape(g, 128, split, cat_stage_bytes(128, A, in, out), 2 * 128 * A * in, groups, &di, &ls))
        got = ws_plan(ls.tiles, ls.grid, 128 * (2 * A * in + 20), ls.in_flight,
                      companion_pays(A, split, B * T, 2 * A * in + 20, 128, ls.tiles, ls.grid, ls.in_flight, out)).companion;
    if (got == want) return;
    ++bad;
    printf("B=%lld T=%lld A=%d in=%zu out=%zu groups=%d split=%d: %d\n", B, T, A, in, out, groups, (int)split, (int)got);
}

int main() {
    for (int A : {8, 9, 12, 16, 18}) {
        expect(A <= 12, 16, 4096, A, 4, 4, 4, true);
        expect(true, 24, 4096, A, 4, 4, 4, true);
        expect(true, 31, 4000, A, 4, 4, 4, true);
    }
    expect(true, 16, 4096, 18, 2, 2, 4, true);
    expect(true, 31, 4000, 18, 2, 2, 4, true);
    expect(false, 16, 4096, 20, 2, 2, 3, true);
    expect(false, 16, 4096, 28, 4, 4, 3, true);
    expect(true, 20, 4096, 24, 4, 4, 3, true);
    expect(false, 24, 4096, 33, 2, 2, 4, true);
    expect(false, 600, 128, 18, 4, 4, 4, false);
    expect(false, 600, 128, 9, 4, 4, 4, false);
    expect(true, 1024, 128, 18, 4, 4, 5, false);
    expect(true, 1024, 128, 18, 4, 4, 4, false);
    expect(true, 1180, 128, 18, 4, 4, 5, false);
    expect(true, 1024, 128, 20, 4, 4, 4, false);
    expect(false, 1180, 128, 20, 4, 4, 4, false);
    expect(true, 1180, 128, 20, 4, 2, 4, false);
    expect(true, 800, 128, 24, 4, 4, 4, false);
    expect(false, 900, 128, 24, 4, 4, 4, false);
    expect(true, 700, 128, 28, 4, 4, 4, false);
    expect(false, 800, 128, 28, 4, 4, 4, false);
    expect(false, 1024, 128, 32, 4, 4, 3, false);
    printf("%d wrong\n", bad);
    return bad;
}
