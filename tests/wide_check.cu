// How rows of more than 32 actions are laid on lanes, for every count: each element belongs to one lane, the vectors that the
// kernels read without a look at them are there, a form of that many vectors is compiled.  Then what split launches keep in a
// workspace's spare slots.  Prints the first few that fail and returns their number (255 at most).
#include <stdio.h>

#include "impact_categorical.cuh"

using namespace impact;

int main() {
    int bad = 0;
    auto check = [&](bool ok, const char* what, int A, long long x) {
        if (!ok && bad++ < 5) printf("%s: A=%d %lld\n", what, A, x);
    };
    DeviceInfo di;
    di.sm_count = 148;
    di.max_smem_optin = 227 * 1024;
    for (int A = 33; A <= 512; ++A) {
        const int elements = wide_elements(A), vecs = A / elements, single = A % 2;
        const WideWidth w = wide_width(A);
        const int lanes = 1 << w.log_lanes, sure = elements == 4 ? w.vectors - 1 : w.vectors - 2;
        check(vecs * elements + single == A, "elements", A, elements);
        check(w.log_lanes >= 1 && w.log_lanes <= 4, "lanes", A, lanes);
        check(w.vectors * lanes >= vecs && w.vectors * elements <= 32, "vectors", A, w.vectors);
        check(sure * lanes <= vecs, "vectors that are there", A, sure);
        check(elements == 4 ? w.vectors >= 5 && w.vectors <= 8 : w.vectors >= 10 && w.vectors <= 16 && w.vectors % 2 == 0, "form", A, w.vectors);
        for (size_t in : {2, 4})
            for (size_t out : {2, 4})
                for (long long T : {20ll, 65ll, 300ll, 4096ll, 100000ll})
                    for (long long B : {1ll, 7ll, 60ll, 160ll, 5000ll}) {
                        BatchGeometry g = {};
                        g.B = B;
                        g.T = T;
                        for (bool split : {false, true}) {
                            const int nt = wide_tile_rows(g, split, A, in, out, &di), groups = split ? 3 : 4;
                            check(nt * lanes == 128 || nt * lanes == 256, "rows", A, nt);
                            LaunchShape ls;
                            check(launch_shape(g, nt, split, cat_stage_bytes(nt, A, in, out), 2 * nt * A * in, groups, &di, &ls), "shape", A, nt);
                        }
                    }
    }
    // where either way of working on few trajectories was found the faster one by a twentieth and more
    const struct { int A; long long B, T; bool split; } found[] = {
        {60, 20, 300, true}, {60, 32, 300, true}, {64, 28, 300, true}, {60, 38, 500, true}, {60, 50, 500, true}, {64, 54, 1000, true},
        {36, 50, 1000, true}, {100, 50, 300, true}, {100, 58, 1000, true}, {64, 62, 2000, true}, {64, 66, 4000, true}, {100, 20, 100, true},
        {40, 50, 300, false}, {40, 40, 200, false}, {64, 40, 200, false}, {100, 50, 100, false}, {64, 160, 100, false}, {180, 58, 100, false}};
    for (const auto& f : found) {
        BatchGeometry g = {};
        g.B = f.B;
        g.T = f.T;
        check(splits_trajectories(g, true, 128 >> wide_width(f.A).log_lanes, &di, f.A) == f.split, "split", f.A, f.B * f.T);
    }
    // (rows of one lane, tiles of 128: trajectories of three tiles stay whole, but for one or two with every switch)
    for (long long B : {1ll, 2ll, 3ll, 44ll})
        for (long long T : {200ll, 256ll, 257ll, 384ll, 385ll, 600ll})
            for (bool plain : {false, true}) {
                BatchGeometry g = {};
                g.B = B;
                g.T = T;
                check(splits_trajectories(g, true, 128, &di, 0, 0, 0, plain) == (T > (plain || B > 2 ? 384 : 256)), "split of three", (int)B, T);
            }
    printf("%d\n", bad);
    return bad > 255 ? 255 : bad;
}
