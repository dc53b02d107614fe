// The shape in which a lattice is stepped two steps per launch (k_step2.cu); host code.
#pragma once
#include <cmath>

#include "internal.h"

namespace hlbm {

// Tile and planes per block with the least time, in phases of one plane of the 32 x 7 tile (about
// 1.75 us for a phase pair with every SM full): a block of zc planes runs zc + 2 planes of phase 1 and zc of
// phase 2, and starts and ends with a wait; a plane of the 24 x 9 tile takes 0.945 of that; the
// blocks of a single wave run in step and take 1.03; a last wave that is partly full saves a fifth of
// what is missing. Two steps, 32 x 7 / 24 x 9, us: 128^3 88.7 / 94.6, 160^3 177 / 167, 240^3
// 541 / 501, 256^3 617 / 615, 288^3 864 / 840. Over 60 lattices with two to four measured plans
// each, the plan chosen here took 0.6 % more than the best of them. Slower: 16 x 14 (256^3 671),
// and with two blocks per SM 48 x 7 (721) and 32 x 11 (651, though 163 at 160^3).
// A plan is made for each call, so the loop visits each number of planes per block once (up to
// 2 sqrt(nz) of them; 8 x 8 x 65535 cells: 7 us, with every number of blocks 73), and no tile
// whose cover of x and y alone leaves it below `need` or the best so far.
constexpr int kStep2BlocksPerSM = 3;
struct Step2Plan {
    bool wide;      // 32 x 7, else 24 x 9
    int zc;
    double useful;  // cells over the cells that the waves' blocks have room for
};
inline Step2Plan step2_plan(const LaunchCtx& c, double need = 0.0) {
    constexpr int kSlots = kStep2BlocksPerSM * 152;
    Step2Plan best{true, c.nz, 0.0};
    for (const bool wide : {true, false}) {
        const int tx = wide ? 32 : 24, ty = wide ? 7 : 9;
        const long long bxy = (long long)((c.nx + tx - 1) / tx) * ((c.ny + ty - 1) / ty);
        const double cover = (double)c.nx * c.ny / (bxy * 32 * 7 * (wide ? 1.0 : 0.945));  // useful is less than this
        if (cover < need || cover <= best.useful) continue;
        for (int zc = c.nz;;) {
            const int bz = (c.nz + zc - 1) / zc;
            const double full = (double)(bxy * bz) / kSlots, waves = std::ceil(full);
            const double turns = waves > 1.0 ? waves - 0.2 * (waves - full) : 1.03;
            const double time = turns * (2.0 * zc + 3.0) * (wide ? 1.0 : 0.945);
            const double useful = 2.0 * c.nx * c.ny * c.nz / (time * kSlots * 32 * 7);
            if (useful > best.useful) best = {wide, zc, useful};
            if (zc <= 8) break;
            const int k = (c.nz + zc - 2) / (zc - 1);  // the fewest blocks with fewer planes each
            zc = (c.nz + k - 1) / k;
        }
    }
    return best;
}

}  // namespace hlbm
