// The plan of two steps per launch (csrc/step2_plan.h) on the CPU: the best over every number of
// blocks along z, found in a fraction of the time that trying them all takes.
#include <cuda_runtime.h>

#include <chrono>
#include <cstdio>

#include "step2_plan.h"

using namespace hlbm;

static Step2Plan every_number(const LaunchCtx& c) {
    constexpr int kSlots = kStep2BlocksPerSM * 152;
    Step2Plan best{true, c.nz, 0.0};
    for (const bool wide : {true, false}) {
        const int tx = wide ? 32 : 24, ty = wide ? 7 : 9;
        const long long bxy = (long long)((c.nx + tx - 1) / tx) * ((c.ny + ty - 1) / ty);
        for (int k = 1; k <= c.nz; ++k) {
            const int zc = (c.nz + k - 1) / k, bz = (c.nz + zc - 1) / zc;
            const double full = (double)(bxy * bz) / kSlots, waves = std::ceil(full);
            const double turns = waves > 1.0 ? waves - 0.2 * (waves - full) : 1.03;
            const double useful = 2.0 * c.nx * c.ny * c.nz / (turns * (2.0 * zc + 3.0) * (wide ? 1.0 : 0.945) * kSlots * 32 * 7);
            if (useful > best.useful) best = {wide, zc, useful};
            if (zc <= 8) break;
        }
    }
    return best;
}

int main() {
    int failed = 0;
    LaunchCtx c{};
    const auto check = [&](int nx, int ny, int nz) {
        c.nx = nx, c.ny = ny, c.nz = nz;
        const Step2Plan a = step2_plan(c), b = every_number(c);
        bool same = a.wide == b.wide && a.zc == b.zc && std::fabs(a.useful - b.useful) <= 1e-12 * b.useful;
        for (const double need : {0.78, 0.83, 0.86}) same = same && (step2_plan(c, need).useful >= need) == (b.useful >= need);
        if (same) return;
        if (++failed < 10) std::fprintf(stderr, "%d x %d x %d: %d planes instead of %d\n", nx, ny, nz, a.zc, b.zc);
    };
    for (int n = 4; n < 700; ++n) check(8 + 4 * (n % 90), 4 + n % 301, n);
    for (const int n : {96, 128, 160, 192, 240, 256, 288, 384, 512}) check(n, n, n);
    for (int nz = 1000; nz <= 65535; nz += 977) check(8, 8, nz), check(32, 7, nz), check(64, 63, nz);

    c.nx = c.ny = 8, c.nz = 65535;
    double seconds[2], sink = 0.0;
    for (int k = 0; k < 2; ++k) {
        const auto t = std::chrono::steady_clock::now();
        for (int i = 0; i < 200; ++i) {
            c.nx = 8 + 4 * (i & 1);
            sink += (k ? every_number(c) : step2_plan(c)).useful;
        }
        seconds[k] = std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count();
    }
    std::fprintf(stderr, "a plan of 8 x 8 x 65535: %.1f us, with every number of blocks %.1f us (%g)\n", seconds[0] * 5e3, seconds[1] * 5e3, sink);
    return failed != 0 || seconds[0] > 0.25 * seconds[1];
}
