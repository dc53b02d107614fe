// The block shapes of csrc/internal.h on the CPU: every y axis that one grid of the general
// shape (whole warps of up to 128 cells, 256 threads) covers is covered by one grid of theirs.
#include <cuda_runtime.h>

#include <cstdio>

#include "internal.h"

int main() {
    int failed = 0;
    const auto check = [&](const char* rule, int nx, int ny, dim3 blk, unsigned most) {
        const unsigned grid_y = (ny + blk.y - 1) / blk.y, threads = blk.x * blk.y * blk.z;
        if (grid_y <= 65535 && threads <= most && blk.x >= 1 && blk.z == 1) return;
        if (++failed < 20) std::fprintf(stderr, "%s nx %d ny %d: block %u x %u, grid.y %u\n", rule, nx, ny, blk.x, blk.y, grid_y);
    };
    for (int nx = 1; nx <= 1100; ++nx) {
        const int general_x = nx > 96 ? 128 : (nx + 31) / 32 * 32, rows = 65535 * (256 / general_x);
        for (const int ny : {1, 2, 7, 65535, 65536, 70000, 131070, 262140, 524280}) {
            if (ny > rows) continue;
            check("row_block", nx, ny, hlbm::row_block(nx, ny), 256);
            if (nx % 2) continue;
            for (const int cap : {128, 256}) check("pair_block", nx, ny, hlbm::pair_block(nx, ny, cap), cap);
        }
    }
    return failed != 0;
}
