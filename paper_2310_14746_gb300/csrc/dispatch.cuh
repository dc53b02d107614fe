// Host-side helpers of the kernels over a stored state (observables, reductions,
// state conversion): geometry, force coefficients, and the dispatch from a
// launch's run-time settings to template arguments.
#pragma once
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"

namespace hlbm {

static Geometry geom(const LaunchCtx& c) {
    return Geometry{c.nx, c.ny, c.nz, c.wall[0], c.wall[1], c.wall[2], (size_t)c.nx * c.ny * c.nz};
}

template <class C, int Q>
static Phys<C> phys(const LaunchCtx& c) {
    return make_phys<C, Q>(c.tau, c.F);
}

// The layout as a template argument while 32-bit indices fit, else -1.
template <class Fn>
static void with_layout(size_t values, int lay, Fn&& fn) {
    if (values >= ((size_t)1 << 31)) fn.template operator()<-1>();
    else if (lay == NATURAL) fn.template operator()<NATURAL>();
    else if (lay == STREAMED) fn.template operator()<STREAMED>();
    else fn.template operator()<SWAPPED>();
}

// ---------------------------------------------------------------------------
// dispatch on (q, storage, walls)
// ---------------------------------------------------------------------------
template <int Q, class S, class Fn>
static cudaError_t with_walls(const LaunchCtx& c, Fn&& fn) {
    const bool walls = c.wall[0] || c.wall[1] || c.wall[2] || c.links;
    return walls ? fn.template operator()<Q, S, true>() : fn.template operator()<Q, S, false>();
}
template <int Q, class Fn>
static cudaError_t with_storage(const LaunchCtx& c, Fn&& fn) {
    switch (c.storage) {
        case 0: return with_walls<Q, StoreF64>(c, fn);
        case 1: return with_walls<Q, StoreF32>(c, fn);
        case 2: return with_walls<Q, StoreF16>(c, fn);
        case 3: return with_walls<Q, StoreBF16>(c, fn);
    }
    return cudaErrorInvalidValue;
}
template <class Fn>
static cudaError_t dispatch(const LaunchCtx& c, Fn&& fn) {
    if (c.q == 9) return with_storage<9>(c, fn);
    if (c.q == 19) return with_storage<19>(c, fn);
    return cudaErrorInvalidValue;
}


}  // namespace hlbm
