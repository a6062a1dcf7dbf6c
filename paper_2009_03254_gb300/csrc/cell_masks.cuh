// A block's 64 cells as 64-bit masks (bit x + 4y + 16z): from the below masks
// of a block and its +group, which corners of which cells are below the
// isovalue, and which cells the surface crosses.
#pragma once

#include <cstdint>

#include "common.cuh"
#include "kernels.cuh"

namespace bcmc {

// candidates the triangle stage visits: none once the cache update failed
// (both bits are final before the count kernel starts)
__device__ __forceinline__ uint32_t mc_candidates(const Ctl *c) {
    return (c->status & (kStatusBudget | kStatusTimeout | kStatusTimeoutLru)) ? 0u : c->n_cand;
}

// cells of a block per axis inside the volume (0 to 4), 4 bits each
__device__ __forceinline__ uint32_t cell_limits(const Geom &g, uint32_t bx, uint32_t by, uint32_t bz) {
    const uint32_t lx = min(4u, g.nx - 1 - min(g.nx - 1, 4 * bx));
    const uint32_t ly = min(4u, g.ny - 1 - min(g.ny - 1, 4 * by));
    const uint32_t lz = min(4u, g.nz - 1 - min(g.nz - 1, 4 * bz));
    return lx | (ly << 4) | (lz << 8);
}

__device__ __forceinline__ unsigned long long in_x(unsigned long long a, unsigned long long n) {   // sample (x+1, y, z)
    return ((a >> 1) & 0x7777777777777777ull) | ((n << 3) & 0x8888888888888888ull);
}
__device__ __forceinline__ unsigned long long in_y(unsigned long long a, unsigned long long n) {   // (x, y+1, z)
    return ((a >> 4) & 0x0FFF0FFF0FFF0FFFull) | ((n << 12) & 0xF000F000F000F000ull);
}
__device__ __forceinline__ unsigned long long in_z(unsigned long long a, unsigned long long n) {   // (x, y, z+1)
    return (a >> 16) | (n << 48);
}

// the corner masks m[c] of block b's cells; cells outside the volume (not in
// the returned mask `valid`) hold anything
__device__ __forceinline__ void corner_masks(const DevState &s, const Geom &g, uint32_t b, unsigned long long (&m)[8],
                                             uint32_t &lim) {
    uint32_t bx, by, bz;
    block_coords(g, b, bx, by, bz);
    const bool e[3] = {bx + 1 < g.nbx, by + 1 < g.nby, bz + 1 < g.nbz};
    lim = cell_limits(g, bx, by, bz);
    const uint32_t slab = g.nbx * g.nby;
    int32_t sl[8];
#pragma unroll
    for (int o = 0; o < 8; o++) {                        // slots of the +group, all loads first
        const bool in = (!(o & 1) || e[0]) && (!(o & 2) || e[1]) && (!(o & 4) || e[2]);
        const uint32_t id = b + ((o & 1) ? 1u : 0u) + ((o & 2) ? g.nbx : 0u) + ((o & 4) ? slab : 0u);
        sl[o] = in && in_bounds(id < g.nb, &s.ctl->status) ? s.islot[id] : -1;
    }
    unsigned long long n[8];
#pragma unroll
    for (int o = 0; o < 8; o++)
        n[o] = sl[o] >= 0 && in_bounds((uint32_t)sl[o] < s.ctl->cap, &s.ctl->status) ? s.bmask[sl[o]] : 0ull;
    const unsigned long long x23 = in_x(n[2], n[3]), x45 = in_x(n[4], n[5]), x67 = in_x(n[6], n[7]);
    m[0] = n[0];
    m[1] = in_x(n[0], n[1]);
    m[2] = in_y(n[0], n[2]);
    m[3] = in_y(m[1], x23);
    m[4] = in_z(n[0], n[4]);
    m[5] = in_z(m[1], x45);
    m[6] = in_z(m[2], in_y(n[4], n[6]));
    m[7] = in_z(m[3], in_y(x45, x67));
}

// cells with x < lim.x, y < lim.y, z < lim.z
__device__ __forceinline__ unsigned long long valid_cells(uint32_t lim) {
    if (lim == 0x444u) return ~0ull;
    const uint32_t lx = lim & 15u, ly = (lim >> 4) & 15u, lz = lim >> 8;
    return ((1ull << lx) - 1ull) * 0x1111111111111111ull & (((1ull << (4 * ly)) - 1ull) * 0x0001000100010001ull) &
           (lz >= 4u ? ~0ull : (1ull << (16 * lz)) - 1ull);
}

__device__ __forceinline__ unsigned long long crossing_cells(const unsigned long long (&m)[8],
                                                             unsigned long long valid) {
    return ((m[0] | m[1] | m[2] | m[3] | m[4] | m[5] | m[6] | m[7]) &
            ~(m[0] & m[1] & m[2] & m[3] & m[4] & m[5] & m[6] & m[7])) & valid;
}

}  // namespace bcmc
