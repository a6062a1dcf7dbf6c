// Implicit isosurface ray casting over the block grid as a macrocell grid
// (the future work Section 4.6.2 proposes: the blocks as macrocells for
// space skipping, the isosurface of the trilinear interpolant found inside
// them), reading the decoded-block cache of Sections 4.1-4.2.
//
// iso_raycast runs the extraction's front for the isovalue (range test,
// cache update, decode: every block whose 2x2x2 group range holds the
// isovalue is active, and so is its whole group, so every sample a ray can
// need is cached, and its below mask with it), then cross_kernel finds each
// candidate's crossing cells from the masks (a bit per block, 64 bits per
// slot), and one thread per pixel (16 x 16 pixel tiles per CTA) casts its
// ray:
//   - a slab test against the volume box gives the start; the block, then
//     the cell, holding the current point starts each level;
//   - each box's interval comes from its own slab test (not an
//     incremental update; the direction's reciprocal is taken once per
//     ray), and the next box is one step along the exit axis, so the
//     visited boxes and their intervals are fixed by the ray;
//   - a block is searched when its precomputed group range (hull8) holds
//     the isovalue; a cell when its 8 corners' range does, i.e. when it is a
//     crossing cell (so blocks without any are passed by at once, and only
//     the samples of crossing cells are read): 5 samples of the trilinear
//     interpolant on its interval, then 12 bisection steps at the first
//     change of side;
//   - a step changes one coordinate, so only that axis' interval is computed
//     again, by the same operations on the same numbers;
//   - the hit is shaded from the interpolant's gradient (two-sided Lambert).
// Every float operation is one IEEE float32 operation (this file is built
// without multiply-add contraction), so the depths equal the CPU oracle's
// bit for bit.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "bcmc.h"
#include "cell_masks.cuh"
#include "volume.cuh"

namespace bcmc {

namespace {

constexpr int kTile = 16;                               // pixels per tile side (four CTAs, 8 x 4 pixels a warp)
constexpr int kCastThreads = 64;

struct CastArgs {
    const int32_t *islot;
    const float *slots;
    const uint32_t *occ;          // a bit per block: some cell crosses
    const unsigned long long *cross;   // per slot of such a block: its crossing cells
    const Ctl *ctl;
    unsigned long long *hits;
    uint32_t *rgba;
    unsigned long long *nhit;
    uint32_t *err;
    uint32_t nx, ny, nz, nbx, nby, nbz;
    uint32_t width, height;
    float iso;
    float eye[3], fwd[3], right[3], up[3], light[3];
};

struct Ray {
    float o[3], d[3], inv[3];     // inv = 1 / d (0 where d == 0: unused)
};

__device__ __forceinline__ float inf_f() { return __int_as_float(0x7f800000); }

// interval of the ray inside box [lo, hi]; false if an axis parallel to
// the ray misses it.  The exit axis is the first whose upper value is the
// interval's end (-1 if the ray is parallel to every axis).
__device__ __forceinline__ bool slab(const Ray &r, const float lo[3], const float hi[3], float &tin, float &tout,
                                     int &ax) {
    float a = -inf_f(), b = inf_f();
    ax = -1;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        if (r.d[k] == 0.0f) {
            if (r.o[k] < lo[k] || r.o[k] > hi[k]) return false;
            continue;
        }
        const float t0 = (lo[k] - r.o[k]) * r.inv[k], t1 = (hi[k] - r.o[k]) * r.inv[k];
        const float mn = t0 < t1 ? t0 : t1, mx = t0 < t1 ? t1 : t0;
        if (mn > a) a = mn;
        if (mx < b) {
            b = mx;
            ax = k;
        }
    }
    tin = a;
    tout = b;
    return true;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ float clamp01(float x) { return fminf(fmaxf(x, 0.0f), 1.0f); }

__device__ __forceinline__ float trilinear(const float c[8], float fx, float fy, float fz) {
    const float c00 = c[0] + fx * (c[1] - c[0]), c10 = c[2] + fx * (c[3] - c[2]);
    const float c01 = c[4] + fx * (c[5] - c[4]), c11 = c[6] + fx * (c[7] - c[6]);
    const float c0 = c00 + fy * (c10 - c00), c1 = c01 + fy * (c11 - c01);
    return c0 + fz * (c1 - c0);
}

__device__ __forceinline__ float g_at(const Ray &r, const float c[8], const float cell[3], float iso, float t) {
    const float fx = clamp01(r.o[0] + t * r.d[0] - cell[0]);
    const float fy = clamp01(r.o[1] + t * r.d[1] - cell[1]);
    const float fz = clamp01(r.o[2] + t * r.d[2] - cell[2]);
    return trilinear(c, fx, fy, fz) - iso;
}

__device__ __forceinline__ bool cell_root(const Ray &r, const float c[8], const float cell[3], float iso, float a, float b,
                          float &thit) {
    const float h = (b - a) * 0.25f;
    float tk = a;
    bool sk = g_at(r, c, cell, iso, tk) < 0.0f;
    for (int k = 1; k <= 4; k++) {
        const float tn = k == 4 ? b : a + h * (float)k;
        const bool sn = g_at(r, c, cell, iso, tn) < 0.0f;
        if (sn != sk) {
            float lo = tk, hi = tn;
            for (int it = 0; it < 12; it++) {
                const float m = (lo + hi) * 0.5f;
                const bool sm = g_at(r, c, cell, iso, m) < 0.0f;
                if (sm == sk) lo = m;
                else hi = m;
            }
            thit = (lo + hi) * 0.5f;
            return true;
        }
        tk = tn;
        sk = sn;
    }
    return false;
}

// The ray's interval on each axis of a box, and the box's own by slab()'s
// rule: an axis parallel to the ray bounds nothing (the caller has seen that
// it does not miss the box).
struct Axes {
    float mn[3], mx[3];
    __device__ __forceinline__ void meet(float &tin, float &tout, int &ax) const {
        float a = -inf_f(), b = inf_f();
        ax = -1;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            if (mn[k] > a) a = mn[k];
            if (mx[k] < b) {
                b = mx[k];
                ax = k;
            }
        }
        tin = a;
        tout = b;
    }
};

__device__ __forceinline__ void axis_interval(float o, float d, float inv, float lo, float hi, float &mn, float &mx) {
    const float t0 = (lo - o) * inv, t1 = (hi - o) * inv;
    mn = d == 0.0f ? -inf_f() : (t0 < t1 ? t0 : t1);
    mx = d == 0.0f ? inf_f() : (t0 < t1 ? t1 : t0);
}

// v[ax] without an indexed array
template <class T>
__device__ __forceinline__ T pick(const T v[3], int ax) {
    return ax == 0 ? v[0] : (ax == 1 ? v[1] : v[2]);
}

// The first hit of any ray; the hit cell's corners in cv.  Box by box, every
// interval from all its planes: for the rays cast() does not take.
__device__ __noinline__ bool cast_any(const CastArgs &a, const Ray &r, float &thit, float hc[3], uint32_t &hb, float cv[8]) {
    const int n[3] = {(int)a.nx, (int)a.ny, (int)a.nz};
    int ncb[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        if (n[k] < 2) return false;
        ncb[k] = (n[k] - 2) / 4 + 1;
    }
    const float vlo[3] = {0.0f, 0.0f, 0.0f};
    const float vhi[3] = {(float)(n[0] - 1), (float)(n[1] - 1), (float)(n[2] - 1)};
    float t0, t1;
    int ax;
    if (!slab(r, vlo, vhi, t0, t1, ax)) return false;
    if (t0 < 0.0f) t0 = 0.0f;
    if (!(t0 <= t1)) return false;
    int b[3];
    Axes ba;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        b[k] = clampi((int)floorf((r.o[k] + t0 * r.d[k]) * 0.25f), 0, ncb[k] - 1);
        const float lo = (float)(4 * b[k]), hi = (float)min(4 * b[k] + 4, n[k] - 1);
        if (r.d[k] == 0.0f && (r.o[k] < lo || r.o[k] > hi)) return false;   // and so for every block on the way
        axis_interval(r.o[k], r.d[k], r.inv[k], lo, hi, ba.mn[k], ba.mx[k]);
    }
    float t = t0;
    for (;;) {
        float bin, bout;
        int bax;
        ba.meet(bin, bout, bax);
        if (bax < 0) return false;
        if (bin < t) bin = t;
        const uint32_t bid = (uint32_t)b[0] + a.nbx * ((uint32_t)b[1] + a.nby * (uint32_t)b[2]);
        if (bin <= bout && ((__ldg(a.occ + (bid >> 5)) >> (bid & 31u)) & 1u)) {
            const unsigned long long cross = __ldg(a.cross + __ldg(a.islot + bid));
            int c[3];
            Axes ca;
            bool miss = false;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                c[k] = clampi((int)floorf(r.o[k] + bin * r.d[k]), 4 * b[k], min(4 * b[k] + 3, n[k] - 2));
                const float lo = (float)c[k], hi = (float)(c[k] + 1);
                miss = miss || (r.d[k] == 0.0f && (r.o[k] < lo || r.o[k] > hi));
                axis_interval(r.o[k], r.d[k], r.inv[k], lo, hi, ca.mn[k], ca.mx[k]);
            }
            while (!miss) {
                float cin, cout;
                int cax;
                ca.meet(cin, cout, cax);
                if (cax < 0) break;
                if (cin < bin) cin = bin;
                const uint32_t cell = (uint32_t)(c[0] & 3) | ((uint32_t)(c[1] & 3) << 2) | ((uint32_t)(c[2] & 3) << 4);
                if (cin <= cout && ((cross >> cell) & 1ull)) {
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const int x = c[0] + (k & 1), y = c[1] + ((k >> 1) & 1), z = c[2] + (k >> 2);
                        const int32_t sl = __ldg(a.islot + ((uint32_t)(x >> 2) + a.nbx * ((uint32_t)(y >> 2) +
                                                                                          a.nby * (uint32_t)(z >> 2))));
                        float v = 0.0f;
                        if (sl >= 0) v = __ldg(a.slots + (size_t)sl * 64 + (x & 3) + 4 * (y & 3) + 16 * (z & 3));
                        else atomicOr(a.err, 1u);       // never: every group member is cached
                        cv[k] = v;
                    }
                    const float lo[3] = {(float)c[0], (float)c[1], (float)c[2]};
                    if (cell_root(r, cv, lo, a.iso, cin, cout, thit)) {
                        hb = bid;
#pragma unroll
                        for (int k = 0; k < 3; k++) hc[k] = lo[k];
                        return true;
                    }
                }
                // one step along the exit axis (selects, not an indexed array)
                const float d = pick(r.d, cax);
                const int cn = pick(c, cax) + (d > 0.0f ? 1 : -1), c0 = 4 * pick(b, cax);
                if (cn < c0 || cn > min(c0 + 3, pick(n, cax) - 2)) break;
                float mn, mx;
                axis_interval(pick(r.o, cax), d, pick(r.inv, cax), (float)cn, (float)(cn + 1), mn, mx);
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (k == cax) {
                        c[k] = cn;
                        ca.mn[k] = mn;
                        ca.mx[k] = mx;
                    }
            }
        }
        const float d = pick(r.d, bax);
        const int bn = pick(b, bax) + (d > 0.0f ? 1 : -1);
        if (bn < 0 || bn >= pick(ncb, bax)) return false;
        float mn, mx;
        axis_interval(pick(r.o, bax), d, pick(r.inv, bax), (float)(4 * bn), (float)min(4 * bn + 4, pick(n, bax) - 1), mn, mx);
#pragma unroll
        for (int k = 0; k < 3; k++)
            if (k == bax) {
                b[k] = bn;
                ba.mn[k] = mn;
                ba.mx[k] = mx;
            }
        t = bout;
    }
}

// A ray's place on one level of the grid (blocks, or the cells of one
// block): per axis the plane the current box is left through, the ray's
// parameter there and the boxes left on that side; the box's entry, and its
// index (block id, or the cell's bit).
struct Place {
    float plane[3], exit[3], entry;
    int left[3], index;
};

// The first hit of the ray; the hit cell's corners in cv and its low corner
// in hc.  Called by all lanes of a warp (`live`: this lane has a ray).  For
// rays whose reciprocals are finite in volumes whose coordinates are exact in
// float32: no interval is NaN, on every axis a box's entry value is at most
// its exit value, and the next box's entry value along the exit axis is this
// box's exit value.  So a box's entry is the larger of the last box's entry
// and exit, and a step computes one new exit, by axis_interval()'s operations.
//
// One loop steps blocks and cells alike, so that the lanes of a warp step
// together whichever they are at.  A lane at a block to be searched waits
// until a quarter of the warp's rays do (or none steps), and then all such
// lanes go into their blocks; a lane at a crossing cell waits for half of
// them, and then the cells' roots are looked for together.  (Waiting for all
// of them adds up the longest paths of every stage: 3000 steps for a warp
// whose longest ray takes 300.)
// Bound by instruction issue (14 of 32 lanes step at a time) and, at the end,
// by the latency of the longest rays (68% of issue slots; the benchmark's view
// of 384^3 noise, 534 M warp instructions, takes 810 us).  1080p over another
// 384^3 noise volume, where the variants were timed: 588 us; nested loops that tested every cell's samples took 1080 and had 6 lanes
// active.  Picking the stepped axis' numbers by selects instead of a branch
// per axis took 650.
__device__ __forceinline__ bool cast(const CastArgs &a, const Ray &r, bool live, float &thit, float hc[3], uint32_t &hb,
                                     float cv[8]) {
    const int n[3] = {(int)a.nx, (int)a.ny, (int)a.nz};
    if (n[0] < 2 || n[1] < 2 || n[2] < 2) return false;
    const float vlo[3] = {0.0f, 0.0f, 0.0f};
    const float vhi[3] = {(float)(n[0] - 1), (float)(n[1] - 1), (float)(n[2] - 1)};
    float t0 = 0.0f, t1 = 0.0f;
    int ax;
    if (!slab(r, vlo, vhi, t0, t1, ax)) live = false;
    if (t0 < 0.0f) t0 = 0.0f;
    if (!(t0 <= t1)) live = false;
    const int stride[3] = {1, (int)a.nbx, (int)(a.nbx * a.nby)};
    Place w, blk;                                          // where the ray is; its block while it is in the cells
    w.entry = -inf_f();
    w.index = 0;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int last = (n[k] - 2) / 4, b = clampi((int)floorf((r.o[k] + t0 * r.d[k]) * 0.25f), 0, last);
        const bool up = r.d[k] > 0.0f;
        const float lo = (float)(4 * b), hi = (float)min(4 * b + 4, n[k] - 1);
        if (r.d[k] == 0.0f && (r.o[k] < lo || r.o[k] > hi)) live = false;   // and so for every block on the way
        float mn;
        axis_interval(r.o[k], r.d[k], r.inv[k], lo, hi, mn, w.exit[k]);
        if (mn > w.entry) w.entry = mn;
        w.plane[k] = (float)(up ? 4 * b + 4 : 4 * b);
        w.left[k] = up ? last - b : b;
        w.index += b * stride[k];
    }
    if (w.entry < t0) w.entry = t0;
    blk = w;
    bool found = false, cells = false, searched = false;   // searched: this block is done, step on
    unsigned long long cross = 0;
    float tout = 0.0f;
    auto step = [&]() {
        const bool p0 = w.exit[0] == tout, p1 = !p0 && w.exit[1] == tout;   // the first axis with the smallest exit
        const float size = cells ? 1.0f : 4.0f;
        if (w.entry < tout) w.entry = tout;
        int out = 0;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const bool go = k == 0 ? p0 : (k == 1 ? p1 : (!p0 && !p1));
            const bool up = r.d[k] > 0.0f;
            if (go) {
                w.plane[k] = __fadd_rn(w.plane[k], up ? size : -size);
                w.exit[k] = (fminf(w.plane[k], vhi[k]) - r.o[k]) * r.inv[k];
                w.left[k] -= 1;
                out = w.left[k];
                const int by = cells ? 1 << (2 * k) : stride[k];
                w.index += up ? by : -by;
            }
        }
        if (out < 0 || !(tout < inf_f())) {
            if (cells) {                                   // out of the block's cells: back to the block
                w = blk;
                cells = false;
                searched = true;
            } else {
                live = false;
            }
        }
    };
    bool root = false, enter = false;                      // what the lane waits for
    for (;;) {
        if (live && !root && !enter) {
            tout = fminf(fminf(w.exit[0], w.exit[1]), w.exit[2]);
            const bool inside = w.entry <= tout;
            if (cells) root = inside && ((cross >> w.index) & 1ull);
            else enter = !searched && inside && ((__ldg(a.occ + ((uint32_t)w.index >> 5)) >> (w.index & 31)) & 1u);
            if (!(tout < inf_f())) root = enter = false;       // parallel to every axis: step() ends the search
            if (!root && !enter) {
                if (!cells) searched = false;
                step();
            }
        }
        const uint32_t rays = __ballot_sync(0xffffffffu, live), at_cell = __ballot_sync(0xffffffffu, root),
                       at_block = __ballot_sync(0xffffffffu, enter);
        if (!rays) return found;
        const bool stuck = rays == (at_cell | at_block);
        if (at_block && (stuck || 4 * __popc(at_block) >= __popc(rays))) {
            if (enter) {
                enter = false;
                cross = __ldg(a.cross + __ldg(a.islot + w.index));
                blk = w;
                float entry = -inf_f();
                bool miss = false;
                int bit = 0;
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const bool up = r.d[k] > 0.0f;
                    const int b4 = (int)w.plane[k] - (up ? 4 : 0), last = min(b4 + 3, n[k] - 2);
                    const int q = clampi((int)floorf(r.o[k] + blk.entry * r.d[k]), b4, last);
                    const float lo = (float)q, hi = (float)(q + 1);
                    miss = miss || (r.d[k] == 0.0f && (r.o[k] < lo || r.o[k] > hi));
                    float mn;
                    axis_interval(r.o[k], r.d[k], r.inv[k], lo, hi, mn, w.exit[k]);
                    if (mn > entry) entry = mn;
                    w.plane[k] = up ? hi : lo;
                    w.left[k] = up ? last - q : q - b4;
                    bit += (q - b4) << (2 * k);
                }
                w.index = bit;
                w.entry = entry < blk.entry ? blk.entry : entry;
                cells = !miss;
                if (miss) {
                    w = blk;
                    searched = true;
                }
            }
            continue;
        }
        if (at_cell && (stuck || 2 * __popc(at_cell) >= __popc(rays)) && root) {
            root = false;
            float lo[3];
            int c[3];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                lo[k] = w.plane[k] - (r.d[k] > 0.0f ? 1.0f : 0.0f);
                c[k] = (int)lo[k];
            }
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int x = c[0] + (k & 1), y = c[1] + ((k >> 1) & 1), z = c[2] + (k >> 2);
                const int32_t sl = __ldg(a.islot + ((uint32_t)(x >> 2) + a.nbx * ((uint32_t)(y >> 2) +
                                                                                  a.nby * (uint32_t)(z >> 2))));
                float v = 0.0f;
                if (sl >= 0) v = __ldg(a.slots + (size_t)sl * 64 + (x & 3) + 4 * (y & 3) + 16 * (z & 3));
                else atomicOr(a.err, 1u);               // never: every group member is cached
                cv[k] = v;
            }
            if (cell_root(r, cv, lo, a.iso, w.entry, tout, thit)) {
                found = true;
                live = false;
                hb = (uint32_t)blk.index;
#pragma unroll
                for (int k = 0; k < 3; k++) hc[k] = lo[k];
            } else {
                step();
            }
        }
    }
}

// The crossing cells of every candidate (blocks without one are not marked),
// a candidate per thread; `occ` was cleared.
__global__ void __launch_bounds__(256) cross_kernel(DevState s, Geom g, uint32_t *occ, unsigned long long *cross) {
    const uint32_t n = mc_candidates(s.ctl);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t b = s.icand[i];
        unsigned long long m[8];
        uint32_t lim;
        corner_masks(s, g, b, m, lim);
        const unsigned long long x = crossing_cells(m, valid_cells(lim));
        const int32_t sl = s.islot[b];
        if (x && sl >= 0) {
            cross[sl] = x;
            atomicOr(occ + (b >> 5), 1u << (b & 31u));
        }
    }
}

__global__ void __launch_bounds__(kCastThreads) raycast_kernel(CastArgs a) {
    if (a.ctl->status & (kStatusBudget | kStatusAnyTimeout)) return;   // the cache update failed
    const uint32_t tiles_x = (a.width + kTile - 1) / kTile;
    // a warp takes 8 x 4 pixels of the tile: nearby rays take similar steps
    constexpr uint32_t kParts = kTile * kTile / kCastThreads;
    const uint32_t tile = blockIdx.x / kParts, w = (blockIdx.x % kParts) * (kCastThreads / 32) + (threadIdx.x >> 5),
                   l = threadIdx.x & 31u;
    const int i = (int)((tile % tiles_x) * kTile + 8 * (w & 1u) + (l & 7u));
    const int j = (int)((tile / tiles_x) * kTile + 4 * (w >> 1) + (l >> 3));
    const bool inside = i < (int)a.width && j < (int)a.height;
    bool hit = false;
    {
        const float u = ((float)i + 0.5f) / (float)a.width * 2.0f - 1.0f;
        const float v = ((float)j + 0.5f) / (float)a.height * 2.0f - 1.0f;
        Ray r;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            r.o[k] = a.eye[k];
            r.d[k] = a.fwd[k] + u * a.right[k] + v * a.up[k];
            r.inv[k] = r.d[k] == 0.0f ? 0.0f : 1.0f / r.d[k];
        }
        const size_t px = (size_t)j * a.width + i;
        float t, cv[8];
        float c[3];
        uint32_t b;
        bool regular = max(max(a.nx, a.ny), a.nz) < (1u << 24);
#pragma unroll
        for (int k = 0; k < 3; k++) regular = regular && fabsf(r.inv[k]) < inf_f() && fabsf(r.d[k]) < inf_f();
        hit = cast(a, r, inside && regular, t, c, b, cv);
        if (inside && !regular) hit = cast_any(a, r, t, c, b, cv);
        if (!inside) {
        } else if (!hit) {
            a.hits[px] = ~0ull;
            if (a.rgba) a.rgba[px] = 0u;
        } else {
            a.hits[px] = ((unsigned long long)__float_as_uint(t) << 32) | b;
            if (a.rgba) {
                const float base[3] = {0.85f, 0.75f, 0.55f};
                const float l2 = a.light[0] * a.light[0] + a.light[1] * a.light[1] + a.light[2] * a.light[2];
                const float linv = 1.0f / sqrtf(l2);
                const float L[3] = {a.light[0] * linv, a.light[1] * linv, a.light[2] * linv};
                const float fx = clamp01(r.o[0] + t * r.d[0] - c[0]);
                const float fy = clamp01(r.o[1] + t * r.d[1] - c[1]);
                const float fz = clamp01(r.o[2] + t * r.d[2] - c[2]);
                const float gx = (1.0f - fz) * ((1.0f - fy) * (cv[1] - cv[0]) + fy * (cv[3] - cv[2])) +
                                 fz * ((1.0f - fy) * (cv[5] - cv[4]) + fy * (cv[7] - cv[6]));
                const float gy = (1.0f - fz) * ((1.0f - fx) * (cv[2] - cv[0]) + fx * (cv[3] - cv[1])) +
                                 fz * ((1.0f - fx) * (cv[6] - cv[4]) + fx * (cv[7] - cv[5]));
                const float gz = (1.0f - fy) * ((1.0f - fx) * (cv[4] - cv[0]) + fx * (cv[5] - cv[1])) +
                                 fy * ((1.0f - fx) * (cv[6] - cv[2]) + fx * (cv[7] - cv[3]));
                const float n2 = gx * gx + gy * gy + gz * gz;
                float inten = 0.2f;
                if (n2 > 0.0f) {
                    const float cth = fabsf(gx * L[0] + gy * L[1] + gz * L[2]) / sqrtf(n2);
                    inten = 0.2f + 0.8f * cth;
                    if (inten > 1.0f) inten = 1.0f;
                }
                uint32_t out = 255u << 24;
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const float x = inten * base[k] * 255.0f + 0.5f;
                    out |= ((uint32_t)x & 255u) << (8 * k);
                }
                a.rgba[px] = out;
            }
        }
    }
    const uint32_t nh = __reduce_add_sync(0xffffffffu, hit ? 1u : 0u);
    if ((threadIdx.x & 31) == 0 && nh) atomicAdd(a.nhit, (unsigned long long)nh);
}

}  // namespace

}  // namespace bcmc

extern "C" int iso_raycast(iso_volume *v, float isovalue, const iso_pinhole *cam, uint64_t *d_hits, uint32_t *d_rgba,
                           iso_raycast_stats *stats) {
    using namespace bcmc;
    using namespace bcmc_host;
    NvtxRange nvtx("iso_raycast");
    if (!v || !cam || !d_hits || !std::isfinite(isovalue) || cam->width == 0 || cam->height == 0 ||
        cam->width > 32768 || cam->height > 32768 || misaligned(d_hits, 8) || misaligned(d_rgba, 4))
        return ISO_ERR_INVALID_ARG;
    const float *vecs[5] = {cam->eye, cam->forward, cam->right, cam->up, cam->light};
    for (const float *p : vecs)
        for (int k = 0; k < 3; k++)
            if (!std::isfinite(p[k])) return ISO_ERR_INVALID_ARG;
    const double l2 = (double)cam->light[0] * cam->light[0] + (double)cam->light[1] * cam->light[1] +
                      (double)cam->light[2] * cam->light[2];
    if (!(l2 > 1e-30) || !(l2 < 1e30)) return ISO_ERR_INVALID_ARG;
    DeviceGuard dg(v->device);
    ISO_CK_RC(finish_upload(v));
    cudaStream_t st = v->stream;
    // the extraction's front for this isovalue: range test, cache update, decode
    *v->host_params = Params{isovalue, kVertexFloat4, 0u, 0u, 0u, 0u, 0ull, 0ull, 0ull, 0ull, 0ull};
    ISO_CK(cudaMemcpyAsync(&v->s.ctl->params, v->host_params, sizeof(Params), cudaMemcpyHostToDevice, st));
    const Launch L{nullptr, 1u, single_counters(v), VolEntry{v->s, v->g, v->n_cull_desc, v->n_lru_desc}};
    launch_front(L, v->plan, st, nullptr);
    // counters, then a bit per block.  The slots' crossing cells go where an
    // extraction keeps its occupied candidates' (no emission follows, and there
    // are as many entries as slots), so a cast holds next to nothing of its own
    void *scratch = nullptr;
    const size_t occ_at = 256, occ_bytes = ((size_t)v->g.nb + 31) / 32 * 4;
    int rc = dalloc_bytes(&scratch, occ_at + occ_bytes, v->device, st);
    if (rc) return rc;
    uint32_t *occ = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + occ_at);
    unsigned long long *cross = v->s.ocross;
    CastArgs a{};
    a.islot = v->s.islot;
    a.slots = v->s.slots;
    a.occ = occ;
    a.cross = cross;
    a.ctl = v->s.ctl;
    a.hits = reinterpret_cast<unsigned long long *>(d_hits);
    a.rgba = d_rgba;
    a.nhit = static_cast<unsigned long long *>(scratch);
    a.err = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + 8);
    a.nx = v->g.nx;
    a.ny = v->g.ny;
    a.nz = v->g.nz;
    a.nbx = v->g.nbx;
    a.nby = v->g.nby;
    a.nbz = v->g.nbz;
    a.width = cam->width;
    a.height = cam->height;
    a.iso = isovalue;
    for (int k = 0; k < 3; k++) {
        a.eye[k] = cam->eye[k];
        a.fwd[k] = cam->forward[k];
        a.right[k] = cam->right[k];
        a.up[k] = cam->up[k];
        a.light[k] = cam->light[k];
    }
    unsigned long long counters[2] = {0, 0};
    cudaError_t e = cudaMemsetAsync(scratch, 0, occ_at + occ_bytes, st);
    if (e == cudaSuccess) {
        cross_kernel<<<v->plan.mc_scan, 256, 0, st>>>(v->s, v->g, occ, cross);
        const uint32_t tiles = ((cam->width + kTile - 1) / kTile) * ((cam->height + kTile - 1) / kTile);
        raycast_kernel<<<tiles * (kTile * kTile / kCastThreads), kCastThreads, 0, st>>>(a);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(v->host_ctl, v->s.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(counters, scratch, 16, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    dfree_on(scratch, st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? ISO_ERR_OOM : ISO_ERR_CUDA;
    }
    keep_pass(v, *v->host_ctl, false);               // (no triangles are counted)
    v->last_tris = 0;
    rc = status_to_error(v, v->host_ctl->status);
    if (rc) return rc;
    if ((uint32_t)(counters[1] & 0xFFFFFFFFu)) return ISO_ERR_CUDA;
    if (stats) {
        stats->hits = counters[0];
        stats->n_active = v->host_ctl->n_active;
        stats->n_new = v->host_ctl->n_new;
        stats->n_slots = v->host_ctl->S;
    }
    return ISO_OK;
}
