// Triangle stage (paper Sections 4.3-4.5) over the candidate blocks, in
// the paper's two passes.
//
// Candidates are the active blocks whose 2x2x2 "+group" (the block and its
// +x/+y/+z face, edge and corner neighbours, the only blocks its cells
// read) has a range containing the isovalue; any block with a crossing
// cell is one (its cell's below and above corners lie in the +group), so
// no triangle is lost, and every +neighbour of a candidate is itself
// active and therefore cached.  This is the refinement Section 4.4 notes
// as possible ("checking which side the neighbor was on").
//
//   count and scan   Section 4.4, one pass, one candidate per thread: from
//           the 64-bit below masks of its +group (made by the decode for
//           the new blocks and by lru_b for the cached ones) each
//           candidate's triangle count, by bit logic on all 64 cells at
//           once; the counts' prefix sums (block offsets and the total) and
//           the compaction of the occupied candidates, by decoupled
//           look-backs side by side
//   emit    Section 4.5, over the occupied candidates only: stage the
//           samples, classify, list the triangles, then one vertex per lane
//
// Emit gives each warp 4 consecutive occupied candidates at a time (a "warp
// tile") and no warp ever waits for another one:
//   A  slots of each block's 8 blocks of the +group (8 lanes per block),
//      loaded two tiles ahead
//   B  stage the samples in shared memory by asynchronous copies, one tile
//      ahead, a sample per lane: the 5x5x5 window of each block unpadded
//      (sample (x, y, z) at x + 5y + 25z)
//   C  list the crossing cells (the count kept a mask of them), then, one of
//      them per lane, take their cases from their eight samples and list
//      their triangles in order
//   D  write: lane by output vertex, so that every store of the warp is 512
//      contiguous bytes without passing through shared memory: the vertex's
//      triangle from the list, its edge from the case table, two samples
//
// Over a batch, warp tiles are numbered volume after volume; a warp tile
// never spans two volumes.
//
// Indexed mesh (the alternative output Section 4.5 mentions: vertices
// shared within a block).  A block's vertices are the cut edges of its
// 5x5x5 window: edges between two window samples, exactly one of them
// below the isovalue, that belong to at least one of the block's cells
// inside the volume.  The case table uses every cut edge of a cell, so
// these are exactly the edges the block's triangles use.  An edge is named
// by its axis a and lower sample s = x + 5y + 25z; a block's vertices are
// ordered by a, then s.  The cut edges of one axis form a 125-bit mask:
// the below mask XOR itself shifted by the axis step (1, 5, 25), limited
// to the window; lane 4a + r of a warp holds word r of axis a.  Count adds
// the number of cut edges, scan a third prefix sum, and emit lists the
// tile's vertices in shared memory, computes one vertex per lane (the
// triangle soup's arithmetic) and writes each triangle corner as its
// edge's rank: the vertices before its word plus a popcount.
#include <algorithm>
#include <cstdint>

#include <cuda_fp16.h>

#include "common.cuh"
#include "kernels.cuh"
#include "cell_masks.cuh"
#include "launch.cuh"
#include "mc_tables.cuh"
#include "tile_scan.cuh"

namespace bcmc {

namespace {

constexpr int kBPW = kTileBlocks;                     // blocks per warp tile
constexpr int kTmap = 256;                            // triangles the list holds (32 cells have at most 160)
constexpr int kCells = kBPW * 64;                     // crossing cells a tile can have
constexpr int kVmap = 2 * kTmap + kCells;             // indexed meshes: vertices the same memory holds
constexpr int kWinWords = 3 * 6 * 4;                  // window rows (indexed meshes), then
constexpr int kWinTable = kWinWords + 32;             // a per-lane word for blocks inside the volume
constexpr uint32_t kNoBlock = 0xFFFFFFFFu;

// One warp's shared-memory area: two tiles' samples and lists (one being
// copied in while the other is used), the crossing cells and the triangle
// list.
template <bool kIdx>
struct EmitWarp {
    float halo[2][kBPW][kWindow];
    alignas(16) unsigned long long cross[2][kBPW];    // the blocks' crossing cells
    unsigned long long first[2][2];                   // the tile's first triangle and first vertex
    uint32_t bid[2][kBPW];
    // table row (byte offset) | q << 13 | byte offset of the cell's lower corner in the tile's windows << 16
    alignas(16) uint32_t tmap[kTmap];
    uint16_t cells[kCells];                           // crossing cells in order: place of the lower corner | q << 11
    // indexed: per block, the 12 cut-edge words, then (from word 12) the
    // vertices of the tile before each word; cells per axis inside the volume
    uint32_t cut[kIdx ? kBPW : 1][kIdx ? 24 : 2];
    uint32_t lim[kIdx ? 2 : 1][kIdx ? kBPW : 2];
};

template <bool kIdx>
struct EmitTab {                                      // a CTA's copy of what it reads of EmitTables
    uint16_t info[256];
    uint16_t corner[kCaseTriangles][4];
    uint16_t coord[kIdx ? 4 : kBPW * kWindow][4];
};

template <int kW, bool kIdx>                          // kW warps per CTA
struct EmitSmem {
    EmitWarp<kIdx> w[kW];
    EmitTab<kIdx> tab;
    uint32_t win[kIdx ? kWinTable : 4];               // window rows
    // a batch's kMaxBatch + 1 prefix words follow, as many as it has volumes
};

// Copy job of window sample j (0..124): the +group member it lies in (3) |
// its float offset inside that block (6) << 3.
__device__ __forceinline__ uint32_t halo_job(int j) {
    const int x = j % 5, y = (j / 5) % 5, z = j / 25;
    return (x >> 2) | ((y >> 2) << 1) | ((z >> 2) << 2) | (uint32_t)(((x & 3) + 4 * (y & 3) + 16 * (z & 3)) << 3);
}

// Per-lane constants.
struct LaneConst {
    uint32_t job[4];                    // copy jobs of samples lane + 32r
    uint32_t cell[2];                   // place of the lower corners of cells lane and lane + 32
    __device__ __forceinline__ void init(int lane) {
#pragma unroll
        for (int r = 0; r < 4; r++) job[r] = halo_job(min(lane + 32 * r, kWindow - 1));
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int c = lane + 32 * h;
            cell[h] = (c & 3) + 5 * ((c >> 2) & 3) + 25 * (c >> 4);
        }
    }
};

// 16-byte global -> shared copy that completes asynchronously; `dst` is a
// shared-window address
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest group
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ uint32_t shared_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 8 and 4 bytes
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(gmem) : "memory");
}
// `off` bytes into shared memory at `base`
template <class T>
__device__ __forceinline__ const T &at(const void *base, uint32_t off) {
    return *reinterpret_cast<const T *>(static_cast<const char *>(base) + off);
}

// the 128-bit below-iso mask of a staged block: bit i of word r says
// sample s = 32r + i (s = x + 5y + 25z, s < 125) is below the isovalue
__device__ __forceinline__ void below_mask(const float *hb, float iso, uint32_t m[4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int i = lane + 32 * r;
        m[r] = __ballot_sync(0xffffffffu, i < kWindow && hb[i] < iso);
    }
}

// Window rows: word r of row k of axis a has bit i set when sample
// s = 32r + i (s < 125) has coordinate <= k - 1 along a (row 0: none).
__host__ __device__ constexpr uint32_t window_row_word(int a, int k, int r) {
    uint32_t w = 0;
    for (int i = 0; i < 32; i++) {
        const int s = 32 * r + i, c = a == 0 ? s % 5 : (a == 1 ? (s / 5) % 5 : s / 25);
        if (s < 125 && c <= k - 1) w |= 1u << i;
    }
    return w;
}

// copy of the window rows into shared memory (word a*24 + k*4 + r), then
// at word 72 + lane the window word lane_cut_word takes for a block with
// all its cells inside the volume (0 for lanes 12-31)
__device__ __forceinline__ void load_window_rows(uint32_t *win) {
    for (int i = threadIdx.x; i < kWinTable; i += blockDim.x) {
        if (i < kWinWords) {
            win[i] = window_row_word(i / 24, (i / 4) % 6, i % 4);
        } else {
            const int k = i - kWinWords, a = k >> 2, r = k & 3;
            win[i] = k < 12 ? window_row_word(0, a == 0 ? 4 : 5, r) & window_row_word(1, a == 1 ? 4 : 5, r) &
                                  window_row_word(2, a == 2 ? 4 : 5, r)
                            : 0u;
        }
    }
}

// This lane's word of a block's cut edges (lanes 0-11: axis lane / 4,
// word lane % 4; 0 in the other lanes), from the block's below mask m: bit
// i is set when the edge from sample 32r + i along axis a (steps 1, 5, 25)
// crosses the isovalue and belongs to one of the block's cells inside the
// volume (lim: cells per axis inside, 4 bits each).  Such an edge exists
// when every axis has a cell; its samples lie in [0, l] on the other axes
// and it starts below l along its own.
__device__ __forceinline__ uint32_t lane_cut_word(const uint32_t m[4], uint32_t lim, const uint32_t *win) {
    const int lane = threadIdx.x & 31, a = min(lane >> 2, 2), r = lane & 3;
    const uint32_t lo = (r & 2) ? ((r & 1) ? m[3] : m[2]) : ((r & 1) ? m[1] : m[0]);
    const uint32_t hi = (r & 2) ? ((r & 1) ? 0u : m[3]) : ((r & 1) ? m[2] : m[1]);
    const uint32_t far = __funnelshift_r(lo, hi, a == 0 ? 1 : (a == 1 ? 5 : 25));   // bit i: sample s + step
    uint32_t w;
    if (lim == 0x444u) {                                // warp-uniform: the common case
        w = win[kWinWords + lane];
    } else {
        const uint32_t lx = lim & 15u, ly = (lim >> 4) & 15u, lz = lim >> 8;
        w = win[(a == 0 ? lx : lx + 1) * 4 + r] & win[24 + (a == 1 ? ly : ly + 1) * 4 + r] &
            win[48 + (a == 2 ? lz : lz + 1) * 4 + r];
        w = (lane < 12 && lx && ly && lz) ? w : 0u;
    }
    return (lo ^ far) & w;
}

}  // namespace

// ================================================================ count and scan (Section 4.4)
//
// One candidate per thread.  Its 64 cells are handled together as 64-bit
// masks: corner c's mask says, per cell, whether that corner is below the
// isovalue; the eight masks are the block's own below mask and its
// neighbours' shifted in.  A crossing cell's triangles follow from its
// corners without the table.  Its segments link into C cycles through its E
// cut edges, and a cycle of length l is fanned into l - 2 triangles: E - 2C.
// The cycles separate the regions of the cube's surface, one fewer than
// there are regions: C = B + A - 1 with B the groups of below corners joined
// by cube edges and A those of above corners joined by edges and face
// diagonals (a face with two diagonal below corners cuts each off on its
// own).  With k below corners and J edges between them, E = 3k - 2J and
// B = k - J + (the cycles of those edges), which leaves
//   k - 2 (cycles of the below edges) - 2 (A - 1):
// the cycles are the faces with all four corners below (F), and the ring of
// six around two opposite above corners (H), where A is 2:  k - 2F - 4H.
// Over 64 cells the terms are carry-save sums of masks and five popcounts.
//
// The counting reads 8 bytes a block of each +group (L2 holds most of them)
// instead of staging 5x5x5 samples.  Three loads in a row and these
// instructions bound it: with E and C counted edge by edge (44 popcounts, at a
// quarter of the rate) the 411 k candidates of a 384^3 channel took 8.25
// million instructions and a tile of three rounds (768 candidates) 7 to 14 us,
// now 6.35 and 6.

__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) { return lop3<0x96>(a, b, c); }
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return lop3<0xE8>(a, b, c); }

// triangles of 32 cells with corner masks m; sets the crossing cells
__device__ __forceinline__ int count_triangles32(const uint32_t (&m)[8], uint32_t valid, uint32_t &cross) {
    // faces (d, side) with all corners below, and their count as bits s, tw
    // (at most three in a crossing cell)
    const uint32_t p01 = m[0] & m[1], p23 = m[2] & m[3], p45 = m[4] & m[5], p67 = m[6] & m[7];
    const uint32_t f0 = m[0] & m[2] & m[4] & m[6], f1 = m[1] & m[3] & m[5] & m[7];
    const uint32_t f2 = p01 & p45, f3 = p23 & p67, f4 = p01 & p23, f5 = p45 & p67;
    const uint32_t sa = xor3(f0, f1, f2), sb = xor3(f3, f4, f5);
    const uint32_t s = sa ^ sb, tw = (maj3(f0, f1, f2) | maj3(f3, f4, f5)) | (sa & sb);
    cross = (m[0] | m[1] | m[2] | m[3] | m[4] | m[5] | m[6] | m[7]) & ~(f4 & f5) & valid;
    // below corners as bits o, t, f
    const uint32_t oa = xor3(m[0], m[1], m[2]), ob = xor3(m[3], m[4], m[5]), oc = xor3(oa, ob, m[6]);
    const uint32_t ta = maj3(m[0], m[1], m[2]), tb = maj3(m[3], m[4], m[5]), tc = maj3(oa, ob, m[6]);
    const uint32_t td = oc & m[7], te = xor3(ta, tb, tc);
    const uint32_t o = oc ^ m[7], t = te ^ td, f = maj3(ta, tb, tc) ^ (te & td);
    const uint32_t ring = f & t & ~o & ~(s | tw);
    return __popc(o & cross) + 2 * (__popc(t & cross) - __popc(s & cross)) +
           4 * (__popc(f & ~ring & cross) - __popc(tw & cross));
}

__device__ __forceinline__ uint32_t count_triangles(const unsigned long long (&m)[8], unsigned long long valid,
                                                    unsigned long long &cross) {
    uint32_t lo[8], hi[8], clo, chi;
#pragma unroll
    for (int c = 0; c < 8; c++) {
        lo[c] = (uint32_t)m[c];
        hi[c] = (uint32_t)(m[c] >> 32);
    }
    const int n = count_triangles32(lo, (uint32_t)valid, clo) + count_triangles32(hi, (uint32_t)(valid >> 32), chi);
    cross = ((unsigned long long)chi << 32) | clo;
    return (uint32_t)n;
}

// the cut edges of the block's 5x5x5 window: a cell counts its three edges at
// its lower corner and, as the last one along an axis, those on its far side
__device__ __forceinline__ uint32_t count_vertices(const unsigned long long (&m)[8], unsigned long long valid,
                                                   uint32_t lim) {
    unsigned long long last[3];
    if (lim == 0x444u) {
        last[0] = 0x8888888888888888ull;
        last[1] = 0xF000F000F000F000ull;
        last[2] = 0xFFFF000000000000ull;
    } else {
        const uint32_t lx = lim & 15u, ly = (lim >> 4) & 15u, lz = lim >> 8;
        if (!lx || !ly || !lz) return 0u;
        last[0] = valid & ~valid_cells(lim - 1u);
        last[1] = valid & ~valid_cells(lim - 16u);
        last[2] = valid & ~valid_cells(lim - 256u);
    }
    uint32_t n = 0;
#pragma unroll
    for (int half = 0; half < 2; half++) {
        uint32_t e[4][3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int p = (a + 1) % 3, q = (a + 2) % 3;  // the other two axes
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int c = ((k & 1) << p) | ((k >> 1) << q);
                unsigned long long w = (m[c] ^ m[c | (1 << a)]) & valid;
                if (k & 1) w &= last[p];
                if (k & 2) w &= last[q];
                e[k][a] = (uint32_t)(w >> (32 * half));
            }
        }
        uint32_t o[4], t[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            o[k] = xor3(e[k][0], e[k][1], e[k][2]);
            t[k] = maj3(e[k][0], e[k][1], e[k][2]);
        }
        n += __popc(xor3(o[0], o[1], o[2])) + __popc(o[3]) +
             2 * (__popc(maj3(o[0], o[1], o[2])) + __popc(xor3(t[0], t[1], t[2])) + __popc(t[3])) +
             4 * __popc(maj3(t[0], t[1], t[2]));
    }
    return n;
}

// Tiles of at most kCountTile candidates, smaller ones while that gives more
// CTAs a tile (the counting outweighs the look-backs: 11.8 -> 6.7 us for a
// 64^3 sphere, 24.4 -> 18.9 for 397 x 301 x 259 noise, the same where every
// CTA had a tile before): counts, the tile's prefixes from up to three
// look-backs side by side, then the occupied candidates' ids and offsets;
// the last tile of a volume writes the totals.  Every volume has at least
// one item; its item 0 records how many look-back descriptors the volume
// used (the next prep clears them).
struct ScanSmem {
    static constexpr int kR = kCountTile / kThreads;
    TileScan<kR> tri, occ, vtx;
    uint32_t val[kR][kThreads];       // triangles (9 bits), vertices (9), triangles before in the warp (14)
    unsigned long long cross[kR][kThreads];   // crossing cells
};

// rounds of 256 candidates a tile; batches share the CTAs among volumes and
// take full tiles
template <bool kOne>
__device__ __forceinline__ uint32_t count_rounds(uint32_t n) {
    constexpr uint32_t kMax = ScanSmem::kR;
    return kOne ? min(kMax, max(1u, ceil_div(n, gridDim.x * kThreads))) : kMax;
}

template <bool kOne, bool kIdx>
__global__ void __launch_bounds__(kThreads, 4) mc_scan_kernel(Launch L) {
    constexpr uint32_t kR = ScanSmem::kR;
    __shared__ ScanSmem sm;
    __shared__ uint32_t pre[kMaxBatch + 1];
    __shared__ uint32_t s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    after_previous_stage();
    const uint32_t total = launch_prefix<kOne>(
        L, [&](uint32_t v) {
            const uint32_t n = mc_candidates(vol_of<kOne>(L, v).s.ctl);
            return max(1u, ceil_div(n, count_rounds<kOne>(n) * kThreads));
        },
        pre);
    while (true) {
        const uint32_t x = next_item(&L.ctr[kLcScan], &s_item);
        if (x >= total) break;
        const uint32_t v = item_vol<kOne>(pre, L.n, x);
        const DevState &s = vol_of<kOne>(L, v).s;
        const Geom &g = vol_of<kOne>(L, v).g;
        Ctl *c = s.ctl;
        const uint32_t tile = x - item_base<kOne>(pre, v);
        const uint32_t n = mc_candidates(c);
        const uint32_t rounds = count_rounds<kOne>(n), tile_size = rounds * kThreads;
        const uint32_t ntiles = ceil_div(n, tile_size);
        if (tile == 0 && threadIdx.x == 0) c->mc_tiles = ntiles;
        if (ntiles == 0) continue;                        // block-uniform
        const uint32_t i0 = tile * tile_size + threadIdx.x;
#pragma unroll 1
        for (uint32_t r = 0; r < rounds; r++) {
            const uint32_t i = i0 + r * kThreads;
            uint32_t nt = 0, nv = 0;
            if (i < n) {
                unsigned long long m[8];
                uint32_t lim;
                corner_masks(s, g, s.icand[i], m, lim);
                const unsigned long long valid = valid_cells(lim);
                nt = count_triangles(m, valid, sm.cross[r][threadIdx.x]);
                if (kIdx) nv = count_vertices(m, valid, lim);
            }
            uint32_t incl = nt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t ob = __ballot_sync(0xffffffffu, nt != 0u);
            const uint32_t vsum = kIdx ? __reduce_add_sync(0xffffffffu, nv) : 0u;
            if (lane == 31) {
                sm.tri.cnt[r][warp] = incl;
                sm.occ.cnt[r][warp] = __popc(ob);
                if (kIdx) sm.vtx.cnt[r][warp] = vsum;
            }
            sm.val[r][threadIdx.x] = nt | (nv << 9) | ((incl - nt) << 18);
        }
        __syncthreads();
        // warp 0: triangle offsets; warp 1: occupied positions; warp 2: vertex offsets
        if (warp < (kIdx ? 3 : 2)) {
            TileScan<ScanSmem::kR> &ts = warp == 0 ? sm.tri : (warp == 1 ? sm.occ : sm.vtx);
            const uint32_t tot = scan_tile_counts(ts, rounds);
            unsigned long long *desc = warp == 0 ? s.desc_mc : (warp == 1 ? s.desc_occ : s.desc_vtx);
            const unsigned long long excl = lookback_exclusive(desc, tile, tot, &c->status, kStatusTimeoutScan);
            if (lane == 0) {
                ts.excl = excl;
                if (tile == ntiles - 1) {
                    if (warp == 0) c->n_tri = excl + tot;
                    else if (warp == 1) c->n_occ = (uint32_t)(excl + tot);
                    else c->n_vtx = excl + tot;
                }
            }
        }
        __syncthreads();
#pragma unroll 1
        for (uint32_t r = 0; r < rounds; r++) {
            const uint32_t i = i0 + r * kThreads;
            const uint32_t val = sm.val[r][threadIdx.x], nt = val & 511u, nv = (val >> 9) & 511u;
            const unsigned long long run = sm.tri.excl + sm.tri.cnt[r][warp] + (val >> 18);
            const uint32_t ob = __ballot_sync(0xffffffffu, nt != 0u);
            unsigned long long vrun = 0;
            if (kIdx) {
                uint32_t vincl = nv;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, vincl, o);
                    if (lane >= o) vincl += t;
                }
                vrun = sm.vtx.excl + sm.vtx.cnt[r][warp] + (vincl - nv);
            }
            const uint32_t at = (uint32_t)sm.occ.excl + sm.occ.cnt[r][warp] + __popc(ob & lt);
            if (nt && in_bounds(at < s.list_cap, &c->status)) {
                s.iocc[at] = s.icand[i];
                s.ooff[at] = run;
                s.ocross[at] = sm.cross[r][threadIdx.x];
                if (kIdx) s.voff[at] = vrun;
            }
        }
        __syncthreads();
    }
}

// debug volumes: the 64 cell cases of every candidate
__global__ void __launch_bounds__(kThreads) debug_cases_kernel(Launch L) {
    const DevState &s = L.one.s;
    const uint32_t n = mc_candidates(s.ctl);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        unsigned long long m[8];
        uint32_t lim;
        corner_masks(s, L.one.g, s.icand[i], m, lim);
        const unsigned long long valid = valid_cells(lim);
        for (int cell = 0; cell < 64; cell++) {
            uint32_t cs = 0;
#pragma unroll
            for (int c = 0; c < 8; c++) cs |= (uint32_t)(((m[c] & valid) >> cell) & 1ull) << c;
            s.cases[(size_t)i * 64 + cell] = (uint8_t)cs;
        }
    }
}

// ================================================================ emit (Section 4.5)
//
// What bounds it: instruction issue (58% of slots) and the latency of the
// shared-memory gathers (51% of its wavefronts, the first of the stalls),
// beside the vertices' 48 bytes a triangle (39% of the DRAM peak), counted on a
// 384^3 noise surface of 2.95 M triangles: 66 us, 40.7 M warp instructions.
// The variants below were timed on a surface of 4.3 M triangles (24 warps an
// SM): 72 us, 45 M warp instructions.  A triangle per lane with its vertices passed
// through shared memory, on cases found for every cell, took 85 us and
// 65 M.  Staging rows of 8 floats by 16-byte copies (x of 5 to 7 unused)
// left bank conflicts: 82 us.  32 warps an SM (64 registers) 79 us and a
// larger shared-memory share of the L1 79 us: the L1 serves the windows'
// shared rows, so the warps' areas are kept small.

// The warp tiles of one launch, as a lane of a warp sees them
template <bool kOne>
struct TileWalk {
    const Launch &L;
    const uint32_t *pre;
    uint32_t total;

    // volume, first occupied candidate and blocks of tile t < total
    __device__ __forceinline__ void locate(uint32_t t, uint32_t &v, uint32_t &base, uint32_t &nb_w) const {
        v = item_vol<kOne>(pre, L.n, t);
        base = (t - item_base<kOne>(pre, v)) * kBPW;
        nb_w = min((uint32_t)kBPW, vol_of<kOne>(L, v).s.ctl->n_occ - base);
    }
    // this lane's block of tile t (block lane / 8 of the tile)
    __device__ __forceinline__ uint32_t block_at(uint32_t t) const {
        if (t >= total) return kNoBlock;
        uint32_t v, base, nb_w;
        locate(t, v, base, nb_w);
        const uint32_t q = (threadIdx.x & 31) >> 3;
        return q < nb_w ? vol_of<kOne>(L, v).s.iocc[base + q] : kNoBlock;
    }
    // The slot of member lane % 8 of block b's +group (-1: none).  Where the
    // volume ends the ids run on into the next row: cells that read such a
    // block are outside the volume and never cross, so any slot will do.
    __device__ __forceinline__ int32_t slot_at(uint32_t t, uint32_t b) const {
        if (b == kNoBlock) return -1;
        const uint32_t v = item_vol<kOne>(pre, L.n, t), o = threadIdx.x & 7;
        const DevState &s = vol_of<kOne>(L, v).s;
        const Geom &g = vol_of<kOne>(L, v).g;
        const unsigned long long id = (unsigned long long)b + ((o & 1) ? 1u : 0u) + ((o & 2) ? g.nbx : 0u) +
                                      ((o & 4) ? g.nbx * g.nby : 0u);
        if (id >= g.nb) return -1;
        const int32_t sl = s.islot[id];
        return sl >= 0 && in_bounds((uint32_t)sl < s.ctl->cap, &s.ctl->status) ? sl : -1;
    }
};

// Phase B: queue the copies of a tile's samples and lists and write down its
// blocks (this lane's block b and slot from the two functions above)
template <bool kOne, bool kIdx>
__device__ __forceinline__ void stage_tile(const TileWalk<kOne> &walk, uint32_t t, uint32_t b, int32_t slot, int buf,
                                           EmitWarp<kIdx> &wt, const LaneConst &lc) {
    const int lane = threadIdx.x & 31;
    const uint32_t v = item_vol<kOne>(walk.pre, walk.L.n, t);
    const DevState &s = vol_of<kOne>(walk.L, v).s;
    const uint32_t base = (t - item_base<kOne>(walk.pre, v)) * kBPW;
    const uint32_t halo = shared_u32(&wt.halo[buf][0][0]);
    if ((lane & 7) == 0) {
        const uint32_t q = lane >> 3;
        wt.bid[buf][q] = b;
        if (kIdx && b != kNoBlock) {
            const Geom &g = vol_of<kOne>(walk.L, v).g;
            uint32_t bx, by, bz;
            block_coords(g, b, bx, by, bz);
            wt.lim[kIdx ? buf : 0][q] = cell_limits(g, bx, by, bz);
        }
    }
    if (lane < 2) cp_async16(shared_u32(&wt.cross[buf][2 * lane]), s.ocross + base + 2 * lane);
    if (lane == 2) cp_async8(shared_u32(&wt.first[buf][0]), s.ooff + base);
    if (kIdx && lane == 3) cp_async8(shared_u32(&wt.first[buf][1]), s.voff + base);
    const uint32_t dst = halo + 4 * lane;
#pragma unroll
    for (int q = 0; q < kBPW; q++)
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int32_t sl = __shfl_sync(0xffffffffu, slot, 8 * q + (lc.job[r] & 7u));
            if (sl >= 0 && (r < 3 || lane < kWindow - 96))
                cp_async4(dst + 4 * (q * kWindow + 32 * r), s.slots + (size_t)(uint32_t)sl * 64 + (lc.job[r] >> 3));
        }
}

// Phase D: the vertices of the `n` listed triangles, the first of them
// triangle t0 of the surface.  Lane l of round r writes vertex 32r + l of a
// chunk of 32 triangles, i.e. corner (32r + l) % 3 of triangle (32r + l) / 3.
// With kSafe every difference of two samples is in the reciprocal's range (the
// caller looked at the samples).  Vertices are stored evict-first (a surface
// is several times the L2, and the hulls, slot map and cached blocks the
// next extraction reads should stay there).
template <bool kPacked, bool kSafe, bool kDebug, bool kIdx>
__device__ __forceinline__ void write_soup(const DevState &s, const Geom &g, float iso, const EmitWarp<kIdx> &wt,
                                           const EmitTab<kIdx> &tab, int buf, uint32_t n, unsigned long long t0) {
    const uint32_t lane = threadIdx.x & 31;
    const Ctl *c = s.ctl;
    const unsigned long long cap = c->params.tri_cap;
    // vertices of the list that fit the output
    const int fit = t0 >= cap ? 0 : 3 * (int)min((unsigned long long)n, cap - t0);
    float4 *out4 = reinterpret_cast<float4 *>(c->params.out) + 3 * t0 + lane;
    uint2 *out2 = reinterpret_cast<uint2 *>(c->params.out) + 3 * t0 + lane;
    const uint32_t last = 4 * (n - 1);
    uint32_t tri[3];                                       // byte offsets in the list
#pragma unroll
    for (int r = 0; r < 3; r++) tri[r] = 4 * ((32 * r + lane) / 3);
    for (int left = fit - (int)lane; left > -(int)lane; left -= 96) {
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const uint32_t e = at<uint32_t>(wt.tmap, min(tri[r], last));
            const uint32_t info = at<uint16_t>(tab.corner, (e & 0x1FFFu) | (2 * ((32 * r + lane) % 3)));
            const uint32_t bid = wt.bid[buf][(e >> 13) & 3u];
            const uint32_t smp = (e >> 16) + (info & 0xFFu), step = info >> 8;   // byte offsets
            const float vlo = at<float>(wt.halo[buf], smp), vhi = at<float>(wt.halo[buf], smp + step);
            const uint2 h = at<uint2>(tab.coord, 2 * smp);
            const float2 xy = __half22float2(*reinterpret_cast<const __half2 *>(&h.x));
            float px = xy.x, py = xy.y, pz = __low2float(*reinterpret_cast<const __half2 *>(&h.y));
            const float tt = edge_fraction<kPacked, kSafe>(iso, vlo, vhi);
            if (step == 4u) px = __fadd_rn(px, tt);
            if (step == 20u) py = __fadd_rn(py, tt);
            if (step == 100u) pz = __fadd_rn(pz, tt);
            const bool write = left > 32 * r;
            if (!kPacked) {
                if (write) __stcs(out4 + 32 * r, make_float4(px, py, pz, __uint_as_float(bid)));
            } else {
                // the 10-bit code round(p / 4 * 1023) decides an integer, so every
                // step is one IEEE float32 operation (the division correctly
                // rounded), as the oracle computes it
                const uint32_t qx = (uint32_t)__float2int_rn(__fmul_rn(px, 255.75f));
                const uint32_t qy = (uint32_t)__float2int_rn(__fmul_rn(py, 255.75f));
                const uint32_t qz = (uint32_t)__float2int_rn(__fmul_rn(pz, 255.75f));
                if (write) __stcs(out2 + 32 * r, make_uint2(qx | (qy << 10) | (qz << 20), bid));
            }
            if (kDebug) {
                uint32_t bx, by, bz;
                block_coords(g, bid, bx, by, bz);
                const uint32_t i = smp / 4 % kWindow, a = step == 4u ? 0u : (step == 20u ? 1u : 2u);
                const unsigned long long x = 4ull * bx + i % 5u, y = 4ull * by + (i / 5u) % 5u, z = 4ull * bz + i / 25u;
                if (write)
                    s.dbg_edges[3 * t0 + (unsigned)(fit - left) + 32 * r] =
                        3ull * (x + (unsigned long long)g.nx * (y + (unsigned long long)g.ny * z)) + a;
            }
            tri[r] += 128;
        }
        out4 += 96;
        out2 += 96;
    }
}

// Phase D of an indexed mesh: the three vertex indices of each listed
// triangle, `vt` that of the tile's first vertex; lanes as above.  A corner's
// index is the rank of its edge among the tile's vertices: those before its
// cut-edge word, then the word's bits below it.
template <bool kDebug>
__device__ __forceinline__ void write_indices(const DevState &s, const Geom &g, const EmitWarp<true> &wt,
                                              const EmitTab<true> &tab, int buf, uint32_t n, unsigned long long t0,
                                              unsigned long long vt) {
    const int lane = threadIdx.x & 31;
    const Ctl *c = s.ctl;
    const unsigned long long cap = c->params.tri_cap;
    const uint32_t fit = t0 >= cap ? 0u : (uint32_t)min((unsigned long long)n, cap - t0);
    uint32_t *out = reinterpret_cast<uint32_t *>(c->params.idx_out) + 3 * t0 + lane;
    for (uint32_t c0 = 0; c0 < n; c0 += 32) {
#pragma unroll
        for (int r = 0; r < 3; r++) {
            const uint32_t f = 32 * r + lane, tri = min(c0 + f / 3u, n - 1), e = wt.tmap[tri];
            const uint32_t info = at<uint16_t>(tab.corner, (e & 0x1FFFu) | (2 * (f % 3u)));
            const uint32_t q = (e >> 13) & 3u, step = info >> 8, a = step == 4u ? 0u : (step == 20u ? 1u : 2u);
            const uint32_t smp = (e >> 18) - q * kWindow + ((info & 0xFFu) >> 2);
            const uint32_t *cw = wt.cut[q] + 4 * a + (smp >> 5);
            const uint32_t rank = cw[12] + __popc(cw[0] & ((1u << (smp & 31)) - 1u));
            const bool write = 3 * c0 + f < 3 * fit;
            if (write) out[32 * r] = (uint32_t)(vt + rank);
            if (kDebug) {
                uint32_t bx, by, bz;
                block_coords(g, wt.bid[buf][q], bx, by, bz);
                const unsigned long long x = 4ull * bx + smp % 5u, y = 4ull * by + (smp / 5u) % 5u, z = 4ull * bz + smp / 25u;
                if (write)
                    s.dbg_edges[3 * (t0 + c0) + f] =
                        3ull * (x + (unsigned long long)g.nx * (y + (unsigned long long)g.ny * z)) + a;
            }
        }
        out += 96;
    }
}

// The vertices of an indexed tile, in order (block, axis, sample).  Lanes
// 0-11 (and 12-23 for a second block) take one word each of a block's cut
// edges, leave the vertices of the tile before it in cut[q][12..23], and list
// its edges in the vertex map; then one vertex per lane, the triangle soup's
// arithmetic, consecutive lanes writing consecutive vertices.  The map holds
// two blocks (at most 600 vertices); it is written out when full.
__device__ __forceinline__ void write_vertices(const DevState &s, float iso, EmitWarp<true> &wt, int buf, int nb_w,
                                               unsigned long long vt) {
    const int lane = threadIdx.x & 31;
    const Ctl *c = s.ctl;
    const bool packed = c->params.format == kVertexPacked;     // warp-uniform
    const unsigned long long vcap = c->params.vert_cap;
    float4 *out = reinterpret_cast<float4 *>(c->params.out);
    uint16_t *vm = reinterpret_cast<uint16_t *>(wt.tmap);      // block (2) | sample (7) | axis (2)
    uint32_t nvt = 0, first = 0;                               // vertices so far; the map's first one
    for (int qq = 0; qq < nb_w; qq += 2) {
        const int q = qq + (lane >= 12 ? 1 : 0), lk = lane % 12, la = lk >> 2, lr = lk & 3;
        uint32_t w = (lane < 24 && q < nb_w) ? wt.cut[q][lk] : 0u;
        const uint32_t n = __popc(w);
        uint32_t incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t rank = nvt + incl - n;                        // the tile's vertices before this word
        if (lane < 24 && q < nb_w) wt.cut[q][12 + lk] = rank;
        // listed now, or after what the map holds has been written
        for (int pass = 0; pass < 2; pass++) {
            const bool room = nvt - first + tot <= (uint32_t)kVmap;
            if (room) {
                while (w) {
                    const uint32_t i = __ffs(w) - 1;
                    w &= w - 1;
                    vm[rank++ - first] = (uint16_t)((q << 9) | ((32 * lr + i) << 2) | la);
                }
            }
            __syncwarp();
            if (room && qq + 2 < nb_w) break;                  // go on listing
            const uint32_t to = room ? nvt + tot : nvt;
            for (uint32_t k = first + lane; k < to; k += 32) {
                const uint32_t e = vm[k - first], q2 = e >> 9, smp = (e >> 2) & 127u, ax = e & 3u;
                const uint32_t sx = smp % 5u, sy = (smp / 5u) % 5u, sz = smp / 25u;
                const float *hp = &wt.halo[buf][q2][smp];
                const float vlo = hp[0], vhi = hp[ax == 0 ? 1 : (ax == 1 ? 5 : 25)];
                float px = (float)sx, py = (float)sy, pz = (float)sz;
                const float tt = packed ? edge_fraction<true>(iso, vlo, vhi) : edge_fraction<false>(iso, vlo, vhi);
                if (ax == 0) px = __fadd_rn(px, tt);
                else if (ax == 1) py = __fadd_rn(py, tt);
                else pz = __fadd_rn(pz, tt);
                if (vt + k < vcap) {
                    const uint32_t bid = wt.bid[buf][q2];
                    if (!packed) {
                        out[vt + k] = make_float4(px, py, pz, __uint_as_float(bid));
                    } else {
                        const uint32_t qx = (uint32_t)__float2int_rn(__fmul_rn(px, 255.75f));
                        const uint32_t qy = (uint32_t)__float2int_rn(__fmul_rn(py, 255.75f));
                        const uint32_t qz = (uint32_t)__float2int_rn(__fmul_rn(pz, 255.75f));
                        reinterpret_cast<uint2 *>(out)[vt + k] = make_uint2(qx | (qy << 10) | (qz << 20), bid);
                    }
                }
            }
            first = to;
            __syncwarp();                                      // the map is read
            if (room) break;
        }
        nvt += tot;
    }
}

template <int kW, bool kDebug, bool kOne, bool kIdx>
__device__ __forceinline__ void emit_body(const Launch &L) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EmitSmem<kW, kIdx> &sm = *reinterpret_cast<EmitSmem<kW, kIdx> *>(smem_raw);
    uint32_t *pre = reinterpret_cast<uint32_t *>(&sm + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    after_previous_stage();
    // all failure bits are final before this kernel starts
    const uint32_t total = launch_prefix<kOne>(
        L, [&](uint32_t v) {
            const Ctl *c = vol_of<kOne>(L, v).s.ctl;
            return (c->status & (kStatusBudget | kStatusAnyTimeout | kStatusSkip)) ? 0u : ceil_div(c->n_occ, kBPW);
        },
        pre);
    // one tile's samples are copied in while the tile before it is written;
    // its slots were loaded a tile earlier, and its block ids two (the first
    // ones before the tables, so that their latencies pass together)
    const TileWalk<kOne> walk{L, pre, total};
    const uint32_t stride = gridDim.x * kW;
    uint32_t t = blockIdx.x * kW + warp;
    const uint32_t b0 = walk.block_at(t);
    uint32_t b1 = walk.block_at(t + stride), b2 = walk.block_at(t + 2 * stride);
    const EmitTables *tables = vol_of<kOne>(L, 0).s.tables;
    auto fill = [&](void *dst, const void *src, uint32_t bytes) {
        for (uint32_t i = threadIdx.x; i < bytes / 16; i += 32 * kW)
            static_cast<uint4 *>(dst)[i] = __ldg(static_cast<const uint4 *>(src) + i);
    };
    static_assert(sizeof(EmitWarp<kIdx>) % 16 == 0 && sizeof(tables->info) % 16 == 0 &&
                      sizeof(tables->corner) % 16 == 0 && sizeof(tables->coord) % 16 == 0, "16-byte copies");
    fill(sm.tab.info, tables->info, sizeof(tables->info));
    fill(sm.tab.corner, tables->corner, sizeof(tables->corner));
    if (!kIdx) fill(sm.tab.coord, tables->coord, sizeof(tables->coord));
    if (kIdx) load_window_rows(sm.win);
    const int32_t s0 = walk.slot_at(t, b0);
    int32_t s1 = walk.slot_at(t + stride, b1);
    __syncthreads();                                      // the tables
    if (t >= total) return;
    LaneConst lc;
    lc.init(lane);
    EmitWarp<kIdx> &wt = sm.w[warp];
    stage_tile<kOne, kIdx>(walk, t, b0, s0, 0, wt, lc);
    cp_async_commit();
    const uint32_t lt = (1u << lane) - 1u;
    for (int buf = 0; t < total; t += stride, buf ^= 1) {
        if (t + stride < total) stage_tile<kOne, kIdx>(walk, t + stride, b1, s1, buf ^ 1, wt, lc);
        cp_async_commit();
        s1 = walk.slot_at(t + 2 * stride, b2);
        b1 = b2;
        b2 = walk.block_at(t + 3 * stride);
        uint32_t v, base, nb_w;
        walk.locate(t, v, base, nb_w);
        const DevState &s = vol_of<kOne>(L, v).s;
        const Geom &g = vol_of<kOne>(L, v).g;
        const Ctl *c = s.ctl;
        const float iso = c->params.iso;
        const bool packed = c->params.format == kVertexPacked;     // warp-uniform
        // subtracting -0 instead of 0 leaves a sample of -0 at +0, not below
        const float iso_sub = iso == 0.0f ? -0.0f : iso;
        cp_async_wait_prev();
        __syncwarp();
        // consecutive occupied candidates have adjacent outputs: the tile
        // starts at its first block's
        unsigned long long t0 = wt.first[buf][0], vt = 0;
        if constexpr (kIdx) {
            vt = wt.first[buf][1];
            for (uint32_t q = 0; q < nb_w; q++) {
                uint32_t m[4];
                below_mask(&wt.halo[buf][q][0], iso, m);
                const uint32_t w = lane_cut_word(m, wt.lim[buf][q], sm.win);
                if (lane < 12) wt.cut[q][lane] = w;
            }
            __syncwarp();
            write_vertices(s, iso, wt, buf, (int)nb_w, vt);
            vt += c->params.vtx_base;                  // indices count the vertices of earlier waves
        }
        // ---- C: the crossing cells in order
        uint32_t ncell = 0;
#pragma unroll
        for (int q = 0; q < kBPW; q++) {
            const unsigned long long w2 = q < (int)nb_w ? wt.cross[buf][q] : 0ull;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t w = h ? (uint32_t)(w2 >> 32) : (uint32_t)w2;
                if ((w >> lane) & 1u) wt.cells[ncell + __popc(w & lt)] = (uint16_t)((lc.cell[h] + q * kWindow) | (q << 11));
                ncell += __popc(w);
            }
        }
        __syncwarp();
        // 32 cells at a time: their triangles while they fit the list, then D
        uint32_t n = 0, k0 = 0;
        bool safe = true;
        for (;;) {
            for (; k0 < ncell; k0 += 32) {
                const uint32_t cell = wt.cells[min(k0 + lane, ncell - 1)];
                const float *hb = &wt.halo[buf][0][0] + (cell & 0x7FFu);
                float d[8];
                float mx = 0.0f, mn = INFINITY;
                uint32_t cs = 0;
#pragma unroll
                for (int k = 7; k >= 0; k--) {
                    d[k] = __fsub_rn(hb[(k & 1) + 5 * ((k >> 1) & 1) + 25 * (k >> 2)], iso_sub);
                    cs = __funnelshift_l(__float_as_uint(d[k]), cs, 1);      // below: the difference's sign
                    mx = fmaxf(mx, fabsf(d[k]));
                    mn = fminf(mn, fabsf(d[k]));
                }
                const uint32_t row = sm.tab.info[cs];
                const uint32_t k = k0 + lane < ncell ? row >> 13 : 0u;
                uint32_t incl = k;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
                if (n + tot > (uint32_t)kTmap) break;
                // the two samples of a cut edge lie on either side of iso, each
                // between 2^-100 and 2^124 away: their difference is in range
                safe = safe && __all_sync(0xffffffffu, mn >= 0x1p-100f && mx < 0x1p124f);
                uint32_t *to = wt.tmap + n + incl - k;
                const uint32_t e = ((cell & 0x7FFu) << 18) | ((cell >> 11) << 13) | (row & 0x1FFFu);
                if (k > 0) to[0] = e;
                if (k > 1) to[1] = e + 8;
                if (k > 2) to[2] = e + 16;
                if (k > 3) to[3] = e + 24;
                if (k > 4) to[4] = e + 32;
                n += tot;
            }
            __syncwarp();
            if (n) {                              // warp-uniform
                if constexpr (kIdx) write_indices<kDebug>(s, g, wt, sm.tab, buf, n, t0, vt);
                else if (packed) write_soup<true, false, kDebug, kIdx>(s, g, iso, wt, sm.tab, buf, n, t0);
                else if (safe) write_soup<false, true, kDebug, kIdx>(s, g, iso, wt, sm.tab, buf, n, t0);
                else write_soup<false, false, kDebug, kIdx>(s, g, iso, wt, sm.tab, buf, n, t0);
            }
            __syncwarp();                         // the list (and, at the end, the samples) are read
            if (k0 >= ncell) break;
            t0 += n;
            n = 0;
            safe = true;
        }
    }
    cp_async_wait_all();
}

// the triangle soup; registers bounded for 24 warps per SM, what the shared
// memory of two tiles' samples a warp allows
template <int kW, bool kDebug, bool kOne>
__global__ void __launch_bounds__(32 * kW, kW == 16 ? 1 : 24 / kW) mc_emit_kernel(Launch L) {
    emit_body<kW, kDebug, kOne, false>(L);
}

// the indexed mesh (single volumes)
template <int kW, bool kDebug>
__global__ void __launch_bounds__(32 * kW, kW == 16 ? 1 : 24 / kW) mc_emit_indexed_kernel(Launch L) {
    emit_body<kW, kDebug, true, true>(L);
}

// ================================================================ launchers

namespace {

// dynamic shared memory of an emission: the warps' areas and tables, then a
// batch's prefix words
template <int kW, bool kIdx>
size_t emit_smem(const Launch &L) {
    return sizeof(EmitSmem<kW, kIdx>) + (L.vols ? ((size_t)L.n + 1) * 4 : 0);
}

template <int kW, bool kOne, bool kIdx>
void emit_w(const Launch &L, bool debug, int grid, cudaStream_t st) {
    const size_t bytes = emit_smem<kW, kIdx>(L);
    if constexpr (kIdx) {
        if (debug) launch_next(L, mc_emit_indexed_kernel<kW, true>, grid, 32 * kW, bytes, st);
        else launch_next(L, mc_emit_indexed_kernel<kW, false>, grid, 32 * kW, bytes, st);
    } else if constexpr (kOne) {
        if (debug) launch_next(L, mc_emit_kernel<kW, true, true>, grid, 32 * kW, bytes, st);
        else launch_next(L, mc_emit_kernel<kW, false, true>, grid, 32 * kW, bytes, st);
    } else {                                          // debug volumes are not batched
        launch_next(L, mc_emit_kernel<kW, false, false>, grid, 32 * kW, bytes, st);
    }
}

// resident CTAs per SM of `kernel` (at least 1)
template <class K>
int occupancy(K kernel, int threads, size_t smem) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess) {
        (void)cudaGetLastError();
        occ = 1;
    }
    return std::max(1, occ);
}

template <class K>
void raise_smem(K kernel, size_t bytes) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int kW>
int emit_occupancy(bool single) {
    constexpr size_t soup = sizeof(EmitSmem<kW, false>), idx = sizeof(EmitSmem<kW, true>);
    constexpr size_t table = (kMaxBatch + 1) * 4;         // the largest batch's prefix words
    raise_smem(mc_emit_kernel<kW, false, false>, soup + table);
    raise_smem(mc_emit_kernel<kW, false, true>, soup);
    raise_smem(mc_emit_kernel<kW, true, true>, soup);
    raise_smem(mc_emit_indexed_kernel<kW, false>, idx);
    raise_smem(mc_emit_indexed_kernel<kW, true>, idx);
    // every kernel launched with this CTA count must fit it: a CTA beyond
    // the resident ones would start only when a whole CTA has finished, and
    // its statically assigned tiles would trail the rest (batches of so many
    // volumes that their prefix words cost a CTA are the exception)
    if (single)
        return std::min({occupancy(mc_emit_kernel<kW, false, true>, 32 * kW, soup),
                         occupancy(mc_emit_kernel<kW, true, true>, 32 * kW, soup),
                         occupancy(mc_emit_indexed_kernel<kW, false>, 32 * kW, idx),
                         occupancy(mc_emit_indexed_kernel<kW, true>, 32 * kW, idx)});
    return occupancy(mc_emit_kernel<kW, false, false>, 32 * kW, soup + 65 * 4);
}

template <bool kOne, bool kIdx>
void emit_any(const Launch &L, bool debug, const Plan &pl, cudaStream_t st) {
    if (pl.emit_tile == 16) emit_w<4, kOne, kIdx>(L, debug, pl.mc_emit, st);
    else if (pl.emit_tile == 64) emit_w<16, kOne, kIdx>(L, debug, pl.mc_emit, st);
    else emit_w<8, kOne, kIdx>(L, debug, pl.mc_emit, st);
}

}  // namespace

void launch_mc_scan(const Launch &L, bool debug, const Plan &pl, cudaStream_t st, bool indexed) {
    if (L.vols) launch_next(L, mc_scan_kernel<false, false>, pl.mc_scan, kThreads, 0, st);
    else if (indexed) launch_next(L, mc_scan_kernel<true, true>, pl.mc_scan, kThreads, 0, st);
    else launch_next(L, mc_scan_kernel<true, false>, pl.mc_scan, kThreads, 0, st);
    if (debug && !L.vols) debug_cases_kernel<<<pl.mc_scan, kThreads, 0, st>>>(L);
}

// the indexed mesh is made for single volumes only
void launch_mc_emit(const Launch &L, bool debug, const Plan &pl, cudaStream_t st, bool indexed) {
    if (L.vols) emit_any<false, false>(L, debug, pl, st);
    else if (indexed) emit_any<true, true>(L, debug, pl, st);
    else emit_any<true, false>(L, debug, pl, st);
}

void mc_occupancy(Plan *pl, bool single) {
    // every variant's shared-memory limit is raised, whichever is asked for
    const int e4 = emit_occupancy<4>(single), e8 = emit_occupancy<8>(single), e16 = emit_occupancy<16>(single);
    pl->mc_emit = std::max(1, pl->emit_tile == 16 ? e4 : (pl->emit_tile == 64 ? e16 : e8));
    // the soup's and the indexed mesh's counts share the CTA count
    pl->mc_scan = single ? std::min(occupancy(mc_scan_kernel<true, false>, kThreads, 0),
                                    occupancy(mc_scan_kernel<true, true>, kThreads, 0))
                         : occupancy(mc_scan_kernel<false, false>, kThreads, 0);
}

}  // namespace bcmc
