// Fixed-rate 4x4x4 block codec, device side (paper Section 4.2.1: each new
// block is decoded by one thread straight into its cache slot; the format
// follows ZFP's fixed-rate mode as summarised in Section 3.3.4).
//
// Block format, rate*64 bits in `rate` little-endian 64-bit words, bits
// taken LSB first:
//   bit 0      non-zero flag (0: all 64 samples are +0, the rest is padding)
//   bits 1..8  emax + 127, emax = largest binary exponent in the block
//              (frexp convention, at least -126)
//   then       the 32 bit planes, most significant first, of 64 negabinary
//              coefficients listed in sequency order.  In each plane, the
//              coefficients already reached are sent verbatim; then group
//              tests: a 1 means some later coefficient has a one in this
//              plane, followed by the later bits one by one up to and
//              including that one (a one in the last coefficient is not
//              sent); a 0 ends the plane.  Coding stops exactly when the
//              block's bits are used up; unread bits count as zero.
// Samples are q = trunc(v * 2^(27 - emax)) integers, decorrelated by a
// two-level integer S-transform along x, then y, then z; the decoder runs
// the exact inverse in 32-bit wrap-around arithmetic and returns the
// float32 of q (rounded to nearest even) times 2^(emax - 27): exact while
// the result is normal, rounded once more when it is subnormal.
#pragma once

#include "common.cuh"

namespace bcmc {

__device__ __forceinline__ uint64_t low_mask(uint32_t n) { return n >= 64 ? ~0ull : ((1ull << n) - 1ull); }

// ---------------------------------------------------------------- staging
//
// A warp decodes up to 32 blocks at a time, one per lane (Section 4.2.1
// decodes one block per thread).  The blocks' words are first copied into
// a per-warp staging area of shared memory by coalesced loads: in each
// round consecutive lanes load consecutive 8-byte words, block after block,
// so a warp instruction reads 256 contiguous bytes of every block it
// touches.  Each lane then parses its own block from shared memory.
//
// A staged block takes 2R + 1 32-bit words (its 2R words, then a zero pad
// word; the odd stride spreads the lanes' reads over the banks), and the
// area ends with two more words, so a window may read up to two words past
// the block's last one (bits past the budget are never used).

__host__ __device__ constexpr uint32_t stage_words(uint32_t rate) { return 32u * (2u * rate + 1u) + 2u; }

// Copy block `id` of each lane that has one (`have`) into the warp's
// staging area `stage` (stage_words(rate) words).  Called by all 32 lanes.
__device__ __forceinline__ void stage_blocks(const uint64_t *__restrict__ bits, uint32_t rate, uint32_t id, bool have,
                                             uint32_t *stage) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t stride = 2u * rate + 1u;
    const uint32_t magic = (65535u + rate) / rate;          // ceil(2^16 / rate): j / rate = (j * magic) >> 16, j < 1024
    const uint32_t have_mask = __ballot_sync(0xffffffffu, have);
    // Rounds of kInFlight words per lane: every load of a round is issued
    // before the first shared store, so a lane waits for one memory latency
    // per round rather than one per word.  Round k of lane j copies word
    // j + 32k of the warp's 32 * rate, i.e. word w of block q.
    constexpr uint32_t kInFlight = 8;
    for (uint32_t k0 = 0; k0 < rate; k0 += kInFlight) {      // the same number of rounds in every lane
        uint64_t v[kInFlight];
#pragma unroll
        for (uint32_t k = 0; k < kInFlight; k++) {
            const uint32_t j = lane + 32u * (k0 + k);
            const uint32_t q = (j * magic) >> 16, w = j - q * rate;
            const uint32_t bq = __shfl_sync(0xffffffffu, id, (int)(q & 31u));
            v[k] = 0ull;
            if (k0 + k < rate && ((have_mask >> q) & 1u)) v[k] = __ldg(bits + (size_t)bq * rate + w);
        }
#pragma unroll
        for (uint32_t k = 0; k < kInFlight; k++) {
            const uint32_t j = lane + 32u * (k0 + k);
            const uint32_t q = (j * magic) >> 16, w = j - q * rate;
            if (k0 + k < rate) {
                stage[q * stride + 2u * w] = (uint32_t)v[k];
                stage[q * stride + 2u * w + 1u] = (uint32_t)(v[k] >> 32);
            }
        }
    }
    stage[lane * stride + 2u * rate] = 0u;
    if (lane < 2) stage[32u * stride + lane] = 0u;
    __syncwarp();
}

// fetch block id's words into L2 (a later stage_blocks call reads them)
__device__ __forceinline__ void prefetch_block(const uint64_t *__restrict__ bits, uint32_t rate, uint32_t id) {
    const uint64_t *p = bits + (size_t)id * rate;
    for (uint32_t w = 0; w < rate; w += 16) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + w));
}

// Shared-memory accesses by 32-bit shared-window address (the decoder's
// loops address the staging area and plane columns this way, so every
// access is a plain shared-memory load or store).
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void lds_u64(uint32_t a, uint32_t &lo, uint32_t &hi) {
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(lo), "=r"(hi) : "r"(a));
}
__device__ __forceinline__ void sts_u64(uint32_t a, uint32_t lo, uint32_t hi) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(lo), "r"(hi));
}

// The mask of the lowest n bits (n > 32: all of them)
__device__ __forceinline__ uint32_t bit_mask(uint32_t n) {
    uint32_t r;
    asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(r) : "r"(n));
    return r;
}

// Bit windows over staged blocks.  A position is a bit's place in shared
// memory (8 x its byte's shared address + its place in the byte), so a
// window needs no base address; staged blocks start at whole words.
__device__ __forceinline__ uint32_t win32(uint32_t pos) {     // the 32 bits from pos on
    const uint32_t a = (pos >> 3) & ~3u;
    return __funnelshift_r(lds_u32(a), lds_u32(a + 4), pos);
}
__device__ __forceinline__ void win64(uint32_t pos, uint32_t &lo, uint32_t &hi) {   // 64 bits, as two halves
    const uint32_t a = (pos >> 3) & ~3u;
    const uint32_t x = lds_u32(a), y = lds_u32(a + 4), z = lds_u32(a + 8);
    lo = __funnelshift_r(x, y, pos);
    hi = __funnelshift_r(y, z, pos);
}

// inverse of one two-level S-transform step on (ll, hh, h0, h1) -> (a, b, c, d), two's-complement words
// held as uint32 (wrap-around arithmetic)
__device__ __forceinline__ void inv_lift4u(uint32_t &p0, uint32_t &p1, uint32_t &p2, uint32_t &p3) {
    const uint32_t ll = p0, hh = p1, h0 = p2, h1 = p3;
    const uint32_t l1 = ll - (uint32_t)((int32_t)hh >> 1);
    const uint32_t l0 = hh + l1;
    const uint32_t b = l0 - (uint32_t)((int32_t)h0 >> 1);
    const uint32_t a = h0 + b;
    const uint32_t d = l1 - (uint32_t)((int32_t)h1 >> 1);
    const uint32_t c = h1 + d;
    p0 = a; p1 = b; p2 = c; p3 = d;
}

// forward step (a, b, c, d) -> (ll, hh, h0, h1); inputs |x| < 2^29
__device__ __forceinline__ void fwd_lift4(int32_t &p0, int32_t &p1, int32_t &p2, int32_t &p3) {
    const int32_t a = p0, b = p1, c = p2, d = p3;
    const int32_t h0 = a - b, l0 = b + (h0 >> 1);
    const int32_t h1 = c - d, l1 = d + (h1 >> 1);
    const int32_t hh = l0 - l1, ll = l1 + (hh >> 1);
    p0 = ll; p1 = hh; p2 = h0; p3 = h1;
}

// out[l] = float32(q[l]) * 2^e, e in [-154, 101]: the conversion rounds to
// nearest even; the scaling is exact while the result is normal and rounds
// once more when it is subnormal.  One branch per block (uniform in a warp
// unless some of its blocks have tiny exponents).
__device__ __forceinline__ void scale_block(const uint32_t (&q)[64], int e, float (&out)[64]) {
    if (e >= -126) {
        const float sc = __int_as_float((e + 127) << 23);
#pragma unroll
        for (int l = 0; l < 64; l++) out[l] = __fmul_rn(__int2float_rn((int32_t)q[l]), sc);
    } else {
        // f * 2^(e+64) is exact and normal; the final multiply rounds once
        const float sc = __int_as_float((e + 64 + 127) << 23), down = __int_as_float((127 - 64) << 23);
#pragma unroll
        for (int l = 0; l < 64; l++) out[l] = __fmul_rn(__fmul_rn(__int2float_rn((int32_t)q[l]), sc), down);
    }
}

// ---------------------------------------------------------------- group-test steps
//
// The group tests of a plane (after its verbatim bits) are read eight bits
// at a time through a 512-entry table: for a state (0: the next bit is a
// group test, 1: it is a run bit) and a byte of the stream, the entry holds
// what reading those bits one by one does --
//   bits 0-7    the run bits met, in order (coefficient n, n + 1, ...)
//   bit  10     the state after the consumed bits (its place in the entry's
//               byte offset in the table: state * 1024 + byte * 4)
//   bit  15     a 0 test ended the plane
//   bits 16-23  how many run bits that is
//   bits 24-31  bits consumed (8, or fewer when a 0 test ends the plane)
// A group test is a 1 followed by the run of later coefficients' bits up to
// and including the next one, or the 0 that ends the plane, so without the
// budget and coefficient 63's implied one the table step is exactly eight
// steps of that rule.  The decoder checks the two exceptions around it.
constexpr uint32_t kGroupState = 1u << 10, kGroupEnd = 1u << 15;
__host__ __device__ constexpr uint32_t group_step_entry(uint32_t state, uint32_t byte) {
    uint32_t runbits = 0, count = 0, consumed = 8, ended = 0;
    for (uint32_t i = 0; i < 8; i++) {
        const uint32_t bit = (byte >> i) & 1u;
        if (state == 0) {
            if (!bit) {
                ended = 1;
                consumed = i + 1;
                break;
            }
            state = 1;
        } else {
            runbits |= bit << count;
            count++;
            if (bit) state = 0;
        }
    }
    return runbits | (state ? kGroupState : 0u) | (ended ? kGroupEnd : 0u) | (count << 16) | (consumed << 24);
}

constexpr uint32_t kGroupTableEntries = 512;

struct GroupTable {
    uint32_t e[kGroupTableEntries];
};
__host__ __device__ constexpr GroupTable make_group_table() {
    GroupTable t{};
    for (uint32_t i = 0; i < kGroupTableEntries; i++) t.e[i] = group_step_entry(i >> 8, i & 255u);
    return t;
}
__device__ const GroupTable kGroupTable = make_group_table();

// fill a block's copy of the table (all threads; the caller synchronises).
// Made at compile time: working the entries out took a CTA of 128 some 600
// instructions a warp, where a chunk of blocks takes 3700.
__device__ __forceinline__ void load_group_table(uint32_t *tab) {
    for (uint32_t i = threadIdx.x; i < kGroupTableEntries; i += blockDim.x) tab[i] = __ldg(&kGroupTable.e[i]);
}

// Parse the bit planes of a staged block of `rate` words at shared address
// `words`: plane k (most significant first) goes to shared address
// planes + k * stride as a 64-bit word whose bit i belongs to the i-th coded
// coefficient.  A zero block (flag bit 0: the rest is not read) has all
// planes zero.  Sets emax.
//
// The lanes of a warp parse different blocks.  One loop of uniform steps
// keeps them together: a step takes the plane's verbatim bits when it opens
// a plane, then up to kSteps table steps of its group tests out of one
// 32-bit window, all predicated; a lane whose block is done sits the
// remaining steps out.  Where a table step would reach coefficient 63, whose
// one is implied, a step takes one group test and its run instead.  Bits
// past the budget read as zero: the staged block is followed by a zero word,
// and a window is used only as far as 9 bits past the budget's last.
// Once every coefficient is reached (n = 64) a plane is its 64 verbatim
// bits, which a short loop of its own copies.
//
// Bound by issue, and half of a decode's instructions: some 16 turns of the
// loop at 8 bits a value, half of the lanes at work (blocks differ in their
// planes and tests).  With two window reads a turn, 64-bit masks made by
// compares, and bit-by-bit events in half of the turns it took some 2700 of
// the 4400 warp instructions of 32 blocks, now 1850 of 3700 (333 k new blocks
// of 384^3 noise: decode 79 -> 61 us with the stores below).  One or three table steps a turn
// and selects instead of branches came out slower.
template <int kSteps = 2>
__device__ __forceinline__ void parse_planes(uint32_t words, uint32_t rate, uint32_t tab, uint32_t planes,
                                             uint32_t stride, int &emax) {
    static_assert(kSteps <= 3, "a window of 30 bits holds three steps of 9");
    const uint32_t head = lds_u32(words);
    emax = (int)((head >> 1) & 0xFFu) - 127;
    uint32_t pos = words * 8u;
    const uint32_t end = pos + ((head & 1u) ? rate * 64u : 0u);
    pos += 9;
    uint32_t n = 0;                        // coefficients reached by the group tests
    int k = 31;                            // plane, most significant first
    if (head & 1u) {
        // Until a coefficient is reached, a plane has no verbatim bits and a
        // 0 group test ends it: each 0 bit here is a whole empty plane
        // (end - pos >= 55 at every rate, so the window is inside the budget).
        const uint32_t win = win32(pos);
        const uint32_t z = win ? (uint32_t)__ffs(win) - 1u : 32u;
        for (uint32_t j = 0; j < z; j++) sts_u64(planes + (31u - j) * stride, 0u, 0u);
        k -= (int)z;
        pos += z;
    }
    uint32_t xlo = 0u, xhi = 0u, at = tab; // at: the state's half of the table
    bool opening = true;
    while (k >= 0 && pos < end && n < 64u) {
        if (opening) {                     // the verbatim bits of the n coefficients reached so far
            const uint32_t m = min(n, end - pos);
            uint32_t wlo, whi;
            win64(pos, wlo, whi);
            xlo = wlo & bit_mask(m);
            xhi = whi & bit_mask(max(m, 32u) - 32u);
            pos += m;
            at = tab;
        }
        bool done = pos >= end;
        uint32_t w = win32(pos) << 2;      // (at pos == end: the zero word, and not used)
#pragma unroll
        for (int t = 0; t < kSteps; t++) {
            if (done) continue;
            const uint32_t e = lds_u32(at + (w & 0x3FCu));
            const uint32_t cnt = __byte_perm(e, 0u, 0x4442);
            if (n + cnt <= 62u) {
                const uint64_t bits = (uint64_t)(e & 0xFFu) << n;
                xlo |= (uint32_t)bits;
                xhi |= (uint32_t)(bits >> 32);
                n += cnt;
                pos += e >> 24;
                at = tab + (e & kGroupState);
                w >>= 8;
                done = (e & kGroupEnd) != 0u || pos >= end;
            } else {                       // one event; here n >= 55
                const bool test = at == tab;
                const bool ended = test && !(w & 4u);
                uint32_t used = test ? 1u : 0u;
                if (!ended) {
                    const uint32_t lim = 63u - n, run = w >> (2u + used);       // run bits that may be sent
                    const uint32_t z = (uint32_t)__ffs(run | (1u << lim)) - 1u;  // zeros before the run's one
                    const bool implied = z == lim;                              // none sent: 63's one is implied
                    xhi |= 1u << (n + z - 32u);
                    n += z + 1u;
                    used += implied ? z : z + 1u;
                    // the budget ran out inside the run: no one was read
                    if (pos + used > end) xhi &= 0x7FFFFFFFu;
                }
                pos += used;
                at = tab;
                w >>= used;
                done = ended || pos >= end || n >= 64u;
            }
        }
        if (done) {
            sts_u64(planes + (uint32_t)k * stride, xlo, xhi);
            k--;
        }
        opening = done;
    }
    // every coefficient reached: each remaining plane is the next 64 bits,
    // read two words a plane
    uint32_t column = planes + (uint32_t)k * stride;        // (k < 0: not used)
    if (k >= 0 && pos < end) {
        uint32_t a = (pos >> 3) & ~3u, x = lds_u32(a);
        for (; k >= 0 && pos + 64u <= end; k--, pos += 64u, a += 8, column -= stride) {
            const uint32_t y = lds_u32(a + 4), z = lds_u32(a + 8);
            sts_u64(column, __funnelshift_r(x, y, pos), __funnelshift_r(y, z, pos));
            x = z;
        }
        if (k >= 0 && pos < end) {         // the budget ends inside this plane
            const uint32_t m = end - pos;
            uint32_t wlo, whi;
            win64(pos, wlo, whi);
            sts_u64(column, wlo & bit_mask(m), whi & bit_mask(max(m, 32u) - 32u));
            k--;
            column -= stride;
        }
    }
    for (; k >= 3; k -= 4, column -= 4u * stride) {
        sts_u64(column, 0u, 0u);
        sts_u64(column - stride, 0u, 0u);
        sts_u64(column - 2u * stride, 0u, 0u);
        sts_u64(column - 3u * stride, 0u, 0u);
    }
    for (; k >= 0; k--, column -= stride) sts_u64(column, 0u, 0u);
}

// 32 words of bit planes to the coefficients' two's complement: a transpose
// whose odd planes (the negabinary digits of negative weight) are inverted on
// the way in, then one subtraction each
__device__ __forceinline__ void coefficients(uint32_t (&a)[32]) {
    transpose_round<1, true>(a);
    transpose_round<2>(a);
    transpose_round<4>(a);
    transpose_round<8>(a);
    transpose_round<16>(a);
#pragma unroll
    for (int p = 0; p < 32; p++) a[p] -= kNegaMask;
}

// The second half of decoding a block, after parse_planes has written its
// bit planes (plane k at planes + k * stride bytes, shared-window address)
// and its exponent: two 32x32 bit transposes turn the planes into the 64
// negabinary coefficients, which are mapped back to integers, put in
// block order, inverse-lifted along z, y and x and scaled into out[64].
__device__ __forceinline__ void finish_planes(uint32_t pa, uint32_t ps, int emax, float (&out)[64]) {
    constexpr CodingOrder order = make_coding_order();
    uint32_t q[64];
    {
        uint32_t a[32], b[32];             // coded coefficients 0..31 and 32..63
#pragma unroll
        for (int j = 0; j < 32; j++) lds_u64(pa + (uint32_t)j * ps, a[j], b[j]);
        coefficients(a);
        coefficients(b);
#pragma unroll
        for (int p = 0; p < 32; p++) {
            q[order.perm[p]] = a[p];
            q[order.perm[32 + p]] = b[p];
        }
    }
#pragma unroll
    for (int i = 0; i < 16; i++) inv_lift4u(q[i], q[i + 16], q[i + 32], q[i + 48]);             // z
#pragma unroll
    for (int z = 0; z < 4; z++)
#pragma unroll
        for (int x = 0; x < 4; x++) inv_lift4u(q[x + 16 * z], q[x + 4 + 16 * z], q[x + 8 + 16 * z], q[x + 12 + 16 * z]);  // y
#pragma unroll
    for (int i = 0; i < 16; i++) inv_lift4u(q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);  // x
    scale_block(q, emax - kPrecision, out);
}

// Decode a staged block of `rate` words into out[64] (block-local order).
// `planes` is this thread's column of a shared-memory area: plane k lives at
// planes[k * stride].  A zero block decodes to 64 samples of +0.
__device__ __forceinline__ void decode_staged(const uint32_t *staged, uint32_t rate, const uint32_t *tab,
                                              float (&out)[64], uint64_t *planes, uint32_t stride) {
    int emax = 0;
    const uint32_t pa = smem_u32(planes), ps = stride * 8u;
    parse_planes(smem_u32(staged), rate, smem_u32(tab), pa, ps, emax);
    finish_planes(pa, ps, emax, out);
}

// Write a warp's decoded blocks, 256 contiguous bytes each: lane i's v[64] to
// row `to` of 64 floats at `base` if bit i of `have` is set.  A lane's own
// 16-byte stores would touch 32 lines an instruction and half of each
// 32-byte sector, so the blocks pass through the warp's plane columns (plane
// k of its lanes is 256 bytes; the planes are used up), 16-byte pieces
// swizzled against bank conflicts, and every store writes two whole blocks.
// A caller's buffer that is not 16-byte aligned (`aligned` false, the same in
// every lane) takes 4-byte stores.  Called by all 32 lanes.
__device__ __forceinline__ void store_blocks(float *base, uint32_t to, uint32_t have, const float (&v)[64],
                                             uint64_t *planes, uint32_t stride, bool aligned = true) {
    const uint32_t lane = threadIdx.x & 31u, rows = smem_u32(planes) - lane * 8u, ps = stride * 8u;
    __syncwarp();                          // every lane has read its planes
#pragma unroll
    for (uint32_t c = 0; c < 16; c++)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(rows + lane * ps + ((c ^ (lane & 15u)) << 4)),
                     "f"(v[4 * c]), "f"(v[4 * c + 1]), "f"(v[4 * c + 2]), "f"(v[4 * c + 3]));
    __syncwarp();
    const uint32_t half = lane >> 4, piece = lane & 15u;
#pragma unroll
    for (uint32_t i = 0; i < 16; i++) {
        const uint32_t b = 2 * i + half;
        float4 d;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w)
                     : "r"(rows + b * ps + ((piece ^ (b & 15u)) << 4)));
        const uint32_t row = __shfl_sync(0xffffffffu, to, (int)b);
        if (aligned) {
            if ((have >> b) & 1u) *reinterpret_cast<float4 *>(base + (size_t)row * 64 + 4 * piece) = d;
        } else if ((have >> b) & 1u) {
            float *dst = base + (size_t)row * 64 + 4 * piece;
            dst[0] = d.x;
            dst[1] = d.y;
            dst[2] = d.z;
            dst[3] = d.w;
        }
    }
}

// Dynamic shared memory of a decoding kernel of `threads` threads: the
// plane columns (32 words of 8 bytes per thread), the group-step table, then
// one staging area per warp for blocks of up to `rate` words.
struct DecodeSmem {
    uint64_t *planes;
    uint32_t *tab;
    uint32_t *stage;          // this warp's staging area
};

__host__ __device__ constexpr size_t decode_smem_bytes(uint32_t threads, uint32_t rate) {
    return 32u * 8u * (size_t)threads + kGroupTableEntries * 4u + (size_t)(threads / 32u) * stage_words(rate) * 4u;
}

__device__ __forceinline__ DecodeSmem decode_smem_layout(uint64_t *base, uint32_t threads, uint32_t rate) {
    uint32_t *tab = reinterpret_cast<uint32_t *>(base + 32u * threads);
    return DecodeSmem{base, tab, tab + kGroupTableEntries + (threadIdx.x >> 5) * stage_words(rate)};
}

// ---------------------------------------------------------------- encoder (input generation)
//
// The encoder mirrors the decoder: a lane's 64 coefficients become 32 bit
// planes in its column of shared memory, one loop of uniform steps writes
// their code into the lane's staged block, and the warp copies its 32 staged
// blocks out together.  The bits past the budget are simply not kept: the
// code is a prefix of the unlimited one.  On the way each plane is cut down
// to what the kept bits say, so the columns end up holding what parse_planes
// would read back, and finish_planes gives the decoded samples without a
// parse.

// 32-bit words of a staged block being written (bits appended LSB first)
struct StagedWriter {
    uint32_t w, left;                      // shared address of the next word; words that may be kept
    uint64_t acc;                          // bits not yet stored
    uint32_t cnt;                          // how many (below 32 between calls)
    __device__ __forceinline__ void word(uint32_t v) {
        if (left) {
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(w), "r"(v));
            w += 4;
            left--;
        }
    }
    __device__ __forceinline__ void put(uint32_t bits, uint32_t n) {   // n <= 32; bits beyond n are zero
        acc |= (uint64_t)bits << cnt;
        cnt += n;
        if (cnt >= 32u) {
            word((uint32_t)acc);
            acc >>= 32;
            cnt -= 32u;
        }
    }
    __device__ __forceinline__ void finish() {                         // the rest of the block is zero
        if (left) word((uint32_t)acc);
        while (left) word(0u);
    }
};

// the inverse of `coefficients` but for the addition
__device__ __forceinline__ void digit_planes(uint32_t (&a)[32]) {
    transpose_round<16>(a);
    transpose_round<8>(a);
    transpose_round<4>(a);
    transpose_round<2>(a);
    transpose_round<1, false, true>(a);
}

// Turn v[64] into bit planes at `planes` + k * stride (plane k, shared-window
// address) and an exponent; false: the block is zero (no planes written).
__device__ __forceinline__ bool make_planes(const float (&v)[64], uint32_t planes, uint32_t stride, int &emax) {
    int maxe = 0;
    bool nonzero = false;
#pragma unroll
    for (int i = 0; i < 64; i++) {
        const uint32_t b = __float_as_uint(v[i]);
        nonzero |= (b & 0x7FFFFFFFu) != 0;
        maxe = max(maxe, (int)((b >> 23) & 0xFFu));
    }
    emax = maxe - 126;                     // frexp exponent of the largest sample, >= -126
    if (!nonzero) return false;
    int32_t q[64];
#pragma unroll
    for (int i = 0; i < 64; i++) {
        const uint32_t b = __float_as_uint(v[i]);
        const int E = (int)((b >> 23) & 0xFFu);
        const uint32_t M = E ? ((b & 0x7FFFFFu) | 0x800000u) : (b & 0x7FFFFFu);
        const int s = max(E, 1) - 150 + kPrecision - emax;   // |v| * 2^(P-emax) = M * 2^s
        uint32_t mag = s >= 0 ? (M << s) : (s > -32 ? (M >> -s) : 0u);
        q[i] = (b >> 31) ? -(int32_t)mag : (int32_t)mag;
    }
#pragma unroll
    for (int i = 0; i < 16; i++) fwd_lift4(q[4 * i], q[4 * i + 1], q[4 * i + 2], q[4 * i + 3]);  // x
#pragma unroll
    for (int z = 0; z < 4; z++)
#pragma unroll
        for (int x = 0; x < 4; x++) fwd_lift4(q[x + 16 * z], q[x + 4 + 16 * z], q[x + 8 + 16 * z], q[x + 12 + 16 * z]);  // y
#pragma unroll
    for (int i = 0; i < 16; i++) fwd_lift4(q[i], q[i + 16], q[i + 32], q[i + 48]);             // z
    constexpr CodingOrder order = make_coding_order();
    uint32_t lo[32], hi[32];
#pragma unroll
    for (int p = 0; p < 64; p++) {
        const uint32_t u = (uint32_t)q[order.perm[p]] + kNegaMask;   // (its odd digits are inverted as planes)
        if (p < 32) lo[p] = u; else hi[p - 32] = u;
    }
    digit_planes(lo);                      // lo[k] = plane k of coefficients 0-31
    digit_planes(hi);
#pragma unroll
    for (int k = 0; k < 32; k++) sts_u64(planes + (uint32_t)k * stride, lo[k], hi[k]);
    return true;
}

// Write the code of a block's planes to its staged words and cut the planes
// down to what the kept bits hold.  One loop for all lanes: a step opens a
// plane (its verbatim bits), then takes group-test events one by one: a
// test bit, the zeros and the one of the run up to the next coefficient
// reached (a one in the last coefficient is not sent), or the 0 test that
// ends the plane.
__device__ __forceinline__ void code_planes(StagedWriter &out, uint32_t rate, uint32_t planes, uint32_t stride,
                                            bool nonzero, int emax) {
    const uint32_t end = nonzero ? rate * 64u : 0u;
    uint32_t pos = 9, n = 0;               // n: coefficients reached
    int k = 31;
    if (nonzero) out.put(1u | ((uint32_t)(emax + 127) << 1), 9);
    uint64_t x = 0, kept = 0, rest = 0;    // the plane, what the kept bits say of it, its ones from n on
    bool opening = true;
    while (k >= 0 && pos < end) {
        if (opening) {
            uint32_t xlo, xhi;
            lds_u64(planes + (uint32_t)k * stride, xlo, xhi);
            x = ((uint64_t)xhi << 32) | xlo;
            const uint64_t low = low_mask(n);
            out.put(xlo & (uint32_t)low, min(n, 32u));
            if (n > 32u) out.put(xhi & (uint32_t)(low >> 32), n - 32u);
            kept = x & low & low_mask(min(64u, end - pos));
            rest = x & ~low;
            pos += n;
        }
        bool done = n >= 64u || pos >= end;
        if (!done) {
            if (rest == 0) {               // nothing more in this plane
                out.put(0u, 1);
                pos += 1;
                done = true;
            } else {
                const uint32_t p = (uint32_t)__ffsll((long long)rest) - 1u, z = p - n;
                // the test's 1, z zeros and, unless p is the last coefficient, its 1
                const uint32_t len = z + (p < 63u ? 2u : 1u);
                const uint64_t code = 1ull | (p < 63u && z < 63u ? 2ull << z : 0ull);
                out.put((uint32_t)code, min(len, 32u));
                if (len > 32u) out.put((uint32_t)(code >> 32), min(len, 64u) - 32u);
                pos += len;
                if (pos <= end) kept |= rest & (0ull - rest);
                rest &= rest - 1;
                n = p + 1;
                done = n >= 64u || pos >= end;
            }
        }
        if (done) {
            if (pos > end) sts_u64(planes + (uint32_t)k * stride, (uint32_t)kept, (uint32_t)(kept >> 32));
            else if (pos == end && kept != x) sts_u64(planes + (uint32_t)k * stride, (uint32_t)kept, (uint32_t)(kept >> 32));
            k--;
        }
        opening = done;
    }
    for (; k >= 0; k--) sts_u64(planes + (uint32_t)k * stride, 0u, 0u);
    out.finish();
}

}  // namespace bcmc
