// Stand-alone codec kernels: encode a device field (input generation),
// decode an explicit list of blocks, and decode a whole volume into a
// dense field (the full-volume baseline of the paper's ZFP decompression
// measurements).
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "codec.cuh"
#include "kernels.cuh"

namespace bcmc {

constexpr uint32_t kCodecThreads = 128;

// the codec kernels' dynamic shared memory (plane columns, group-step
// table, staging areas), with the table filled
__device__ __forceinline__ DecodeSmem codec_smem(uint64_t *base, uint32_t rate) {
    const DecodeSmem sm = decode_smem_layout(base, kCodecThreads, rate);
    load_group_table(sm.tab);
    __syncthreads();
    return sm;
}

// One lane per block, a warp's 32 blocks in id order: gather the 4x4x4
// samples (repeating the last sample past the volume edge; a warp's rows are
// contiguous, so 16 bytes a lane where rows are aligned), make and code the
// planes, copy the 32 staged blocks out as one contiguous span of the
// bitstream, and take each block's range over its in-volume samples as the
// kept bits decode.  Bound by instruction issue and latency at 16 warps an SM
// (56% of issue slots, 62% of the ALU pipe): the coding loop is a few dozen
// steps of some 40 instructions, beside the two transforms.  499 x 333 x 218
// samples at 6 bits a value: 273 us.  A thread per block that wrote its
// words to memory one by one and parsed them again for the range took 1160.
__global__ void __launch_bounds__(kCodecThreads, 4) encode_kernel(const float *__restrict__ field, Geom g, uint64_t *bits,
                                                               float *bmin, float *bmax) {
    extern __shared__ __align__(16) uint64_t dsm[];
    const DecodeSmem sm = decode_smem_layout(dsm, kCodecThreads, g.rate);
    const uint32_t planes = smem_u32(sm.planes + threadIdx.x), ps = 8u * kCodecThreads;
    const uint32_t lane = threadIdx.x & 31u, stride = 2u * g.rate + 1u;   // words a staged block takes
    const uint32_t mine = smem_u32(sm.stage + lane * stride);
    const bool rows16 = (g.nx & 3u) == 0 && (reinterpret_cast<uintptr_t>(field) & 15u) == 0;
    for (uint32_t b0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b0 < g.nb; b0 += gridDim.x * blockDim.x) {
        const uint32_t b = b0 + lane;
        uint32_t bx = 0, by = 0, bz = 0;
        int emax = 0;
        bool nonzero = false;
        if (b < g.nb) {
            block_coords(g, b, bx, by, bz);
            float v[64];
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const uint32_t y = min(4 * by + j, g.ny - 1), z = min(4 * bz + k, g.nz - 1);
                    const float *row = field + (size_t)g.nx * ((size_t)y + (size_t)g.ny * z);
                    if (rows16) {
                        const float4 r = __ldg(reinterpret_cast<const float4 *>(row + 4 * bx));
                        v[4 * j + 16 * k] = r.x;
                        v[4 * j + 16 * k + 1] = r.y;
                        v[4 * j + 16 * k + 2] = r.z;
                        v[4 * j + 16 * k + 3] = r.w;
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; i++) v[i + 4 * j + 16 * k] = __ldg(row + min(4 * bx + i, g.nx - 1));
                    }
                }
            nonzero = make_planes(v, planes, ps, emax);
            StagedWriter out{mine, 2u * g.rate, 0ull, 0u};
            code_planes(out, g.rate, planes, ps, nonzero, emax);
        }
        __syncwarp();                                   // the staged blocks are written
        const uint32_t words = min(32u, g.nb - b0) * g.rate, magic = (65535u + g.rate) / g.rate;   // as in stage_blocks
        for (uint32_t j = lane; j < words; j += 32u) {
            const uint32_t q = (j * magic) >> 16, w = q * stride + 2u * (j - q * g.rate);
            bits[(size_t)b0 * g.rate + j] = (uint64_t)sm.stage[w] | ((uint64_t)sm.stage[w + 1] << 32);
        }
        __syncwarp();                                   // they are read
        if (b >= g.nb) continue;
        float d[64];
        finish_planes(planes, ps, nonzero ? emax : -127, d);
        float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000);   // +inf, -inf
#pragma unroll
        for (int k = 0; k < 4; k++)
#pragma unroll
            for (int j = 0; j < 4; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    if (4 * bx + i >= g.nx || 4 * by + j >= g.ny || 4 * bz + k >= g.nz) continue;
                    const float x = d[i + 4 * j + 16 * k];
                    if (x < lo) lo = x;
                    if (x > hi) hi = x;
                }
        bmin[b] = lo;
        bmax[b] = hi;
    }
}

__global__ void __launch_bounds__(kCodecThreads, 5) decode_list_kernel(const uint64_t *__restrict__ bits, uint32_t rate,
                                                                    const uint32_t *__restrict__ ids, uint64_t n,
                                                                    float *out) {
    extern __shared__ __align__(16) uint64_t dsm[];
    const DecodeSmem sm = codec_smem(dsm, rate);
    const uint32_t lane = threadIdx.x & 31u;
    const bool aligned = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
    for (uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); i0 < n;
         i0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = i0 + lane;
        const bool have = i < n;
        stage_blocks(bits, rate, have ? ids[i] : 0u, have, sm.stage);
        float v[64];                       // (a lane without a block decodes a zero one)
        decode_staged(sm.stage + lane * (2u * rate + 1u), rate, sm.tab, v, sm.planes + threadIdx.x, blockDim.x);
        store_blocks(out + i0 * 64, lane, __ballot_sync(0xffffffffu, have), v, sm.planes + threadIdx.x, blockDim.x,
                     aligned);
    }
}

// One block per lane, blocks in id order: decode, then write the block's
// in-volume samples into the dense x-fastest field.  Lanes of a warp hold
// consecutive blocks along x, so each row store of the warp covers one
// contiguous span of the field, and the staging loads read one contiguous
// span of the bitstream.
__global__ void __launch_bounds__(kCodecThreads, 5) decode_volume_kernel(const uint64_t *__restrict__ bits, Geom g,
                                                                      float *field, uint32_t skew) {
    extern __shared__ __align__(16) uint64_t dsm[];
    const DecodeSmem sm = codec_smem(dsm, g.rate);
    const bool rows16 = (skew & 3u) == 0;       // every row starts 16-byte aligned
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t b0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b0 < g.nb; b0 += gridDim.x * blockDim.x) {
        const uint32_t b = b0 + lane;
        const bool have = b < g.nb;
        stage_blocks(bits, g.rate, b, have, sm.stage);
        const uint64_t ahead = (uint64_t)b + gridDim.x * blockDim.x;       // its latency passes during this decode
        if (ahead < g.nb) prefetch_block(bits, g.rate, (uint32_t)ahead);
        if (!have) continue;
        uint32_t bx, by, bz;
        block_coords(g, b, bx, by, bz);
        float v[64];
        decode_staged(sm.stage + lane * (2u * g.rate + 1u), g.rate, sm.tab, v, sm.planes + threadIdx.x, blockDim.x);
        const uint32_t x0 = 4 * bx;
        const bool full_x = x0 + 4 <= g.nx;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t z = 4 * bz + k;
            if (z >= g.nz) break;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t y = 4 * by + j;
                if (y >= g.ny) break;
                float *row = field + (size_t)x0 + (size_t)g.nx * ((size_t)y + (size_t)g.ny * z);
                if (rows16 && full_x) {
                    *reinterpret_cast<float4 *>(row) =
                        make_float4(v[16 * k + 4 * j], v[16 * k + 4 * j + 1], v[16 * k + 4 * j + 2], v[16 * k + 4 * j + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++)
                        if (x0 + i < g.nx) row[i] = v[16 * k + 4 * j + i];
                }
            }
        }
    }
}

// Launch a codec kernel over n blocks, a lane each, with no more CTAs than
// the device holds at once: each fills its group-step table once (a CTA per
// 128 blocks spent a part of its time on that, and the launch on 20 waves of
// them: 474 us for the 512^3 decode at 8 bits a value, 385 with resident CTAs,
// 310 with the present parse).  The
// resident count is looked up once per kernel, device and rate.
template <class K, class... A>
void launch_codec(K kernel, std::atomic<uint32_t> (*known)[33], uint32_t rate, uint64_t n, cudaStream_t st, A... args) {
    constexpr int kDevices = 64;
    const size_t bytes = decode_smem_bytes(kCodecThreads, rate);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;      // the caller reads the error
    uint32_t resident = dev < kDevices ? known[dev][rate].load(std::memory_order_acquire) : 0u;
    if (resident == 0) {
        // the limit is set for the largest rate, so any launch fits
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)decode_smem_bytes(kCodecThreads, 32));
        int sms = 1, occ = 1;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kCodecThreads, bytes) != cudaSuccess)
            return;
        resident = (uint32_t)(std::max(1, sms) * std::max(1, occ));
        if (dev < kDevices) known[dev][rate].store(resident, std::memory_order_release);
    }
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((n + kCodecThreads - 1) / kCodecThreads, resident));
    kernel<<<(unsigned)blocks, kCodecThreads, bytes, st>>>(args...);
}

std::atomic<uint32_t> g_known[3][64][33];               // decode_volume, encode, decode_list

void launch_decode_volume(const uint64_t *bits, const Geom &g, float *field, cudaStream_t st) {
    // rows are aligned when they hold a multiple of four floats and the field,
    // which may start at any float, is
    const uint32_t skew = g.nx | (uint32_t)((reinterpret_cast<uintptr_t>(field) & 15u) / 4u);
    launch_codec(decode_volume_kernel, g_known[0], g.rate, g.nb, st, bits, g, field, skew);
}

void launch_encode(const float *field, const Geom &g, uint64_t *bits, float *bmin, float *bmax, cudaStream_t st) {
    launch_codec(encode_kernel, g_known[1], g.rate, g.nb, st, field, g, bits, bmin, bmax);
}

void launch_decode_list(const uint64_t *bits, uint32_t rate, const uint32_t *ids, uint64_t n, float *out,
                        cudaStream_t st) {
    if (n == 0) return;
    launch_codec(decode_list_kernel, g_known[2], rate, n, st, bits, rate, ids, n, out);
}

}  // namespace bcmc
