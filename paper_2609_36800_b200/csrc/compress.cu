// The step before the product: bits = [W_fine - W_base > 0], alpha[b] = mean |W_fine - W_base|.
//
// The matrices are taken flat: K is a multiple of 32, so the words of all rows are one run of N K / 32.  A block takes tiles of 8192
// elements, a fixed stride apart.  Its producer thread streams a tile of W_base and then the same tile of every tenant through a ring in shared
// memory (bulk copies of 16 KB); eight warps, 32 elements per lane, keep the base in registers (as floats) for all tenants, so that it is read
// once.  The comparison is taken on the exact bf16 values (as fp32), through the sign of (base - fine); |delta| is formed in fp32, four at
// a time, and summed in double: per thread, then across the warp (shuffles), over the warp's tiles and the block (fixed order) into
// one partial per block and tenant; a second kernel adds the partials of a tenant in a fixed order.  Nothing depends on the order
// in which blocks run, nor on the device (the grid is a fixed number of blocks).
// Bound by DRAM: 8 x 4096 x 14336 in 166 us, 6.7 TB/s (6.2 with plain loads of 64 bytes per lane and row tiles of 1024 k, which waited for
// their latency), 8 x 4096 x 4096 52.6 us (60.5), and a K that is not a multiple of 1024 leaves no lanes idle: 12 x 3000 x 2080 34 us (46).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "gemm_common.cuh"
#include "gemm_tc.h"
#include "ptx.cuh"

namespace bd {

constexpr int kCompressWarps = 8;                          // consumers; the warp behind them is the producer
constexpr int kCompressTile = kCompressWarps * 1024, kCompressTileWords = kCompressTile / 32;   // elements, sign words
// 16 KB each, two blocks a multiprocessor: about 100 KB in flight.  More is slower, less too (8 x 4096 x 14336, two / three / four / six stages:
// 193 / 175 / 172 / 186 us with a contiguous run of tiles per block; three and four with strided tiles 166; one block of six 185).
constexpr int kCompressStages = 3;
constexpr int kCompressTenantChunk = 32;                   // tenants whose warp sums are staged in shared memory at once
constexpr uint32_t kCompressStageBytes = kCompressTile * 2;

struct CompressCtl {
    uint64_t full[kCompressStages], empty[kCompressStages];
    double warp_sum[kCompressTenantChunk][kCompressWarps];
    uint32_t abort_flag;
};
constexpr uint32_t kCompressSmem = kCompressStages * kCompressStageBytes + 128 + sizeof(CompressCtl);

__device__ __forceinline__ float bf16lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__global__ void __launch_bounds__((kCompressWarps + 1) * 32, 2)
compress_kernel(const uint8_t* __restrict__ Wf, const uint8_t* __restrict__ Wb, uint32_t* __restrict__ bits, double* __restrict__ partial, int B,
                long long words) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw), base = (raw + 127u) & ~127u;
    CompressCtl* ctl = reinterpret_cast<CompressCtl*>(smem_raw + (base - raw) + kCompressStages * kCompressStageBytes);
    volatile uint32_t* abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kCompressStages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), kCompressWarps);
        }
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) grid_launch_dependents();   // (the finishing kernel may become resident; it waits for this grid's end)
    // This block's tiles (first word): a fixed stride apart, so that the blocks are in one part of every matrix at any time.
    const long long lo = (long long)blockIdx.x * kCompressTileWords, step = (long long)gridDim.x * kCompressTileWords;
    int slot = 0;
    uint32_t phase = 0;
    if (warp == kCompressWarps) {
        if (lane == 0) {
            bool ok = true;
            grid_dependency_wait();
            for (int b0 = 0; b0 < B; b0 += kCompressTenantChunk) {
                const int nb = min(kCompressTenantChunk, B - b0);
                for (long long first = lo; ok && first < words; first += step) {
                    const uint32_t bytes = (uint32_t)min((long long)kCompressStageBytes, (words - first) * 64);
                    for (int j = -1; j < nb; ++j) {   // W_base, then the tenants
                        ok = wait_bar(smem_u32(&ctl->empty[slot]), phase ^ 1, abort_flag, 70);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&ctl->full[slot]);
                        mbar_arrive_expect_tx(bar, bytes);
                        bulk_load(base + (uint32_t)slot * kCompressStageBytes, (j < 0 ? Wb : Wf + (size_t)(b0 + j) * (size_t)words * 64) + first * 64, bytes, bar);
                        if (++slot == kCompressStages) { slot = 0; phase ^= 1; }
                    }
                }
            }
        }
    } else {
        // Lane l's 64 bytes of a tile, in the order 16-byte piece c ^ ((l >> 1) & 3), c = 0..3: eight lanes of a shared-memory phase hit
        // different banks.
        const uint32_t turn = (uint32_t)(lane >> 1) & 3u;
        const uint32_t off = (uint32_t)threadIdx.x * 64u;
        bool ok = true;
        grid_dependency_wait();   // the results may still be in use by the previous kernel
        auto load = [&](uint4 (&v)[4]) {
            // (one answer per warp: its lanes leave the wait one by one, and the votes below need all of them)
            ok = warp_all(ok && wait_bar(smem_u32(&ctl->full[slot]), phase, abort_flag, 71));
            const uint32_t st = base + (uint32_t)slot * kCompressStageBytes + off;
#pragma unroll
            for (uint32_t c = 0; c < 4; ++c)
                asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v[c].x), "=r"(v[c].y), "=r"(v[c].z), "=r"(v[c].w) : "r"(st + ((c ^ turn) << 4)) : "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->empty[slot]));
            if (++slot == kCompressStages) { slot = 0; phase ^= 1; }
        };
        for (int b0 = 0; b0 < B; b0 += kCompressTenantChunk) {
            const int nb = min(kCompressTenantChunk, B - b0);
            if (lane < nb) ctl->warp_sum[lane][warp] = 0.0;
            __syncwarp();
            for (long long first = lo; first < words; first += step) {
                const long long w = first + threadIdx.x;   // this lane's sign word
                const bool live = w < words;
                // This lane's 32 base weights as floats, once for all tenants of the chunk; x + 0 turns a -0 into +0 (see the
                // sign rule below).
                float gf[32];
                {
                    uint4 v[4];
                    load(v);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t g[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            gf[i * 8 + q * 2] = __fadd_rn(bf16lo(g[q]), 0.f);
                            gf[i * 8 + q * 2 + 1] = __fadd_rn(bf16hi(g[q]), 0.f);
                        }
                    }
                }
                uint32_t* dst = bits + (size_t)b0 * (size_t)words + w;
                for (int j = 0; j < nb; ++j, dst += words) {
                    uint4 v[4];
                    load(v);
                    // Sign bit k of the word = (fine > base) for element k = the sign of (base - fine), which is +0 when
                    // the two are equal (a base of -0 was made +0 above): a piece's elements are taken from the last to the
                    // first and each difference's sign bit is shifted in from the right (one funnel shift per element
                    // instead of a compare and a predicated OR).
                    uint32_t word = 0;
                    double acc = 0.0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t f[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
                        float s4[2] = {0.f, 0.f};
                        uint32_t byte = 0;
#pragma unroll
                        for (int q = 3; q >= 0; --q) {
                            const float d1 = gf[i * 8 + q * 2 + 1] - bf16hi(f[q]);
                            byte = __funnelshift_l(__float_as_uint(d1), byte, 1);
                            const float d0 = gf[i * 8 + q * 2] - bf16lo(f[q]);
                            byte = __funnelshift_l(__float_as_uint(d0), byte, 1);
                            s4[q >> 1] += fabsf(d0) + fabsf(d1);
                        }
                        word |= byte << (8 * ((uint32_t)i ^ turn));
                        acc += (double)s4[0] + (double)s4[1];
                    }
                    if (!live) acc = 0.0;
                    if (ok && live) *dst = word;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                    if (lane == 0) ctl->warp_sum[j][warp] += acc;
                }
            }
            named_bar_sync(1, kCompressWarps * 32);
            for (int j = (int)threadIdx.x; j < nb; j += kCompressWarps * 32) {
                double t = 0.0;
#pragma unroll
                for (int i = 0; i < kCompressWarps; ++i) t += ctl->warp_sum[j][i];
                partial[(size_t)(b0 + j) * gridDim.x + blockIdx.x] = t;
            }
            named_bar_sync(1, kCompressWarps * 32);
        }
    }
    __syncthreads();
    if (*abort_flag) {
        // A wait was abandoned: copies still in flight get a bounded time to land before shared memory is released.
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) {
        }
    }
}

// alpha[b] = (sum of the tenant's block partials, in a fixed order) / (N K), rounded to fp32.
__global__ void compress_finish_kernel(const double* __restrict__ partial, float* __restrict__ alpha, int nblocks,
                                       double inv_count) {
    // Launched with an early start behind compress_kernel (which releases it at once): resident and waiting when the
    // partials are complete, instead of a launch gap later.  It releases nothing itself: a product queued behind it with an early start fetches
    // sign words and scales at once, so it may begin only when they are written.
    grid_dependency_wait();
    const int b = blockIdx.x, lane = threadIdx.x;
    double t = 0.0;
    for (int i = lane; i < nblocks; i += 32) t += partial[(size_t)b * nblocks + i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) alpha[b] = (float)(t * inv_count);
}

// Blocks of the compress kernel: one per tile, but never more than a B200 holds at once (148 multiprocessors x 2): a fixed number, so
// that the order of the sums does not depend on the device.
constexpr long long kCompressMaxBlocks = 148 * 2;
long long compress_blocks(int N, int K) {
    const long long tiles = ((long long)N * K + kCompressTile - 1) / kCompressTile;
    return tiles < kCompressMaxBlocks ? tiles : kCompressMaxBlocks;
}

cudaError_t launch_compress(const void* Wf, const void* Wb, uint32_t* bits, float* alpha, double* partial, int B, int N,
                            int K, cudaStream_t stream) {
    const long long blocks = compress_blocks(N, K);
    static std::atomic<unsigned char> attr_done[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_done[dev].load()) {
        e = cudaFuncSetAttribute(compress_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCompressSmem);
        if (e != cudaSuccess) return e;
        attr_done[dev].store(1);
    }
    // (both kernels with an early start: they wait for their predecessor before they touch anything.  The first one's is worth 2 us of a call in
    // a row, 8 x 4096 x 4096 53.9 -> 51.9, and nothing in a graph.)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.stream = stream;
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((kCompressWarps + 1) * 32);
    cfg.dynamicSmemBytes = kCompressSmem;
    e = cudaLaunchKernelEx(&cfg, compress_kernel, static_cast<const uint8_t*>(Wf), static_cast<const uint8_t*>(Wb), bits, partial, B, (long long)N * (K / 32));
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((unsigned)B);
    cfg.blockDim = dim3(32u);
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, compress_finish_kernel, const_cast<const double*>(partial), alpha, (int)blocks,
                              1.0 / ((double)N * (double)K));
}

cudaError_t read_compress_status(unsigned int out[2]) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_device_status, sizeof(unsigned int) * 2);
    if (e != cudaSuccess) return e;
    if (out[0] != 0u) {
        const unsigned int zero[2] = {0u, 0u};
        e = cudaMemcpyToSymbol(g_device_status, zero, sizeof(zero));
    }
    return e;
}

}  // namespace bd
