// BitDelta fused GEMM, row-stream decode kernel (few token rows): ONE launch, nothing but the call's own arrays.
//
//   Y[b,t,n] = act( sum_k X[b,t,k] W[n,k] + alpha[b] sum_k X[b,t,k] S[b,n,k] + bias[n] )
//
// A unit is up to sixteen weight rows, all of K, up to eight tenants.  A producer thread streams W_base, sign words and
// activations through shared memory in stages of 1024 k (bulk-tensor copies, 128-byte rows); eight consumer warps take 128 k
// of a stage each and keep fp32 sums in registers; at the end of a unit the eight partial sums are added in shared memory.
// There is no activation pre-pass, no tensor-memory hand-over, no workspace and no sum across blocks: for few tenants
// those latencies are most of a call of the other decode kernels (1 x 8 x 1024 x 1024: 2.3 us, 5.3 there; 8 x 1 x 2048 x 2048:
// 6.2 and 14.3; 1 x 1 x 4096 x 4096: 8.3 and 10.3, 4.3 TB/s).
//
// The products run on mma.sync (m16n8k16, the weights on the 16-row side), because its A operand comes from registers, where the
// decoded signs are; that path is a quarter as fast as tcgen05, which is what limits the kernel to few tenants.
//   * k is dealt to the threads of a fragment by words: thread t of a quad owns word t of the warp's 128 k, in both operands.
//   * Signs are operands +-1, exactly: bits p and p + 16 of a word, shifted to the two halves' sign bits, flip the signs of a pair of
//     ones (a shift and a logic operation per two of them).  Every product is exact, so the sums are as good as fp32 accumulation
//     makes them, and infinities and NaN come out by themselves.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "gemm_common.cuh"
#include "gemm_row.h"
#include "ptx.cuh"

namespace bd {

constexpr int kRowWarps = 8;                                  // consumers; warp 8 is the producer
constexpr int kRowThreads = (kRowWarps + 1) * 32;

// The matrix unit truncates as it accumulates, so a long chain of MMAs drifts: at most this many stages (of eight MMAs per sum and
// warp) are one chain, then a rounded addition takes over.  Error of the delta's sum against 64 bits, relative, 2 x 8 x 14336 x 1024 in
// binary16, in one chain, in chains of four and of two stages (8-bit kernel): N(0, 1) 1.7e-7, 8.6e-8, 8.8e-8 (8.2e-7); heavy-tailed,
// N(0, 1) times exp(1.5 N(0, 1)), 1.5e-6, 3.1e-7, 1.9e-7 (1.8e-7).  Time, 2 x 1 x 6656 x 9920: 27.4, 27.6, 28.2 us; a form of its own
// for K within one chain, which does not pay for the additions (2 x 1 x 4096 x 4096 9.3 us, 9.6 with them).
constexpr int kRowChainStages = 4;

struct RowCtl {
    uint64_t full[kRowMaxStages], empty[kRowMaxStages];
    uint32_t abort_flag;
};
static_assert(sizeof(RowCtl) <= 1024, "control block too large");

// (not volatile: the compiler may interleave independent sums)
template <bool kF16>
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    if constexpr (kF16)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// Signs p and p + 16 of a word as a pair of +-1 in the I/O type (`minus_one2`: two of -1, in a register: and_xor).
__device__ __forceinline__ uint32_t row_sign_pair(uint32_t w, int p, uint32_t minus_one2) {   // (p: a constant after unrolling)
    return and_xor(w << (15 - p), 0x80008000u, minus_one2);
}

// kTpt: tenants per activation tile, kNt: activation tiles per unit, kLong: K beyond one chain.
template <bool kF16, int kTpt, int kNt, bool kLong>
__global__ void __launch_bounds__(kRowThreads, 1)
bitdelta_gemm_row_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                         const __grid_constant__ CUtensorMap tmBits, const RowArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw);
    const uint32_t red_off = (uint32_t)a.stages * a.stage_bytes;
    constexpr int kRedBufs = kNt < 4 ? 2 : 1;
    constexpr int kRedFloats = kNt * kRowWarps * 128;                            // [warp][tile][column][16 rows]
    RowCtl* ctl = reinterpret_cast<RowCtl*>(smem + red_off + kRedBufs * kRedFloats * 4);
    volatile uint32_t* abort_flag = &ctl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRowMaxStages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), kRowWarps);
        }
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) grid_launch_dependents();

    if (warp == kRowWarps) {
        // ------------------------------------------------------------ producer (one thread)
        if (lane == 0) {
            prefetch_tensormap(&tmW);
            prefetch_tensormap(&tmBits);
            prefetch_tensormap(&tmX);
            const uint32_t tx = (uint32_t)a.rows * 2048u + (uint32_t)(a.TB * a.rows) * 128u + (uint32_t)kNt * 16384u;
            auto weights = [&](int unit, int s, int slot) {
                const int tile = unit / a.groups, g = unit - tile * a.groups;
                const uint32_t bar = smem_u32(&ctl->full[slot]), dst = base + (uint32_t)slot * a.stage_bytes;
                mbar_arrive_expect_tx(bar, tx);
                tma_load_3d(dst, &tmW, bar, 0, tile * a.rows, s * (kRowStageK / kAtomK));
                tma_load_3d(dst + a.s_off, &tmBits, bar, s * (kRowStageK / 32), tile * a.rows, g * kTpt * kNt);
            };
            auto activations = [&](int unit, int s, int slot) {
                const int g = unit % a.groups;
                const uint32_t bar = smem_u32(&ctl->full[slot]), dst = base + (uint32_t)slot * a.stage_bytes + a.x_off;
#pragma unroll
                for (int i = 0; i < kNt; ++i)
                    tma_load_3d(dst + i * 16384u, &tmX, bar, 0, (g * kNt + i) * kTpt * a.m, s * (kRowStageK / kAtomK));
            };
            // the weights do not depend on the kernel before this one: as many stages as there is room for, then the rest
            int unit = (int)blockIdx.x, s = 0, n = 0;
            auto advance = [&](int& un, int& st) { if (++st == a.k_stages) { st = 0; un += (int)gridDim.x; } };
            for (; n < a.stages && unit < a.units; ++n, advance(unit, s)) weights(unit, s, n);
            grid_dependency_wait();
            int xu = (int)blockIdx.x, xs = 0;
            for (int i = 0; i < n; ++i, advance(xu, xs)) activations(xu, xs, i);
            int slot = 0;
            uint32_t phase = 0;
            for (; unit < a.units; advance(unit, s)) {
                if (!wait_bar(smem_u32(&ctl->empty[slot]), phase, abort_flag, 40)) break;
                weights(unit, s, slot);
                activations(unit, s, slot);
                if (++slot == a.stages) { slot = 0; phase ^= 1; }
            }
        }
    } else {
        // ------------------------------------------------------------ consumers
        const int g = lane >> 2, t = lane & 3;
        // this thread's four 16-byte chunks of a row's 128 k (slot i: chunk i, for t >= 2 chunk i ^ 2: the eight lanes of a
        // shared-memory phase then hit different banks; its sign words are turned by sixteen bits to match)
        const int atom = 2 * warp + (t >> 1), c0 = (t & 1) * 4, flip = t & 2;
        const int turn = flip ? 16 : 0;
        const uint32_t xrow = (uint32_t)(atom * 8 + g);
        // (rows past a short unit's last one read what follows in the stage: they only reach their own outputs, not written)
        const uint32_t wrow0 = (uint32_t)(atom * a.rows + g), wrow1 = wrow0 + 8;
        bool ok = true;
        int slot = 0;
        uint32_t phase = 0, minus_one2 = kF16 ? 0xBC00BC00u : 0xBF80BF80u;
        asm volatile("" : "+r"(minus_one2));
        const int m = a.m;
        const int jc[2] = {2 * t / m, (2 * t + 1) / m};   // the tenant of the tile that this thread's two columns belong to
        // The partial results of successive units go to two buffers in turn: a warp that writes a buffer again has passed the
        // barrier of the unit between, which the others reach only after they have read it, so one barrier a unit is enough
        // (2 x 1 x 4096 x 4096 10.5 -> 9.9 us then, 2 x 4 x 1024 x 8192 8.4 -> 7.8).  Four activation tiles leave no room for two.
        for (int unit = (int)blockIdx.x, odd = 0; unit < a.units; unit += (int)gridDim.x, odd ^= 1) {
            float* red = reinterpret_cast<float*>(smem + red_off) + (kRedBufs == 2 ? odd * kRedFloats : 0);
            const int tile = unit / a.groups, grp = unit - tile * a.groups;
            const int n0 = tile * a.rows, tenant0 = grp * kTpt * kNt;
            const int nten = min(kTpt * kNt, a.B - tenant0);
            float accb[kNt][4], accd[kNt][kTpt][4], sum[kNt][4], al[kNt][2];
#pragma unroll
            for (int i = 0; i < kNt; ++i) {
#pragma unroll
                for (int e = 0; e < 4; ++e) sum[i][e] = 0.f;
#pragma unroll
                for (int e = 0; e < 2; ++e) al[i][e] = (jc[e] < kTpt && i * kTpt + jc[e] < nten) ? __ldg(a.alpha + tenant0 + i * kTpt + jc[e]) : 0.f;
            }
            // this warp's 128 k of a stage
            auto stage = [&] {
                const uint32_t st = base + (uint32_t)slot * a.stage_bytes;
#pragma unroll
                for (int i = 0; i < kNt; ++i) {
                    uint4 x[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        x[q] = lds128(st + a.x_off + i * 16384u + xrow * 128u + (uint32_t)(((c0 + (q ^ flip)) ^ (xrow & 7)) << 4));
                    // the tenants' sign words of the rows g, g + 8 (tenants past the unit's own: the first one's, not used)
                    uint32_t sw[kTpt][2];
#pragma unroll
                    for (int j = 0; j < kTpt; ++j) {
                        const int jj = i * kTpt + j < nten ? i * kTpt + j : 0;
                        const uint32_t r0 = (uint32_t)(jj * a.rows + g), r1 = r0 + 8;
                        const uint32_t sb = st + a.s_off + (uint32_t)(t * 4);
                        sw[j][0] = lds32(sb + r0 * 128u + ((warp ^ (r0 & 7)) << 4));
                        sw[j][1] = lds32(sb + r1 * 128u + ((warp ^ (r1 & 7)) << 4));
                    }
                    // the activations as pairs (k, k + 16) of the thread's word, like the signs
                    uint32_t xp[16];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const uint32_t lo[4] = {x[q].x, x[q].y, x[q].z, x[q].w}, hi[4] = {x[q + 2].x, x[q + 2].y, x[q + 2].z, x[q + 2].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            xp[8 * q + 2 * e] = __byte_perm(lo[e], hi[e], 0x5410);
                            xp[8 * q + 2 * e + 1] = __byte_perm(lo[e], hi[e], 0x7632);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kTpt; ++j) {
                        sw[j][0] = __funnelshift_l(sw[j][0], sw[j][0], turn);
                        sw[j][1] = __funnelshift_l(sw[j][1], sw[j][1], turn);
                    }
                    // (independent sums next to one another: a sum's MMAs wait for each other.  No test in here: with one per MMA
                    // 8 x 1 x 4096 x 4096 took 48 us instead of 20)
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if ((q & 1) == 0) {
                            const int c = q >> 1;
                            const uint4 w0 = lds128(st + wrow0 * 128u + (uint32_t)(((c0 + (c ^ flip)) ^ (wrow0 & 7)) << 4));
                            const uint4 w1 = lds128(st + wrow1 * 128u + (uint32_t)(((c0 + (c ^ flip)) ^ (wrow1 & 7)) << 4));
                            mma16816<kF16>(accb[i], w0.x, w1.x, w0.y, w1.y, x[c].x, x[c].y);
                            mma16816<kF16>(accb[i], w0.z, w1.z, w0.w, w1.w, x[c].z, x[c].w);
                        }
#pragma unroll
                        for (int j = 0; j < kTpt; ++j)
                            mma16816<kF16>(accd[i][j], row_sign_pair(sw[j][0], 2 * q, minus_one2), row_sign_pair(sw[j][1], 2 * q, minus_one2),
                                           row_sign_pair(sw[j][0], 2 * q + 1, minus_one2), row_sign_pair(sw[j][1], 2 * q + 1, minus_one2),
                                           xp[2 * q], xp[2 * q + 1]);
                    }
                }
            };
            int s = 0;
            do {
                const int end = kLong ? min(s + kRowChainStages, a.k_stages) : a.k_stages;
#pragma unroll
                for (int i = 0; i < kNt; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        accb[i][e] = 0.f;
#pragma unroll
                        for (int j = 0; j < kTpt; ++j) accd[i][j][e] = 0.f;
                    }
                for (; s < end; ++s) {
                    // (one answer per warp: its lanes leave the wait one by one, and the matrix instructions below need all of them)
                    ok = warp_all(ok && wait_bar(smem_u32(&ctl->full[slot]), phase, abort_flag, 41));
                    if (ok && s * kRowStageK + warp * 128 < a.K) stage();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->empty[slot]));
                    if (++slot == a.stages) { slot = 0; phase ^= 1; }
                }
                // this warp's share of every output: base + alpha * delta
#pragma unroll
                for (int i = 0; i < kNt; ++i) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float d[kTpt];   // (selected bit by bit of the tenant's number: of a chain of tests the compiler makes an array in local memory)
#pragma unroll
                        for (int j = 0; j < kTpt; ++j) d[j] = accd[i][j][e];
#pragma unroll
                        for (int w = kTpt / 2; w > 0; w /= 2)
#pragma unroll
                            for (int j = 0; j < w; ++j) d[j] = (jc[e & 1] & w) ? d[j + w] : d[j];
                        const float v = fmaf(al[i][e & 1], d[0], accb[i][e]);
                        sum[i][e] = kLong ? sum[i][e] + v : v;
                    }
                }
            } while (kLong && s < a.k_stages);
#pragma unroll
            for (int i = 0; i < kNt; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) red[((warp * kNt + i) * 8 + 2 * t + (e & 1)) * 16 + g + 8 * (e >> 1)] = sum[i][e];
            named_bar_sync(1, kRowWarps * 32);
            grid_dependency_wait();   // Y may still be in use by the previous kernel
#pragma unroll
            for (int o = 0; o < kNt * 128; o += kRowWarps * 32) {
                const int idx = o + (int)threadIdx.x;
                if (idx < kNt * 128) {   // (whole warps)
                    const int i = idx >> 7, col = (idx >> 4) & 7, row = idx & 15;
                    float v = 0.f;
#pragma unroll
                    for (int w = 0; w < kRowWarps; ++w) v += red[((w * kNt + i) * 8 + col) * 16 + row];
                    const int jt = col / m, n = n0 + row, b = tenant0 + i * kTpt + jt;
                    const bool live = ok && jt < kTpt && b < a.B && row < a.rows && n < a.N;
                    const int tok = b * m + col - jt * m;
                    if (a.bias && n < a.N) v += from_io16(__ldg(static_cast<const uint16_t*>(a.bias) + n), kF16);
                    uint16_t* Y = static_cast<uint16_t*>(a.Y);
                    if (a.act == 2) {
                        // SiLU gate: rows 2i (gate) and 2i + 1 (up) are neighbouring lanes
                        const float up = __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                        if (live && !(n & 1)) Y[(size_t)tok * (a.N >> 1) + (n >> 1)] = to_io16(__fdividef(v, 1.f + __expf(-v)) * up, kF16);
                    } else if (live) {
                        Y[(size_t)tok * a.N + n] = finish_io16(v, 0.f, a.act, kF16);
                    }
                }
            }
            if constexpr (kRedBufs == 1) named_bar_sync(1, kRowWarps * 32);   // the partial sums are read: the next unit's may come
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

typedef void (*RowKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const RowArgs);
template <bool kF16, bool kLong> static RowKernel row_kernel(int tpt, int nt) {
    switch (tpt * 8 + nt) {
        case 65: return bitdelta_gemm_row_kernel<kF16, 8, 1, kLong>;
        case 33: return bitdelta_gemm_row_kernel<kF16, 4, 1, kLong>;
        case 34: return bitdelta_gemm_row_kernel<kF16, 4, 2, kLong>;
        case 17: return bitdelta_gemm_row_kernel<kF16, 2, 1, kLong>;
        case 18: return bitdelta_gemm_row_kernel<kF16, 2, 2, kLong>;
        case 20: return bitdelta_gemm_row_kernel<kF16, 2, 4, kLong>;
        case 9: return bitdelta_gemm_row_kernel<kF16, 1, 1, kLong>;
        case 10: return bitdelta_gemm_row_kernel<kF16, 1, 2, kLong>;
        case 12: return bitdelta_gemm_row_kernel<kF16, 1, 4, kLong>;
    }
    return nullptr;
}

cudaError_t launch_gemm_row(const CUtensorMap& tmW, const CUtensorMap& tmX, const CUtensorMap& tmBits, const RowArgs& args,
                            const RowPlan& p, bool early_start, cudaStream_t stream) {
    const bool long_k = p.k_stages > kRowChainStages;
    const RowKernel k = args.f16 ? (long_k ? row_kernel<true, true>(p.tpt, p.nt) : row_kernel<true, false>(p.tpt, p.nt))
                                 : (long_k ? row_kernel<false, true>(p.tpt, p.nt) : row_kernel<false, false>(p.tpt, p.nt));
    if (!k) return cudaErrorInvalidValue;
    static std::atomic<unsigned char> attr_done[64][4][72];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::atomic<unsigned char>& done = attr_done[dev][(args.f16 ? 2 : 0) + (long_k ? 1 : 0)][p.tpt * 8 + p.nt];
    if (!done.load()) {
        e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
        if (e != cudaSuccess) return e;
        done.store(1);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid);
    cfg.blockDim = dim3((unsigned)kRowThreads);
    cfg.dynamicSmemBytes = p.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early_start ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, tmW, tmX, tmBits, args);
}

cudaError_t read_row_status(unsigned int out[2]) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_device_status, sizeof(unsigned int) * 2);
    if (e != cudaSuccess) return e;
    if (out[0] != 0u) {
        const unsigned int zero[2] = {0u, 0u};
        e = cudaMemcpyToSymbol(g_device_status, zero, sizeof(zero));
    }
    return e;
}

}  // namespace bd
