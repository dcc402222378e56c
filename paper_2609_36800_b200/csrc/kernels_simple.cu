// Plain CUDA-core kernels: sign packing / unpacking and a diagnostic GEMM.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include "gemm_tc.h"
#include "ptx.cuh"

namespace bd {

// One thread per output word: reads 32 consecutive int8 (two 16-byte loads, so
// a warp reads 1 KiB contiguously) and sets bit j when element j is positive.
__global__ void pack_kernel(const int8_t* __restrict__ S, uint32_t* __restrict__ bits, long long words) {
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= words) return;
    const uint4* src = reinterpret_cast<const uint4*>(S + w * 32);
    uint32_t word = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint4 v = __ldg(src + h);
        const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int byte = 0; byte < 4; ++byte) {
                const int8_t s = (int8_t)((q[i] >> (8 * byte)) & 0xFF);
                if (s > 0) word |= 1u << (h * 16 + i * 4 + byte);
            }
        }
    }
    bits[w] = word;
}

__global__ void unpack_kernel(const uint32_t* __restrict__ bits, int8_t* __restrict__ S, long long words) {
    const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= words) return;
    const uint32_t word = __ldg(bits + w);
    uint4* dst = reinterpret_cast<uint4*>(S + w * 32);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t v = 0;
#pragma unroll
            for (int byte = 0; byte < 4; ++byte) {
                const uint32_t bit = (word >> (h * 16 + i * 4 + byte)) & 1u;
                v |= (bit ? 0x01u : 0xFFu) << (8 * byte);
            }
            q[i] = v;
        }
        dst[h] = make_uint4(q[0], q[1], q[2], q[3]);
    }
}

// One warp per (tenant, weight row); lanes stride over the sign words, so lane l
// owns k = 32w .. 32w+31 for w = l, l+32, ...  fp32 accumulation, shuffle reduce.
// 16-bit values of the I/O type (bf16, or IEEE binary16 when `f16`) <-> fp32.
__device__ __forceinline__ float io16_to_float(uint16_t h, int f16) {
    return f16 ? __half2float(__ushort_as_half(h)) : __uint_as_float((uint32_t)h << 16);
}
__device__ __forceinline__ uint16_t float_to_io16(float v, int f16) {
    return f16 ? __half_as_ushort(__float2half_rn(v)) : __bfloat16_as_ushort(__float2bfloat16_rn(v));
}

__global__ void gemm_simt_kernel(const uint16_t* __restrict__ X, const uint16_t* __restrict__ W,
                                 const uint32_t* __restrict__ bits, const float* __restrict__ alpha,
                                 const uint16_t* __restrict__ bias, uint16_t* __restrict__ Y, int B, int m, int N,
                                 int K, int f16, int act) {
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (gw >= (long long)B * N) return;
    const int b = (int)(gw / N);
    const int n = (int)(gw % N);
    const int words = K >> 5;
    const float al = alpha[b];
    if (act == 2) {
        // SiLU gate over interleaved (gate, up) rows: the warp of the gate row computes both rows of its pair
        if (n & 1) return;
        for (int t = 0; t < m; ++t) {
            const uint16_t* xrow = X + ((size_t)b * m + t) * K;
            float z[2];
            for (int r = 0; r < 2; ++r) {
                const uint32_t* brow2 = bits + ((size_t)b * N + n + r) * words;
                const uint16_t* wrow2 = W + (size_t)(n + r) * K;
                float base = 0.f, delta = 0.f;
                for (int w = lane; w < words; w += 32) {
                    const uint32_t word = brow2[w];
#pragma unroll 8
                    for (int j = 0; j < 32; ++j) {
                        const float x = io16_to_float(xrow[w * 32 + j], f16);
                        base = fmaf(x, io16_to_float(wrow2[w * 32 + j], f16), base);
                        delta += ((word >> j) & 1u) ? x : -x;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    base += __shfl_xor_sync(0xFFFFFFFFu, base, o);
                    delta += __shfl_xor_sync(0xFFFFFFFFu, delta, o);
                }
                z[r] = fmaf(al, delta, base) + (bias ? io16_to_float(bias[n + r], f16) : 0.f);
            }
            if (lane == 0) Y[((size_t)b * m + t) * (N >> 1) + (n >> 1)] = float_to_io16(z[0] / (1.f + __expf(-z[0])) * z[1], f16);
        }
        return;
    }
    const uint32_t* brow = bits + ((size_t)b * N + n) * words;
    const uint16_t* wrow = W + (size_t)n * K;
    const float bias_n = bias ? io16_to_float(bias[n], f16) : 0.f;
    for (int t = 0; t < m; ++t) {
        const uint16_t* xrow = X + ((size_t)b * m + t) * K;
        float base = 0.f, delta = 0.f;
        for (int w = lane; w < words; w += 32) {
            const uint32_t word = brow[w];
#pragma unroll 8
            for (int j = 0; j < 32; ++j) {
                const float x = io16_to_float(xrow[w * 32 + j], f16);
                base = fmaf(x, io16_to_float(wrow[w * 32 + j], f16), base);
                delta += ((word >> j) & 1u) ? x : -x;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            base += __shfl_xor_sync(0xFFFFFFFFu, base, o);
            delta += __shfl_xor_sync(0xFFFFFFFFu, delta, o);
        }
        if (lane == 0) {
            float v = fmaf(al, delta, base) + bias_n;
            if (act == 1) v = v / (1.f + __expf(-v));   // SiLU
            Y[((size_t)b * m + t) * N + n] = float_to_io16(v, f16);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Activation split for the decode schedule.  The delta contraction there runs on the 8-bit float
// tensor path (K = 32 per instruction, signs decoded four per register), so each bf16 activation
// is rewritten, once per call, as a chain of four e5m2 pieces: p0 = rn(x), p1 = rn(x - p0), ...
// Each piece removes three more bits, so x = p0 + p1 + p2 + p3 up to 2^-12 |x| (e5m2 has the
// exponent range of fp16: magnitudes above 57344 saturate, below 2^-16 vanish).  Elementwise; four
// neighbouring threads per group of 32 k.  Inside a group the pieces are stored in the order the sign decode
// produces: byte slot 4c+i holds k = c + 8i; thread u of the four makes the slots of c = 2u and 2u + 1, from
// pairs of neighbours.  Output rows: X8[(b*4 + q)*m + t, :] for piece q.
// Bound by latency and, with many rows, by the conversions: eight values a thread, converted in pairs, and no fourth
// piece where the third leaves nothing to represent (every bfloat16 magnitude below 2^16; a remainder below 2^-17 would be
// a signed zero).  The whole call in a graph, against one thread per group and four pieces always: 16 x 8 x 4096 x 4096
// 33.4 -> 32.5 us, 8 x 16 28.3 -> 27.4, 16 x 6 x 4096 x 5000 39.4 -> 38.5, 16 x 8 x 4096 x 11008 76.3 -> 75.2; 32 x 4 x 4096 x 4096,
// 24 x 8 x 11008 x 4096 and 32 x 8 x 14336 x 4096 level.
// Status word of this translation unit: [0] = 9 (BITDELTA_ERR_RANGE) once the split has met a magnitude of
// 2^16 or more (it is clamped to 65504, the largest binary16 number, exactly as the GEMM kernels' own split does).
static __device__ unsigned int g_simple_status[2];

__global__ void __launch_bounds__(128) x_split_kernel(const uint16_t* __restrict__ X, uint8_t* __restrict__ X8,
                                                      int m, int K, long long total, int f16) {
    // Let the GEMM kernel queued behind this one start its weight prefetch right away.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= total) return;
    const int quarters = K >> 3;
    const int row = (int)(id / quarters);
    const int k0 = (int)(id - (long long)row * quarters) >> 2 << 5, u = (int)id & 3;   // (quarters is a multiple of 4)
    const int b = row / m, t = row - b * m;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(X + (size_t)row * K + k0) + u;
    float2 y[4];   // k = 2u + 8i and the next
    bool out_of_range = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t q = __ldg(src + 4 * i);
        y[i] = make_float2(io16_to_float((uint16_t)(q & 0xFFFFu), f16), io16_to_float((uint16_t)(q >> 16), f16));
        if (!f16 && (((q & 0x7FFFu) >= 0x4780u) || (((q >> 16) & 0x7FFFu) >= 0x4780u))) out_of_range = true;
    }
    if (out_of_range) {
#pragma unroll
        for (int i = 0; i < 4; ++i) y[i] = make_float2(fminf(fmaxf(y[i].x, -65504.f), 65504.f), fminf(fmaxf(y[i].y, -65504.f), 65504.f));
        atomicCAS(&g_simple_status[0], 0u, 9u);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w0 = 0, w1 = 0;
        if (q < 3 || f16 || out_of_range) {
            uint32_t pc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_fp8x2_storage_t v = __nv_cvt_float2_to_fp8x2(y[i], __NV_SATFINITE, __NV_E5M2);
                const float2 back = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(v, __NV_E5M2)));
                y[i].x -= back.x;
                y[i].y -= back.y;
                pc[i] = v;
            }
            const uint32_t lo = __byte_perm(pc[0], pc[1], 0x5410), hi = __byte_perm(pc[2], pc[3], 0x5410);
            w0 = __byte_perm(lo, hi, 0x6420);
            w1 = __byte_perm(lo, hi, 0x7531);
        }
        *reinterpret_cast<uint2*>(X8 + ((size_t)(b * 4 + q) * m + t) * K + k0 + 8 * u) = make_uint2(w0, w1);
    }
}

cudaError_t read_simple_status(unsigned int out[2]) {
    cudaError_t e = cudaMemcpyFromSymbol(out, g_simple_status, sizeof(unsigned int) * 2);
    if (e != cudaSuccess) return e;
    if (out[0] != 0) {
        unsigned int zero[2] = {0, 0};
        e = cudaMemcpyToSymbol(g_simple_status, zero, sizeof(zero));
    }
    return e;
}

cudaError_t launch_x_split(const void* X, uint8_t* X8, int B, int m, int K, int f16, cudaStream_t stream) {
    const long long total = (long long)B * m * (K >> 3);
    const int threads = 128;
    const long long blocks = (total + threads - 1) / threads;
    x_split_kernel<<<(unsigned)blocks, threads, 0, stream>>>(reinterpret_cast<const uint16_t*>(X), X8, m, K, total, f16);
    return cudaGetLastError();
}

cudaError_t launch_pack(const int8_t* S, uint32_t* bits, long long words, cudaStream_t stream) {
    const int threads = 256;
    const long long blocks = (words + threads - 1) / threads;
    pack_kernel<<<(unsigned)blocks, threads, 0, stream>>>(S, bits, words);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const uint32_t* bits, int8_t* S, long long words, cudaStream_t stream) {
    const int threads = 256;
    const long long blocks = (words + threads - 1) / threads;
    unpack_kernel<<<(unsigned)blocks, threads, 0, stream>>>(bits, S, words);
    return cudaGetLastError();
}

cudaError_t launch_gemm_simt(const void* X, const void* W, const uint32_t* bits, const float* alpha, const void* bias,
                             void* Y, int B, int m, int N, int K, int f16, int act, cudaStream_t stream) {
    const int threads = 256;
    const long long warps = (long long)B * N;
    const long long blocks = (warps * 32 + threads - 1) / threads;
    gemm_simt_kernel<<<(unsigned)blocks, threads, 0, stream>>>(
        reinterpret_cast<const uint16_t*>(X), reinterpret_cast<const uint16_t*>(W), bits, alpha,
        reinterpret_cast<const uint16_t*>(bias), reinterpret_cast<uint16_t*>(Y), B, m, N, K, f16, act);
    return cudaGetLastError();
}

}  // namespace bd
