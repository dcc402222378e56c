// extern "C" entry points of libbitdelta.so: argument checks, tensor-map
// construction and kernel launches.  See include/bitdelta.h for the contract.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "../../include/bitdelta.h"
#include "early_start.h"
#include "gemm_row.h"
#include "gemm_tc.h"
#include "plan.h"

// Scratch of bitdelta_gemm_noalloc: lives in the library's device image (zero at load), one copy per GPU
// that loads the library.  In host code this name is only a handle for cudaGetSymbolAddress, never an
// address a kernel could use.
static __device__ __align__(256) unsigned char g_noalloc_scratch[BITDELTA_NOALLOC_SCRATCH_BYTES];

namespace {

std::atomic<unsigned long long> g_launches{0};
// The entry points that PRODUCE what the GEMM prefetches before its grid dependency is resolved (sign words, alpha: bitdelta_pack,
// bitdelta_compress) note it here; the next GEMM call on each stream (or in the same capture) then launches fully serialised, once.
bd::ProducerNote g_producers;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            fn = reinterpret_cast<EncodeTiledFn>(p);
        }
    });
    return fn;
}

struct DeviceInfo {
    int device = -1;
    int cc_major = 0, cc_minor = 0, sms = 0;
};

// Properties of the current device, cached per device id.
int device_info(DeviceInfo* out) {
    static DeviceInfo cache[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return BITDELTA_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64) return BITDELTA_ERR_CUDA;
    if (cache[dev].device != dev) {
        DeviceInfo d;
        if (cudaDeviceGetAttribute(&d.cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.cc_minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            return BITDELTA_ERR_CUDA;
        }
        d.device = dev;
        cache[dev] = d;
    }
    *out = cache[dev];
    return BITDELTA_OK;
}

int check_arch(DeviceInfo* d) {
    int st = device_info(d);
    if (st != BITDELTA_OK) return st;
    if (d->cc_major != 10 || d->cc_minor != 0) return BITDELTA_ERR_ARCH;
    return BITDELTA_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_pack_args(const void* a, const void* b, int B, int N, int K) {
    if (!a || !b) return BITDELTA_ERR_NULL;
    if (B <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return BITDELTA_ERR_SHAPE;
    if (!aligned16(a) || !aligned16(b)) return BITDELTA_ERR_ALIGN;
    return BITDELTA_OK;
}

int check_gemm_args(const void* X, const void* W, const void* bits, const void* alpha, const void* Y, int B, int m,
                    int N, int K) {
    if (!X || !W || !bits || !alpha || !Y) return BITDELTA_ERR_NULL;
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return BITDELTA_ERR_SHAPE;
    if ((long long)B * m > 0x7FFFFFFFll / 2 || (long long)B * N > 0x7FFFFFFFll) return BITDELTA_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(W) || !aligned16(bits) || !aligned16(Y)) return BITDELTA_ERR_ALIGN;
    if ((reinterpret_cast<uintptr_t>(alpha) & 3u) != 0) return BITDELTA_ERR_ALIGN;
    return BITDELTA_OK;
}

// bf16 [rows, K] row-major, seen as [K/64 atoms][rows][64]: one box = two 64-column atoms (128 bytes per
// row each, swizzled) x box_rows, i.e. a whole 128-k stage tile in ONE bulk-tensor operation, landing in
// shared memory atom after atom.  (The number of bulk operations a CTA keeps in flight is what limits
// its load throughput, not their size.)  Coordinates: (0, first row, k / 64).
bool encode_bf16_tile(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t K, uint32_t box_rows, uint32_t atoms = 2) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {64, rows, K / 128 * 2};   // (whole 128-k steps)
    cuuint64_t strides[2] = {K * 2, 128};
    cuuint32_t box[3] = {64, box_rows, atoms};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The last K % 128 columns of a bf16 [rows, K] matrix (`ptr`: their first one), box = one 64-column atom x box_rows;
// columns past the matrix are zero-filled.  (x = 0 or 64: 128-byte aligned.)
bool encode_bf16_tail(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t K, uint32_t box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {K % 128, rows};
    cuuint64_t strides[1] = {K * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D bytes [rows, K] row-major (e5m2 activation pieces), box = 128 bytes (swizzled) x box_rows.
bool encode_u8_2d(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t K, uint32_t box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {K, rows};
    cuuint64_t strides[1] = {K};
    cuuint32_t box[2] = {128, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D uint32 [B, N, K/32], box = `box_words` words (8: the signs of 256 k, 32 bytes; 4: of 128 k) x 128 rows x tenants.
bool encode_bits_3d(CUtensorMap* map, const void* ptr, uint64_t B, uint64_t N, uint64_t words, uint32_t tenants,
                    uint32_t box_words = 8, uint32_t box_rows = 128) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {words, N, B};
    cuuint64_t strides[2] = {words * 4, words * 4 * N};
    cuuint32_t box[3] = {box_words, box_rows, tenants};   // (32 words = 128 bytes: swizzled, the rows are read by lanes)
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, box_words == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// BITDELTA_TB=<n> overrides the tenants per decode tile (experiments); read once.
int tb_override() {
    static int v = 0;
    static std::once_flag once;
    std::call_once(once, [] { const char* e = getenv("BITDELTA_TB"); v = e ? atoi(e) : 0; });
    return v;
}

// BITDELTA_WHOLE (experiments, read once): 1 forces, 2 forbids the whole-unit work order; 3 forces one team of CTAs
// per tenant group, 4 forces the plain even cut.
int whole_override() {
    static int v = 0;
    static std::once_flag once;
    std::call_once(once, [] { const char* e = getenv("BITDELTA_WHOLE"); v = e ? atoi(e) : 0; });
    return v;
}

// BITDELTA_EARLY_START=0 launches the GEMM kernel fully serialised behind its predecessor
// (for experiments; the default lets it begin its weight prefetch early).
bool early_start_enabled() {
    const char* e = getenv("BITDELTA_EARLY_START");   // (read at every call: bench.py times both settings in one process)
    return !(e && e[0] == '0');
}

// The stream of a call, for the producers' note.  The default stream cannot be captured; the per-thread one is another in every thread.
bool stream_key(int device, cudaStream_t stream, bd::StreamKey* key) {
    static thread_local char this_thread;
    key->device = device;
    key->stream = stream == cudaStreamPerThread ? static_cast<const void*>(&this_thread) : static_cast<const void*>(stream);
    key->capture = 0;
    if (stream == nullptr || stream == cudaStreamLegacy) return true;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(stream, &status, &id) != cudaSuccess || status == cudaStreamCaptureStatusInvalidated) {
        cudaGetLastError();   // (the launch reports what is wrong with the stream)
        return false;
    }
    if (status == cudaStreamCaptureStatusActive) key->capture = id;
    return true;
}

// The row-stream decode kernel: by default where it pays (row_plan.h); BITDELTA_ROW=1: wherever it applies, =0: never.  A choice
// of the other decode kernels (BITDELTA_FP4 and its variants, BITDELTA_CLUSTER) leaves the call to them.
bool take_row_kernel(int B, int m, int N, int K, int sms, bool plain, int cluster) {
    const char* e = getenv("BITDELTA_ROW");
    if (e && e[0] == '0') return false;
    const bd::RowPlan p = bd::make_row_plan(B, m, N, K, sms);
    if (e && e[0] == '1') return p.ok;
    if (!bd::row_kernel_pays(p, B, m, N, K, plain, cluster)) return false;
    return bd::fp4_mode() == 2 && bd::cluster_enabled() && !getenv("BITDELTA_FP4_INKERNEL") && !getenv("BITDELTA_FP4_RESIDENT") &&
           !getenv("BITDELTA_FP4_COOP");
}

// Whether a call has no options (the 4-bit decode kernel takes none).
bool is_plain(int dtype, bool has_bias, int act) { return dtype == BITDELTA_DTYPE_BF16 && !has_bias && act == BITDELTA_ACT_NONE; }

// Encoded tensor maps, kept per (kind, pointer, shape, box): encoding one costs a microsecond or two of host time,
// a GEMM call needs three or four, and a serving loop calls with the same few weight and activation buffers.
struct MapKey {
    int kind;
    const void* ptr;
    uint64_t d0, d1, d2;
    uint32_t b0, b1;
    bool operator==(const MapKey& o) const {
        return kind == o.kind && ptr == o.ptr && d0 == o.d0 && d1 == o.d1 && d2 == o.d2 && b0 == o.b0 && b1 == o.b1;
    }
};
// (a table of sets of four by a hash of the key, so that a look-up compares four keys however many are held)
constexpr int kMapSets = 64, kMapWays = 4;
struct MapCache {
    std::mutex mu;
    MapKey keys[kMapSets][kMapWays];
    CUtensorMap maps[kMapSets][kMapWays];
    uint8_t used[kMapSets] = {}, next[kMapSets] = {};
};
inline unsigned map_set(const MapKey& k) {
    uint64_t h = reinterpret_cast<uint64_t>(k.ptr) ^ (k.d0 * 0x9E3779B97F4A7C15ull) ^ (k.d1 << 20) ^ ((uint64_t)k.b0 << 44) ^ ((uint64_t)k.kind << 60);
    h *= 0x9E3779B97F4A7C15ull;
    return (unsigned)(h >> 58);   // 64 sets
}
MapCache& map_cache() {
    static MapCache c;
    return c;
}
template <class Encode>
bool cached_map(CUtensorMap* out, const MapKey& key, Encode encode) {
    MapCache& c = map_cache();
    const unsigned s = map_set(key);
    {
        std::lock_guard<std::mutex> lock(c.mu);
        for (int i = 0; i < c.used[s]; ++i)
            if (c.keys[s][i] == key) {
                *out = c.maps[s][i];
                return true;
            }
    }
    if (!encode(out)) return false;
    std::lock_guard<std::mutex> lock(c.mu);
    const int i = c.next[s];
    c.next[s] = (uint8_t)((i + 1) % kMapWays);
    if (c.used[s] <= i) c.used[s] = (uint8_t)(i + 1);
    c.keys[s][i] = key;
    c.maps[s][i] = *out;
    return true;
}

}  // namespace

extern "C" {

int bitdelta_pack(const int8_t* S, uint32_t* bits, int B, int N, int K, void* cuda_stream) {
    int st = check_pack_args(S, bits, B, N, K);
    if (st != BITDELTA_OK) return st;
    DeviceInfo d;
    st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    const long long words = (long long)B * N * (K / 32);
    const bd::Producing producing(g_producers, [&](bd::StreamKey* k) { return stream_key(d.device, static_cast<cudaStream_t>(cuda_stream), k); });
    if (bd::launch_pack(S, bits, words, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    g_launches++;
    return BITDELTA_OK;
}

int bitdelta_unpack(const uint32_t* bits, int8_t* S, int B, int N, int K, void* cuda_stream) {
    int st = check_pack_args(bits, S, B, N, K);
    if (st != BITDELTA_OK) return st;
    DeviceInfo d;
    st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    const long long words = (long long)B * N * (K / 32);
    if (bd::launch_unpack(bits, S, words, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    g_launches++;
    return BITDELTA_OK;
}

size_t bitdelta_compress_workspace_bytes(int B, int N, int K) {
    if (B <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return 0;
    return (size_t)B * (size_t)bd::compress_blocks(N, K) * sizeof(double);
}

int bitdelta_compress(const void* W_fine, const void* W_base, uint32_t* bits, float* alpha, int B, int N, int K,
                      void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!W_fine || !W_base || !bits || !alpha) return BITDELTA_ERR_NULL;
    if (B <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return BITDELTA_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(W_fine) | reinterpret_cast<uintptr_t>(W_base) | reinterpret_cast<uintptr_t>(bits)) & 15)
        return BITDELTA_ERR_ALIGN;
    if (!workspace || workspace_bytes < bitdelta_compress_workspace_bytes(B, N, K) ||
        (reinterpret_cast<uintptr_t>(workspace) & 7))
        return BITDELTA_ERR_WORKSPACE;
    DeviceInfo d;
    int st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    const bd::Producing producing(g_producers, [&](bd::StreamKey* k) { return stream_key(d.device, static_cast<cudaStream_t>(cuda_stream), k); });
    if (bd::launch_compress(W_fine, W_base, bits, alpha, static_cast<double*>(workspace), B, N, K,
                            static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    g_launches += 2;
    return BITDELTA_OK;
}

size_t bitdelta_gemm_workspace_bytes(int B, int m, int N, int K) {
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return 0;
    bd::Plan p = bd::make_plan(B, m, N, K, 148, tb_override(), whole_override());
    if ((K % 128) != 0 && !p.ok) return 256;   // CUDA-core path: no scratch needed, keep the pointer non-NULL
    if (!p.ok) return 0;
    size_t need = p.ws_bytes;
    if (p.pair) {   // ... and without pairs, for a device (or a part of one) that cannot hold them all at once
        bd::Plan o = bd::make_plan(B, m, N, K, 148, tb_override(), whole_override(), false);
        if (o.ok && o.ws_bytes > need) need = o.ws_bytes;
    }
    if (p.decode) {   // the same shape on the tiled schedule (BITDELTA_DTYPE_WIDE_RANGE) may need more
        bd::Plan w = bd::make_plan(B, m, N, K, 148, tb_override(), whole_override(), true, true);
        if (w.ok && w.ws_bytes > need) need = w.ws_bytes;
        // ... and a call with options (binary16, bias, activation) never takes the 4-bit decode kernel
        bd::Plan o = bd::make_plan(B, m, N, K, 148, tb_override(), whole_override(), true, false, false);
        if (o.ok && o.ws_bytes > need) need = o.ws_bytes;
    }
    return need;
}

int bitdelta_workspace_init(void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!workspace) return BITDELTA_ERR_NULL;
    if (workspace_bytes == 0) return BITDELTA_ERR_WORKSPACE;
    if (cudaMemsetAsync(workspace, 0, workspace_bytes, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    return BITDELTA_OK;
}

int bitdelta_gemm_simt(const void* X, const void* W_base, const uint32_t* bits, const float* alpha, void* Y, int B,
                       int m, int N, int K, void* cuda_stream) {
    int st = check_gemm_args(X, W_base, bits, alpha, Y, B, m, N, K);
    if (st != BITDELTA_OK) return st;
    DeviceInfo d;
    st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    if (bd::launch_gemm_simt(X, W_base, bits, alpha, nullptr, Y, B, m, N, K, 0, 0,
                             static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    g_launches++;
    return BITDELTA_OK;
}

int bitdelta_gemm(const void* X, const void* W_base, const uint32_t* bits, const float* alpha, void* Y, int B, int m,
                  int N, int K, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return bitdelta_gemm_ex(X, W_base, bits, alpha, nullptr, Y, B, m, N, K, BITDELTA_DTYPE_BF16, BITDELTA_ACT_NONE,
                            workspace, workspace_bytes, cuda_stream);
}

// (allow_pair: the tiled schedule may run on pairs of blocks)
static int run_gemm(const void* X, const void* W_base, const uint32_t* bits, const float* alpha, const void* bias, void* Y, int B, int m, int N,
                    int K, int dtype, int act, void* workspace, size_t workspace_bytes, void* cuda_stream, bool allow_pair) {
    int st = check_gemm_args(X, W_base, bits, alpha, Y, B, m, N, K);
    if (st != BITDELTA_OK) return st;
    const bool wide = (dtype & BITDELTA_DTYPE_WIDE_RANGE) != 0;
    dtype &= ~BITDELTA_DTYPE_WIDE_RANGE;
    if ((dtype != BITDELTA_DTYPE_BF16 && dtype != BITDELTA_DTYPE_F16) || (act != BITDELTA_ACT_NONE && act != BITDELTA_ACT_SILU && act != BITDELTA_ACT_SILU_GATE))
        return BITDELTA_ERR_OPTION;
    if (act == BITDELTA_ACT_SILU_GATE && (N % 2) != 0) return BITDELTA_ERR_SHAPE;
    if (bias && (reinterpret_cast<uintptr_t>(bias) & 1)) return BITDELTA_ERR_ALIGN;
    const int f16 = (dtype == BITDELTA_DTYPE_F16) ? 1 : 0;
    DeviceInfo d;
    st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);

    const bool plain = is_plain(dtype, bias != nullptr, act);
    bd::Plan p = bd::make_plan(B, m, N, K, d.sms, tb_override(), whole_override(), allow_pair, wide, plain);
    if (!wide && p.ok && workspace && workspace_bytes >= p.ws_bytes && aligned16(workspace) && take_row_kernel(B, m, N, K, d.sms, plain, p.cluster)) {
        // (the row-stream kernel needs no scratch; a call that is refused for its workspace stays refused)
        const bd::RowPlan rp = bd::make_row_plan(B, m, N, K, d.sms);
        CUtensorMap rW, rX, rB;
        if (!cached_map(&rW, MapKey{4, W_base, (uint64_t)N, (uint64_t)K, 0, (uint32_t)rp.rows, 16u},
                        [&](CUtensorMap* mp) { return encode_bf16_tile(mp, W_base, (uint64_t)N, (uint64_t)K, (uint32_t)rp.rows, 16u); }) ||
            !cached_map(&rX, MapKey{4, X, (uint64_t)B * m, (uint64_t)K, 0, 8u, 16u},
                        [&](CUtensorMap* mp) { return encode_bf16_tile(mp, X, (uint64_t)B * m, (uint64_t)K, 8u, 16u); }) ||
            !cached_map(&rB, MapKey{5, bits, (uint64_t)B, (uint64_t)N, (uint64_t)(K / 32), (uint32_t)rp.TB, (uint32_t)rp.rows},
                        [&](CUtensorMap* mp) { return encode_bits_3d(mp, bits, (uint64_t)B, (uint64_t)N, (uint64_t)(K / 32), (uint32_t)rp.TB, 32u, (uint32_t)rp.rows); }))
            return BITDELTA_ERR_CUDA;
        bd::RowArgs ra{};
        ra.B = B; ra.m = m; ra.N = N; ra.K = K; ra.f16 = f16; ra.act = act;
        ra.TB = rp.TB; ra.rows = rp.rows; ra.groups = rp.groups; ra.units = rp.units; ra.stages = rp.stages; ra.k_stages = rp.k_stages;
        ra.s_off = rp.s_off; ra.x_off = rp.x_off; ra.stage_bytes = rp.stage_bytes;
        ra.bias = bias; ra.alpha = alpha; ra.Y = Y;
        bd::ProductStart start(g_producers, early_start_enabled(), [&](bd::StreamKey* k) { return stream_key(d.device, stream, k); });
        if (bd::launch_gemm_row(rW, rX, rB, ra, rp, start.early, stream) != cudaSuccess) return BITDELTA_ERR_CUDA;
        start.launched();
        g_launches++;
        return BITDELTA_OK;
    }
    if (p.ok && p.pair) {
        // The pair schedule wants every pair resident at once (a cluster of two needs two free SMs of one
        // cluster-capable group); where the device cannot do that, run the one-CTA schedule.  Asked once per device.
        static std::mutex mu_pairs;
        static int pairs_cache[64][2] = {};   // [device]: {shared memory bytes asked with, pairs that fit + 1}
        const int di = (d.device >= 0 && d.device < 64) ? d.device : 0;
        int fit;
        {
            std::lock_guard<std::mutex> lock(mu_pairs);
            if (pairs_cache[di][1] == 0 || pairs_cache[di][0] != (int)p.smem_bytes) {
                pairs_cache[di][0] = (int)p.smem_bytes;
                pairs_cache[di][1] = bd::max_active_pairs(p.smem_bytes) + 1;
            }
            fit = pairs_cache[di][1] - 1;
        }
        if (2 * fit < p.grid) p = bd::make_plan(B, m, N, K, d.sms, tb_override(), whole_override(), false, wide, plain);
    }
    if (p.ok && p.cluster > 1) {
        // The cluster form wants all its clusters resident at once (clusters are independent, so this is about
        // speed, not progress); where the device cannot hold them, the flat work list is planned.
        static std::mutex mu;
        static int fit_cache[64][4] = {};   // [device][log2 cluster]: 0 unknown, else clusters that fit + 1
        const int di = (d.device >= 0 && d.device < 64) ? d.device : 0;
        const int ci = p.cluster == 8 ? 3 : (p.cluster == 4 ? 2 : 1);
        int n;
        {
            std::lock_guard<std::mutex> lock(mu);
            if (fit_cache[di][ci] == 0) fit_cache[di][ci] = bd::fp4_max_active_clusters(p.smem_bytes, p.cluster) + 1;
            n = fit_cache[di][ci] - 1;
        }
        const int need = p.grid / p.cluster;
        if (n < need) p = bd::make_plan(B, m, N, K, d.sms, tb_override(), whole_override(), false, false, plain);
    }
    if ((K % 128) != 0 && (!p.ok || !workspace || workspace_bytes < p.ws_bytes || !aligned16(workspace))) {
        // K < 128, a work list beyond the split arithmetic, or no scratch for the tiled schedule (the no-allocation
        // entry point with a large shape): the CUDA-core kernel, which needs none.
        if (bd::launch_gemm_simt(X, W_base, bits, alpha, bias, Y, B, m, N, K, f16, act, stream) != cudaSuccess)
            return BITDELTA_ERR_CUDA;
        g_launches++;
        return BITDELTA_OK;
    }
    if (!p.ok) return BITDELTA_ERR_SHAPE;
    if (!workspace || workspace_bytes < p.ws_bytes) return BITDELTA_ERR_WORKSPACE;
    if (!aligned16(workspace)) return BITDELTA_ERR_ALIGN;

    CUtensorMap tmW, tmX, tmX8, tmBits;
    if (!cached_map(&tmW, MapKey{0, W_base, (uint64_t)N, (uint64_t)K, 0, (uint32_t)bd::kTileN, 0u},
                    [&](CUtensorMap* mp) { return encode_bf16_tile(mp, W_base, (uint64_t)N, (uint64_t)K, bd::kTileN); }))
        return BITDELTA_ERR_CUDA;
    if (!p.stream && !cached_map(&tmX, MapKey{0, X, (uint64_t)B * m, (uint64_t)K, 0, (uint32_t)p.x_rows, 0u},
                                 [&](CUtensorMap* mp) { return encode_bf16_tile(mp, X, (uint64_t)B * m, (uint64_t)K, (uint32_t)p.x_rows); }))
        return BITDELTA_ERR_CUDA;
    const uint32_t box_words = (p.fp4 && p.bits_row == 16) ? 4u : 8u;
    if (!p.ragged && !cached_map(&tmBits, MapKey{1, bits, (uint64_t)B, (uint64_t)N, (uint64_t)(K / 32), (uint32_t)p.TB, box_words},
                    [&](CUtensorMap* mp) { return encode_bits_3d(mp, bits, (uint64_t)B, (uint64_t)N, (uint64_t)(K / 32), (uint32_t)p.TB, box_words); }))
        return BITDELTA_ERR_CUDA;
    if (p.ragged) {
        // the short last k-step of W_base and of the activations
        const uint64_t k_full = (uint64_t)(K / bd::kPairK * bd::kPairK);
        const uint16_t* Wt = static_cast<const uint16_t*>(W_base) + k_full;
        const uint16_t* Xt = static_cast<const uint16_t*>(X) + k_full;
        if (!cached_map(&tmX8, MapKey{3, Wt, (uint64_t)N, (uint64_t)K, 0, (uint32_t)bd::kTileN, 0u},
                        [&](CUtensorMap* mp) { return encode_bf16_tail(mp, Wt, (uint64_t)N, (uint64_t)K, bd::kTileN); }) ||
            !cached_map(&tmBits, MapKey{3, Xt, (uint64_t)B * m, (uint64_t)K, 0, (uint32_t)p.x_rows, 0u},
                        [&](CUtensorMap* mp) { return encode_bf16_tail(mp, Xt, (uint64_t)B * m, (uint64_t)K, (uint32_t)p.x_rows); }))
            return BITDELTA_ERR_CUDA;
    } else if (p.fp4) {
        // 4-bit decode kernel: the activation operands of every (tenant group, 128-k step) as shared-memory images, and
        // the token rows' fixed-point units; then the GEMM, which prefetches weights while this is still running.
        uint8_t* img = bd::ws_x8(p, workspace);
        // (its early start is always safe: it waits for its predecessor before it touches anything)
        if (!p.convert && !p.coop && bd::launch_x_split_fp4(X, img, p, early_start_enabled(), stream) != cudaSuccess)
            return BITDELTA_ERR_CUDA;
        if (!p.convert && !p.coop) g_launches++;
        tmX8 = tmW;   // not read
    } else if (p.decode && !p.convert) {
        // Decode schedule with many token rows per tile: split the activations into e5m2 pieces first
        // (tiny), then the GEMM, which may start prefetching weights while the split is still running.
        uint8_t* x8 = bd::ws_x8(p, workspace);
        if (!cached_map(&tmX8, MapKey{2, x8, (uint64_t)B * bd::kPieces * m, (uint64_t)K, 0, (uint32_t)p.x8_rows, 0u},
                        [&](CUtensorMap* mp) { return encode_u8_2d(mp, x8, (uint64_t)B * bd::kPieces * m, (uint64_t)K, (uint32_t)p.x8_rows); }))
            return BITDELTA_ERR_CUDA;
        if (bd::launch_x_split(X, x8, B, m, K, f16, stream) != cudaSuccess)
            return BITDELTA_ERR_CUDA;
        g_launches++;
    } else {
        tmX8 = tmX;   // not read: the kernel splits the activations itself, or runs the tiled schedule
    }

    bd::GemmArgs args = bd::make_args(p, alpha, Y, workspace);
    args.f16 = f16; args.act = act; args.bias = bias;
    args.X = X; args.bits = bits;
    { static int h = -1; if (h < 0) { const char* e = getenv("BITDELTA_HOLD"); h = (e && e[0] == '0') ? 0 : 1; } args.hold_prefetch = h; }
    // (a GEMM queued right behind the library's own pack / compress must not prefetch what they are still writing)
    bd::ProductStart start(g_producers, early_start_enabled(), [&](bd::StreamKey* k) { return stream_key(d.device, stream, k); });
    const cudaError_t le = p.fp4
        ? bd::launch_gemm_fp4(tmW, tmBits, args, p.grid, p.smem_bytes, start.early, stream)
        : bd::launch_gemm_tc(tmW, tmX, tmX8, tmBits, args, p.grid, p.smem_bytes, start.early, stream);
    if (le != cudaSuccess) return BITDELTA_ERR_CUDA;
    start.launched();
    g_launches++;
    return BITDELTA_OK;
}

int bitdelta_gemm_ex(const void* X, const void* W_base, const uint32_t* bits, const float* alpha, const void* bias,
                     void* Y, int B, int m, int N, int K, int dtype, int act, void* workspace,
                     size_t workspace_bytes, void* cuda_stream) {
    return run_gemm(X, W_base, bits, alpha, bias, Y, B, m, N, K, dtype, act, workspace, workspace_bytes, cuda_stream, true);
}

size_t bitdelta_gemm_host_arena_bytes(int B, int m, int N, int K) {
    size_t ws = bitdelta_gemm_workspace_bytes(B, m, N, K);
    if (ws == 0) return 0;
    size_t total = 0;
    total += align_up((size_t)B * m * K * 2, 256);
    total += align_up((size_t)N * K * 2, 256);
    total += align_up((size_t)B * N * (K / 32) * 4, 256);
    total += align_up((size_t)B * 4, 256);
    total += align_up((size_t)B * m * N * 2, 256);
    total += align_up(ws, 256);
    return total;
}

int bitdelta_gemm_host(const void* X_host, const void* W_base_host, const uint32_t* bits_host,
                       const float* alpha_host, void* Y_host, int B, int m, int N, int K, void* arena,
                       size_t arena_bytes, void* cuda_stream) {
    if (!X_host || !W_base_host || !bits_host || !alpha_host || !Y_host || !arena) return BITDELTA_ERR_NULL;
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 32) != 0) return BITDELTA_ERR_SHAPE;
    const size_t need = bitdelta_gemm_host_arena_bytes(B, m, N, K);
    if (need == 0) return BITDELTA_ERR_SHAPE;
    if (arena_bytes < need) return BITDELTA_ERR_WORKSPACE;
    if ((reinterpret_cast<uintptr_t>(arena) & 255u) != 0) return BITDELTA_ERR_ALIGN;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);

    const size_t xb = (size_t)B * m * K * 2, wb = (size_t)N * K * 2, bb = (size_t)B * N * (K / 32) * 4;
    const size_t ab = (size_t)B * 4, yb = (size_t)B * m * N * 2;
    const size_t ws = bitdelta_gemm_workspace_bytes(B, m, N, K);
    char* p = static_cast<char*>(arena);
    void* dX = p;      p += align_up(xb, 256);
    void* dW = p;      p += align_up(wb, 256);
    void* dBits = p;   p += align_up(bb, 256);
    void* dAlpha = p;  p += align_up(ab, 256);
    void* dY = p;      p += align_up(yb, 256);
    void* dWs = p;

    if (cudaMemcpyAsync(dX, X_host, xb, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(dW, W_base_host, wb, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(dBits, bits_host, bb, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(dAlpha, alpha_host, ab, cudaMemcpyHostToDevice, stream) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    // Only the arrival counters at the start of the workspace have to be clear.
    bd::Plan plan = bd::make_plan(B, m, N, K, 148, tb_override(), whole_override());
    const size_t header = plan.ok ? plan.ws_header_bytes : (ws < 256 ? ws : 256);
    if (cudaMemsetAsync(dWs, 0, header, stream) != cudaSuccess) return BITDELTA_ERR_CUDA;
    int st = bitdelta_gemm(dX, dW, static_cast<const uint32_t*>(dBits), static_cast<const float*>(dAlpha), dY, B, m,
                           N, K, dWs, ws, cuda_stream);
    if (st != BITDELTA_OK) return st;
    if (cudaMemcpyAsync(Y_host, dY, yb, cudaMemcpyDeviceToHost, stream) != cudaSuccess) return BITDELTA_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return BITDELTA_ERR_CUDA;
    return BITDELTA_OK;
}

int bitdelta_gemm_plan(int B, int m, int N, int K, int num_sms, int* info) {
    if (!info) return BITDELTA_ERR_NULL;
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 32) != 0 || num_sms <= 0) return BITDELTA_ERR_SHAPE;
    for (int i = 0; i < BITDELTA_PLAN_INFO_INTS; ++i) info[i] = 0;
    bd::Plan p = bd::make_plan(B, m, N, K, num_sms, tb_override(), whole_override());
    if ((K % 128) != 0 && !p.ok) { info[0] = 3; return BITDELTA_OK; }
    if (!p.ok) return BITDELTA_ERR_SHAPE;
    info[0] = !p.decode ? (p.pair ? 4 : 0) : p.fp4 ? (p.cluster > 1 ? 8 : 7) : (p.convert ? 2 : 1);
    info[1] = p.grid; info[2] = p.TB; info[3] = p.units; info[4] = p.P;
    info[5] = p.cluster > 1 ? 3 : (p.whole_units ? 1 : (p.teams > 1 ? 2 : 0));
    info[6] = p.teams; info[7] = (int)p.smem_bytes; info[8] = p.n_w; info[9] = p.n_x; info[10] = p.n_x8;
    info[11] = p.a_slots; info[12] = p.halves; info[13] = p.tok_tile; info[14] = p.groups; info[15] = p.n_tiles;
    return BITDELTA_OK;
}

int bitdelta_gemm_row_stream(int B, int m, int N, int K, int num_sms) {
    return bitdelta_gemm_row_stream_ex(B, m, N, K, BITDELTA_DTYPE_BF16, 0, BITDELTA_ACT_NONE, num_sms);
}

int bitdelta_gemm_row_stream_ex(int B, int m, int N, int K, int dtype, int has_bias, int act, int num_sms) {
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 32) != 0 || num_sms <= 0) return 0;
    if ((dtype & BITDELTA_DTYPE_WIDE_RANGE) != 0) return 0;
    const bool plain = is_plain(dtype, has_bias != 0, act);
    const bd::Plan p = bd::make_plan(B, m, N, K, num_sms, tb_override(), whole_override(), true, false, plain);
    return p.ok && take_row_kernel(B, m, N, K, num_sms, plain, p.cluster) ? 1 : 0;
}

int bitdelta_gemm_plan_cta_items(int B, int m, int N, int K, int num_sms, int cta, int* first, int* end) {
    if (!first || !end) return BITDELTA_ERR_NULL;
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 128) != 0 || num_sms <= 0) return BITDELTA_ERR_SHAPE;
    bd::Plan p = bd::make_plan(B, m, N, K, num_sms, tb_override(), whole_override());
    if (!p.ok || cta < 0 || cta >= p.grid) return BITDELTA_ERR_SHAPE;
    if (p.whole_units) {
        *first = cta * p.P;
        *end = *first + p.P;
        return BITDELTA_OK;
    }
    if (p.cluster > 1) {   // block `cta` = rank cta % cluster of the cluster that takes unit cta / cluster
        const int un = cta / p.cluster, r = cta % p.cluster;
        *first = un * p.P + (r * p.P) / p.cluster;
        *end = un * p.P + ((r + 1) * p.P) / p.cluster;
        return BITDELTA_OK;
    }
    const bd::GemmArgs a = bd::make_args(p, nullptr, nullptr, nullptr);
    const int cutter = p.pair ? cta / 2 : cta;   // both blocks of a pair take the pair's items
    *first = bd::cta_first_item(a, cutter);
    *end = bd::cta_first_item(a, cutter + 1);
    return BITDELTA_OK;
}

int bitdelta_gemm_plan_item_cta(int B, int m, int N, int K, int num_sms, int item) {
    if (B <= 0 || m <= 0 || N <= 0 || K <= 0 || (K % 128) != 0 || num_sms <= 0) return -1;
    bd::Plan p = bd::make_plan(B, m, N, K, num_sms, tb_override(), whole_override());
    if (!p.ok || item < 0 || item >= p.T) return -1;
    if (p.cluster > 1) {
        const int un = item / p.P, s = item - un * p.P;
        int r = (int)(((long long)(s + 1) * p.cluster - 1) / p.P);   // largest r with r * P / cluster <= s
        while ((r * p.P) / p.cluster > s) --r;
        while (((r + 1) * p.P) / p.cluster <= s) ++r;
        return un * p.cluster + r;
    }
    if (p.whole_units) return (item / p.P) % p.grid;
    const bd::GemmArgs a = bd::make_args(p, nullptr, nullptr, nullptr);
    return p.pair ? 2 * bd::cta_of_item(a, item) : bd::cta_of_item(a, item);   // (pairs: the pair's first block)
}

int bitdelta_selftest_timeout(long long limit_cycles, int site, void* cuda_stream) {
    if (limit_cycles < 1000 || limit_cycles > 2000000000ll || site < 0) return BITDELTA_ERR_SHAPE;
    DeviceInfo d;
    int st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    if (bd::launch_selftest_timeout(limit_cycles, site, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return BITDELTA_ERR_CUDA;
    g_launches++;
    return BITDELTA_OK;
}

int bitdelta_last_device_status(void* cuda_stream, int* site) {
    unsigned int st[2] = {0, 0};
    if (bd::read_device_status(st, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return BITDELTA_ERR_CUDA;
    if (site) *site = (int)st[1];
    return st[0] == 0 ? BITDELTA_OK : (int)st[0];
}

int bitdelta_gemm_noalloc(const void* X, const void* W_base, const uint32_t* bits, const float* alpha, void* Y, int B,
                          int m, int N, int K, void* cuda_stream) {
    int st = check_gemm_args(X, W_base, bits, alpha, Y, B, m, N, K);
    if (st != BITDELTA_OK) return st;
    DeviceInfo d;
    st = check_arch(&d);
    if (st != BITDELTA_OK) return st;
    const size_t need = bitdelta_gemm_workspace_bytes(B, m, N, K);
    if (need == 0) return BITDELTA_ERR_SHAPE;
    bd::Plan plan = bd::make_plan(B, m, N, K, d.sms, tb_override(), whole_override());
    bool pairs = true;
    if (need > (size_t)BITDELTA_NOALLOC_SCRATCH_BYTES && (K % 128) == 0) {   // (other K: the CUDA-core kernel needs no scratch)
        // (the partial results of pairs' wider token tiles may not fit where those of single blocks do)
        pairs = false;
        if (plan.pair) plan = bd::make_plan(B, m, N, K, d.sms, tb_override(), whole_override(), false);
        else plan.ok = false;
        if (!plan.ok || plan.ws_bytes > (size_t)BITDELTA_NOALLOC_SCRATCH_BYTES) return BITDELTA_ERR_WORKSPACE;
    }

    // Device address of the scratch array, looked up once per device with that device current.
    static void* scratch_ptr[64] = {};
    static std::mutex mu;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (d.device < 0 || d.device >= 64) return BITDELTA_ERR_CUDA;
        if (!scratch_ptr[d.device]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return BITDELTA_ERR_CUDA;
            scratch_ptr[d.device] = p;
        }
        scratch = scratch_ptr[d.device];
    }
    // The arrival counters at the start of the scratch have to be zero when the kernel begins; a call
    // that was cut short could have left them otherwise.
    if (!plan.ok && (K % 128) == 0) return BITDELTA_ERR_SHAPE;
    if (plan.ok && plan.ws_bytes <= (size_t)BITDELTA_NOALLOC_SCRATCH_BYTES) {
        if (cudaMemsetAsync(scratch, 0, plan.ws_header_bytes, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
            return BITDELTA_ERR_CUDA;
    }
    return run_gemm(X, W_base, bits, alpha, nullptr, Y, B, m, N, K, BITDELTA_DTYPE_BF16, BITDELTA_ACT_NONE, scratch,
                    (size_t)BITDELTA_NOALLOC_SCRATCH_BYTES, cuda_stream, pairs);
}

unsigned long long bitdelta_kernel_launch_count(void) { return g_launches.load(); }

const char* bitdelta_status_string(int status) {
    switch (status) {
        case BITDELTA_OK: return "ok";
        case BITDELTA_ERR_NULL: return "null pointer argument";
        case BITDELTA_ERR_SHAPE: return "invalid shape (B, m, N, K must be positive and K a multiple of 32)";
        case BITDELTA_ERR_ALIGN: return "pointer not 16-byte aligned";
        case BITDELTA_ERR_WORKSPACE: return "workspace missing or too small";
        case BITDELTA_ERR_ARCH: return "device is not compute capability 10.0 (sm_100a required)";
        case BITDELTA_ERR_CUDA: return "CUDA runtime or driver call failed";
        case BITDELTA_ERR_TIMEOUT: return "a bounded wait inside a kernel expired";
        case BITDELTA_ERR_OPTION: return "unknown data type or activation code";
        case BITDELTA_ERR_RANGE: return "an activation of magnitude 2^16 or more was clamped in a decode schedule's delta term";
        default: return "unknown status";
    }
}

}  // extern "C"
