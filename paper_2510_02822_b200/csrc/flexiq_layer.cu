// Layer handles: the static part of the method.  Layout post-processing (Sec. 5),
// per-(group, output channel) weight extraction positions (Sec. 4.1, Fig. 4), cached
// 4-bit weights (Sec. 7), and the run-time ratio knob max_4bit_ch (Sec. 7).
#include "flexiq_internal.h"

#include "sm100_ptx.cuh"

#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

namespace flexiq {

static thread_local char g_err[512] = "";

int set_error(int code, const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int check_device_sm100()
{
    static int major_of[64] = {};  // compute capability major per device ordinal, looked up once
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return set_error(FLEXIQ_ERR_CUDA, "cudaGetDevice failed: %s", cudaGetErrorString(e));
    int major = dev < 64 ? major_of[dev] : 0;
    if (major == 0) {
        e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (e != cudaSuccess)
            return set_error(FLEXIQ_ERR_CUDA, "cudaDeviceGetAttribute failed: %s", cudaGetErrorString(e));
        if (dev < 64) major_of[dev] = major;
    }
    if (major != 10)
        return set_error(FLEXIQ_ERR_UNSUPPORTED,
                         "device compute capability %d.x is not sm_100; there is no fallback path", major);
    return FLEXIQ_OK;
}

int device_sm_count(int device)
{
    static int sms_of[64] = {};
    if (device >= 0 && device < 64 && sms_of[device]) return sms_of[device];
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (device >= 0 && device < 64) sms_of[device] = sms;
    return sms;
}

Layer *as_layer(flexiq_layer_t h)
{
    Layer *L = reinterpret_cast<Layer *>(h);
    if (L == nullptr || L->magic != kLayerMagic) return nullptr;
    return L;
}

int check_layer_device(const Layer *L)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_error(FLEXIQ_ERR_CUDA, "cudaGetDevice failed: %s", cudaGetErrorString(e));
    if (dev != L->device)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "the layer lives on device %d but device %d is current: its pointers are not valid there",
                         L->device, dev);
    return FLEXIQ_OK;
}

unsigned long long stream_capture_id(cudaStream_t st)
{
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) { cudaGetLastError(); return 0; }
    return status == cudaStreamCaptureStatusActive ? (id ? id : 1ull) : 0ull;
}

void record_slab(Layer *L, const void *ptr, int K_lo)
{
    if (!ptr) return;
    for (int i = 0; i < 8; ++i)
        if (L->slab_seen[i].ptr == ptr) { L->slab_seen[i].K_lo = K_lo; return; }
    L->slab_seen[L->slab_next] = Layer::SlabRecord{ptr, K_lo};
    L->slab_next = (L->slab_next + 1) & 7;
}

int check_slab(const Layer *L, const void *ptr, const char *what)
{
    if (!L->slab_check || !ptr) return FLEXIQ_OK;
    for (int i = 0; i < 8; ++i)
        if (L->slab_seen[i].ptr == ptr && L->slab_seen[i].K_lo != L->K_lo)
            return set_error(FLEXIQ_ERR_INVALID_ARG,
                             "%s was last written at max_4bit_ch = %d but the layer is now at %d: run flexiq_quantize_lower "
                             "again, or set the ratio the slab was written at", what, L->slab_seen[i].K_lo, L->K_lo);
    return FLEXIQ_OK;
}

// Masked path: the straddle block is read when max_4bit_ch falls inside a K block.
bool straddle_in_use(const Layer *L)
{
    return L->lowbit_path == FLEXIQ_LOWBIT_MASKED_I8 && L->K_lo < L->C && (L->K_lo % choose_bk(L)) != 0;
}
// Does wst hold the block for the current max_4bit_ch at this point of the stream?  Outside a capture the
// host's record decides, unless a captured graph may have rewritten wst since.  Inside a capture only a write
// earlier in the same capture counts, so that every graph is complete in itself and graphs of different
// ratios replay in any order.
bool straddle_stale(const Layer *L, cudaStream_t st)
{
    const unsigned long long cap = stream_capture_id(st);
    if (cap) return !(L->st_cap_id == cap && L->st_cap_K_lo == L->K_lo);
    return L->st_graph_seen || L->st_K_lo != L->K_lo;
}
void straddle_written(Layer *L, cudaStream_t st)
{
    const unsigned long long cap = stream_capture_id(st);
    if (cap) { L->st_cap_id = cap; L->st_cap_K_lo = L->K_lo; L->st_graph_seen = 1; L->st_K_lo = -1; }
    else { L->st_K_lo = L->K_lo; L->st_fresh = 1; }
}

static void *driver_entry(const char *name)
{
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &qres) != cudaSuccess) return nullptr;
    if (qres != cudaDriverEntryPointSuccess) return nullptr;
    return fn;
}

EncodeTiledFn get_encode_tiled()
{
    static EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(driver_entry("cuTensorMapEncodeTiled"));
    return fn;
}

EncodeIm2colFn get_encode_im2col()
{
    static EncodeIm2colFn fn = reinterpret_cast<EncodeIm2colFn>(driver_entry("cuTensorMapEncodeIm2col"));
    return fn;
}

static CUtensorMapSwizzle swizzle_enum(int bytes)
{
    switch (bytes) {
        case 128: return CU_TENSOR_MAP_SWIZZLE_128B;
        case 64: return CU_TENSOR_MAP_SWIZZLE_64B;
        case 32: return CU_TENSOR_MAP_SWIZZLE_32B;
        default: return CU_TENSOR_MAP_SWIZZLE_NONE;
    }
}

int make_map_2d(CUtensorMap *map, const void *base, uint64_t row_bytes, uint64_t rows,
                uint64_t pitch_bytes, uint32_t box_bytes, uint32_t box_rows, int swizzle_bytes)
{
    EncodeTiledFn enc = get_encode_tiled();
    if (!enc) return set_error(FLEXIQ_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    if ((reinterpret_cast<uintptr_t>(base) & 15) != 0 || (pitch_bytes & 15) != 0)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "tensor base %p / pitch %llu not 16-byte aligned", base,
                         (unsigned long long)pitch_bytes);
    cuuint64_t dims[2] = {row_bytes, rows};
    cuuint64_t strides[1] = {pitch_bytes};
    cuuint32_t box[2] = {box_bytes, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box,
                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_enum(swizzle_bytes),
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return set_error(FLEXIQ_ERR_CUDA, "cuTensorMapEncodeTiled failed with CUresult %d (rows %llu x %llu B, box %u x %u)",
                         (int)r, (unsigned long long)rows, (unsigned long long)row_bytes, box_rows, box_bytes);
    return FLEXIQ_OK;
}

int choose_bk(const Layer *L) { return L->C >= 128 ? 128 : 64; }

// ---------------------------------------------------------------------------------
// Weight preparation (Sec. 5, Sec. 4.1): the slab-order weight forms of a handle for a group order, and the
// tables that go with the order.  A selection search lays a layer out once per chromosome, so this runs between
// forward passes and not only once per layer.
//
// Bound by bytes: Wq is read once (K N), w8 and w8m (K N each), w4 (K N / 2) and sw (K N / G) are written, mostly
// in L2.  The original weights of a linear layer are [K][N] and the slab rows [N][K], so a byte transpose lies in
// between: done in registers (4 x 4 bytes by byte permutes) and through a shared-memory tile whose rows leave as
// whole 128-byte segments.  One thread per (group, output channel) with byte loads and byte stores, each store 32
// rows apart from its neighbour lane's, took 59.5 us for 768 x 3072 (2.4 MB in, 6.2 MB out).

// The group order and the activation positions travel in the launch's parameters (at most 4 KB of them) up to
// this many groups, i.e. 16,384 channels at the smallest group size; beyond it they are uploaded beforehand.
constexpr int kInlineGroups = 1024;
struct InlineOrder {
    uint16_t perm[kInlineGroups];
    uint8_t sx[kInlineGroups];   // slab order
};
struct PrepArgs {
    const int8_t *Wq;
    int aligned;          // Wq allows 4-byte (linear) or 16-byte (convolution) loads
    int C, N, G, T;
    int inline_order;     // the order is in InlineOrder and the tables are still to be written, else perm is on the device
    int32_t *perm, *inv_perm, *chunk_ent, *chunk_ent_slab;
    uint8_t *sx;
    int8_t *w8, *w8m;
    uint8_t *w4;
    int w4_pitch;
    uint8_t *sw;
    // linear layers: the straddle block (straddle.cuh) of the max_4bit_ch in force, NULL where that needs none
    int8_t *wst;
    int st_blk0, BK, K_lo;
};

// bytes with their sign folded away (v >= 0 ? v : ~v): the OR of a range's folded values has the bit length of the
// range's used magnitude bits
__device__ __forceinline__ uint32_t fold_signs(uint32_t w)
{
    uint32_t sign;
    asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(sign) : "r"(w));   // 0xff where the byte is negative
    return w ^ sign;
}
// extraction position of a group whose folded values OR to o: sign + 3 bits are kept
__device__ __forceinline__ int position_of(uint32_t o)
{
    const int used = 32 - __clz(o);
    return used > 3 ? used - 3 : 0;
}
// 16 weights of one slab row at position s: w8 as they are, w8m with the bits below s cleared, w4 the nibbles
__device__ __forceinline__ void write_forms(const PrepArgs &a, long long row8, long long row4, int col, const uint4 &v, int s)
{
    const uint32_t mask = ((0xffu << s) & 0xffu) * 0x01010101u;
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t n = (w[k] >> s) & 0x0f0f0f0fu;   // one nibble per byte
        h[k] = n | (n >> 4);                             // bytes 0 and 2 hold two nibbles each
    }
    *reinterpret_cast<uint4 *>(a.w8 + row8 + col) = v;
    *reinterpret_cast<uint4 *>(a.w8m + row8 + col) = make_uint4(w[0] & mask, w[1] & mask, w[2] & mask, w[3] & mask);
    *reinterpret_cast<uint2 *>(a.w4 + row4 + (col >> 1)) = make_uint2(__byte_perm(h[0], h[1], 0x6420), __byte_perm(h[2], h[3], 0x6420));
}
// the tables of an inline order that begins at `at`, by one block
__device__ __forceinline__ void write_tables(const PrepArgs &a, const InlineOrder &o, int at)
{
    const int n_g = a.C / a.G, cpg = a.G / 16;
    for (int j = threadIdx.x; j < n_g; j += blockDim.x) {
        const int g = o.perm[at + j];
        const int sx = o.sx[at + j];
        a.perm[j] = g;
        a.inv_perm[g] = j;
        a.sx[j] = (uint8_t)sx;
        // chunk table: original chunk c lies in original group c * 16 / G, which is slab group j with perm[j] = that group
        for (int i = 0; i < cpg; ++i) {
            const int ent = (j * cpg + i) | (sx << 24);
            a.chunk_ent[g * cpg + i] = ent;
            a.chunk_ent_slab[j * cpg + i] = ent;
        }
    }
}

// Linear weights [K][N].  A block transposes 128 slab channels x 64 output channels: thread (chunk, quad) loads 16
// channels of 4 output channels, so that 16 lanes cover 64 contiguous bytes of a row.  64 and not 128 output channels: 288 blocks
// instead of 144 for 768 x 3072, and 18 for 384 x 384.
constexpr int kPrepN = 64, kPrepChunks = 8;
constexpr int kPrepStatic = 9 * 1024, kPrepSmem = 228 * 1024 / 2 - 1024;   // the kernel's own shared memory, rounded up; what it asks for at most
// Several layers at once (a selection search lays a chain out per chromosome): a layer's blocks are too few to fill the machine, and
// four launches of 3 us each stood before every chain.
constexpr int kPrepLayers = 4;
struct PrepMany {
    PrepArgs a[kPrepLayers];
    int n, first_block[kPrepLayers], first_group[kPrepLayers], nx[kPrepLayers];   // nx: blocks across the output channels
};
__global__ void __launch_bounds__(kPrepN / 4 * kPrepChunks)
prep_linear_kernel(const __grid_constant__ PrepMany many, const __grid_constant__ InlineOrder order)
{
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();   // what runs before may still read the previous layout, or write Wq
    int which = 0;
    while (which + 1 < many.n && (int)blockIdx.x >= many.first_block[which + 1]) ++which;
    const PrepArgs &a = many.a[which];
    const int rel = (int)blockIdx.x - many.first_block[which], by = rel / many.nx[which], bx = rel - by * many.nx[which], at = many.first_group[which];
    __shared__ uint4 tile[kPrepN * kPrepChunks];      // [n][chunk ^ (n / 4)]: neither the writes nor the reads share a bank
    __shared__ uint32_t fold_s[kPrepChunks][kPrepN / 4];
    const int quad = threadIdx.x % (kPrepN / 4), chunk = threadIdx.x / (kPrepN / 4);
    const int n0 = bx * kPrepN + 4 * quad, c16 = by * kPrepChunks + chunk;
    const int cpg = a.G / 16, j = c16 / cpg;
    if (a.inline_order && rel == 0) write_tables(a, order, at);
    uint32_t r[16];
    uint32_t o = 0;
    const bool live = c16 < a.C / 16 && n0 < a.N;
    if (live) {
        const int g = a.inline_order ? (int)order.perm[at + j] : a.perm[j];
        const int8_t *src = a.Wq + (long long)(g * a.G + (c16 % cpg) * 16) * a.N + n0;
        if (a.aligned) {
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = *reinterpret_cast<const uint32_t *>(src + (long long)i * a.N);
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint8_t *b = reinterpret_cast<const uint8_t *>(src + (long long)i * a.N);
                r[i] = (uint32_t)b[0] | (uint32_t)b[1] << 8 | (uint32_t)b[2] << 16 | (uint32_t)b[3] << 24;
            }
        }
        uint32_t t[4][4];                               // [output channel][word of 4 channels]
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t *q = r + 4 * i;
            const uint32_t lo01 = __byte_perm(q[0], q[1], 0x5140), lo23 = __byte_perm(q[2], q[3], 0x5140);
            const uint32_t hi01 = __byte_perm(q[0], q[1], 0x7362), hi23 = __byte_perm(q[2], q[3], 0x7362);
            t[0][i] = __byte_perm(lo01, lo23, 0x5410);
            t[1][i] = __byte_perm(lo01, lo23, 0x7632);
            t[2][i] = __byte_perm(hi01, hi23, 0x5410);
            t[3][i] = __byte_perm(hi01, hi23, 0x7632);
            o |= fold_signs(q[0]) | fold_signs(q[1]) | fold_signs(q[2]) | fold_signs(q[3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) tile[(4 * quad + e) * kPrepChunks + (chunk ^ (quad & 7))] = make_uint4(t[e][0], t[e][1], t[e][2], t[e][3]);
    }
    fold_s[chunk][quad] = o;
    __syncthreads();
    // the whole group's folded OR, one byte per output channel (a group's chunks never span two blocks: 128 % G == 0)
    uint32_t go = 0;
    for (int i = 0; i < cpg; ++i) go |= fold_s[chunk - chunk % cpg + i][quad];
    __syncthreads();
    uint32_t pos = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) pos |= (uint32_t)position_of((go >> (8 * e)) & 0xffu) << (8 * e);
    fold_s[chunk][quad] = pos;
    if (live && chunk % cpg == 0) *reinterpret_cast<uint32_t *>(a.sw + (long long)j * a.N + n0) = pos;
    __syncthreads();
    // eight lanes write 128 contiguous bytes of one slab row
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int u = threadIdx.x + it * (kPrepN / 4 * kPrepChunks);
        const int nl = u / kPrepChunks, ch = u % kPrepChunks;
        const int n = bx * kPrepN + nl, c = by * kPrepChunks + ch;
        const bool here = n < a.N && c < a.C / 16;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        uint32_t mask = 0;
        if (here) {
            v = tile[nl * kPrepChunks + (ch ^ ((nl >> 2) & 7))];
            const int s = (int)((fold_s[ch][nl >> 2] >> (8 * (nl & 3))) & 0xffu);
            write_forms(a, (long long)n * a.C, (long long)n * a.w4_pitch, c * 16, v, s);
            mask = c * 16 < a.K_lo ? ((0xffu << s) & 0xffu) * 0x01010101u : 0xffffffffu;
        }
        // the block that max_4bit_ch falls into, from the same registers: channels below it masked, zeros beyond C
        const int col = c * 16 - a.st_blk0;
        if (a.wst != nullptr && n < a.N && col >= 0 && col < a.BK)
            *reinterpret_cast<uint4 *>(a.wst + (long long)n * a.BK + col) = make_uint4(v.x & mask, v.y & mask, v.z & mask, v.w & mask);
    }
}

// Convolution weights [N][T][C]: the slab rows have the same orientation, so 16-byte chunks move whole.  A block owns
// nb output channels and a window of groups; a position needs the group's chunks of every tap, so the chunks are
// folded first and read again (from L1 or L2) when they are written.
constexpr int kPrepGroups = 2048;   // groups per window: bounds the shared memory; one window up to 32,768 channels
__global__ void __launch_bounds__(256) prep_conv_kernel(const __grid_constant__ PrepArgs a, const __grid_constant__ InlineOrder order, int nb)
{
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();   // as above
    extern __shared__ uint32_t prep_s[];                // folded OR [nb][window], then the window's order
    const int g0 = blockIdx.y * kPrepGroups, n_g = min(kPrepGroups, a.C / a.G - g0);
    const int cpg = a.G / 16, n_c16 = n_g * cpg, units = a.T * n_c16;
    const int n_first = blockIdx.x * nb, n_here = min(nb, a.N - n_first);
    uint32_t *perm_s = prep_s + nb * n_g;
    if (a.inline_order && blockIdx.x == 0) write_tables(a, order, 0);   // an inline order is one window
    for (int i = threadIdx.x; i < nb * n_g; i += blockDim.x) prep_s[i] = 0;
    for (int i = threadIdx.x; i < n_g; i += blockDim.x) perm_s[i] = a.inline_order ? (uint32_t)order.perm[i] : (uint32_t)a.perm[g0 + i];
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
        for (int idx = threadIdx.x; idx < n_here * units; idx += blockDim.x) {
            const int nl = idx / units, u = idx - nl * units, t = u / n_c16, c = u - t * n_c16, j = c / cpg;
            const int8_t *src = a.Wq + ((long long)(n_first + nl) * a.T + t) * a.C + perm_s[j] * a.G + (c % cpg) * 16;
            uint4 v;
            if (a.aligned) v = *reinterpret_cast<const uint4 *>(src);
            else {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint8_t *b = reinterpret_cast<const uint8_t *>(src + 4 * k);
                    w[k] = (uint32_t)b[0] | (uint32_t)b[1] << 8 | (uint32_t)b[2] << 16 | (uint32_t)b[3] << 24;
                }
                v = make_uint4(w[0], w[1], w[2], w[3]);
            }
            if (pass == 0) {
                uint32_t o = fold_signs(v.x) | fold_signs(v.y) | fold_signs(v.z) | fold_signs(v.w);
                o |= o >> 16;
                o = (o | o >> 8) & 0xffu;
                if (o) atomicOr(&prep_s[nl * n_g + j], o);
            } else {
                write_forms(a, (long long)(n_first + nl) * a.T * a.C, (long long)(n_first + nl) * a.w4_pitch, t * a.C + g0 * a.G + c * 16, v,
                            position_of(prep_s[nl * n_g + j]));
            }
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < n_here * n_g; i += blockDim.x) {
        const int j = i / n_here, nl = i - j * n_here;
        a.sw[(long long)(g0 + j) * a.N + n_first + nl] = (uint8_t)position_of(prep_s[nl * n_g + j]);
    }
}

// layers[0 .. n): linear, their orders one after the other in `order`
static cudaError_t launch_prep_linear(const Layer *const *layers, const PrepArgs *args, int n, const InlineOrder &order, cudaStream_t stream)
{
    PrepMany many{};
    many.n = n;
    int blocks = 0, groups = 0;
    for (int i = 0; i < n; ++i) {
        const PrepArgs &a = many.a[i] = args[i];
        many.first_block[i] = blocks;
        many.first_group[i] = groups;
        many.nx[i] = (a.N + kPrepN - 1) / kPrepN;
        blocks += many.nx[i] * ((a.C / 16 + kPrepChunks - 1) / kPrepChunks);
        groups += a.C / a.G;
    }
    // spread evenly over the SMs: it is launched while the GEMM before it still runs on most of them
    const int device = layers[0]->device;
    static bool attr_set[64] = {};
    if (device >= 64 || !attr_set[device]) {
        const cudaError_t e = cudaFuncSetAttribute(prep_linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPrepSmem);
        if (e != cudaSuccess) return e;
        if (device < 64) attr_set[device] = true;
    }
    size_t smem = even_share_smem(blocks, device_sm_count(device));
    smem = smem > kPrepStatic ? smem - kPrepStatic : 0;
    return launch_pdl(prep_linear_kernel, (unsigned)blocks, kPrepN / 4 * kPrepChunks, smem, stream, many, order);
}
static cudaError_t launch_prep_conv(const Layer *L, const PrepArgs &a, const InlineOrder &order, cudaStream_t stream)
{
    // as many output channels per block as give every thread a chunk, but blocks enough for the machine
    const int sms = device_sm_count(L->device), window = L->n_g < kPrepGroups ? L->n_g : kPrepGroups;
    int nb = 256 / (a.T * window * (a.G / 16));
    if (nb > (a.N + sms - 1) / sms) nb = (a.N + sms - 1) / sms;
    if (nb < 1) nb = 1;
    const dim3 grid((a.N + nb - 1) / nb, (L->n_g + kPrepGroups - 1) / kPrepGroups);
    return launch_pdl(prep_conv_kernel, grid, 256, sizeof(uint32_t) * (size_t)(nb + 1) * window, stream, a, order, nb);
}

static int validate_perm(const int32_t *perm, int n_g)
{
    char *seen = (char *)calloc((size_t)n_g, 1);
    bool ok = true;
    for (int j = 0; j < n_g && ok; ++j) {
        if (perm[j] < 0 || perm[j] >= n_g || seen[perm[j]]) ok = false;
        else seen[perm[j]] = 1;
    }
    free(seen);
    if (!ok) return set_error(FLEXIQ_ERR_INVALID_ARG, "group_perm_host is not a permutation of 0..%d", n_g - 1);
    return FLEXIQ_OK;
}

static int validate_common(flexiq_layer_t *out, int C, int N, int G, const int8_t *Wq, const float *w_scale,
                           const int32_t *perm)
{
    if (!out) return set_error(FLEXIQ_ERR_INVALID_ARG, "out handle pointer is NULL");
    *out = nullptr;
    if (G != 16 && G != 32 && G != 64)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "group_size %d is not one of 16, 32, 64", G);
    if (C <= 0 || N <= 0) return set_error(FLEXIQ_ERR_INVALID_ARG, "channel counts must be positive (C=%d, N=%d)", C, N);
    if (C % G != 0) return set_error(FLEXIQ_ERR_INVALID_ARG, "input channels %d not a multiple of group_size %d", C, G);
    if (N % 16 != 0) return set_error(FLEXIQ_ERR_INVALID_ARG, "output channels %d not a multiple of 16", N);
    if (!Wq || !w_scale || !perm) return set_error(FLEXIQ_ERR_INVALID_ARG, "Wq_dev, w_scale_dev and group_perm_host must not be NULL");
    return validate_perm(perm, C / G);
}

static void free_layer(Layer *L)
{
    if (!L) return;
    if (L->tables_in_flight) cudaEventSynchronize(L->tables_event);
    cudaFree(L->w8); cudaFree(L->w8m); cudaFree(L->w4); cudaFree(L->wst); cudaFree(L->sw);
    cudaFree(L->tables); cudaFree(L->w_scale); cudaFree(L->bias); cudaFree(L->factor_mem);
    if (L->tables_host) cudaFreeHost(L->tables_host);
    if (L->tables_event) cudaEventDestroy(L->tables_event);
    L->magic = 0;
    free(L);
}

int encode_weight_maps(Layer *L)
{
    const int bk = choose_bk(L);
    const int *bns = kWeightMapRows;
    for (int i = 0; i < kNumWeightMaps; ++i) {
        int rc = make_map_2d(&L->map_w8[i], L->w8, (uint64_t)L->Kw, (uint64_t)L->N, (uint64_t)L->Kw, bk, bns[i], bk);
        if (rc) return rc;
        rc = make_map_2d(&L->map_w8m[i], L->w8m, (uint64_t)L->Kw, (uint64_t)L->N, (uint64_t)L->Kw, bk, bns[i], bk);
        if (rc) return rc;
        const uint64_t st_row = (uint64_t)L->R * L->S * bk;   // the straddle block of every tap
        rc = make_map_2d(&L->map_wst[i], L->wst, st_row, (uint64_t)L->N, st_row, bk, bns[i], bk);
        if (rc) return rc;
        rc = make_map_2d(&L->map_w4[i], L->w4, (uint64_t)L->Kw / 2, (uint64_t)L->N, (uint64_t)L->w4_pitch, bk / 2, bns[i],
                         bk / 2 == 64 ? 64 : 0);  // raw 4-bit tiles: 64-byte rows are read row-per-thread, so they are swizzled
        if (rc) return rc;
    }
    return FLEXIQ_OK;
}

// The layout post-processing of handles for a group order (Sec. 5): the order, the activation positions in slab
// order and the chunk tables, the slab-order weights, their positions and the 4-bit cache, all from the
// original-order weights.  Stream-ordered, allocates nothing on the device, does not wait for the stream: one launch
// that carries the orders in its parameters, or beyond kInlineGroups groups an upload from a pinned mirror before it.
static int plan_layout(Layer *L, const int8_t *Wq, const int32_t *perm, const uint8_t *x_shift, PrepArgs &a, InlineOrder &order, int at, cudaStream_t stream)
{
    const int n_g = L->n_g, C = L->C, G = L->G;
    a = PrepArgs{};
    a.Wq = Wq;
    a.aligned = (reinterpret_cast<uintptr_t>(Wq) & (L->is_conv ? 15u : 3u)) == 0;
    a.C = C; a.N = L->N; a.G = G; a.T = L->R * L->S;
    a.perm = L->perm; a.inv_perm = L->inv_perm; a.chunk_ent = L->chunk_ent; a.chunk_ent_slab = L->chunk_ent_slab; a.sx = L->sx;
    a.w8 = L->w8; a.w8m = L->w8m; a.w4 = L->w4; a.w4_pitch = L->w4_pitch; a.sw = L->sw;
    a.inline_order = n_g <= kInlineGroups;
    a.K_lo = L->K_lo;
    if (!L->is_conv && straddle_in_use(L)) {
        a.wst = L->wst;
        a.BK = choose_bk(L);
        a.st_blk0 = L->K_lo / a.BK * a.BK;
    }
    if (a.inline_order) {
        for (int j = 0; j < n_g; ++j) {
            order.perm[at + j] = (uint16_t)perm[j];
            order.sx[at + j] = x_shift ? x_shift[perm[j]] : 0;
        }
    } else {
        // the pinned mirror is free again once the previous upload has read it (normally long ago)
        if (L->tables_in_flight) FLEXIQ_CUDA_TRY(cudaEventSynchronize(L->tables_event));
        const int n_c = C / 16, cpg = G / 16;
        int32_t *h_perm = static_cast<int32_t *>(L->tables_host), *h_inv = h_perm + n_g, *h_ent = h_inv + n_g, *h_ent_slab = h_ent + n_c;
        uint8_t *h_sx = reinterpret_cast<uint8_t *>(h_ent_slab + n_c);
        // chunk table: original chunk c lies in original group c*16/G, which is slab group j with perm[j] = that group
        for (int j = 0; j < n_g; ++j) {
            h_perm[j] = perm[j];
            h_inv[perm[j]] = j;
            h_sx[j] = x_shift ? x_shift[perm[j]] : 0;  // slab order
            for (int i = 0; i < cpg; ++i) {
                h_ent[perm[j] * cpg + i] = (j * cpg + i) | ((int32_t)h_sx[j] << 24);
                h_ent_slab[j * cpg + i] = (j * cpg + i) | ((int32_t)h_sx[j] << 24);
            }
        }
        FLEXIQ_CUDA_TRY(cudaMemcpyAsync(L->tables, L->tables_host, L->tables_bytes, cudaMemcpyHostToDevice, stream));
        FLEXIQ_CUDA_TRY(cudaEventRecord(L->tables_event, stream));
        L->tables_in_flight = 1;
    }
    return FLEXIQ_OK;
}
static void layout_done(Layer *L, const PrepArgs &a, cudaStream_t stream)
{
    L->st_K_lo = -1;   // the straddle block was cut from the previous order's weights
    L->st_cap_id = 0;
    if (a.wst) straddle_written(L, stream);   // ... and this layout has cut it again
    const unsigned long long cap = stream_capture_id(stream);
    if (cap) { L->weights_cap_id = cap; L->weights_graph_seen = L->st_graph_seen = 1; }   // a replay makes both stale unseen
    else L->weights_fresh = 1;
    L->slab_next = 0;  // slabs written for the previous order are no longer this layer's
    memset(L->slab_seen, 0, sizeof(L->slab_seen));
}
static int layout_layer(Layer *L, const int8_t *Wq, const int32_t *perm, const uint8_t *x_shift, cudaStream_t stream)
{
    InlineOrder order;
    PrepArgs a;
    const int rc = plan_layout(L, Wq, perm, x_shift, a, order, 0, stream);
    if (rc) return rc;
    FLEXIQ_CUDA_TRY(L->is_conv ? launch_prep_conv(L, a, order, stream) : launch_prep_linear(&L, &a, 1, order, stream));
    layout_done(L, a, stream);
    return FLEXIQ_OK;
}

static int create_common(flexiq_layer_t *out, int is_conv, int C, int N, int R, int S, int stride, int pad,
                         int G, const int8_t *Wq, const float *w_scale, const float *bias,
                         const int32_t *perm, const uint8_t *x_shift, void *stream_)
{
    int rc = validate_common(out, C, N, G, Wq, w_scale, perm);
    if (rc) return rc;
    const int n_g = C / G;
    if (x_shift)
        for (int g = 0; g < n_g; ++g)
            if (x_shift[g] > 4) return set_error(FLEXIQ_ERR_INVALID_ARG, "x_shift_host[%d] = %d exceeds 4", g, x_shift[g]);
    if (is_conv && (R <= 0 || S <= 0 || stride <= 0 || pad < 0 || R > 15 || S > 15))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "bad conv geometry R=%d S=%d stride=%d pad=%d", R, S, stride, pad);
    rc = check_device_sm100();
    if (rc) return rc;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);

    Layer *L = (Layer *)calloc(1, sizeof(Layer));
    if (!L) return set_error(FLEXIQ_ERR_CUDA, "out of host memory");
    L->magic = kLayerMagic;
    L->is_conv = is_conv; L->C = C; L->N = N; L->G = G; L->n_g = n_g;
    L->R = R; L->S = S; L->stride = stride; L->pad = pad;
    L->Kw = R * S * C; L->w4_pitch = ((L->Kw / 2 + 15) / 16) * 16; L->K_lo = 0; L->lowbit_path = FLEXIQ_LOWBIT_MASKED_I8;
    cudaGetDevice(&L->device);
    const size_t wbytes = (size_t)N * L->Kw;
#define TRY_OR_FREE(expr)                                                                        \
    do {                                                                                         \
        cudaError_t e__ = (expr);                                                                \
        if (e__ != cudaSuccess) {                                                                \
            free_layer(L);                                                                       \
            return set_error(FLEXIQ_ERR_CUDA, "%s failed: %s", #expr, cudaGetErrorString(e__));  \
        }                                                                                        \
    } while (0)
    TRY_OR_FREE(cudaMalloc(&L->w8, wbytes));
    TRY_OR_FREE(cudaMalloc(&L->w8m, wbytes));
    TRY_OR_FREE(cudaMalloc(&L->wst, (size_t)N * R * S * choose_bk(L)));
    TRY_OR_FREE(cudaMalloc(&L->w4, (size_t)N * L->w4_pitch));
    TRY_OR_FREE(cudaMemsetAsync(L->w4, 0, (size_t)N * L->w4_pitch, stream));
    TRY_OR_FREE(cudaMalloc(&L->sw, (size_t)n_g * N));
    {
        // [perm n_g | inv_perm n_g | chunk_ent n_c | chunk_ent_slab n_c] int32, then sx [n_g] bytes
        const int n_c = C / 16;
        L->tables_bytes = sizeof(int32_t) * (2 * (size_t)n_g + 2 * (size_t)n_c) + (size_t)n_g;
        TRY_OR_FREE(cudaMalloc(&L->tables, L->tables_bytes));
        if (n_g > kInlineGroups) {
            TRY_OR_FREE(cudaMallocHost(&L->tables_host, L->tables_bytes));
            TRY_OR_FREE(cudaEventCreateWithFlags(&L->tables_event, cudaEventDisableTiming));
        }
        L->perm = static_cast<int32_t *>(L->tables);
        L->inv_perm = L->perm + n_g;
        L->chunk_ent = L->inv_perm + n_g;
        L->chunk_ent_slab = L->chunk_ent + n_c;
        L->sx = reinterpret_cast<uint8_t *>(L->chunk_ent_slab + n_c);
    }
    TRY_OR_FREE(cudaMalloc(&L->w_scale, sizeof(float) * N));
    if (bias) TRY_OR_FREE(cudaMalloc(&L->bias, sizeof(float) * N));
    L->st_K_lo = -1;
    L->slab_check = 1;
    TRY_OR_FREE(cudaMalloc(&L->factor_mem, sizeof(float) * 2 * (size_t)N * (Layer::kFactorTables + 1)));
    for (int i = 0; i <= Layer::kFactorTables; ++i) {
        L->factors[i].alpha = L->factor_mem + (size_t)2 * N * i;
        L->factors[i].beta = L->factors[i].alpha + N;
    }
    TRY_OR_FREE(cudaMemcpyAsync(L->w_scale, w_scale, sizeof(float) * N, cudaMemcpyDeviceToDevice, stream));
    if (bias) TRY_OR_FREE(cudaMemcpyAsync(L->bias, bias, sizeof(float) * N, cudaMemcpyDeviceToDevice, stream));
    rc = layout_layer(L, Wq, perm, x_shift, stream);
    if (rc) { free_layer(L); return rc; }
    TRY_OR_FREE(cudaStreamSynchronize(stream));
    L->weights_fresh = 0;   // waited for just now
#undef TRY_OR_FREE
    rc = encode_weight_maps(L);
    if (rc) { free_layer(L); return rc; }
    *out = reinterpret_cast<flexiq_layer_t>(L);
    return FLEXIQ_OK;
}

}  // namespace flexiq

using namespace flexiq;

extern "C" {

const char *flexiq_last_error(void) { return g_err; }

int flexiq_layer_create_linear(flexiq_layer_t *out, int K, int N, int group_size, const int8_t *Wq_dev,
                               const float *w_scale_dev, const float *bias_dev,
                               const int32_t *group_perm_host, const uint8_t *x_shift_host, void *stream)
{
    return create_common(out, 0, K, N, 1, 1, 1, 0, group_size, Wq_dev, w_scale_dev, bias_dev,
                         group_perm_host, x_shift_host, stream);
}

int flexiq_layer_create_conv(flexiq_layer_t *out, int Cin, int Cout, int R, int S, int stride, int pad,
                             int group_size, const int8_t *Wq_dev, const float *w_scale_dev,
                             const float *bias_dev, const int32_t *group_perm_host,
                             const uint8_t *x_shift_host, void *stream)
{
    return create_common(out, 1, Cin, Cout, R, S, stride, pad, group_size, Wq_dev, w_scale_dev, bias_dev,
                         group_perm_host, x_shift_host, stream);
}

static int check_layout(Layer *L, const int8_t *Wq_dev, const int32_t *group_perm_host, const uint8_t *x_shift_host)
{
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    if (!Wq_dev || !group_perm_host) return set_error(FLEXIQ_ERR_INVALID_ARG, "Wq_dev and group_perm_host must not be NULL");
    int rc = validate_perm(group_perm_host, L->n_g);
    if (rc) return rc;
    if (x_shift_host)
        for (int g = 0; g < L->n_g; ++g)
            if (x_shift_host[g] > 4) return set_error(FLEXIQ_ERR_INVALID_ARG, "x_shift_host[%d] = %d exceeds 4", g, x_shift_host[g]);
    return check_layer_device(L);
}

int flexiq_layer_set_group_perm(flexiq_layer_t layer, const int8_t *Wq_dev, const int32_t *group_perm_host,
                                const uint8_t *x_shift_host, void *stream)
{
    Layer *L = as_layer(layer);
    const int rc = check_layout(L, Wq_dev, group_perm_host, x_shift_host);
    if (rc) return rc;
    return layout_layer(L, Wq_dev, group_perm_host, x_shift_host, reinterpret_cast<cudaStream_t>(stream));
}

int flexiq_layers_set_group_perm(int n, const flexiq_layer_t *layers, const int8_t *const *Wq_dev, const int32_t *const *group_perm_host,
                                 const uint8_t *const *x_shift_host, void *stream)
{
    if (n < 0 || (n > 0 && (!layers || !Wq_dev || !group_perm_host)))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "n = %d is negative, or an array is NULL", n);
    int rc;
    for (int i = 0; i < n; ++i) {
        if ((rc = check_layout(as_layer(layers[i]), Wq_dev[i], group_perm_host[i], x_shift_host ? x_shift_host[i] : nullptr))) return rc;
        for (int k = 0; k < i; ++k)
            if (layers[k] == layers[i]) return set_error(FLEXIQ_ERR_INVALID_ARG, "layers[%d] and layers[%d] are the same handle", k, i);
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    InlineOrder order;
    PrepArgs args[kPrepLayers];
    for (int i = 0; i < n;) {
        // as many linear layers as one launch takes
        Layer *taken[kPrepLayers];
        int count = 0, groups = 0;
        for (; i + count < n && count < kPrepLayers; ++count) {
            Layer *L = as_layer(layers[i + count]);
            if (L->is_conv || groups + L->n_g > kInlineGroups) break;
            taken[count] = L;
            groups += L->n_g;
        }
        if (count < 2) {   // nothing to share a launch with
            if ((rc = layout_layer(as_layer(layers[i]), Wq_dev[i], group_perm_host[i], x_shift_host ? x_shift_host[i] : nullptr, st))) return rc;
            ++i;
            continue;
        }
        for (int k = 0, at = 0; k < count; at += taken[k]->n_g, ++k)
            if ((rc = plan_layout(taken[k], Wq_dev[i + k], group_perm_host[i + k], x_shift_host ? x_shift_host[i + k] : nullptr, args[k], order, at, st))) return rc;
        FLEXIQ_CUDA_TRY(launch_prep_linear(taken, args, count, order, st));
        for (int k = 0; k < count; ++k) layout_done(taken[k], args[k], st);
        i += count;
    }
    return FLEXIQ_OK;
}

int flexiq_layer_destroy(flexiq_layer_t layer)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    free_layer(L);
    return FLEXIQ_OK;
}

int flexiq_layer_set_lowbit_path(flexiq_layer_t layer, int lowbit_path)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    if (lowbit_path != FLEXIQ_LOWBIT_MASKED_I8 && lowbit_path != FLEXIQ_LOWBIT_PACKED_U4)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "unknown lowbit_path %d", lowbit_path);
    L->lowbit_path = lowbit_path;
    return FLEXIQ_OK;
}

int flexiq_set_lowbit_ratio(flexiq_layer_t layer, float ratio)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    if (!(ratio >= 0.0f && ratio <= 1.0f))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "ratio %f outside [0, 1]", (double)ratio);
    int n_low = (int)ceil((double)ratio * (double)L->n_g - 1e-4);
    if (n_low < 0) n_low = 0;
    if (n_low > L->n_g) n_low = L->n_g;
    L->K_lo = n_low * L->G;
    return FLEXIQ_OK;
}

int flexiq_layer_set_slab_check(flexiq_layer_t layer, int enabled)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    L->slab_check = enabled != 0;
    return FLEXIQ_OK;
}

int flexiq_get_max_4bit_ch(flexiq_layer_t layer, int *K_lo)
{
    Layer *L = as_layer(layer);
    if (!L || !K_lo) return set_error(FLEXIQ_ERR_INVALID_ARG, "bad handle or NULL output");
    *K_lo = L->K_lo;
    return FLEXIQ_OK;
}

int flexiq_layer_early_loads(flexiq_layer_t layer, int *weights, int *straddle)
{
    Layer *L = as_layer(layer);
    if (!L || !weights || !straddle) return set_error(FLEXIQ_ERR_INVALID_ARG, "bad handle or NULL output");
    *weights = L->early_w;
    *straddle = L->early_st;
    return FLEXIQ_OK;
}

int flexiq_x4_pitch(flexiq_layer_t layer, int K_lo, int64_t *pitch_bytes)
{
    Layer *L = as_layer(layer);
    if (!L || !pitch_bytes) return set_error(FLEXIQ_ERR_INVALID_ARG, "bad handle or NULL output");
    if (K_lo < 0 || K_lo > L->C || K_lo % L->G != 0)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "K_lo %d is not a multiple of the group size within [0, %d]", K_lo, L->C);
    *pitch_bytes = L->lowbit_path == FLEXIQ_LOWBIT_PACKED_U4 ? (int64_t)((K_lo / 2 + 15) / 16) * 16 : (int64_t)L->C;
    return FLEXIQ_OK;
}

int flexiq_layer_export(flexiq_layer_t layer, uint8_t *sw_host, int8_t *w8_host, uint8_t *w4_host)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    const size_t wbytes = (size_t)L->N * L->Kw;
    if (sw_host) FLEXIQ_CUDA_TRY(cudaMemcpy(sw_host, L->sw, (size_t)L->n_g * L->N, cudaMemcpyDeviceToHost));
    if (w8_host) FLEXIQ_CUDA_TRY(cudaMemcpy(w8_host, L->w8, wbytes, cudaMemcpyDeviceToHost));
    if (w4_host)
        FLEXIQ_CUDA_TRY(cudaMemcpy2D(w4_host, (size_t)L->Kw / 2, L->w4, (size_t)L->w4_pitch, (size_t)L->Kw / 2, (size_t)L->N,
                                     cudaMemcpyDeviceToHost));
    return FLEXIQ_OK;
}

}  // extern "C"
