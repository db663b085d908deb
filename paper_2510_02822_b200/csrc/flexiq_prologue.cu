// Activation prologue: quantize (Sec. 2.1, Eq. 1), bit-lower (Sec. 4.1, Fig. 3) and
// gather the channel groups into slab order (Sec. 5), writing the low-bit slab and the
// 8-bit slab that the mainloop consumes.  One pass over X (two in the dynamic
// extraction-position mode of the packed path), one 16-channel chunk per thread.
#include "flexiq_internal.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "sm100_ptx.cuh"
#include "copy_ring.cuh"
#include "eq1_quantize.cuh"
#include "straddle.cuh"


namespace flexiq {

__device__ __forceinline__ int position_from_or(unsigned o)
{
    const int used = 32 - __clz(o);  // highest bit in use among the folded values
    return used > 3 ? used - 3 : 0;
}

__global__ void clear_words_kernel(unsigned *words, int n)
{
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();
    for (int i = threadIdx.x; i < n; i += blockDim.x) words[i] = 0;
}

// Phase 1 of the dynamic mode (Sec. 4.1): OR of the sign-folded quantized values of each
// slab group over all rows.  A thread keeps one chunk column and walks rows; lanes that
// hold the same group merge with a warp reduction, then one shared and one global atomic.
template <int DTYPE>
__global__ void group_or_kernel(const void *X, long long M, int K, int G, float S,
                                const int32_t *perm, unsigned *__restrict__ or_words)
{
    extern __shared__ unsigned or_s[];
    const int n_c16 = K / 16, c_per_g = G / 16, n_g = K / G;
    for (int i = threadIdx.x; i < n_g; i += blockDim.x) or_s[i] = 0;
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();  // the kernel before this one in the stream may still be producing X
    __syncthreads();
    // grid-wide thread count is a multiple of n_c16, so each thread keeps its chunk column
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    const long long rows_per_pass = nthreads / n_c16;
    const int c16 = (int)(tid % n_c16);
    const int j = c16 / c_per_g;
    const Divider div = make_divider(S);
    unsigned o = 0;
    if (tid < rows_per_pass * n_c16) {
        const int src_c = perm[j] * G + (c16 % c_per_g) * 16;
        for (long long m = tid / n_c16; m < M; m += rows_per_pass) {
            unsigned w[4];
            quantize16<DTYPE>(reinterpret_cast<const char *>(X) + ((size_t)m * K + src_c) * elem_bytes<DTYPE>(), div, -128.f, 127.f, w);
            // fold negatives per byte (q >= 0 ? q : ~q): xor with the byte's sign replicated
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned sign = (w[k] >> 7) & 0x01010101u;
                o |= w[k] ^ (sign * 0xffu);
            }
        }
    }
    o = (o | (o >> 8) | (o >> 16) | (o >> 24)) & 0xffu;  // OR of the four byte lanes
    const unsigned peers = __match_any_sync(0xffffffffu, j);
    const unsigned merged = __reduce_or_sync(peers, o);
    if ((threadIdx.x & 31) == (__ffs(peers) - 1) && merged) atomicOr(&or_s[j], merged);
    __syncthreads();
    for (int i = threadIdx.x; i < n_g; i += blockDim.x)
        if (or_s[i]) atomicOr(&or_words[i], or_s[i]);
}

// ---------------------------------------------------------------------------------
// Masked path.
//
// Bound by HBM: every input byte is read once and one byte per value written.  A tile is a few whole rows, contiguous in
// memory, which one bulk copy brings into a ring in shared memory; the gather into slab order is done from there.  Bulk
// copies read at 6.7 TB/s where 128-bit loads by all threads, whatever their number and order, stay at 5.5 to 5.9 (206 MB,
// read only; 38.7 MB: 7.5 us against 8.9 to 10), and the gather costs no sectors (a 16-byte int8 chunk is half of one).
// A thread keeps its row within the tile and its slab chunk from tile to tile, so that a step is the 128-bit reads of its
// chunk, the arithmetic and one 128-bit store; the stores of a warp are contiguous.  Measured, replayed from a graph on buffers
// larger than L2, against one chunk per thread by plain loads: fp16 25216 x 4096 62.3 -> 51.8 us (6.0 TB/s; a plain
// copy of the same bytes reaches 6.2), fp16 25216 x 1024 17.3 -> 15.6, fp32 12608 x 768 10.6 -> 9.4, int8 12608 x 3072 19.8 -> 14.8.
constexpr int kRowWarps = 8;                     // consumer warps per block at most; one more issues the copies
constexpr int kRowStages = 8;                    // ring stages at most
constexpr int kRowRing = 49152;                  // bytes of ring a block aims at: four blocks per SM
constexpr int kRowStageBytes = 65536;            // largest row the ring takes; wider rows go through the packed path's kernels
constexpr int kRowSmem = 3 * kRowStageBytes + 32768;   // three stages of that and the tables of 65,536 channels (int8)
constexpr uint32_t kCopyWaitLimit = 1u << 21;    // parked waits of at most a microsecond each: about two seconds

__device__ unsigned int g_prologue_status = 0;

// Bounded wait; false after the limit or when another warp already gave up.
__device__ __forceinline__ bool wait_copy(uint32_t bar, uint32_t parity, volatile int *gave_up, uint32_t limit = kCopyWaitLimit)
{
    if (ptx::mbar_try_wait_s(bar, parity)) return true;
    for (uint32_t it = 0; it < limit; ++it) {
        if (ptx::mbar_try_wait_hint_s(bar, parity, 1000u)) return true;
        if (*gave_up) return false;
    }
    *gave_up = 1;
    atomicMax(&g_prologue_status, 0x301u);
    return false;
}

// Where slab chunk c comes from and how it is lowered: source chunk | shift << 28.  A low group keeps bits s..s+3 of
// values clipped to what four bits hold at position s; an 8-bit group is the same at position 4 with nothing cleared,
// which is told apart by shift 5: one instruction stream for both, since a warp spans the boundary in most rows.
constexpr unsigned kShift8Bit = 5;
__device__ __forceinline__ unsigned chunk_entry(int c, int log_cpg, int lo_c16, const int32_t *perm, const uint8_t *sx)   // 1 << log_cpg chunks a group
{
    const int j = c >> log_cpg;
    const unsigned shift = c < lo_c16 ? (unsigned)sx[j] : kShift8Bit;
    return (unsigned)((perm[j] << log_cpg) + (c - (j << log_cpg))) | (shift << 28);
}

struct RowsArgs {
    const void *X;
    int8_t *slab;
    long long M, tiles;
    int K, G, K_lo;
    int rows;                  // rows per tile
    int stages, stage_bytes;
    int ahead;                 // tiles a block asks into L2 before its dependency wait
    float S;
    QuotientPlan quot;
    const int32_t *perm;
    const uint8_t *sx;         // static positions, slab order
    unsigned *or_words;        // dynamic: OR of the sign-folded values of every group
    StraddleJob wp;
};

// DYN: phase 1 of the dynamic mode.  Every group is written at 8 bits and the OR of the sign-folded values of every
// group is collected on the way, so that the input is read once.
template <int DTYPE, bool DYN>
__global__ void __launch_bounds__(32 * (kRowWarps + 1)) quantize_rows_kernel(const __grid_constant__ RowsArgs a)
{
    constexpr int kBytes = DTYPE == FLEXIQ_DTYPE_F32 ? 4 : (DTYPE == FLEXIQ_DTYPE_I8 ? 1 : 2);
    constexpr int kPieces = kBytes;                  // 16-byte pieces per chunk: 4, 2 or 1
    extern __shared__ __align__(128) uint8_t rows_smem[];
    __shared__ uint64_t full_bar[kRowStages], empty_bar[kRowStages];
    __shared__ int gave_up;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (blockDim.x >> 5) - 1;
    const int n_c16 = a.K / 16, lo_c16 = DYN ? 0 : a.K_lo / 16, log_cpg = a.G == 16 ? 0 : a.G == 32 ? 1 : 2;
    unsigned *table = reinterpret_cast<unsigned *>(rows_smem + a.stages * a.stage_bytes);
    unsigned *or_s = table + n_c16;
    ptx::pdl_launch_dependents();
    if (blockIdx.x < a.wp.first_block) {
        // Extra blocks in front of the quantizing ones (so that they run beside the first wave, not behind the
        // last): the weight K block that max_4bit_ch falls into, for the GEMM that consumes these slabs -- the
        // only weight data that depends on the ratio -- 16 bytes per thread.
        const StraddleUnit unit(a.wp, (long long)blockIdx.x * blockDim.x + threadIdx.x);
        unit.ask();
        ptx::pdl_wait();
        unit.write();
        return;
    }
    const long long first = blockIdx.x - a.wp.first_block, step = gridDim.x - a.wp.first_block;
    const size_t row_bytes = (size_t)a.K * kBytes, tile_bytes = (size_t)a.rows * row_bytes;
    auto bytes_of = [&](long long tile) { return (uint32_t)(min((long long)a.rows, a.M - tile * a.rows) * (long long)row_bytes); };
    auto copy = [&](long long tile, int stage) {
        const uint32_t bytes = bytes_of(tile);
        const uint32_t bar = ptx::smem_u32(&full_bar[stage]);
        ptx::mbar_expect_tx_s(bar, bytes);
        ptx::bulk_load(ptx::smem_u32(rows_smem) + (uint32_t)(stage * a.stage_bytes),
                       reinterpret_cast<const char *>(a.X) + (size_t)tile * tile_bytes, bytes, bar);
    };
    // Everything that needs no global memory comes before the dependency wait: a small launch is one chain of latencies behind it.
    const int threads = 32 * warps, units = a.rows * n_c16;
    const bool single = units <= threads;            // one chunk per thread and tile, the same in every tile
    const int r0 = (int)threadIdx.x / n_c16, c0 = (int)threadIdx.x - r0 * n_c16;
    long long next = first;                          // the copying thread's next tile
    const bool copier = warp == warps && lane == 0;
    if (copier) {
        for (int i = 0; i < a.stages; ++i) {
            ptx::mbar_init(&full_bar[i], 1);
            ptx::mbar_init(&empty_bar[i], warps);
        }
        gave_up = 0;
        ptx::fence_mbar_init();
        // Where X was there before the previous kernel began, its first tiles can come from memory while that one ends: asked into
        // L2, which is where a write of that kernel would go too, so nothing is read early.
        long long t = first;
        for (int i = 0; i < a.ahead && t < a.tiles; ++i, t += step)
            ptx::bulk_prefetch_l2(reinterpret_cast<const char *>(a.X) + (size_t)t * tile_bytes, bytes_of(t));
    }
    if (DYN)
        for (int j = threadIdx.x; j < a.K / a.G; j += blockDim.x) or_s[j] = 0;
    __syncthreads();
    ptx::pdl_wait();  // the previous kernel may still read the slab this one overwrites, or write X
    if (copier)
        for (int i = 0; i < a.stages && next < a.tiles; ++i, next += step) copy(next, i);
    // A thread with one chunk fetches that chunk's entry itself; otherwise the block makes a table.  (With the entries by shifts and
    // all that needs no memory ahead of the wait: DeiT-S at batch 1, 48 layers, 265.9 -> 254.3 us, one block at batch 8 28.9 -> 27.9,
    // 1001 x 720 bf16 with its GEMM 7.8 -> 7.45; ViT-B sweep level.)
    unsigned ent = 0;
    if (single) {
        if ((int)threadIdx.x < units) ent = chunk_entry(c0, log_cpg, lo_c16, a.perm, a.sx);
    } else {
        for (int c = threadIdx.x; c < n_c16; c += blockDim.x) table[c] = chunk_entry(c, log_cpg, lo_c16, a.perm, a.sx);
        __syncthreads();
    }
    if (warp == warps) {
        if (lane == 0) {
            // refill a stage when every warp has read it
            int stage = 0;
            uint32_t phase = 0;
            for (; next < a.tiles; next += step) {
                if (!wait_copy(ptx::smem_u32(&empty_bar[stage]), phase, &gave_up)) break;
                copy(next, stage);
                if (++stage == a.stages) { stage = 0; phase ^= 1; }
            }
        }
    } else {
        unsigned src = 0, shift = kShift8Bit, mask = 0xffffffffu;
        float lo = -128.f, hi = 127.f;
        auto position = [&](int r, unsigned ent) {   // of the chunk of this entry in row r of a tile
            src = (unsigned)r * (unsigned)row_bytes + (ent & 0x0fffffffu) * (16u * kBytes);
            if (DYN) return;
            shift = ent >> 28;
            const float bound = (float)(8u << min(shift, 4u));
            lo = -bound;
            hi = bound - 1.f;
            mask = shift == kShift8Bit ? 0xffffffffu : ((0xffu << shift) & 0xffu) * 0x01010101u;
        };
        if (single) position(r0, ent);
        unsigned held = 0;                           // DYN: OR of the folded words this thread has seen, four bytes wide
        auto merge = [&](unsigned o, int c) {
            o |= o >> 16;
            o = (o | (o >> 8)) & 0xffu;
            unsigned *seen = or_s + (c >> log_cpg);
            if (o & ~*reinterpret_cast<volatile unsigned *>(seen)) atomicOr(seen, o);   // rare after the first rows
        };
        int stage = 0;
        uint32_t phase = 0;
        for (long long tile = first; tile < a.tiles; tile += step) {
            if (!__all_sync(0xffffffffu, wait_copy(ptx::smem_u32(&full_bar[stage]), phase, &gave_up))) break;
            const uint32_t base = ptx::smem_u32(rows_smem) + (uint32_t)(stage * a.stage_bytes);
            const int here = (int)min((long long)a.rows, a.M - tile * a.rows) * n_c16;
            int r = r0, c = c0;
            for (int u = threadIdx.x; u < here; u += threads) {
                if (!single) position(r, table[c]);
                uint4 raw[kPieces];
                // Neighbouring lanes start at different pieces of their chunks: with one order for all, the 16-byte reads
                // of a quarter warp would share half (16-bit inputs) or a quarter (fp32) of the banks.
                const unsigned turn = kPieces == 1 ? 0u : (unsigned)lane % kPieces;
#pragma unroll
                for (int p = 0; p < kPieces; ++p) raw[p] = ptx::ld_shared_128(base + src + ((p + turn) % kPieces) * 16);
                unsigned w[4];
                if constexpr (DTYPE == FLEXIQ_DTYPE_I8) {
                    const unsigned in[4] = {raw[0].x, raw[0].y, raw[0].z, raw[0].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = DYN ? in[k] : clip_bytes(in[k], min(shift, 4u));
                } else if (a.quot.form == kQuotGeneral) {
                    quantize_raw<DTYPE>(raw, make_divider(a.S), lo, hi, w);
                } else if constexpr (DTYPE == FLEXIQ_DTYPE_F32) {
                    quantize_raw<DTYPE>(raw, TwoTerm{a.quot.r_hi, a.quot.r_lo}, lo, hi, w);
                } else {
                    quantize_raw_magic<DTYPE>(raw, a.quot.r_hi, lo, hi, w);
                }
                // back to channel order: piece p of the chunk is in place (p - turn) mod kPieces
                if constexpr (kPieces == 4) {
                    if (turn & 1) { const unsigned t = w[3]; w[3] = w[2]; w[2] = w[1]; w[1] = w[0]; w[0] = t; }
                    if (turn & 2) { const unsigned t0 = w[0], t1 = w[1]; w[0] = w[2]; w[1] = w[3]; w[2] = t0; w[3] = t1; }
                } else if constexpr (kPieces == 2) {
                    if (turn) { const unsigned t0 = w[0], t1 = w[1]; w[0] = w[2]; w[1] = w[3]; w[2] = t0; w[3] = t1; }
                }
                if (DYN) {
                    unsigned o = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {   // fold negatives per byte (q >= 0 ? q : ~q): xor with the byte's sign replicated
                        unsigned sign;
                        asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(sign) : "r"(w[k]));
                        o |= w[k] ^ sign;
                    }
                    if (single) held |= o;      // its own chunk in every tile: merged once, behind the last
                    else merge(o, c);
                }
                *reinterpret_cast<uint4 *>(a.slab + (size_t)tile * (size_t)(units * 16) + (size_t)u * 16) =
                    make_uint4(w[0] & mask, w[1] & mask, w[2] & mask, w[3] & mask);
                if (!single) {
                    c += threads;
                    while (c >= n_c16) { c -= n_c16; ++r; }
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&empty_bar[stage]);
            if (++stage == a.stages) { stage = 0; phase ^= 1; }
        }
        if (DYN && single && (int)threadIdx.x < units) merge(held, c0);
    }
    __syncthreads();
    if (gave_up) {
        if (copier) drain_ring(full_bar, a.stages, (next - first) / step);   // the tiles it has requested
        return;
    }
    if (DYN) {
        // with many blocks most find nothing new in the end: a read saves the atomic
        const bool look = gridDim.x > 128;
        for (int j = threadIdx.x; j < a.K / a.G; j += blockDim.x) {
            const unsigned o = or_s[j];
            if (o & ~(look ? __ldcg(a.or_words + j) : 0u)) atomicOr(a.or_words + j, o);
        }
    }
}

// Test hook: a ring of two stages given up on with copies in flight.  Three copies are issued, the third into the first
// one's stage; a wait of about a millisecond on a barrier that nothing arrives on gives up; after the drain the stages hold
// what the last copies brought.
constexpr int kDrainBytes = 16384;
__global__ void drain_kernel(const uint8_t *src, int *result)
{
    __shared__ __align__(128) uint8_t ring[2][kDrainBytes];
    __shared__ uint64_t full[2], never;
    __shared__ int gave_up;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) ptx::mbar_init(&full[i], 1);
        ptx::mbar_init(&never, 1);
        gave_up = 0;
        ptx::fence_mbar_init();
        auto copy = [&](int i) {
            const uint32_t bar = ptx::smem_u32(&full[i & 1]);
            ptx::mbar_expect_tx_s(bar, kDrainBytes);
            ptx::bulk_load(ptx::smem_u32(ring[i & 1]), src + (size_t)i * kDrainBytes, kDrainBytes, bar);
        };
        copy(0);
        const bool served = wait_copy(ptx::smem_u32(&full[0]), 0, &gave_up, 4096u);
        const bool starved = wait_copy(ptx::smem_u32(&never), 0, &gave_up, 1024u);
        copy(1);
        if (served) copy(2);
        const bool landed = drain_ring(full, 2, served ? 3 : 2);
        int wrong = 0;
        for (int s = 0; s < 2; ++s)
            for (int b = 0; b < kDrainBytes; ++b) wrong += ring[s][b] != src[(size_t)(2 - s) * kDrainBytes + b];
        result[0] = served;
        result[1] = starved;
        result[2] = gave_up;
        result[3] = landed;
        result[4] = wrong;
    }
}

// Phase 2 of the dynamic mode: the low groups of the slab that phase 1 wrote are lowered in place with the positions
// the OR words give, 16 bytes per thread.  The positions cover every value of the call, so nothing saturates and
// lowering is clearing the bits below the position; a group whose position is 0 is already what it should be and
// is not touched.  The positions go to sx_out (slab order).  Blocks in front: the straddle block of the weights.
__global__ void lower_inplace_kernel(int8_t *__restrict__ slab, long long M, int K, int G, int K_lo,
                                     const unsigned *or_words, uint8_t *__restrict__ sx_out, StraddleJob wp,
                                     int step_m, int step_c)
{
    ptx::pdl_launch_dependents();
    if (blockIdx.x < wp.first_block) {
        const StraddleUnit unit(wp, (long long)blockIdx.x * blockDim.x + threadIdx.x);
        unit.ask();
        ptx::pdl_wait();
        unit.write();
        return;
    }
    ptx::pdl_wait();  // phase 1 has written the slab and the OR words
    const unsigned qblock = blockIdx.x - wp.first_block;
    if (qblock == 0)
        for (int j = threadIdx.x; j < K / G; j += blockDim.x) sx_out[j] = (uint8_t)position_from_or(__ldcg(or_words + j));
    const int lo_c16 = K_lo / 16, c_per_g = G / 16;
    if (lo_c16 == 0) return;
    const long long idx = (long long)qblock * blockDim.x + threadIdx.x;
    long long m = idx / lo_c16;
    int c = (int)(idx - m * lo_c16);
    while (m < M) {
        // four units at a time: their loads are in flight together
        uint4 *ptr[4];
        uint4 v[4];
        unsigned mask[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ptr[i] = nullptr;
            if (m < M) {
                const int s = position_from_or(__ldcg(or_words + c / c_per_g));
                mask[i] = ((0xffu << s) & 0xffu) * 0x01010101u;
                if (s) {
                    ptr[i] = reinterpret_cast<uint4 *>(slab + (size_t)m * K + (size_t)c * 16);
                    v[i] = *ptr[i];
                }
            }
            m += step_m;
            c += step_c;
            if (c >= lo_c16) { c -= lo_c16; ++m; }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (ptr[i]) *ptr[i] = make_uint4(v[i].x & mask[i], v[i].y & mask[i], v[i].z & mask[i], v[i].w & mask[i]);
    }
}

// Dynamic mode in one launch.  A cluster of eight CTAs owns a window of slab chunks (whole groups), each CTA an eighth of the
// rows: it quantizes its part of the columns into shared memory, the CTAs read one another's OR words through
// distributed shared memory, and each lowers and writes what it holds.  The input is read once, the slab written once, and
// nothing is cleared beforehand or read back: 197 x 384 fp16 8.3 -> 3.3 us, 1576 x 1536 fp32 12.4 -> 9.0, 6304 x 768 fp16 14.4 -> 9.4 (graph
// replay, against a clear and two launches).
// The window is 32 bytes of a slab row (64 for groups of 64), so that a row's stores are whole sectors.
constexpr int kColCluster = 8;
constexpr int kColThreads = 256;
constexpr long long kColBytes = 10ll << 20, kColRows = 6144;   // of input, rows: the largest calls it takes (see columns_fit)
constexpr int kColSmem = 228 * 1024 / 2 - 1024;   // one CTA per SM at most (see launch_columns); the rows a CTA holds take up to 48 KB

struct ColumnsArgs {
    const void *X;
    int8_t *slab;
    long long M;
    int K, G, K_lo;
    int window, rows;          // chunks per cluster, rows per CTA
    float S;
    QuotientPlan quot;
    const int32_t *perm;
    uint8_t *sx_out;
    StraddleJob wp;
};

template <int DTYPE>
__global__ void __launch_bounds__(kColThreads) dynamic_columns_kernel(const __grid_constant__ ColumnsArgs a)
{
    constexpr int kBytes = DTYPE == FLEXIQ_DTYPE_F32 ? 4 : (DTYPE == FLEXIQ_DTYPE_I8 ? 1 : 2);
    constexpr int kPieces = kBytes, kAhead = DTYPE == FLEXIQ_DTYPE_F32 ? 2 : 4;   // rows in flight per thread
    extern __shared__ __align__(128) uint8_t cols_smem[];
    __shared__ unsigned or_s[4], all_s[4];
    uint4 *held = reinterpret_cast<uint4 *>(cols_smem);
    ptx::pdl_launch_dependents();
    if (blockIdx.x < a.wp.first_block) {   // whole clusters: the straddle block of the weights
        const StraddleUnit unit(a.wp, (long long)blockIdx.x * blockDim.x + threadIdx.x);
        unit.ask();
        ptx::pdl_wait();
        unit.write();
        return;
    }
    const int n_c16 = a.K / 16, cpg = a.G / 16;
    const int rank = (int)ptx::cluster_ctarank(), first = (int)((blockIdx.x - a.wp.first_block) / kColCluster) * a.window;
    const int cl = threadIdx.x % a.window, c = first + cl, j = c / cpg;
    const bool live = c < n_c16;
    const int r0 = threadIdx.x / a.window, step = kColThreads / a.window;
    const long long m_first = (long long)rank * a.rows;
    const int rows = (int)max(0ll, min((long long)a.rows, a.M - m_first));
    if (threadIdx.x < 4) { or_s[threadIdx.x] = 0; all_s[threadIdx.x] = 0; }
    __syncthreads();
    ptx::pdl_wait();  // the previous kernel may still read the slab this one overwrites, or write X
    if (live) {
        const size_t row_bytes = (size_t)a.K * kBytes;
        const char *src = reinterpret_cast<const char *>(a.X) + (size_t)(m_first + r0) * row_bytes + ((size_t)a.perm[j] * a.G + (c % cpg) * 16) * kBytes;
        unsigned o = 0;
        for (int r = r0; r < rows; r += kAhead * step, src += (size_t)(kAhead * step) * row_bytes) {
            uint4 raw[kAhead][kPieces];
#pragma unroll
            for (int i = 0; i < kAhead; ++i)
                if (r + i * step < rows) {
#pragma unroll
                    for (int p = 0; p < kPieces; ++p) raw[i][p] = reinterpret_cast<const uint4 *>(src + (size_t)(i * step) * row_bytes)[p];
                }
#pragma unroll
            for (int i = 0; i < kAhead; ++i)
                if (r + i * step < rows) {
                    unsigned w[4];
                    if constexpr (DTYPE == FLEXIQ_DTYPE_I8) {
                        w[0] = raw[i][0].x; w[1] = raw[i][0].y; w[2] = raw[i][0].z; w[3] = raw[i][0].w;
                    } else if (a.quot.form == kQuotGeneral) {
                        quantize_raw<DTYPE>(raw[i], make_divider(a.S), -128.f, 127.f, w);
                    } else if constexpr (DTYPE == FLEXIQ_DTYPE_F32) {
                        quantize_raw<DTYPE>(raw[i], TwoTerm{a.quot.r_hi, a.quot.r_lo}, -128.f, 127.f, w);
                    } else {
                        quantize_raw_magic<DTYPE>(raw[i], a.quot.r_hi, -128.f, 127.f, w);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {   // fold negatives per byte
                        unsigned sign;
                        asm("prmt.b32 %0, %1, 0, 0xba98;" : "=r"(sign) : "r"(w[k]));
                        o |= w[k] ^ sign;
                    }
                    held[(r + i * step) * a.window + cl] = make_uint4(w[0], w[1], w[2], w[3]);
                }
        }
        o |= o >> 16;
        o = (o | (o >> 8)) & 0xffu;
        if (o) atomicOr(&or_s[cl], o);
    }
    ptx::cluster_sync_all();       // every CTA's OR words are complete
    if ((int)threadIdx.x < kColCluster * a.window) {
        const unsigned o = ptx::ld_shared_cluster(ptx::mapa(ptx::smem_u32(&or_s[threadIdx.x % a.window]), threadIdx.x / a.window));
        if (o) atomicOr(&all_s[threadIdx.x % a.window], o);
    }
    ptx::cluster_sync_all();       // and read: a CTA may leave
    unsigned o = 0;
    for (int i = 0; i < cpg; ++i) o |= all_s[cl / cpg * cpg + i];
    const int s = position_from_or(o);
    if (!live) return;
    if (rank == 0 && r0 == 0 && c % cpg == 0) a.sx_out[j] = (uint8_t)s;
    const unsigned mask = c < a.K_lo / 16 ? ((0xffu << s) & 0xffu) * 0x01010101u : 0xffffffffu;
    for (int r = r0; r < rows; r += step) {
        const uint4 v = held[r * a.window + cl];
        *reinterpret_cast<uint4 *>(a.slab + (size_t)(m_first + r) * a.K + (size_t)c * 16) = make_uint4(v.x & mask, v.y & mask, v.z & mask, v.w & mask);
    }
}

// Packed path, and the masked path's rows that are too wide for the ring: quantize + lower + gather.  Thread <-> (row m,
// 16-channel slab chunk c16).
//   sx != nullptr : static positions (slab order);  else positions from or_words.
// Lowering works on the packed int8 words: q is first clipped to the range the 4-bit value
// at position s can hold, [-2^(s+3), 2^(s+3) - 1] (identical to clamping q >> s to [-8, 7],
// the shift being monotone); then bits s..s+3 of every byte are the two's-complement nibble (packed path), and
// clearing the s low bits of every byte is (q >> s) << s (masked path: one slab, X8 lies behind the low groups of X4).
template <int DTYPE, bool PACKED>
__global__ void quantize_chunks_kernel(const void *X, long long M, int K, int G, int K_lo, float S,
                                       const int32_t *perm, const uint8_t *sx,
                                       const unsigned *or_words, uint8_t *__restrict__ X4,
                                       long long x4_pitch, int8_t *__restrict__ X8, long long x8_pitch, uint8_t *__restrict__ sx_out)
{
    const int n_c16 = K / 16, c_per_g = G / 16, lo_c16 = K_lo / 16;
    const long long total = M * n_c16;
    const Divider div = make_divider(S);
    ptx::pdl_launch_dependents();
    ptx::pdl_wait();  // the previous kernel may still read the slabs this one overwrites, or write X
    if (sx_out != nullptr && blockIdx.x == 0)
        for (int j = threadIdx.x; j < K / G; j += blockDim.x) sx_out[j] = (uint8_t)position_from_or(or_words[j]);
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const long long m = idx / n_c16;
        const int c16 = (int)(idx - m * n_c16);
        const int j = c16 / c_per_g;
        const int src_c = perm[j] * G + (c16 % c_per_g) * 16;
        const void *src = reinterpret_cast<const char *>(X) + ((size_t)m * K + src_c) * elem_bytes<DTYPE>();
        unsigned w[4];
        if (c16 < lo_c16) {
            const int s = sx ? (int)sx[j] : position_from_or(or_words[j]);
            const float bound = (float)(8 << s);
            quantize16<DTYPE>(src, div, -bound, bound - 1.f, w);
            if (PACKED) {
                unsigned h[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const unsigned n = (w[k] >> s) & 0x0f0f0f0fu;  // one nibble per byte
                    h[k] = n | (n >> 4);                            // bytes 0 and 2 now hold two nibbles each
                }
                *reinterpret_cast<uint2 *>(X4 + m * x4_pitch + (size_t)c16 * 8) =
                    make_uint2(__byte_perm(h[0], h[1], 0x6420), __byte_perm(h[2], h[3], 0x6420));
            } else {
                const unsigned mask = ((0xffu << s) & 0xffu) * 0x01010101u;
                *reinterpret_cast<uint4 *>(X4 + m * x4_pitch + (size_t)c16 * 16) =
                    make_uint4(w[0] & mask, w[1] & mask, w[2] & mask, w[3] & mask);
            }
        } else {
            quantize16<DTYPE>(src, div, -128.f, 127.f, w);
            *reinterpret_cast<uint4 *>(X8 + m * x8_pitch + (size_t)(c16 - lo_c16) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// Scratch of the allocation-free dynamic prologue: one OR word per channel group.  The array
// lives in the library image, so every GPU that loads the library holds these 16 KB until the
// process exits.  All calls on a device share it.
constexpr int kStaticScratchGroups = 4096;
static __device__ __align__(256) unsigned g_static_group_or[kStaticScratchGroups];

// Device address of the array above on the current device.  In host code the array's name is
// only a handle for the runtime, not a device pointer, so the address is looked up with
// cudaGetSymbolAddress -- once per device, with that device current -- and cached.
static int static_scratch_address(unsigned **out)
{
    static unsigned *cached[64] = {};
    int dev = 0;
    FLEXIQ_CUDA_TRY(cudaGetDevice(&dev));   // the caller has checked that this is the layer's device
    if (dev < 0 || dev >= 64) return set_error(FLEXIQ_ERR_UNSUPPORTED, "device ordinal %d is beyond the 64 this entry point tracks", dev);
    if (cached[dev] == nullptr) {
        void *p = nullptr;
        FLEXIQ_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_group_or));
        if (p == nullptr) return set_error(FLEXIQ_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
        cached[dev] = static_cast<unsigned *>(p);
    }
    *out = cached[dev];
    return FLEXIQ_OK;
}

// The plan of the layer's scale (plan_quotient takes about half a microsecond for 16-bit inputs), one per input type.
static QuotientPlan quotient_plan(Layer *L, float S, int dtype)
{
    Layer::Quotient &k = L->quotient[dtype];
    if (k.S != S) {
        const QuotientPlan p = plan_quotient(S, dtype);
        k = Layer::Quotient{S, p.form, p.r_hi, p.r_lo};
    }
    return QuotientPlan{k.form, k.r_hi, k.r_lo};
}

// The masked path's quantizing kernel, static (DYN = false) or phase 1 of the dynamic mode.
template <int DTYPE, bool DYN>
static int launch_rows(Layer *L, const void *X, long long M, float S, int8_t *slab, unsigned *or_words, const StraddleJob &job, cudaStream_t st)
{
    constexpr int kBytes = DTYPE == FLEXIQ_DTYPE_F32 ? 4 : (DTYPE == FLEXIQ_DTYPE_I8 ? 1 : 2);
    const int n_c16 = L->C / 16, sms = device_sm_count(L->device);
    RowsArgs a{};
    a.X = X; a.slab = slab; a.M = M; a.K = L->C; a.G = L->G; a.K_lo = L->K_lo;
    a.S = S;
    a.quot = quotient_plan(L, S, DTYPE);
    a.perm = L->perm; a.sx = L->sx; a.or_words = or_words;
    a.wp = job;
    // Rows per tile and consumer warps: as many chunks as the block has threads, with the fewest threads idle; a row of
    // more than 256 chunks is a tile by itself.  Few rows: smaller tiles, so that they spread over the SMs (not in the
    // dynamic mode, whose blocks meet at the OR words).
    int warps = kRowWarps;
    a.rows = 1;
    if (n_c16 <= 32 * kRowWarps) {
        double best = 0.0;
        for (int w = kRowWarps; w >= 4; --w) {
            const int r = 32 * w / n_c16;
            const double used = (double)(r * n_c16) / (32 * w);
            if (used > best + 1e-9) { best = used; warps = w; a.rows = r; }
        }
        if (!DYN && (M + a.rows - 1) / a.rows < sms) {
            a.rows = (int)((M + sms - 1) / sms);
            warps = (a.rows * n_c16 + 31) / 32;
        }
    }
    a.tiles = (M + a.rows - 1) / a.rows;
    a.stage_bytes = (a.rows * L->C * kBytes + 127) & ~127;
    a.stages = kRowRing / a.stage_bytes;
    if (a.stages > kRowStages) a.stages = kRowStages;
    if (a.stages < 3) a.stages = 3;                   // wide rows: up to 192 KB, down to one block per SM
    size_t smem = (size_t)a.stages * a.stage_bytes + sizeof(unsigned) * (size_t)(n_c16 + (DYN ? L->n_g : 0));
    long long per_sm = (long long)(220 * 1024 / (smem + 1280));
    if (per_sm > 4) per_sm = 4;
    if (per_sm < 1) per_sm = 1;
    const long long blocks = a.tiles < sms * per_sm ? a.tiles : sms * per_sm;
    // Half a ring (14 MB over the machine): ViT-B sweep 701 -> 680 us, DeiT-S at batch 1 279 -> 276; 12 and 48 KB level.  None in the
    // dynamic mode, whose clear comes between: nothing overlaps, and its phase 1 was slower.
    if (!DYN) a.ahead = kRowRing / 2 / (a.rows * L->C * kBytes) > 1 ? kRowRing / 2 / (a.rows * L->C * kBytes) : 1;
    const int threads = 32 * (warps + 1);
    const unsigned extra = job.wst ? (unsigned)(((long long)job.rows * (job.BK >> 4) + threads - 1) / threads) : 0u;
    a.wp.first_block = extra;   // the straddle blocks come first
    // Spread evenly where the bytes decide (prologue + GEMM by graph replay: int8 2033 x 2704 18.4 -> 15.7 us, fp16 38,332 x 528 in front
    // of a 1x3 convolution 22.4 -> 20.0, fp32 14,843 x 832 16.9 -> 15.8, bf16 19,058 x 320 40.1 -> 38.8).  Below 8 MB a grid on few SMs is
    // the better neighbour: the GEMM behind it finds free SMs and has its preamble and first weights done by then (1536 x 768 9.1 us
    // crowded, 9.5 spread; int8 182 x 2224 10.2 and 10.8).
    if (M * L->C * (kBytes + 1) >= 8ll << 20) {
        const size_t even = even_share_smem(blocks, sms);
        if (smem < even) smem = even;
    }
    static bool attr_set[64] = {};   // per instantiation, whatever the size: the 48 KB default covers the static part too
    if (L->device >= 64 || !attr_set[L->device]) {
        FLEXIQ_CUDA_TRY(cudaFuncSetAttribute(quantize_rows_kernel<DTYPE, DYN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem));
        if (L->device < 64) attr_set[L->device] = true;
    }
    FLEXIQ_CUDA_TRY(launch_pdl(quantize_rows_kernel<DTYPE, DYN>, (unsigned)(blocks + extra), (unsigned)threads, smem, st, a));
    return FLEXIQ_OK;
}

// Does the one-launch dynamic kernel take M rows of this layer?  (rows per CTA, chunks per cluster)  The line lies where its columns'
// short pieces (a chunk of each row at a time, rows far apart) begin to cost more than the two phases' launches: at 9.7 MB of
// fp32, 1576 rows take 9.0 us against 12.4, 3152 10.5, 6304 12.1 and 12,608 17.9; 38.7 MB of fp16 in 6304 rows take 24, 77 MB 47 against 39.
static bool columns_fit(const Layer *L, long long M, int elem, int *rows, int *window)
{
    if (M > kColRows || M * L->C * elem > kColBytes) return false;
    *window = L->G == 64 ? 4 : 2;
    *rows = (int)((M + kColCluster - 1) / kColCluster);
    return true;
}

template <int DTYPE>
static int launch_columns(Layer *L, const void *X, long long M, float S, int8_t *slab, uint8_t *sx_out, const StraddleJob &job, int rows, int window, cudaStream_t st)
{
    ColumnsArgs a{};
    a.X = X; a.slab = slab; a.M = M; a.K = L->C; a.G = L->G; a.K_lo = L->K_lo;
    a.window = window; a.rows = rows;
    a.S = S;
    a.quot = quotient_plan(L, S, DTYPE);
    a.perm = L->perm; a.sx_out = sx_out;
    a.wp = job;
    long long extra = job.wst ? ((long long)job.rows * (job.BK >> 4) + kColThreads - 1) / kColThreads : 0;
    extra = (extra + kColCluster - 1) / kColCluster * kColCluster;   // whole clusters
    a.wp.first_block = (unsigned)extra;
    const long long ctas = (long long)((L->C / 16 + window - 1) / window) * kColCluster;
    size_t smem = (size_t)rows * window * 16;
    // Spread evenly where there are rows enough for it to matter and so few clusters that they would crowd onto a part of the machine
    // (clusters of eight find room on about 128 of the SMs): prologue + GEMM by graph replay, crowded and spread, fp32 6144 x 384
    // 26.2 -> 12.8 us, 3152 x 768 20.5 -> 16.2, fp16 6144 x 192 14.3 -> 11.3, 1576 x 384 9.2 -> 8.8.  With fewer rows, or three and more
    // CTAs per SM, the GEMM behind it gains more from the free SMs: 394 x 384 6.8 and 7.4, fp32 394 x 1536 8.6 and 10.7.
    if (M >= 1024 && ctas <= 2 * 128) {
        const size_t even = even_share_smem(ctas, 128);
        if (smem < even) smem = even;
    }
    static bool attr_set[64] = {};   // per instantiation, as above
    if (L->device >= 64 || !attr_set[L->device]) {
        FLEXIQ_CUDA_TRY(cudaFuncSetAttribute(dynamic_columns_kernel<DTYPE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kColSmem));
        if (L->device < 64) attr_set[L->device] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(extra + ctas), 1, 1);
    cfg.blockDim = dim3(kColThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kColCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    FLEXIQ_CUDA_TRY(cudaLaunchKernelEx(&cfg, dynamic_columns_kernel<DTYPE>, a));
    return FLEXIQ_OK;
}

template <int DTYPE>
static int launch_prologue(Layer *L, const void *X, long long M, float S, int dynamic, uint8_t *X4,
                           long long pitch, int8_t *X8, long long pitch8, uint8_t *sx_out, unsigned *scratch, cudaStream_t st)
{
    const int K = L->C, G = L->G;
    const int n_c16 = K / 16;
    const int sms = device_sm_count(L->device);
    const int threads = 256;
    const bool masked = L->lowbit_path == FLEXIQ_LOWBIT_MASKED_I8;
    constexpr size_t elem = DTYPE == FLEXIQ_DTYPE_F32 ? 4 : (DTYPE == FLEXIQ_DTYPE_I8 ? 1 : 2);
    int col_rows = 0, col_window = 0;
    const bool columns = dynamic && masked && columns_fit(L, M, (int)elem, &col_rows, &col_window);
    // a launch, not a memset: the kernel behind it may then start, and do all that comes before its wait, while the one before it ends
    if (dynamic && !columns) FLEXIQ_CUDA_TRY(launch_pdl(clear_words_kernel, 1, 256, 0, st, scratch, L->n_g));
    if (masked && (columns || (size_t)K * elem <= kRowStageBytes)) {
        StraddleJob job{};
        if (straddle_in_use(L) && straddle_stale(L, st)) {
            // the GEMM that consumes these slabs reads the straddle block of the same max_4bit_ch
            job.wst = L->wst; job.w8m = L->w8m; job.w8 = L->w8;
            job.rows = L->N * L->R * L->S;
            job.C = L->C;
            job.BK = choose_bk(L);
            job.blk0 = (L->K_lo / job.BK) * job.BK;
            job.K_lo = L->K_lo;
        }
        int8_t *slab = reinterpret_cast<int8_t *>(X4);
        int rc;
        if (columns) rc = launch_columns<DTYPE>(L, X, M, S, slab, sx_out, job, col_rows, col_window, st);
        else if (!dynamic) rc = launch_rows<DTYPE, false>(L, X, M, S, slab, nullptr, job, st);
        else {
            // the input is read once: phase 1 quantizes, gathers and collects the OR words, phase 2 lowers the low groups of
            // the slab in place (from L2) with the positions those words give
            if ((rc = launch_rows<DTYPE, true>(L, X, M, S, slab, scratch, StraddleJob{}, st))) return rc;
            const int lo_c16 = L->K_lo / 16;
            const long long want = (M * lo_c16 + 4 * threads - 1) / (4 * threads);
            long long blocks = want < (long long)sms * 8 ? want : (long long)sms * 8;
            if (blocks < 1) blocks = 1;   // the positions are written even when no group is low
            const long long extra = job.wst ? ((long long)job.rows * (job.BK >> 4) + threads - 1) / threads : 0;
            job.first_block = (unsigned)extra;
            FLEXIQ_CUDA_TRY(launch_pdl(lower_inplace_kernel, (unsigned)(blocks + extra), threads, 0, st, slab, M, K, G, L->K_lo,
                                       static_cast<const unsigned *>(scratch), sx_out, job, lo_c16 ? (int)(blocks * threads / lo_c16) : 0,
                                       lo_c16 ? (int)(blocks * threads % lo_c16) : 0));
        }
        if (rc) return rc;
        if (job.wst) straddle_written(L, st);
        record_slab(L, X4, L->K_lo);   // remember at which max_4bit_ch this buffer was written (the mixed_* calls check it)
        return FLEXIQ_OK;
    }
    if (dynamic) {
        long long want = (M * n_c16 + threads - 1) / threads;
        long long blocks = want < (long long)sms * 8 ? want : (long long)sms * 8;
        // thread count must cover at least one full row of chunks
        while (blocks * threads < n_c16) ++blocks;
        FLEXIQ_CUDA_TRY(launch_pdl(group_or_kernel<DTYPE>, (unsigned)blocks, threads, sizeof(unsigned) * L->n_g, st, X, M, K, G, S, L->perm, scratch));
    }
    const long long want = (M * n_c16 + threads - 1) / threads;
    const long long blocks = want < (long long)sms * 16 ? want : (long long)sms * 16;
    const uint8_t *sx = dynamic ? nullptr : L->sx;
    uint8_t *sx_to = dynamic ? sx_out : nullptr;
    if (masked)   // (the straddle block of so wide a layer is left to the GEMM, which writes it when it is stale)
        FLEXIQ_CUDA_TRY(launch_pdl(quantize_chunks_kernel<DTYPE, false>, (unsigned)blocks, threads, 0, st, X, M, K, G, L->K_lo, S, L->perm, sx, scratch, X4, pitch, X8, pitch8, sx_to));
    else
        FLEXIQ_CUDA_TRY(launch_pdl(quantize_chunks_kernel<DTYPE, true>, (unsigned)blocks, threads, 0, st, X, M, K, G, L->K_lo, S, L->perm, sx, scratch, X4, pitch, X8, pitch8, sx_to));
    if (masked || L->K_lo > 0) record_slab(L, X4, L->K_lo);
    if (!masked && L->K_lo < L->C) record_slab(L, X8, L->K_lo);
    return FLEXIQ_OK;
}

unsigned prologue_status()
{
    unsigned word = 0;
    const unsigned zero = 0;
    if (cudaMemcpyFromSymbol(&word, g_prologue_status, sizeof(word)) != cudaSuccess) return 0;   // the caller's own read reports it
    if (word) cudaMemcpyToSymbol(g_prologue_status, &zero, sizeof(zero));
    return word;
}

}  // namespace flexiq

using namespace flexiq;

extern "C" int flexiq_quantize_lower(flexiq_layer_t layer, const void *X_dev, int x_dtype, int64_t M, float x_scale,
                                     int dynamic_pos, uint8_t *X4_dev, int8_t *X8_dev, uint8_t *x_shift_out_dev,
                                     uint32_t *scratch_dev, void *stream)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    if (M < 0) return set_error(FLEXIQ_ERR_INVALID_ARG, "M = %lld is negative", (long long)M);
    if (x_dtype < FLEXIQ_DTYPE_F32 || x_dtype > FLEXIQ_DTYPE_I8)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "unknown x_dtype %d", x_dtype);
    if (x_dtype != FLEXIQ_DTYPE_I8 && !(x_scale > 0.0f))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "x_scale %g must be positive", (double)x_scale);
    if (M == 0) return FLEXIQ_OK;
    const int K_lo = L->K_lo, K_hi = L->C - K_lo;
    if (!X_dev) return set_error(FLEXIQ_ERR_INVALID_ARG, "X_dev is NULL");
    const bool packed = L->lowbit_path == FLEXIQ_LOWBIT_PACKED_U4;
    if (!packed && !X4_dev) return set_error(FLEXIQ_ERR_INVALID_ARG, "X4_dev is NULL: on the masked path it is the whole slab [M][K]");
    if (packed && K_lo > 0 && !X4_dev) return set_error(FLEXIQ_ERR_INVALID_ARG, "X4_dev is NULL but K_lo = %d", K_lo);
    if (packed && K_hi > 0 && !X8_dev) return set_error(FLEXIQ_ERR_INVALID_ARG, "X8_dev is NULL but K_hi = %d", K_hi);
    if (dynamic_pos && (!x_shift_out_dev || !scratch_dev))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "dynamic_pos needs x_shift_out_dev and scratch_dev");
    if ((reinterpret_cast<uintptr_t>(X_dev) | reinterpret_cast<uintptr_t>(X4_dev) | reinterpret_cast<uintptr_t>(X8_dev)) & 15)
        return set_error(FLEXIQ_ERR_INVALID_ARG, "X_dev, X4_dev and X8_dev must be 16-byte aligned");
    int rc = check_device_sm100();
    if (rc) return rc;
    if ((rc = check_layer_device(L))) return rc;
    int64_t pitch = 0;
    flexiq_x4_pitch(layer, K_lo, &pitch);
    // masked path: one slab, low groups first, the 8-bit groups behind them in the same rows
    long long pitch8 = K_hi;
    if (!packed) { X8_dev = reinterpret_cast<int8_t *>(X4_dev) + K_lo; pitch8 = L->C; }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    switch (x_dtype) {
        case FLEXIQ_DTYPE_F32: return launch_prologue<FLEXIQ_DTYPE_F32>(L, X_dev, M, x_scale, dynamic_pos, X4_dev, pitch, X8_dev, pitch8, x_shift_out_dev, scratch_dev, st);
        case FLEXIQ_DTYPE_F16: return launch_prologue<FLEXIQ_DTYPE_F16>(L, X_dev, M, x_scale, dynamic_pos, X4_dev, pitch, X8_dev, pitch8, x_shift_out_dev, scratch_dev, st);
        case FLEXIQ_DTYPE_BF16: return launch_prologue<FLEXIQ_DTYPE_BF16>(L, X_dev, M, x_scale, dynamic_pos, X4_dev, pitch, X8_dev, pitch8, x_shift_out_dev, scratch_dev, st);
        default: return launch_prologue<FLEXIQ_DTYPE_I8>(L, X_dev, M, x_scale, dynamic_pos, X4_dev, pitch, X8_dev, pitch8, x_shift_out_dev, scratch_dev, st);
    }
}

extern "C" int flexiq_quantize_lower_dynamic_noalloc(flexiq_layer_t layer, const void *X_dev, int x_dtype, int64_t M,
                                                     float x_scale, uint8_t *X4_dev, int8_t *X8_dev,
                                                     uint8_t *x_shift_out_dev, void *stream)
{
    Layer *L = as_layer(layer);
    if (!L) return set_error(FLEXIQ_ERR_INVALID_ARG, "not a live flexiq layer handle");
    if (L->n_g > kStaticScratchGroups)
        return set_error(FLEXIQ_ERR_INVALID_ARG,
                         "layer has %d channel groups; the built-in scratch of this entry point holds at most %d "
                         "(use flexiq_quantize_lower with caller-provided scratch instead)", L->n_g, kStaticScratchGroups);
    int rc = check_layer_device(L);   // the array's address is per device: look it up on the layer's
    if (rc) return rc;
    unsigned *scratch = nullptr;
    if ((rc = static_scratch_address(&scratch))) return rc;
    return flexiq_quantize_lower(layer, X_dev, x_dtype, M, x_scale, 1, X4_dev, X8_dev, x_shift_out_dev, scratch, stream);
}

extern "C" int flexiq_selftest_copy_drain(const uint8_t *src_dev, int *result_dev, void *stream)
{
    if (!src_dev || !result_dev || (reinterpret_cast<uintptr_t>(src_dev) & 15))
        return set_error(FLEXIQ_ERR_INVALID_ARG, "src_dev or result_dev is NULL, or src_dev is not 16-byte aligned");
    int rc = check_device_sm100();
    if (rc) return rc;
    drain_kernel<<<1, 32, 0, reinterpret_cast<cudaStream_t>(stream)>>>(src_dev, result_dev);
    FLEXIQ_CUDA_TRY(cudaGetLastError());
    return FLEXIQ_OK;
}
