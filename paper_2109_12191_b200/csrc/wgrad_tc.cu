// Per-example convolution weight gradients on the 5th-generation tensor cores (tcgen05 + TMEM),
// operands staged by TMA.  One (example, output tile) at a time per CTA, persistent CTAs.
//
// For example n the gradient is the matrix product  D_n = dY_n^T * Xcol_n  over the output pixels:
//     dY_n   [pixels, K_out]          (channels-last: K_out contiguous)
//     Xcol_n [pixels, R*S*C_in]       (column j = (r*S+s)*C_in + c is the input shifted by tap (r,s))
// Both operands have the reduction index (pixel) as the slow axis, i.e. they are "MN-major" for the
// tensor core.  A TMA box {64 channels, OWt, OHt, 1 example} lands in shared memory as OWt*OHt rows of
// 128 bytes with the 128-byte swizzle, which is exactly the canonical MN-major operand slab; the tap
// shift and the zero padding come from the box start coordinate and TMA's out-of-bounds zero fill.
//
// Roles (224 threads): warps 0 and 6 issue TMA loads (A and B slabs), warp 1 allocates TMEM and issues tcgen05.mma,
// warps 2-5 read accumulators back with tcgen05.ld, square-sum them (the per-example norm) and store.
// Two accumulator buffers in TMEM let the epilogue of one tile overlap the main loop of the next.
// Every wait is bounded: on expiry the CTA sets a status word, drains and returns.
//
// fp32 inputs: the tensor core truncates fp32 to tf32, which biases every norm by about 1e-3.  DP_TF32 lets the copies
// round to tf32 (nearest even) on the way in: TMA's TFLOAT32 element type does that for free, bit for bit like the warps
// that did it in shared memory before (2.4 us a stage).  DP_F32 runs as split tf32: eight more warps write lo = x - hi (hi = x with the low 13 mantissa bits cleared) of each landed
// stage into a second buffer of the same layout; x itself stays in place, where the tensor core's own truncation
// turns it into hi, and the issuer accumulates lo*hi + hi*lo + hi*hi per step.  What is dropped (lo*lo and the truncation of lo) is below 2^-20 relative.
#include "wgrad_tc.cuh"
#include "mbar.cuh"
#include <cuda.h>
#include <mutex>
#include <atomic>
#include <algorithm>
#include <array>
#include <map>
#include <memory>
#include <numeric>
#include <cmath>

namespace dp {

constexpr int kRowBytes = 128;         // one pixel's slab of channels: 64 bf16 or 32 fp32/tf32
constexpr int kMaxStages = 8;
constexpr int kSmemBudget = 200 * 1024;
constexpr int kBatchSmem = 176 * 1024;
constexpr uint32_t kWaitPolls = 1u << 21;   // x ~1 us suspend hint: about two seconds before a wait gives up
static std::atomic<uint32_t> g_wait_polls{kWaitPolls};
void set_wait_polls(uint32_t polls) { g_wait_polls.store(polls, std::memory_order_relaxed); }
uint32_t default_wait_polls() { return kWaitPolls; }
uint32_t wait_polls() { return g_wait_polls.load(std::memory_order_relaxed); }

struct TcPlan {
    bool ok;
    int a_is_x;                 // 1: rows of D are columns j of Xcol, columns of D are output channels k
    int a_ext, b_ext;           // operand extents in elements (multiples of the slab width)
    int m_tiles, n_tiles, NT;   // NT: nominal columns per tile (<= 256)
    int OWt, OHt, tiles_w, tiles_h, Kt, k_tiles;
    int stages, stage_bytes, a_bytes;
    size_t smem;
    double item_cycles;         // rough time of one (example, tile) item in its CTA
    int split;                  // modes 0 / 1: blocks that share an item's pixel tiles (conv_wgrad_split_kernel), 1: one does them all
};

struct TcParams {
    int B, Kout, Ng, Cin, S, stride, pad;   // Ng: row length of G in memory = number of real gradient columns
    int n_pad_cols;             // 1 when the column extent carries zero padding beyond Ng (im2col'd small-channel layers)
    int slab_ch;                // channels per 128-byte row: 64 (bf16) or 32 (fp32 as tf32)
    int krows;                  // reduction rows per MMA: 16 (bf16) or 8 (tf32)
    int a_is_x, a_ext, b_ext, m_tiles, n_tiles, NT;
    int OWt, OHt, tiles_w, Kt, k_tiles, stages, stage_bytes, a_bytes;
    int a_group, b_group;       // slabs of A / B that one copy brings (all of one filter tap)
    int lo_offset;              // split tf32: byte offset of the lo copy inside a stage
    int mode;                   // 0 store + norm, 1 norm only, 2 clipped sum over a range of examples
    float *G_w;
    float *partial;             // [B][slots], slot = (mt*n_tiles + nt)*4 + epilogue warp (split items: *split + block)
    int slots;
    int *status;
    uint32_t wait_polls;        // polls after which a wait gives up
    int total_tiles;            // work items: (example, tile) pairs, or (example range, tile) pairs in mode 2
    // mode 2: item = (split, tile); the CTA walks examples [split*per_split, ...) and keeps sum_n f_n D_n in registers
    int splits, per_split;
    const float *factor;        // [B][2], element 0 = weight factor
    float C_l;
    float *sqnorm; long long sq_stride; float *clip_out;
    float *sum_out;             // splits == 1: the accumulator (added to); else partial sums [splits][Kout*Ng]
    // modes 0 / 1 with a ticket: counters[0] counts the CTAs that are done (zero on entry, left at zero); the last
    // one folds every example's slots [0, w_slots) and [w_slots, slots) into sqnorm (two values when `separate`)
    int *counters; int w_slots; int separate;
    int fold_slots;             // slots that are folded (all of them, or the weights' only)
    float *factor_out;          // with the ticket: also the clip factors against C_l, [B][2] (weight, bias), and clip_out
    // space-to-depth form of a thin strided layer (s2d_st > 0): row j' of D is (r2, s2, dy, dx, c) of the regrouped
    // input and maps to column ((st*r2+dy)*s2d_S + st*s2d+dx)*s2d_Cin + c of the gradient, or to nothing
    int s2d_st, s2d_R, s2d_S, s2d_Cin;
    // which work items a block takes (norm / store / clipped-sum kernel): block b of `blocks` starts at b * run and takes
    // `run` items in a row, or with run == 0 every blocks-th item from b on
    int blocks, run;
    int cluster;                // single-pass kernel: blocks per cluster of the launch (>= tiles of one example)
};

// A launch serves up to N layers: the table of their tensor maps and parameters travels as a kernel parameter, and every
// block finds its layer by its index (first[] ascending).  N = 1 for a call on its own.
constexpr int kTcLayers = 54, kSsumLayers = 44;      // layers per grouped launch: a table stays below the 32 KB a launch may carry
constexpr int kFewLayers = 4;                        // small models: a table of 2 KB instead of 27, all of which every launch carries
template <typename P, int MAPS>
struct alignas(64) TcEntry { CUtensorMap map[MAPS]; P p; };
template <typename P, int MAPS, int N>
struct TcTable { int n; int first[N]; TcEntry<P, MAPS> e[N]; };

template <int N>
__device__ __forceinline__ int table_entry(const int (&first)[N], int n, int blk) {
    if (N == 1) return 0;
    const int lane = threadIdx.x & 31;
    const unsigned lo = __ballot_sync(0xffffffffu, lane < n && blk >= first[lane < N ? lane : 0]);
    const unsigned hi = __ballot_sync(0xffffffffu, lane + 32 < n && blk >= first[lane + 32 < N ? lane + 32 : 0]);
    return __popc(lo) + __popc(hi) - 1;
}

// column of the gradient that row j of the space-to-depth product stands for, or -1 (a tap or channel that does not exist)
__device__ __forceinline__ int s2d_column(const TcParams &p, int j) {
    const int r2 = j >> 6, s2 = (j >> 4) & 3, ch = j & 15;
    const int q = ch / p.s2d_Cin, c = ch - q * p.s2d_Cin;
    const int dy = q / p.s2d_st, dx = q - dy * p.s2d_st;
    const int r = p.s2d_st * r2 + dy, s = p.s2d_st * s2 + dx;
    return (dy < p.s2d_st && r < p.s2d_R && s < p.s2d_S) ? (r * p.s2d_S + s) * p.s2d_Cin + c : -1;
}

struct Item { int mt, nt, n_lo, n_hi, split; };
__device__ __forceinline__ Item decode_item(const TcParams &p, int item) {
    Item it;
    const int tpe = p.m_tiles * p.n_tiles;
    const int outer = item / tpe;          // the example, or in mode 2 the example range
    const int rem = item - outer * tpe;
    it.mt = rem / p.n_tiles;
    it.nt = rem - it.mt * p.n_tiles;
    if (p.mode == 2) { it.split = outer; it.n_lo = outer * p.per_split; it.n_hi = min(p.B, it.n_lo + p.per_split); }
    else { it.split = 0; it.n_lo = outer; it.n_hi = outer + 1; }
    return it;
}

// ----------------------------------------------------------------------------- PTX wrappers
// A box of an activation tensor seen as {slab of channels, W, H, B, slabs}: it lands slab after slab, each OWt*OHt rows of
// 128 bytes, so one copy brings all slabs of an operand that belong to one filter tap.
__device__ __forceinline__ void tma_load_slabs(uint32_t dst, const CUtensorMap *map, uint32_t bar, int w, int h, int n, int slab) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
                 ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(w), "r"(h), "r"(n), "r"(slab) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], fp32 accumulate, issued by one thread; TF32 selects kind::tf32 (fp32 inputs).
// The operand descriptors arrive as (low word, high word): only the low word (start address) changes from step to
// step, which keeps the issuing thread's work per instruction to one 32-bit add.
template <bool TF32>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                     uint32_t accumulate) {
    if (TF32)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                     "tcgen05.mma.cta_group::1.kind::tf32 [%0], da, db, %4, p;\n\t}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate) : "memory");
}
// Issue only: the registers hold the values after tmem_ld_wait32 on the same array.  Two loads in flight per thread
// hide most of the tensor-memory round trip (a load-then-wait per 32 columns left the epilogue warps idle).
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
// Waits for every tensor-memory load of this thread; the array rides along as in/out operands so that no use of its
// registers can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}

// Shared-memory operand descriptor without the start address, for MN-major slabs of 128-byte rows.
//   leading byte offset (between slabs) >> 4 at bit 16 | stride byte offset (between groups of reduction rows) >> 4
//   at bit 32 | descriptor version 1 at bit 46 | layout type at bit 61.
// 16-bit operands use the plain 128-byte swizzle (type 2: 16-byte chunks, pattern repeats every 8 rows = 1024 B).
// 32-bit (tf32) MN-major operands only exist with the 128-byte swizzle of 32-byte chunks (type 1: pattern
// repeats every 4 rows = 512 B); the tensor map then uses the matching SWIZZLE_128B_ATOM_32B mode.
template <bool TF32>
__device__ __forceinline__ uint64_t operand_desc_base(uint32_t slab_stride_bytes) {
    uint64_t d = (uint64_t)((slab_stride_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(((TF32 ? 512u : 1024u) >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(TF32 ? 1 : 2) << 61;
    return d;
}
// Instruction descriptor: fp32 accumulator, A and B of one type (bf16 = 1, tf32 = 2), both MN-major, M = 128, N = n_cols.
__device__ __forceinline__ uint32_t instr_desc(int n_cols, uint32_t fmt) {
    return (1u << 4) | (fmt << 7) | (fmt << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n_cols >> 3) << 17) | ((128u >> 4) << 24);
}

// How a finished block of D leaves: to per-example gradients nobody reads soon, to partial sums, or added to the
// accumulator.  Every element has one owner per launch, so an add needs no order; as a reduction at L2 it does not wait
// for the old value (reading it back row by row took longer than the tile's whole main loop).
enum { kPutStream = 0, kPutPlain, kPutAdd };
__device__ __forceinline__ void red_add(float *dst, float v) {
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(dst), "f"(v) : "memory");
}
template <int MODE>
__device__ __forceinline__ void put4(float *dst, const float4 v) {
    if (MODE == kPutStream) __stcs(reinterpret_cast<float4 *>(dst), v);
    else if (MODE == kPutPlain) *reinterpret_cast<float4 *>(dst) = v;
    else asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// A warp's 32 x 32 block, one row of 32 columns a lane, to 32 rows `ld` floats apart: through 4 KB of shared memory, so that
// eight lanes write 128 neighbouring bytes of one row (16 bytes a lane of 32 different rows ran at a fraction of the rate).
// The 16-byte pieces of a row are permuted by its number: both directions are free of bank conflicts.
template <int MODE, typename V>
__device__ __forceinline__ void put_rows(float4 *buf, const V &value, int lane, float *dst, long long ld, int rows) {
#pragma unroll
    for (int i = 0; i < 8; ++i) buf[lane * 8 + (i ^ (lane & 7))] = make_float4(value(4 * i), value(4 * i + 1), value(4 * i + 2), value(4 * i + 3));
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int row = 4 * i + (lane >> 3);
        const float4 v = buf[row * 8 + ((lane & 7) ^ (row & 7))];
        if (row < rows) put4<MODE>(dst + (long long)row * ld + 4 * (lane & 7), v);
    }
    __syncwarp();
}

// A thread's 32 values along the tile's columns where the block does not go through put_rows: columns of output channels
// (lanes write neighbouring words), or rows of a length that is no multiple of the vectors.
template <typename V>
__device__ __forceinline__ void put_values(const V &value, float *base, bool add, const TcParams &p, int a_idx, int b_idx) {
    const long long ld = p.Ng;
    if (p.a_is_x) {
        float *dst = base + b_idx * ld + a_idx;
        if (add) {
#pragma unroll
            for (int i = 0; i < 32; ++i) red_add(dst + i * ld, value(i));
        } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) dst[i * ld] = value(i);
        }
    } else {
        float *dst = base + a_idx * ld + b_idx;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (b_idx + i < p.Ng) { if (add) red_add(dst + i, value(i)); else dst[i] = value(i); }
    }
}

// slots first, first + 8, ... below end of an example's partial sums, in order, eight loads in flight
__device__ __forceinline__ double slot_sum(const float *slots, int first, int end) {
    double sum = 0.0;
    for (int i = first; i < end; i += 64) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { v[k] = 0.f; if (i + 8 * k < end) v[k] = __ldcg(slots + i + 8 * k); }
#pragma unroll
        for (int k = 0; k < 8; ++k) sum += (double)v[k];
    }
    return sum;
}

// What a producer warp copies for one operand of a tile: lane o holds the origin of copy o (`group` slabs of one tap).
// Issuing a copy costs the issuing warp about a hundred cycles and a barrier wait somewhat more, whatever the copy's size,
// so the fewer copies a stage takes, the smaller the stages (and the shorter their latency) can be.
struct OperandCopies {
    int count, slab, dw, dh, mul;
    uint32_t bytes;             // of one copy
    __device__ __forceinline__ OperandCopies(const TcParams &p, bool is_x, int slab0, int slabs, int group, int slab_bytes, int lane) {
        count = slabs / group;
        bytes = (uint32_t)(group * slab_bytes);
        slab = slab0 + lane * group; dw = 0; dh = 0; mul = 1;
        if (is_x) {
            const int j0 = slab * p.slab_ch;
            const int tap = j0 / p.Cin;
            slab = (j0 - tap * p.Cin) / p.slab_ch;
            const int r = tap / p.S;
            dw = (tap - r * p.S) - p.pad;
            dh = r - p.pad;
            mul = p.stride;
        }
    }
    // the whole warp calls; `leader` issues (origins travel by shuffle, so the copies' operands are uniform)
    __device__ __forceinline__ void issue(bool leader, const CUtensorMap *map, uint32_t dst, uint32_t bar, int ow0, int oh0, int n) const {
        for (int o = 0; o < count; ++o) {
            const int s = __shfl_sync(0xffffffffu, slab, o), w = __shfl_sync(0xffffffffu, dw, o), h = __shfl_sync(0xffffffffu, dh, o);
            if (leader) tma_load_slabs(dst + (uint32_t)o * bytes, map, bar, ow0 * mul + w, oh0 * mul + h, n, s);
            __syncwarp();
        }
    }
};

// The last block to finish: every example's partial squared norms, bias slots included, in slot order; publishes the squared norm(s)
// and, for a clipped-sum pass that follows, the factors.
__device__ __forceinline__ void publish_norms(const TcParams &p, int lane) {
    // eight lanes per example (slot i goes to lane i % 8, the eight sums are added by a butterfly), four
    // examples per warp and trip: the walk is a chain of L2 round trips, so many examples go side by side,
    // with eight loads of each in flight (one by one, 144 slots an example held the launch up for 2 us)
    const int groups = (int)(blockDim.x >> 3), group = (int)(threadIdx.x >> 3), sub = lane & 7;
    for (int n0 = 0; n0 < p.B; n0 += groups) {     // uniform trip count: the shuffles below need whole warps
        const int n = n0 + group;
        double sw = 0.0, sb = 0.0;
        if (n < p.B) {
            const float *pn = p.partial + (long long)n * p.slots;
            sw = slot_sum(pn, sub, p.w_slots);
            sb = slot_sum(pn, p.w_slots + sub, p.fold_slots);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            sw += __shfl_xor_sync(0xffffffffu, sw, o);
            sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
        if (n < p.B && sub == 0) {
            if (p.separate) { p.sqnorm[n * p.sq_stride] = (float)sw; p.sqnorm[n * p.sq_stride + 1] = (float)sb; }
            else p.sqnorm[n * p.sq_stride] = (float)(sw + sb);
            if (p.factor_out) {                    // the clipped-sum pass that follows reads its factors here
                const float fw = clip_factor(p.separate ? sw : sw + sb, p.C_l);
                const float fb = p.separate ? clip_factor(sb, p.C_l) : fw;
                p.factor_out[2 * n] = fw; p.factor_out[2 * n + 1] = fb;
                if (p.clip_out) {
                    if (p.separate) { p.clip_out[2 * n] = fw; p.clip_out[2 * n + 1] = fb; }
                    else p.clip_out[n] = fw;
                }
            }
        }
    }
}

enum { kBf16 = 0, kTf32, kSplit };       // inputs of the tensor cores: bf16, tf32, or fp32 as hi + lo tf32
// NORM: norms only, read back by eight warps instead of four (7-10 too): where an example has few pixels the read-back of a tile, a
// chain of loads from tensor memory and sums, is what the launch waits for.
template <int ARITH, bool CLIP, int N, bool NORM = false>
__global__ void __launch_bounds__(ARITH == kSplit ? 480 : (NORM ? 352 : 224), 1)
conv_wgrad_tc_kernel(const __grid_constant__ TcTable<TcParams, 2, N> tab) {
    constexpr bool TF32 = ARITH != kBf16, SPLIT = ARITH == kSplit;
    constexpr int READERS = NORM ? 8 : 4;
    const int entry = table_entry(tab.first, tab.n, blockIdx.x);
    const CUtensorMap &tmX = tab.e[entry].map[0], &tmY = tab.e[entry].map[1];
    const TcParams &p = tab.e[entry].p;
    const int blk = (int)blockIdx.x - tab.first[entry];
    const int item0 = p.run ? blk * p.run : blk, item_step = p.run ? 1 : p.blocks;
    const int item_end = p.run ? min(p.total_tiles, item0 + p.run) : p.total_tiles;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], ready_bar[kMaxStages], tmem_full[2], tmem_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ float4 xpose[NORM ? 1 : 4][NORM ? 1 : 256];      // per epilogue warp: a 32 x 32 block on its way out (put_rows)

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t tiles_u32 = smem_u32(tiles);

    if (threadIdx.x == 0) {
        // pull both tensor maps into the TMA descriptor cache before the first copy needs them
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmY)) : "memory");
        abort_flag = 0;
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 2); mbar_init(smem_u32(&empty_bar[s]), 1); mbar_init(smem_u32(&ready_bar[s]), 4);
        }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tmem_full[b]), 1); mbar_init(smem_u32(&tmem_empty[b]), READERS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int *abort_p = &abort_flag;

    const int slab_bytes = p.Kt * kRowBytes;
    const int a_slabs_tile = 128 / p.slab_ch, b_slabs_tile = p.NT / p.slab_ch;

    if (warp == 0 || warp == 6) {
        // ------------------------------------------------------------ TMA producers
        // Two warps, so that a stage's copies are issued side by side: warp 0 loads the A slabs of every
        // stage, warp 6 the B slabs; each announces its own bytes on the stage's full barrier (two arrivals).
        const bool leader = elect_one();
        int stage = 0; uint32_t phase = 0;
        bool live = true;
        for (int item = item0; item < item_end && live; item += item_step) {
            const Item it = decode_item(p, item);
            const int mt = it.mt, nt = it.nt;
            const int a_slab0 = mt * a_slabs_tile, a_slabs = min(a_slabs_tile, p.a_ext / p.slab_ch - a_slab0);
            const int b_slab0 = nt * b_slabs_tile, b_slabs = min(b_slabs_tile, p.b_ext / p.slab_ch - b_slab0);
            const bool is_a = warp == 0, is_x = is_a == (p.a_is_x != 0);
            const OperandCopies copies(p, is_x, is_a ? a_slab0 : b_slab0, is_a ? a_slabs : b_slabs, is_a ? p.a_group : p.b_group, slab_bytes, lane);
            const CUtensorMap *map = is_x ? &tmX : &tmY;
            const uint32_t dst = tiles_u32 + (is_a ? 0u : (uint32_t)p.a_bytes);
            const uint32_t tx_bytes = (uint32_t)copies.count * copies.bytes;
            for (int n = it.n_lo; n < it.n_hi && live; ++n) {
                int ow0 = 0, oh0 = 0, tw = 0;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                    if (leader) mbar_expect_tx(smem_u32(&full_bar[stage]), tx_bytes);
                    __syncwarp();
                    copies.issue(leader, map, dst + stage * p.stage_bytes, smem_u32(&full_bar[stage]), ow0, oh0, n);
                    if (++tw == p.tiles_w) { tw = 0; ow0 = 0; oh0 += p.OHt; } else { ow0 += p.OWt; }
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the warp walks together, one lane issues
        const bool leader = elect_one();
        int stage = 0; uint32_t phase = 0;
        uint32_t acc_phase = 0;  // bit b: phase of accumulator buffer b
        int buf = 0;
        bool live = true;
        const uint64_t desc_base = operand_desc_base<TF32>((uint32_t)slab_bytes);
        const uint32_t desc_lo = (uint32_t)desc_base, desc_hi32 = (uint32_t)(desc_base >> 32);
        const int ksteps = p.Kt / p.krows;
        constexpr uint32_t kadvance = (uint32_t)((TF32 ? 8 : 16) * kRowBytes) >> 4;   // start-address units of 16 B per MMA step
        for (int item = item0; item < item_end && live; item += item_step) {
            const Item it = decode_item(p, item);
            const int b_slabs = min(b_slabs_tile, p.b_ext / p.slab_ch - it.nt * b_slabs_tile);
            const uint32_t idesc = instr_desc(b_slabs * p.slab_ch, TF32 ? 2u : 1u);
            for (int n = it.n_lo; n < it.n_hi && live; ++n) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&tmem_empty[buf]), ((acc_phase >> buf) & 1u) ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
                uint32_t accumulate = 0;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(SPLIT ? &ready_bar[stage] : &full_bar[stage]), phase, abort_p, p.wait_polls))) { live = false; break; }
                    tc_fence_after();
                    const uint32_t a_src = tiles_u32 + stage * p.stage_bytes;
                    // descriptor low words: start address >> 4 in bits 0-13, slab stride >> 4 in bits 16-29
                    uint32_t ad = desc_lo | ((a_src & 0x3FFFFu) >> 4);
                    uint32_t bd = desc_lo | (((a_src + p.a_bytes) & 0x3FFFFu) >> 4);
                    // rows of the A tile past the operand's extent hold whatever the stage held before:
                    // they only feed rows of D that the epilogue never reads
                    if (leader) {
                        if (SPLIT) {
                            const uint32_t lo = (uint32_t)p.lo_offset >> 4;
#pragma unroll 2
                            for (int ks = 0; ks < ksteps; ++ks) {
                                umma<TF32>(d_tmem, ad + lo, bd, desc_hi32, idesc, accumulate);      // lo(A) * hi(B)
                                umma<TF32>(d_tmem, ad, bd + lo, desc_hi32, idesc, 1u);              // hi(A) * lo(B)
                                umma<TF32>(d_tmem, ad, bd, desc_hi32, idesc, 1u);                   // hi(A) * hi(B)
                                accumulate = 1;
                                ad += kadvance; bd += kadvance;
                            }
                        } else {
#pragma unroll 4
                            for (int ks = 0; ks < ksteps; ++ks) {
                                umma<TF32>(d_tmem, ad, bd, desc_hi32, idesc, accumulate);
                                accumulate = 1;
                                ad += kadvance; bd += kadvance;
                            }
                        }
                        umma_commit(smem_u32(&empty_bar[stage]));      // frees the stage once these MMAs have read it
                    }
                    accumulate = 1;
                    __syncwarp();
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
                if (!live) break;
                if (leader) umma_commit(smem_u32(&tmem_full[buf]));            // accumulator complete
                __syncwarp();
                acc_phase ^= 1u << buf;
                buf ^= 1;
            }
        }
    } else if (SPLIT && warp >= 7) {
        // ------------------------------------------------------------ split warps (fp32 inputs only)
        // hi stays where TMA put it, lo goes to the same offset of the stage's second half; both keep the
        // swizzled layout because the split is element-wise on identical relative addresses.
        // The eight warps work as two groups of four that take alternate stages, so the proxy fence that ends one
        // group's stage (it waits for that group's stores to drain) overlaps the other group's loads and stores.
        // The number of stages is even, so that a slot always belongs to the same group: a group that skipped every other
        // use of a slot could find the parity of the use before last and take a copy still under way for its own (stages
        // fill in any order), which with three stages left a launch in some thousands waiting in vain.
        const int group = (warp - 7) >> 2;
        const int tid = (threadIdx.x - 224) & 127;
        int stage = 0; uint32_t phase = 0;
        int turn = 0;                       // global stage counter modulo 2: whose stage is it
        bool live = true;
        for (int item = item0; item < item_end && live; item += item_step) {
            const Item it = decode_item(p, item);
            const int a_slabs = min(a_slabs_tile, p.a_ext / p.slab_ch - it.mt * a_slabs_tile);
            const int b_slabs = min(b_slabs_tile, p.b_ext / p.slab_ch - it.nt * b_slabs_tile);
            const int a_chunks = a_slabs * (slab_bytes >> 4), chunks = a_chunks + b_slabs * (slab_bytes >> 4);
            const int stage_count = (it.n_hi - it.n_lo) * p.k_tiles;
            for (int kt = 0; kt < stage_count; ++kt) {
                if (turn == group) {
                    const bool arrived = mbar_wait(smem_u32(&full_bar[stage]), phase, abort_p, p.wait_polls);
                    if (!__all_sync(0xffffffffu, arrived)) { live = false; break; }
                    uint8_t *base = tiles + (size_t)stage * p.stage_bytes;
                    // four 16-byte groups per thread and trip with all loads first, A region and B region in turn
                    for (int region = 0; region < 2; ++region) {
                        uint8_t *rbase = region ? base + p.a_bytes : base;
                        const int rchunks = region ? chunks - a_chunks : a_chunks;
                        for (int i0 = tid; i0 < rchunks; i0 += 512) {
                            float4 x[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                if (i0 + 128 * u < rchunks) x[u] = *reinterpret_cast<const float4 *>(rbase + ((size_t)(i0 + 128 * u) << 4));
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (i0 + 128 * u < rchunks) {
                                    uint8_t *ptr = rbase + ((size_t)(i0 + 128 * u) << 4);
                                    float4 hi, lo;
                                    hi.x = __uint_as_float(__float_as_uint(x[u].x) & 0xFFFFE000u); lo.x = x[u].x - hi.x;
                                    hi.y = __uint_as_float(__float_as_uint(x[u].y) & 0xFFFFE000u); lo.y = x[u].y - hi.y;
                                    hi.z = __uint_as_float(__float_as_uint(x[u].z) & 0xFFFFE000u); lo.z = x[u].z - hi.z;
                                    hi.w = __uint_as_float(__float_as_uint(x[u].w) & 0xFFFFE000u); lo.w = x[u].w - hi.w;
                                    *reinterpret_cast<float4 *>(ptr + p.lo_offset) = lo;     // x stays: truncated by the MMA itself, it is hi
                                }
                            }
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the tensor core
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ready_bar[stage]));
                }
                turn ^= 1;
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            }
        }
    } else if ((warp >= 2 && warp <= 5) || (NORM && warp >= 7)) {
        // ------------------------------------------------------------ epilogue (a TMEM lane quadrant to each warp, or to two)
        const int q = warp & 3, half = NORM && warp >= 7;
        const int row = q * 32 + lane;
        uint32_t full_phase = 0;     // bit b: parity to wait for on accumulator buffer b
        int buf = 0;
        bool live = true;
        for (int item = item0; item < item_end && live; item += item_step) {
            const Item it = decode_item(p, item);
            const int mt = it.mt, nt = it.nt;
            const int a_rows = min(128, p.a_ext - mt * 128);
            const int n_cols = min(p.NT, p.b_ext - nt * p.NT);
            int a_idx = mt * 128 + row;                  // index along the A operand's extent
            bool row_ok = row < a_rows && (!p.a_is_x || a_idx < p.Ng);
            if (!TF32 && p.s2d_st) {                     // (rows are input columns in this form)
                a_idx = row < a_rows ? s2d_column(p, a_idx) : -1;
                row_ok = a_idx >= 0;
            }
            float run[CLIP ? 128 : 1];                   // clip mode: this thread's row of sum_n f_n D_n (NT <= 128)
            if (CLIP) {
#pragma unroll
                for (int i = 0; i < 128; ++i) run[CLIP ? i : 0] = 0.f;
            }
            float f_lane = 0.f;     // clip mode, known factors: lane l holds the factor of example n_base + l
            int n_base = it.n_lo - 32;
            for (int n = it.n_lo; n < it.n_hi; ++n) {
                if (CLIP && n >= n_base + 32) {
                    n_base = n;
                    f_lane = (n + lane < it.n_hi) ? p.factor[2 * (n + lane)] : 0.f;    // one coalesced load per 32 examples
                }
                const bool arrived = mbar_wait(smem_u32(&tmem_full[buf]), (full_phase >> buf) & 1u, abort_p, p.wait_polls);
                if (!__all_sync(0xffffffffu, arrived)) { live = false; break; }   // the whole warp leaves together
                full_phase ^= 1u << buf;
                tc_fence_after();
                const uint32_t t_addr = tmem_base + (uint32_t)(buf * 256) + ((uint32_t)(q * 32) << 16);
                if (CLIP) {
                    const float f = __shfl_sync(0xffffffffu, f_lane, n - n_base);
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) {           // columns in pairs of 32: both loads in flight before the wait
                        if (c2 * 64 < n_cols) {
                            uint32_t v0[32], v1[32];
                            tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64), v0);
                            tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64 + 32), v1);     // (NT is a multiple of 64 here)
                            tmem_ld_wait32(v0); tmem_ld_wait32(v1);
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                run[CLIP ? c2 * 64 + i : 0] = fmaf(f, __uint_as_float(v0[i]), run[CLIP ? c2 * 64 + i : 0]);
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                run[CLIP ? c2 * 64 + 32 + i : 0] = fmaf(f, __uint_as_float(v1[i]), run[CLIP ? c2 * 64 + 32 + i : 0]);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
                } else {
                    float sq4[4] = {0.f, 0.f, 0.f, 0.f};      // four chains: one accumulator would serialise 256 dependent FMAs
                    float *Gn = p.G_w + (long long)n * p.Kout * p.Ng;
                    auto consume = [&](uint32_t (&v)[32], int cc) {
                        if (row_ok) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) { const float f = __uint_as_float(v[i]); sq4[i & 3] = fmaf(f, f, sq4[i & 3]); }
                            if (!NORM && p.mode == 0) {
                                const int b_idx = nt * p.NT + cc;
                                if (p.a_is_x) {      // row = column j of G, tile column = output channel k: lanes write consecutive j
                                    float *dst = Gn + (long long)b_idx * p.Ng + a_idx;
#pragma unroll
                                    for (int i = 0; i < 32; ++i) __stcs(dst + (long long)i * p.Ng, __uint_as_float(v[i]));
                                }
                            }
                        }
                        if (!NORM && p.mode == 0 && !p.a_is_x) {
                            // row = output channel k, tile columns = 32 consecutive j: each lane holds one row
                            const int col0 = nt * p.NT + cc, rows_here = min(32, a_rows - q * 32);
                            float *dst = Gn + (long long)(mt * 128 + q * 32) * p.Ng + col0;
                            if (!p.n_pad_cols) {
                                put_rows<kPutStream>(xpose[NORM ? 0 : warp - 2], [&](int i) { return __uint_as_float(v[i]); }, lane, dst, p.Ng, rows_here);
                            } else if (lane < rows_here) {           // rows of any length: element by element
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    if (col0 + i < p.Ng) dst[(long long)lane * p.Ng + i] = __uint_as_float(v[i]);
                            }
                        }
                    };
                    // columns in pairs of 32 with both loads in flight before the wait.  The second load of a tile with
                    // an odd number of 32-column blocks reads columns of this accumulator buffer that nobody uses.
                    for (int cc = 64 * half; cc < n_cols; cc += 64 * (READERS / 4)) {
                        uint32_t v0[32], v1[32];
                        tmem_ld32_issue(t_addr + (uint32_t)cc, v0);
                        tmem_ld32_issue(t_addr + (uint32_t)(cc + 32), v1);
                        tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                        consume(v0, cc);
                        if (cc + 32 < n_cols) consume(v1, cc + 32);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
                    const float sq = warp_sum((sq4[0] + sq4[1]) + (sq4[2] + sq4[3]));
                    if (lane == 0) p.partial[(long long)n * p.slots + (mt * p.n_tiles + nt) * READERS + half * 4 + q] = sq;
                }
                buf ^= 1;
            }
            if (!CLIP && p.counters && lane == 0 && item + item_step >= item_end)
                __threadfence();          // after this warp's last item: its partial sums are visible to the CTA that folds them
            if (CLIP && live) {
                // added to the accumulator, or left as a partial sum for the fold
                const bool add = p.splits == 1;
                float *base = p.sum_out + (add ? 0ll : (long long)it.split * p.Kout * p.Ng);
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {
                    if (c4 * 32 < n_cols) {
                        const int b_idx = nt * p.NT + c4 * 32;
                        auto value = [&](int i) { return run[CLIP ? c4 * 32 + i : 0]; };
                        if (!p.a_is_x && !p.n_pad_cols) {
                            float *dst = base + (long long)(mt * 128 + q * 32) * p.Ng + b_idx;
                            if (add) put_rows<kPutAdd>(xpose[NORM ? 0 : warp - 2], value, lane, dst, p.Ng, min(32, a_rows - q * 32));
                            else put_rows<kPutPlain>(xpose[NORM ? 0 : warp - 2], value, lane, dst, p.Ng, min(32, a_rows - q * 32));
                        } else if (row_ok) {
                            put_values(value, base, add, p, a_idx, b_idx);
                        }
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (!CLIP && p.counters && !abort_flag) {
        // The last CTA to finish (one ticket per CTA, nobody waits) folds every example's partial squared norms,
        // bias slots included, in slot order and publishes the squared norm(s): no finalising launch.
        __shared__ int last_cta;
        if (threadIdx.x == 0) {
            __threadfence();
            last_cta = atomicAdd(&p.counters[0], 1) == p.blocks - 1;
            if (last_cta) p.counters[0] = 0;
        }
        __syncthreads();
        if (last_cta) {
            __threadfence();
            publish_norms(p, lane);
        }
        __syncthreads();
    }
    if (abort_flag) {
        // give copies still in flight time to land before shared memory is released
        if (threadIdx.x == 0) { *p.status = DP_ERR_TIMEOUT; __threadfence(); }
        __nanosleep(200000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}


// ----------------------------------------------------------------------------- single-pass fused clip (bf16)
// Per-layer clipping needs an example's whole squared norm before any entry of its gradient can be scaled, so the
// kernel above runs every contraction twice (a norm pass, then the clipped sum).  Here each contraction runs once:
// a thread-block cluster owns ALL tiles of one example's gradient of this layer, one tile per CTA, kept in the CTA's
// tensor memory.  Every CTA square-sums its tile, the CTAs exchange their sums through distributed shared memory
// (one remote store per pair of CTAs that reports its bytes to the receiver's barrier; every CTA loads its own
// operands, nothing is multicast), every CTA then knows the example's norm and factor, scales its tile into a running
// sum held in registers, and moves on to the cluster's next example while the tensor core already fills the other
// accumulator buffer.  Clusters split the batch; with more than one cluster the running sums leave as partial sums,
// folded in cluster order by the launch that follows.  Given the factors beforehand (norms from the Gram-matrix kernel
// below) the same kernel runs without clusters and without the norm pass: one tile a CTA, any number of tiles.
//
// Roles (384 threads): warp 0 issues the TMA loads of the A slabs, warp 2 those of the B slabs, warp 1 allocates tensor
// memory and issues the MMAs, warp 3 idles; warps 4-11 are the epilogue: warp w reads TMEM lanes 32*(w%4).. and the
// 128-column half (w-4)/4 of the tile, so a thread holds 128 running sums.  The first warpgroup gives registers up
// (setmaxnreg) and the epilogue warpgroups take them: 128*56 + 256*224 = 384*168, the launch's allocation; beside normalisation
// layers 128*24 + 256*216 = 384*152, which leaves a warp of 56 registers a thread to each quarter of the SM (see affine_batch.cu)
// and keeps all but one value in registers (128*40 + 256*208 spilled ten values: 794 us a chunk of 32 ResNet-50 examples on
// the GPU that takes 786 this way).
constexpr int kClipThreads = 384;
template <bool BESIDE> struct ClipRegs {
    static constexpr int kLaunch = BESIDE ? 152 : 168, kControl = BESIDE ? 24 : 56, kEpilogue = BESIDE ? 216 : 224;
    static_assert(128 * kControl + 256 * kEpilogue == kClipThreads * kLaunch, "register split must add up");
};
constexpr int kMaxCluster = 8;
constexpr int kMaxExamplesPerCluster = 32;   // examples a cluster walks through when an SM target is set (calls run side by side)

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}
// one-way remote store that reports its bytes to a barrier of the receiving CTA (no separate arrival to release it)
__device__ __forceinline__ void st_async_f32(uint32_t cluster_addr, float v, uint32_t cluster_bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                 ::"r"(cluster_addr), "r"(__float_as_uint(v)), "r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
                 "selp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(1000u) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t polls) {
    for (uint32_t it = 0; it < polls; ++it) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if ((it & 63u) == 63u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// ----------------------------------------------------------------------------- pixels of an item shared by a cluster (bf16)
// Few examples of a layer with few tiles leave most SMs without an item, and a large plane keeps the others busy for long.  Here
// the blocks of a cluster share the pixel tiles of one (example, tile) item.  Their accumulators meet through shared memory:
// every block lays its tile out there (the stages are free by then), each takes an equal share of the gradient's rows (or of its
// columns, where the tile's rows are input columns) and adds that of all blocks in their order, squares and stores it.  What it
// costs is the tile's way through shared memory, some 2 us.  4 examples of 1 x 1 64 -> 64 on 50 x 50, stored: 14.6 us the call,
// 10.3 here; norms of 32 of the 7 x 7 stem on 224 x 224: 44 us, 35 on twice the SMs (its overlapping rows come from the L2 at
// 9 TB/s then, which bounds it).
// Roles until the accumulators are done: warp 0 / 6 TMA, warp 1 MMA, warps 2-5 read tensor memory; then all warps add up.
constexpr int kMaxSplit = 8, kSplitPad = 4;                 // floats between rows of a tile in shared memory: no bank conflicts
__global__ void __launch_bounds__(224, 1)
conv_wgrad_split_kernel(const __grid_constant__ TcTable<TcParams, 2, 1> tab) {
    const CUtensorMap &tmX = tab.e[0].map[0], &tmY = tab.e[0].map[1];
    const TcParams &p = tab.e[0].p;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], done_bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, last_cta;
    __shared__ float warp_sq[7];

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t tiles_u32 = smem_u32(tiles);
    const int rank = (int)cluster_rank(), split = p.splits;
    const Item it = decode_item(p, (int)blockIdx.x / split);
    const int mt = it.mt, nt = it.nt, n = it.n_lo;
    const int kt0 = (int)((long long)p.k_tiles * rank / split), kt1 = (int)((long long)p.k_tiles * (rank + 1) / split);

    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmY)) : "memory");
        abort_flag = 0;
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 2); mbar_init(smem_u32(&empty_bar[s]), 1); }
        mbar_init(smem_u32(&done_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int *abort_p = &abort_flag;

    const int slab_bytes = p.Kt * kRowBytes;
    const int a_slabs = min(128 / p.slab_ch, p.a_ext / p.slab_ch - mt * (128 / p.slab_ch));
    const int b_slabs = min(p.NT / p.slab_ch, p.b_ext / p.slab_ch - nt * (p.NT / p.slab_ch));
    const int a_rows = min(128, p.a_ext - mt * 128), n_cols = b_slabs * p.slab_ch;
    // the tile in shared memory: lines that are contiguous in the gradient, rows of it or (input columns as rows) its columns
    float *tile = reinterpret_cast<float *>(tiles);
    const int lines = p.a_is_x ? n_cols : a_rows, width = p.a_is_x ? 128 : n_cols, pitch = width + kSplitPad;

    if (warp == 0 || warp == 6) {
        const bool leader = elect_one(), is_a = warp == 0, is_x = is_a == (p.a_is_x != 0);
        const OperandCopies copies(p, is_x, is_a ? mt * (128 / p.slab_ch) : nt * (p.NT / p.slab_ch), is_a ? a_slabs : b_slabs,
                                   is_a ? p.a_group : p.b_group, slab_bytes, lane);
        const CUtensorMap *map = is_x ? &tmX : &tmY;
        const uint32_t dst = tiles_u32 + (is_a ? 0u : (uint32_t)p.a_bytes), tx_bytes = (uint32_t)copies.count * copies.bytes;
        int stage = 0; uint32_t phase = 0;
        int tw = kt0 % p.tiles_w, ow0 = tw * p.OWt, oh0 = kt0 / p.tiles_w * p.OHt;
        for (int kt = kt0; kt < kt1; ++kt) {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, abort_p, p.wait_polls))) break;
            if (leader) mbar_expect_tx(smem_u32(&full_bar[stage]), tx_bytes);
            __syncwarp();
            copies.issue(leader, map, dst + stage * p.stage_bytes, smem_u32(&full_bar[stage]), ow0, oh0, n);
            if (++tw == p.tiles_w) { tw = 0; ow0 = 0; oh0 += p.OHt; } else { ow0 += p.OWt; }
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        const uint64_t desc_base = operand_desc_base<false>((uint32_t)slab_bytes);
        const uint32_t desc_lo = (uint32_t)desc_base, desc_hi32 = (uint32_t)(desc_base >> 32);
        const int ksteps = p.Kt / p.krows;
        constexpr uint32_t kadvance = (uint32_t)(16 * kRowBytes) >> 4;
        const uint32_t idesc = instr_desc(n_cols, 1u);
        int stage = 0; uint32_t phase = 0, accumulate = 0;
        bool live = true;
        for (int kt = kt0; kt < kt1; ++kt) {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[stage]), phase, abort_p, p.wait_polls))) { live = false; break; }
            tc_fence_after();
            const uint32_t a_src = tiles_u32 + stage * p.stage_bytes;
            uint32_t ad = desc_lo | ((a_src & 0x3FFFFu) >> 4), bd = desc_lo | (((a_src + p.a_bytes) & 0x3FFFFu) >> 4);
            if (leader) {
#pragma unroll 4
                for (int ks = 0; ks < ksteps; ++ks) {
                    umma<false>(tmem_base, ad, bd, desc_hi32, idesc, accumulate);
                    accumulate = 1;
                    ad += kadvance; bd += kadvance;
                }
                umma_commit(smem_u32(&empty_bar[stage]));
            }
            accumulate = 1;
            __syncwarp();
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
        if (live && leader) umma_commit(smem_u32(&done_bar));
        __syncwarp();
    } else {
        const int q = warp & 3, row = q * 32 + lane;
        // (the last MMA has read its stage: nothing else is left in the stages, whose place the tile takes)
        if (__all_sync(0xffffffffu, mbar_wait(smem_u32(&done_bar), 0u, abort_p, p.wait_polls))) {
            tc_fence_after();
            const uint32_t t_addr = tmem_base + ((uint32_t)(q * 32) << 16);
            for (int cc = 0; cc < n_cols; cc += 64) {                                    // (a multiple of 64)
                uint32_t v0[32], v1[32];
                tmem_ld32_issue(t_addr + (uint32_t)cc, v0);
                tmem_ld32_issue(t_addr + (uint32_t)(cc + 32), v1);
                tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                if (p.a_is_x) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) { tile[(cc + i) * pitch + row] = __uint_as_float(v0[i]); tile[(cc + 32 + i) * pitch + row] = __uint_as_float(v1[i]); }
                } else if (row < a_rows) {
                    float4 *dst = reinterpret_cast<float4 *>(tile + row * pitch + cc);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        dst[i] = make_float4(__uint_as_float(v0[4 * i]), __uint_as_float(v0[4 * i + 1]), __uint_as_float(v0[4 * i + 2]), __uint_as_float(v0[4 * i + 3]));
                        dst[8 + i] = make_float4(__uint_as_float(v1[4 * i]), __uint_as_float(v1[4 * i + 1]), __uint_as_float(v1[4 * i + 2]), __uint_as_float(v1[4 * i + 3]));
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    // A block whose wait gave up has no tile to add: the whole cluster leaves its share of the gradient alone and NaN for a norm.
    if (*abort_p && (int)threadIdx.x < split) asm volatile("st.shared::cluster.u32 [%0], 1;" ::"r"(map_to_cta(smem_u32(&abort_flag), threadIdx.x)) : "memory");
    __syncwarp();
    cluster_sync_all();                                   // every block's tile is in place
    const bool failed = *abort_p != 0;                    // here or in a peer

    // this block's share of the lines, of all blocks in their order; a thread takes four neighbouring values of a line
    const int line0 = lines * rank / split, line1 = lines * (rank + 1) / split, quads = width / 4;
    uint32_t peer[kMaxSplit];
#pragma unroll
    for (int r = 0; r < kMaxSplit; ++r) peer[r] = map_to_cta(tiles_u32, (uint32_t)min(r, split - 1));
    float sq4[4] = {0.f, 0.f, 0.f, 0.f};
    float *Gn = p.G_w + (long long)n * p.Kout * p.Ng;
    for (int e = threadIdx.x; !failed && e < (line1 - line0) * quads; e += 224) {
        const int line = line0 + e / quads, x = (e % quads) * 4;
        const uint32_t off = (uint32_t)(line * pitch + x) * 4u;
        float4 v[kMaxSplit];
#pragma unroll
        for (int r = 0; r < kMaxSplit; ++r)
            if (r < split)
                asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[r].x), "=f"(v[r].y), "=f"(v[r].z), "=f"(v[r].w) : "r"(peer[r] + off));
        float a[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
        for (int r = 1; r < kMaxSplit; ++r)
            if (r < split) { a[0] += v[r].x; a[1] += v[r].y; a[2] += v[r].z; a[3] += v[r].w; }
        // where the four values lie in the gradient; those that stand for nothing count for nothing
        const long long row0 = p.a_is_x ? nt * p.NT + line : mt * 128 + line;
        const int col0 = (p.a_is_x ? mt * 128 : nt * p.NT) + x;
        const bool whole = !p.s2d_st && col0 + 4 <= p.Ng && (!p.a_is_x || x + 4 <= a_rows);
        if (whole && !p.n_pad_cols) {
#pragma unroll
            for (int i = 0; i < 4; ++i) sq4[i] = fmaf(a[i], a[i], sq4[i]);
            if (p.mode == 0) __stcs(reinterpret_cast<float4 *>(Gn + row0 * p.Ng + col0), make_float4(a[0], a[1], a[2], a[3]));
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int col = col0 + i;
                if (p.a_is_x && x + i >= a_rows) col = -1;
                else if (p.s2d_st) col = s2d_column(p, col);
                if (col < 0 || col >= p.Ng) continue;
                sq4[i] = fmaf(a[i], a[i], sq4[i]);
                if (p.mode == 0) Gn[row0 * p.Ng + col] = a[i];
            }
        }
    }
    const float sq = warp_sum((sq4[0] + sq4[1]) + (sq4[2] + sq4[3]));
    if (lane == 0) warp_sq[warp] = failed ? __int_as_float(0x7fffffff) : sq;
    __syncthreads();
    cluster_sync_all();                                   // nobody leaves while a peer may still read its tile
    if (threadIdx.x == 0) {
        p.partial[(long long)n * p.slots + (mt * p.n_tiles + nt) * split + rank] =
            ((warp_sq[0] + warp_sq[1]) + (warp_sq[2] + warp_sq[3])) + ((warp_sq[4] + warp_sq[5]) + warp_sq[6]);
        __threadfence();
        last_cta = atomicAdd(&p.counters[0], 1) == p.blocks - 1;
        if (last_cta) p.counters[0] = 0;
    }
    __syncthreads();
    if (last_cta) { __threadfence(); publish_norms(p, lane); }
    __syncthreads();
    if (abort_flag) {
        if (threadIdx.x == 0) { *p.status = DP_ERR_TIMEOUT; __threadfence(); }
        __nanosleep(200000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 256); }
}

// sum of non-negative floats with its rounding errors; past the range of float it is infinite, as in plain floats
__device__ __forceinline__ float sum8(const float4 &x, const float4 &y) {
    float e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;
    const float a = two_sum(x.x, x.y, e0), b = two_sum(x.z, x.w, e1), c = two_sum(y.x, y.y, e2), d = two_sum(y.z, y.w, e3);
    const float ab = two_sum(a, b, e0), cd = two_sum(c, d, e2);
    const float s = two_sum(ab, cd, e0);
    return s <= kFloatMax ? s + ((e0 + e1) + (e2 + e3)) : s;
}

template <int N, bool BESIDE = false>
__global__ void __maxnreg__(ClipRegs<BESIDE>::kLaunch)
conv_wgrad_clip1_kernel(const __grid_constant__ TcTable<TcParams, 2, N> tab) {
    const int entry = table_entry(tab.first, tab.n, blockIdx.x);
    const CUtensorMap &tmX = tab.e[entry].map[0], &tmY = tab.e[entry].map[1];
    const TcParams &p = tab.e[entry].p;
    const int blk = (int)blockIdx.x - tab.first[entry];
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tmem_full[2], tmem_empty[2], norm_bar[4], warp_bar[4];
    __shared__ float warp_part[4][8];                   // [example mod 4][epilogue warp]: this CTA's partial sums
    __shared__ __align__(16) float norm_part[4][kMaxCluster];         // [example mod 4][source CTA]: every CTA's sum, sent by its first epilogue warp
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t tiles_u32 = smem_u32(tiles);
    const int cs = p.m_tiles * p.n_tiles;                 // cluster size = tiles of one example's gradient
    // With the factors known beforehand (p.factor) nothing is exchanged: the launch has no clusters and any number of tiles
    const bool known = p.factor != nullptr;
    // A cluster of the launch may hold several examples' sets of tiles (layers of different sizes share a launch): blocks
    // [set * cs, set * cs + cs) of it are one set; blocks left over, and sets past the last example range, have no work.
    const int sets = p.cluster / cs, crank = known ? 0 : (int)cluster_rank(), set = crank / cs;
    const int rank = known ? blk % cs : crank - set * cs;
    const int mt = rank / p.n_tiles, nt = rank - mt * p.n_tiles;
    const int split = known ? blk / cs : (set < sets ? blk / p.cluster * sets + set : p.splits);
    const int n_lo = min(p.B, split * p.per_split), n_hi = min(p.B, n_lo + p.per_split);

    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmY)) : "memory");
        abort_flag = 0;
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 2); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tmem_full[b]), 1); mbar_init(smem_u32(&tmem_empty[b]), 8); }
        for (int b = 0; b < 4; ++b) { mbar_init(smem_u32(&norm_bar[b]), 1); mbar_init(smem_u32(&warp_bar[b]), 8); }
        for (int i = 0; i < 4 * kMaxCluster; ++i) norm_part[0][i] = 0.f;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                   // every CTA's barriers exist before anyone arrives on them
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int *abort_p = &abort_flag;

    const int slab_bytes = p.Kt * kRowBytes;
    const int a_slabs_tile = 128 / p.slab_ch, b_slabs_tile = p.NT / p.slab_ch;
    const int a_slabs = min(a_slabs_tile, p.a_ext / p.slab_ch - mt * a_slabs_tile);
    const int b_slabs = min(b_slabs_tile, p.b_ext / p.slab_ch - nt * b_slabs_tile);

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(ClipRegs<BESIDE>::kControl));
        if (warp == 0 || warp == 2) {
            // ------------------------------------------------------------ TMA producers (A slabs / B slabs)
            const bool leader = elect_one();
            const bool is_a = warp == 0, is_x = is_a == (p.a_is_x != 0);
            const OperandCopies copies(p, is_x, is_a ? mt * a_slabs_tile : nt * b_slabs_tile, is_a ? a_slabs : b_slabs,
                                       is_a ? p.a_group : p.b_group, slab_bytes, lane);
            const CUtensorMap *map = is_x ? &tmX : &tmY;
            const uint32_t dst = tiles_u32 + (is_a ? 0u : (uint32_t)p.a_bytes);
            const uint32_t tx_bytes = (uint32_t)copies.count * copies.bytes;
            const int stages = p.stages, stage_bytes = p.stage_bytes, k_tiles = p.k_tiles, tiles_w = p.tiles_w, OWt = p.OWt, OHt = p.OHt;
            int stage = 0; uint32_t phase = 0;
            bool live = true;
            for (int n = n_lo; n < n_hi && live; ++n) {
                int ow0 = 0, oh0 = 0, tw = 0;
                for (int kt = 0; kt < k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                    if (leader) mbar_expect_tx(smem_u32(&full_bar[stage]), tx_bytes);
                    __syncwarp();
                    copies.issue(leader, map, dst + stage * stage_bytes, smem_u32(&full_bar[stage]), ow0, oh0, n);
                    if (++tw == tiles_w) { tw = 0; ow0 = 0; oh0 += OHt; } else { ow0 += OWt; }
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------ MMA issuer: the warp walks together, one lane issues
            const bool leader = elect_one();
            int stage = 0; uint32_t phase = 0, acc_phase = 0;
            int buf = 0;
            bool live = true;
            const uint64_t desc_base = operand_desc_base<false>((uint32_t)slab_bytes);
            const uint32_t desc_lo = (uint32_t)desc_base, desc_hi32 = (uint32_t)(desc_base >> 32);
            const int ksteps = p.Kt / p.krows, k_tiles = p.k_tiles, stages = p.stages, stage_bytes = p.stage_bytes, a_bytes = p.a_bytes;
            constexpr uint32_t kadvance = (uint32_t)(16 * kRowBytes) >> 4;
            const uint32_t idesc = instr_desc(b_slabs * p.slab_ch, 1u);
            for (int n = n_lo; n < n_hi && live; ++n) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&tmem_empty[buf]), ((acc_phase >> buf) & 1u) ^ 1u, abort_p, p.wait_polls))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
                uint32_t accumulate = 0;
                for (int kt = 0; kt < k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[stage]), phase, abort_p, p.wait_polls))) { live = false; break; }
                    tc_fence_after();
                    const uint32_t a_src = tiles_u32 + stage * stage_bytes;
                    uint32_t ad = desc_lo | ((a_src & 0x3FFFFu) >> 4);
                    uint32_t bd = desc_lo | (((a_src + a_bytes) & 0x3FFFFu) >> 4);
                    if (leader) {
#pragma unroll 4
                        for (int ks = 0; ks < ksteps; ++ks) {
                            umma<false>(d_tmem, ad, bd, desc_hi32, idesc, accumulate);
                            accumulate = 1;
                            ad += kadvance; bd += kadvance;
                        }
                        umma_commit(smem_u32(&empty_bar[stage]));
                    }
                    accumulate = 1;
                    __syncwarp();
                    if (++stage == stages) { stage = 0; phase ^= 1u; }
                }
                if (!live) break;
                if (leader) umma_commit(smem_u32(&tmem_full[buf]));
                __syncwarp();
                acc_phase ^= 1u << buf;
                buf ^= 1;
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(ClipRegs<BESIDE>::kEpilogue));
        // ---------------------------------------------------------------- epilogue (8 warps)
        const int e = warp - 4, q = e & 3, half = e >> 2;
        const int row = q * 32 + lane;
        const int a_rows = min(128, p.a_ext - mt * 128);
        const int n_cols = min(p.NT, p.b_ext - nt * p.NT);
        const int my_cols = max(0, min(128, n_cols - half * 128));     // columns of this warp's half that exist
        int a_idx = mt * 128 + row;
        bool row_ok = row < a_rows && (!p.a_is_x || a_idx < p.Ng);
        if (p.s2d_st) {                                    // (rows are input columns in this form)
            a_idx = row < a_rows ? s2d_column(p, a_idx) : -1;
            row_ok = a_idx >= 0;
        }
        float run[128];
#pragma unroll
        for (int i = 0; i < 128; ++i) run[i] = 0.f;
        bool live = true;
        // One step behind, with two tiles of tensor memory: step s first finishes example s - 1 (waits for its partial sums
        // from the whole cluster, scales its tile into the running sum and hands the tile's columns back to the MMA warp,
        // which starts on example s + 1), then square-sums example s and sends its partial sums on their way.
        // Slots and barriers of the exchange come in fours: a slot of example j is overwritten by example j + 4, which a
        // warp sends only after it has scaled example j + 3, i.e. after every warp of the cluster has sent example
        // j + 3, which each of them did after scaling (and so after reading the slots of) example j + 2 and before it j.
        const int count = n_hi - n_lo;
        const float threshold = __double2float_rd((double)p.C_l * (double)p.C_l);
        for (int step = 0; known && step < count && live; ++step) {
            // factors known: one read of the finished tile per example, scaled into the running sum
            const int buf = step & 1;
            const bool arrived = mbar_wait(smem_u32(&tmem_full[buf]), (uint32_t)((step >> 1) & 1), abort_p, p.wait_polls);
            if (!__all_sync(0xffffffffu, arrived)) { live = false; break; }
            tc_fence_after();
            const float f = __ldg(p.factor + 2 * (n_lo + step));
            const uint32_t t_addr = tmem_base + (uint32_t)(buf * 256 + half * 128) + ((uint32_t)(q * 32) << 16);
#pragma unroll
            for (int c2 = 0; c2 < 2; ++c2) {
                if (c2 * 64 < my_cols) {
                    uint32_t v0[32], v1[32];
                    tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64), v0);
                    tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64 + 32), v1);
                    tmem_ld_wait32(v0); tmem_ld_wait32(v1);
#pragma unroll
                    for (int i = 0; i < 32; ++i) run[c2 * 64 + i] = fmaf(f, __uint_as_float(v0[i]), run[c2 * 64 + i]);
#pragma unroll
                    for (int i = 0; i < 32; ++i) run[c2 * 64 + 32 + i] = fmaf(f, __uint_as_float(v1[i]), run[c2 * 64 + 32 + i]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
        }
        for (int step = 0; !known && step <= count && live; ++step) {
            if (step >= 1) {
                // finish example step - 1 first: its tile leaves tensor memory before this step's tile is touched, so the
                // MMAs of the example after this one run while this step's tile is being square-summed
                const int j = step - 1, n = n_lo + j, buf = j & 1, slot = j & 3;
                // half of the tile is on its way to registers while the norm is still being exchanged
                const uint32_t t_addr = tmem_base + (uint32_t)(buf * 256 + half * 128) + ((uint32_t)(q * 32) << 16);
                uint32_t v0[32], v1[32];
                tmem_ld32_issue(t_addr, v0);
                tmem_ld32_issue(t_addr + 32u, v1);
                const bool all_in = mbar_wait_cluster(smem_u32(&norm_bar[slot]), (uint32_t)((j >> 2) & 1), abort_p, p.wait_polls);
                // the same tree in every thread of every CTA (slots past the cluster's size hold zeros): all of them apply
                // the identical factor.  The sum carries its rounding errors along (as good as double, whose pipe is so
                // narrow that the same tree takes it some 800 cycles on the path every example waits on); the factor
                // min(1, C_l / sqrt(sn)) is in single precision.
                const float4 lo = *reinterpret_cast<const float4 *>(norm_part[slot]), hi = *reinterpret_cast<const float4 *>(norm_part[slot] + 4);
                const float sn = sum8(lo, hi);
                float f = (sn <= threshold) ? 1.0f : p.C_l * rsqrtf(sn);
                if (sn > kFloatMax) {                      // nothing is left of the example unless C_l is as large
                    const double s = (((double)lo.x + (double)lo.y) + ((double)lo.z + (double)lo.w)) +
                                     (((double)hi.x + (double)hi.y) + ((double)hi.z + (double)hi.w));
                    f = s <= (double)p.C_l * (double)p.C_l ? 1.0f : 0.0f;
                }
                tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                if (!__all_sync(0xffffffffu, all_in)) { live = false; break; }
                if (rank == 0 && e == 0 && lane == 0) {
                    p.sqnorm[n * p.sq_stride] = sn;
                    if (p.clip_out) p.clip_out[n] = f;
                }
                // pass 2: scale the tile into the running sum
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {
                    if (c2 * 64 < my_cols) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) run[c2 * 64 + i] = fmaf(f, __uint_as_float(v0[i]), run[c2 * 64 + i]);
                        if (c2 == 0 && my_cols > 64) tmem_ld32_issue(t_addr + 64u, v0);
#pragma unroll
                        for (int i = 0; i < 32; ++i) run[c2 * 64 + 32 + i] = fmaf(f, __uint_as_float(v1[i]), run[c2 * 64 + 32 + i]);
                        if (c2 == 0 && my_cols > 64) {
                            tmem_ld32_issue(t_addr + 96u, v1);
                            tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
            }
            if (step < count) {
                const int buf = step & 1, slot = step & 3;
                const bool arrived = mbar_wait(smem_u32(&tmem_full[buf]), (uint32_t)((step >> 1) & 1), abort_p, p.wait_polls);
                if (!__all_sync(0xffffffffu, arrived)) { live = false; break; }
                tc_fence_after();
                const uint32_t t_addr = tmem_base + (uint32_t)(buf * 256 + half * 128) + ((uint32_t)(q * 32) << 16);
                // pass 1: this warp's share of the example's squared norm
                float sq4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2) {           // columns in pairs of 32, both loads in flight before the wait
                    if (c2 * 64 < my_cols) {                // (my_cols is a multiple of 64)
                        uint32_t v0[32], v1[32];
                        tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64), v0);
                        tmem_ld32_issue(t_addr + (uint32_t)(c2 * 64 + 32), v1);
                        tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                        if (row_ok) {      // (columns past the real ones of an unfolded thin layer hold exact zeros)
#pragma unroll
                            for (int i = 0; i < 32; ++i) { const float f = __uint_as_float(v0[i]); sq4[i & 3] = fmaf(f, f, sq4[i & 3]); }
#pragma unroll
                            for (int i = 0; i < 32; ++i) { const float f = __uint_as_float(v1[i]); sq4[i & 3] = fmaf(f, f, sq4[i & 3]); }
                        }
                    }
                }
                const float sq = warp_sum((sq4[0] + sq4[1]) + (sq4[2] + sq4[3]));
                // The CTA's eight partial sums meet in its own shared memory first; its first epilogue warp adds them and
                // tells the cluster: lane r sends the sum to CTA r with a store that reports its bytes to that CTA's barrier
                // (one way; a plain remote store followed by a releasing remote arrival costs a round trip more).
                if (lane == 0) { warp_part[slot][e] = sq; mbar_arrive(smem_u32(&warp_bar[slot])); }
                if (e == 0) {
                    const bool mine_in = mbar_wait(smem_u32(&warp_bar[slot]), (uint32_t)((step >> 2) & 1), abort_p, p.wait_polls);
                    if (!__all_sync(0xffffffffu, mine_in)) { live = false; break; }
                    const float *w = warp_part[slot];
                    const float cta_sq = ((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]));
                    // this CTA expects one float from every CTA of the cluster (its own included) in this slot's phase
                    if (lane == 0) mbar_expect_tx(smem_u32(&norm_bar[slot]), (uint32_t)(cs * 4));
                    if (lane < cs)
                        st_async_f32(map_to_cta(smem_u32(&norm_part[slot][rank]), (uint32_t)(set * cs + lane)), cta_sq,
                                     map_to_cta(smem_u32(&norm_bar[slot]), (uint32_t)(set * cs + lane)));
                }
            }
        }
        if (live && split < p.splits) {
            // added to the accumulator, or left as a partial sum for the fold; every tile has been read, so the stages'
            // memory is free to carry the blocks out
            const bool add = p.splits == 1;
            float *base = p.sum_out + (add ? 0ll : (long long)split * p.Kout * p.Ng);
            float4 *buf = reinterpret_cast<float4 *>(tiles) + e * 256;
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4) {
                if (c4 * 32 < my_cols) {
                    const int b_idx = nt * p.NT + half * 128 + c4 * 32;
                    auto value = [&](int i) { return run[c4 * 32 + i]; };
                    if (!p.a_is_x && !p.n_pad_cols) {
                        float *dst = base + (long long)(mt * 128 + q * 32) * p.Ng + b_idx;
                        if (add) put_rows<kPutAdd>(buf, value, lane, dst, p.Ng, a_rows - q * 32);
                        else put_rows<kPutPlain>(buf, value, lane, dst, p.Ng, a_rows - q * 32);
                    } else if (row_ok) {
                        put_values(value, base, add, p, a_idx, b_idx);
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (abort_flag) {
        if (threadIdx.x == 0) { *p.status = DP_ERR_TIMEOUT; __threadfence(); }
        __nanosleep(200000);
        __syncthreads();
    }
    cluster_sync_all();                                   // nobody leaves while a peer may still write to its shared memory
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}



// ----------------------------------------------------------------------------- clipped sum as ONE matrix product (bf16)
// With the factors known, sum_n f_n dY_n^T Xcol_n is a single matrix product whose reduction runs over (example, pixel)
// once every row of dY carries its example's factor: the tensor core then adds all examples into one accumulator and
// nothing is read back from tensor memory per example (reading a 128 x 256 tile back costs as much as eight MMAs,
// which is what bounds a per-example clipped sum on layers with few pixels).  f_n * dY does not fit bf16, so a small
// launch before this one splits it into hi + lo (both bf16, hi = the rounded product, lo = the rounded remainder: what
// is lost is below 2^-17 of each product) and every k-step issues two MMAs, X with hi and X with lo.  A work item is a
// tile for a range of examples; with more than one range the tiles leave as partial sums for the fold.
// Roles as in the kernel at the top: warp 0 / 6 TMA (the warp that loads dY loads both copies), warp 1 MMA, warps 2-5 epilogue.
template <int N>
__global__ void __launch_bounds__(224, 1)
conv_wgrad_ssum_kernel(const __grid_constant__ TcTable<TcParams, 3, N> tab) {
    const int entry = table_entry(tab.first, tab.n, blockIdx.x);
    const CUtensorMap &tmX = tab.e[entry].map[0], &tmYhi = tab.e[entry].map[1], &tmYlo = tab.e[entry].map[2];
    const TcParams &p = tab.e[entry].p;
    const int blk = (int)blockIdx.x - tab.first[entry];
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tmem_full[2], tmem_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ float4 xpose[4][256];        // per epilogue warp: a 32 x 32 block on its way out (put_rows)

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t tiles_u32 = smem_u32(tiles);

    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmYhi)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmYlo)) : "memory");
        abort_flag = 0;
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 2); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tmem_full[b]), 1); mbar_init(smem_u32(&tmem_empty[b]), 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int *abort_p = &abort_flag;

    const int slab_bytes = p.Kt * kRowBytes;
    const int a_slabs_tile = 128 / p.slab_ch, b_slabs_tile = p.NT / p.slab_ch;
    const bool a_is_y = p.a_is_x == 0;                        // which operand is dY (and so has a lo copy)

    if (warp == 0 || warp == 6) {
        // ------------------------------------------------------------ TMA producers
        const bool leader = elect_one();
        const bool is_a = warp == 0, is_y = is_a == a_is_y;
        int stage = 0; uint32_t phase = 0;
        bool live = true;
        for (int item = blk; item < p.total_tiles && live; item += p.blocks) {
            const Item it = decode_item(p, item);
            const int slab0 = is_a ? it.mt * a_slabs_tile : it.nt * b_slabs_tile;
            const int slabs = min(is_a ? a_slabs_tile : b_slabs_tile, (is_a ? p.a_ext : p.b_ext) / p.slab_ch - slab0);
            const OperandCopies copies(p, !is_y, slab0, slabs, is_a ? p.a_group : p.b_group, slab_bytes, lane);
            const CUtensorMap *map = is_y ? &tmYhi : &tmX;
            const uint32_t dst = tiles_u32 + (is_a ? 0u : (uint32_t)p.a_bytes), dst_lo = tiles_u32 + (uint32_t)p.lo_offset;
            const uint32_t tx_bytes = (uint32_t)copies.count * copies.bytes * (is_y ? 2u : 1u);       // dY comes as hi and lo
            for (int n = it.n_lo; n < it.n_hi && live; ++n) {
                int ow0 = 0, oh0 = 0, tw = 0;
                for (int kt = 0; kt < p.k_tiles; ++kt) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                    if (leader) mbar_expect_tx(smem_u32(&full_bar[stage]), tx_bytes);
                    __syncwarp();
                    copies.issue(leader, map, dst + stage * p.stage_bytes, smem_u32(&full_bar[stage]), ow0, oh0, n);
                    if (is_y) copies.issue(leader, &tmYlo, dst_lo + stage * p.stage_bytes, smem_u32(&full_bar[stage]), ow0, oh0, n);
                    if (++tw == p.tiles_w) { tw = 0; ow0 = 0; oh0 += p.OHt; } else { ow0 += p.OWt; }
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the warp walks together, one lane issues
        const bool leader = elect_one();
        int stage = 0; uint32_t phase = 0, acc_phase = 0;
        int buf = 0;
        bool live = true;
        const uint64_t desc_base = operand_desc_base<false>((uint32_t)slab_bytes);
        const uint32_t desc_lo = (uint32_t)desc_base, desc_hi32 = (uint32_t)(desc_base >> 32);
        const int ksteps = p.Kt / p.krows;
        constexpr uint32_t kadvance = (uint32_t)(16 * kRowBytes) >> 4;
        for (int item = blk; item < p.total_tiles && live; item += p.blocks) {
            const Item it = decode_item(p, item);
            const int b_slabs = min(b_slabs_tile, p.b_ext / p.slab_ch - it.nt * b_slabs_tile);
            const uint32_t idesc = instr_desc(b_slabs * p.slab_ch, 1u);
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&tmem_empty[buf]), ((acc_phase >> buf) & 1u) ^ 1u, abort_p, p.wait_polls))) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * 256);
            uint32_t accumulate = 0;
            const int trips = (it.n_hi - it.n_lo) * p.k_tiles;
            for (int kt = 0; kt < trips; ++kt) {
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[stage]), phase, abort_p, p.wait_polls))) { live = false; break; }
                tc_fence_after();
                const uint32_t src = tiles_u32 + stage * p.stage_bytes;
                uint32_t ad = desc_lo | ((src & 0x3FFFFu) >> 4);
                uint32_t bd = desc_lo | (((src + p.a_bytes) & 0x3FFFFu) >> 4);
                uint32_t ld = desc_lo | (((src + p.lo_offset) & 0x3FFFFu) >> 4);
                if (leader) {
#pragma unroll 2
                    for (int ks = 0; ks < ksteps; ++ks) {
                        umma<false>(d_tmem, ad, bd, desc_hi32, idesc, accumulate);                               // X with hi(f dY)
                        if (a_is_y) umma<false>(d_tmem, ld, bd, desc_hi32, idesc, 1u);                           // X with lo(f dY)
                        else umma<false>(d_tmem, ad, ld, desc_hi32, idesc, 1u);
                        accumulate = 1;
                        ad += kadvance; bd += kadvance; ld += kadvance;
                    }
                    umma_commit(smem_u32(&empty_bar[stage]));
                }
                accumulate = 1;
                __syncwarp();
                if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            }
            if (!live) break;
            if (leader) umma_commit(smem_u32(&tmem_full[buf]));
            __syncwarp();
            acc_phase ^= 1u << buf;
            buf ^= 1;
        }
    } else if (warp >= 2 && warp <= 5) {
        // ------------------------------------------------------------ epilogue: one read of the finished tile per item
        const int q = warp & 3;
        const int row = q * 32 + lane;
        uint32_t full_phase = 0;
        int buf = 0;
        for (int item = blk; item < p.total_tiles; item += p.blocks) {
            const Item it = decode_item(p, item);
            const int mt = it.mt, nt = it.nt;
            const int a_rows = min(128, p.a_ext - mt * 128);
            const int n_cols = min(p.NT, p.b_ext - nt * p.NT);
            const int a_idx = mt * 128 + row;
            const bool row_ok = row < a_rows && (!p.a_is_x || a_idx < p.Ng);
            const bool arrived = mbar_wait(smem_u32(&tmem_full[buf]), (full_phase >> buf) & 1u, abort_p, p.wait_polls);
            if (!__all_sync(0xffffffffu, arrived)) break;
            full_phase ^= 1u << buf;
            tc_fence_after();
            const uint32_t t_addr = tmem_base + (uint32_t)(buf * 256) + ((uint32_t)(q * 32) << 16);
            const bool add = p.splits == 1;
            float *base = p.sum_out + (add ? 0ll : (long long)it.split * p.Kout * p.Ng);
            auto put = [&](uint32_t (&v)[32], int cc) {
                const int b_idx = nt * p.NT + cc;
                auto value = [&](int i) { return __uint_as_float(v[i]); };
                if (!p.a_is_x) {
                    float *dst = base + (long long)(mt * 128 + q * 32) * p.Ng + b_idx;
                    if (add) put_rows<kPutAdd>(xpose[warp - 2], value, lane, dst, p.Ng, a_rows - q * 32);
                    else put_rows<kPutPlain>(xpose[warp - 2], value, lane, dst, p.Ng, a_rows - q * 32);
                } else if (row_ok) {
                    float *dst = base + (long long)b_idx * p.Ng + a_idx;
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        if (add) red_add(dst + (long long)i * p.Ng, value(i)); else dst[(long long)i * p.Ng] = value(i);
                    }
                }
            };
            for (int cc = 0; cc < n_cols; cc += 64) {
                uint32_t v0[32], v1[32];
                tmem_ld32_issue(t_addr + (uint32_t)cc, v0);
                tmem_ld32_issue(t_addr + (uint32_t)(cc + 32), v1);
                tmem_ld_wait32(v0); tmem_ld_wait32(v1);
                put(v0, cc);
                if (cc + 32 < n_cols) put(v1, cc + 32);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
            buf ^= 1;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (abort_flag) {
        if (threadIdx.x == 0) { *p.status = DP_ERR_TIMEOUT; __threadfence(); }
        __nanosleep(200000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}

// ----------------------------------------------------------------------------- norms from Gram matrices
// For a layer whose gradient is far larger than its pixel count squared, the squared norm of example n comes cheaper
// from the identity  ||dY_n^T Xcol_n||_F^2 = sum_{p,q} (dY_n dY_n^T)[p,q] (Xcol_n Xcol_n^T)[p,q]  over pixel pairs
// (the norm the clip factor of the paper's section 2 needs, without the gradient itself): two Gram matrices of
// [pixels x pixels], each a product over channels, and Xcol's is the sum over the taps of the Gram matrices of the
// shifted inputs.  Here the SAME shared-memory tiles as above (one TMA box = pixels x 64 channels, 128-byte rows,
// 128-byte swizzle) are read as K-major operands: the pixel is the M / N index and the channel the reduction index,
// and one tile serves as both A and B.  One CTA per example; a plane of up to 256 pixels (box rows, a multiple of 16)
// is one or two row tiles of 128, and since both matrices are symmetric the second row tile only needs the columns
// from 128 on, the first one counting its columns from 128 on twice.  Planes of 64 box pixels go two examples to a tile
// (one TMA box over two examples): the small MMAs of a single 64-pixel example are bound by their issue rate.
// Roles (192 threads): warp 0 TMA, warp 1 MMA issue, warps 2-5 read both matrices back and sum their products.
struct GramParams {
    int B, Cin, Kout, S, taps, stride, pad;
    int rows;                   // pixels of the box (zero rows past the plane included), a multiple of 16, <= 256
    int pack;                   // examples per tile: 2 when rows == 64 (two examples fill the 128 rows of an MMA; only the
                                // diagonal 64 x 64 blocks of the products are read), else 1
    int m_tiles, stages, stage_bytes;
    float C_l;
    float *sqnorm; long long sq_stride; float *factor_out; float *clip_out;
    int *status;
    uint32_t wait_polls;
    int blocks;                 // blocks of the launch that work on this layer
};

// K-major operand of 128-byte rows with the 128-byte swizzle: 8-row groups 1024 B apart; the leading offset is unused
// because one instruction's 32 bytes of K lie inside one swizzle row.
__device__ __forceinline__ uint64_t kmajor_desc_base() {
    uint64_t d = (uint64_t)1 << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n_cols
__device__ __forceinline__ uint32_t instr_desc_kmajor(int n_cols) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n_cols >> 3) << 17) | ((128u >> 4) << 24);
}

template <int N>
__global__ void __launch_bounds__(192, 1)
conv_gram_norm_kernel(const __grid_constant__ TcTable<GramParams, 2, N> tab) {
    const int entry = table_entry(tab.first, tab.n, blockIdx.x);
    const CUtensorMap &tmX = tab.e[entry].map[0], &tmY = tab.e[entry].map[1];
    const GramParams &p = tab.e[entry].p;
    const int blk = (int)blockIdx.x - tab.first[entry];
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], tmem_full[2], tmem_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ __align__(8) uint64_t norm_bar;
    __shared__ double warp_part[4][4];      // [example & 3][quadrant]: a warp may run up to three examples ahead of the one that adds up

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t tiles_u32 = smem_u32(tiles);

    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmY)) : "memory");
        abort_flag = 0;
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&tmem_full[b]), 1); mbar_init(smem_u32(&tmem_empty[b]), 4); }
        mbar_init(smem_u32(&norm_bar), 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    volatile int *abort_p = &abort_flag;

    // tensor memory: one or two buffers of 256 columns; in a buffer dY's matrix first, then Xcol's
    const int nbuf = p.rows > 128 ? 1 : 2;
    const uint32_t x_col = p.rows > 128 ? 256u : 128u;
    const int y_slabs = p.Kout / 64, c_slabs = p.Cin / 64;
    const int slabs = y_slabs + p.taps * c_slabs;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer: one box per stage
        const bool leader = elect_one();
        int stage = 0; uint32_t phase = 0;
        bool live = true;
        const uint32_t tx_bytes = (uint32_t)(p.pack * p.rows * kRowBytes);
        for (int n = blk * p.pack; n < p.B && live; n += p.blocks * p.pack) {
            for (int mt = 0; mt < p.m_tiles && live; ++mt) {
                int r = 0, sx = 0, cs = 0;                   // tap (r, sx) and slab of X
                for (int s = 0; s < slabs; ++s) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                    const bool is_y = s < y_slabs;
                    if (leader) {
                        mbar_expect_tx(smem_u32(&full_bar[stage]), tx_bytes);
                        tma_load_slabs(tiles_u32 + stage * p.stage_bytes, is_y ? &tmY : &tmX, smem_u32(&full_bar[stage]), is_y ? 0 : sx - p.pad,
                                       is_y ? 0 : r - p.pad, n, is_y ? s : cs);
                    }
                    __syncwarp();
                    if (!is_y && ++cs == c_slabs) { cs = 0; if (++sx == p.S) { sx = 0; ++r; } }
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer: the warp walks together, one lane issues
        const bool leader = elect_one();
        int stage = 0; uint32_t phase = 0, acc_phase = 0;
        int buf = 0;
        bool live = true;
        const uint64_t desc_base = kmajor_desc_base();
        const uint32_t desc_lo = (uint32_t)desc_base, desc_hi32 = (uint32_t)(desc_base >> 32);
        for (int n = blk * p.pack; n < p.B && live; n += p.blocks * p.pack) {
            for (int mt = 0; mt < p.m_tiles && live; ++mt) {
                const int col0 = mt * 128;                       // the tile's columns start at its own first row
                const uint32_t idesc = instr_desc_kmajor(p.pack * p.rows - col0);
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&tmem_empty[buf]), ((acc_phase >> buf) & 1u) ^ 1u, abort_p, p.wait_polls))) { live = false; break; }
                tc_fence_after();
                const uint32_t d_y = tmem_base + (uint32_t)(buf * 256), d_x = d_y + x_col;
                for (int s = 0; s < slabs; ++s) {
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[stage]), phase, abort_p, p.wait_polls))) { live = false; break; }
                    tc_fence_after();
                    const uint32_t src = tiles_u32 + stage * p.stage_bytes + (uint32_t)(col0 * kRowBytes);
                    uint32_t ad = desc_lo | ((src & 0x3FFFFu) >> 4);
                    const uint32_t d_tmem = s < y_slabs ? d_y : d_x;
                    uint32_t accumulate = (s == 0 || s == y_slabs) ? 0u : 1u;
                    if (leader) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {             // 64 channels = four steps of 16, 32 bytes apart in the row
                            umma<false>(d_tmem, ad, ad, desc_hi32, idesc, accumulate);
                            accumulate = 1;
                            ad += 2;
                        }
                        umma_commit(smem_u32(&empty_bar[stage]));
                    }
                    __syncwarp();
                    if (++stage == p.stages) { stage = 0; phase ^= 1u; }
                }
                if (!live) break;
                if (leader) umma_commit(smem_u32(&tmem_full[buf]));
                __syncwarp();
                acc_phase ^= 1u << buf;
                if (nbuf == 2) buf ^= 1;
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue: sum over the tile of G_Y .* G_X
        const int q = warp & 3;
        uint32_t full_phase = 0;
        int buf = 0;
        bool live = true;
        int trip = 0;
        for (int n = blk * p.pack; n < p.B && live; n += p.blocks * p.pack) {
            double acc = 0.0;
            for (int mt = 0; mt < p.m_tiles; ++mt) {
                const int col0 = mt * 128;
                const bool arrived = mbar_wait(smem_u32(&tmem_full[buf]), (full_phase >> buf) & 1u, abort_p, p.wait_polls);
                if (!__all_sync(0xffffffffu, arrived)) { live = false; break; }
                full_phase ^= 1u << buf;
                tc_fence_after();
                const int row = col0 + q * 32 + lane;
                // packed: quadrants 0, 1 hold the first example (columns 0..63), quadrants 2, 3 the second (64..127)
                const int c_lo = p.pack == 2 ? (q >> 1) * 64 : 0;
                const int c_hi = p.pack == 2 ? c_lo + 64 : p.rows - col0;
                if (col0 + q * 32 < p.pack * p.rows) {               // warps whose rows all lie past the box read nothing
                    const uint32_t t_y = tmem_base + (uint32_t)(buf * 256) + ((uint32_t)(q * 32) << 16), t_x = t_y + x_col;
                    float s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};     // columns below / from 128
                    for (int cc = c_lo; cc < c_hi; cc += 32) {
                        uint32_t vy[32], vx[32];
                        tmem_ld32_issue(t_y + (uint32_t)cc, vy);
                        tmem_ld32_issue(t_x + (uint32_t)cc, vx);
                        tmem_ld_wait32(vy); tmem_ld_wait32(vx);
                        const bool twice = cc >= 128;
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const float pr = (cc + i < c_hi) ? __uint_as_float(vy[i]) * __uint_as_float(vx[i]) : 0.f;
                            if (twice) s2[i & 3] += pr; else s1[i & 3] += pr;
                        }
                    }
                    if (row < p.pack * p.rows)
                        acc += ((double)s1[0] + (double)s1[1]) + ((double)s1[2] + (double)s1[3]) +
                               2.0 * (((double)s2[0] + (double)s2[1]) + ((double)s2[2] + (double)s2[3]));
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tmem_empty[buf]));
                if (nbuf == 2) buf ^= 1;
            }
            if (!live) break;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            // the four warps hand their sums to the one that publishes through a barrier word (no warp waits for
            // another except that one, and its wait is bounded like every other)
            if (lane == 0) { warp_part[trip & 3][q] = acc; mbar_arrive(smem_u32(&norm_bar)); }
            if (q == 0) {
                if (!mbar_wait(smem_u32(&norm_bar), (uint32_t)(trip & 1), abort_p, p.wait_polls)) { live = false; break; }
                if (lane < p.pack && n + lane < p.B) {
                    const double *w = warp_part[trip & 3];
                    const double sq = p.pack == 2 ? w[2 * lane] + w[2 * lane + 1] : (w[0] + w[1]) + (w[2] + w[3]);
                    const int m = n + lane;
                    p.sqnorm[m * p.sq_stride] = (float)sq;
                    const float f = clip_factor(sq, p.C_l);
                    if (p.factor_out) { p.factor_out[2 * m] = f; p.factor_out[2 * m + 1] = f; }
                    if (p.clip_out) p.clip_out[m] = f;
                }
            }
            ++trip;
        }
    }

    tc_fence_before();
    __syncthreads();
    if (abort_flag) {
        if (threadIdx.x == 0) { *p.status = DP_ERR_TIMEOUT; __threadfence(); }
        __nanosleep(200000);
        __syncthreads();
    }
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}

// hi[i] = bf16(f_n y[i]), lo[i] = bf16(f_n y[i] - hi[i]) for every entry of example n (eight entries per thread)
struct SplitSeg { const __nv_bfloat16 *y; const float *factor; long long per_example, total8; __nv_bfloat16 *hi, *lo; };
struct SplitTable { int n; int first[kTcLayers]; SplitSeg s[kTcLayers]; };
__global__ void __launch_bounds__(256)
scale_split_kernel(const __grid_constant__ SplitTable tab) {
    const int entry = table_entry(tab.first, tab.n, blockIdx.x);
    const SplitSeg &sg = tab.s[entry];
    const long long i8 = (long long)(blockIdx.x - tab.first[entry]) * 256 + threadIdx.x;
    if (i8 >= sg.total8) return;
    const long long i = i8 * 8;
    const float f = sg.factor[2 * (i / sg.per_example)];
    __nv_bfloat16 v[8], h[8], l[8];
    *reinterpret_cast<uint4 *>(v) = *reinterpret_cast<const uint4 *>(sg.y + i);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float x = f * __bfloat162float(v[e]);
        h[e] = __float2bfloat16_rn(x);
        l[e] = __float2bfloat16_rn(x - __bfloat162float(h[e]));
    }
    *reinterpret_cast<uint4 *>(sg.hi + i) = *reinterpret_cast<const uint4 *>(h);
    *reinterpret_cast<uint4 *>(sg.lo + i) = *reinterpret_cast<const uint4 *>(l);
}

static dp_status launch_scale_split(const std::vector<SplitSeg> &segs, cudaStream_t stream) {
    for (size_t i = 0; i < segs.size();) {
        SplitTable tab;
        long long blocks = 0;
        for (tab.n = 0; i < segs.size() && tab.n < kTcLayers; ++i) {
            tab.first[tab.n] = (int)blocks;
            tab.s[tab.n++] = segs[i];
            blocks += (segs[i].total8 + 255) / 256;
        }
        if (blocks > 0x7fffffffll) return DP_ERR_UNSUPPORTED;
        scale_split_kernel<<<(unsigned)blocks, 256, 0, stream>>>(tab);
        DP_LAUNCH_CHECK("scale_split_kernel");
    }
    return DP_OK;
}

// acc[i] += sum over splits of part[s][i], splits in index order; vec: P a multiple of 4 and both 16-byte aligned.
// A layer's sums are few (a 64 x 128 gradient is 16 blocks), so what bounds this is one thread's chain of loads: eight
// in flight and small blocks, which spread over the SMs (30 ranges of such a gradient: 8.4 us with four in flight and
// 256 threads a block).
constexpr int kFoldThreads = 128, kFoldAhead = 8;
struct FoldSeg { const float *part; float *acc; long long P; int splits, vec; };
struct FoldTable { int n; int first[kTcLayers]; FoldSeg s[kTcLayers]; };
__global__ void __launch_bounds__(kFoldThreads)
fold_partial_sums_kernel(const __grid_constant__ FoldTable tab) {
    const int entry = tab.n == 1 ? 0 : table_entry(tab.first, tab.n, blockIdx.x);
    const long long P = tab.s[entry].P, i = ((long long)(blockIdx.x - tab.first[entry]) * kFoldThreads + threadIdx.x) * 4;
    const float *part = tab.s[entry].part + i;
    float *acc = tab.s[entry].acc + i;
    const int splits = tab.s[entry].splits;
    if (i >= P) return;
    if (tab.s[entry].vec) {
        float4 a = *reinterpret_cast<const float4 *>(acc);
        for (int s = 0; s < splits; s += kFoldAhead) {
            float4 v[kFoldAhead];
#pragma unroll
            for (int k = 0; k < kFoldAhead; ++k) {
                v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (s + k < splits) v[k] = __ldcs(reinterpret_cast<const float4 *>(part + (s + k) * P));
            }
#pragma unroll
            for (int k = 0; k < kFoldAhead; ++k) { a.x += v[k].x; a.y += v[k].y; a.z += v[k].z; a.w += v[k].w; }
        }
        *reinterpret_cast<float4 *>(acc) = a;
    } else {
        for (int k = 0; k < (int)min(P - i, 4ll); ++k) {
            float a = acc[k];
            for (int s = 0; s < splits; ++s) a += part[s * P + k];
            acc[k] = a;
        }
    }
}

static FoldSeg fold_seg(const float *part, int splits, long long P, float *acc) {
    return FoldSeg{part, acc, P, splits, (P % 4 == 0 && aligned(part, 16) && aligned(acc, 16)) ? 1 : 0};
}
static dp_status launch_folds(const std::vector<FoldSeg> &segs, cudaStream_t stream) {
    for (size_t i = 0; i < segs.size();) {
        FoldTable tab;
        long long blocks = 0;
        for (tab.n = 0; i < segs.size() && tab.n < kTcLayers; ++i) {
            tab.first[tab.n] = (int)blocks;
            tab.s[tab.n++] = segs[i];
            blocks += (segs[i].P + 4 * kFoldThreads - 1) / (4 * kFoldThreads);
        }
        if (blocks > 0x7fffffffll) return DP_ERR_UNSUPPORTED;
        fold_partial_sums_kernel<<<(unsigned)blocks, kFoldThreads, 0, stream>>>(tab);
        DP_LAUNCH_CHECK("fold_partial_sums_kernel");
    }
    return DP_OK;
}
static dp_status launch_fold_partial_sums(const float *part, int splits, long long P, float *acc, cudaStream_t stream) {
    return launch_folds({fold_seg(part, splits, P, acc)}, stream);
}

// Layers whose input has too few channels for a TMA slab (C_in = 3 stems) are first unfolded:
// Xcol[n, oh, ow, j] = Xpad[n, oh*st + r - pad, ow*st + s - pad, c], j = (r*S + s)*C_in + c, zero for j >= R*S*C_in,
// with rows padded to a whole number of slabs.  The layer then is a 1x1 convolution over Xcol for the kernel above.
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
unfold_small_channels_kernel(const T *__restrict__ X, T *__restrict__ Xcol, const ConvGeom g, int n_pad, long long total) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;       // one 16-byte group of columns each
    if (idx >= total) return;
    const int groups = n_pad / VEC;
    const long long pixel = idx / groups;                                        // (n*OH + oh)*OW + ow
    const int j0 = (int)(idx - pixel * groups) * VEC;
    const int ow = (int)(pixel % g.OW);
    const long long t = pixel / g.OW;
    const int oh = (int)(t % g.OH);
    const long long n = t / g.OH;
    T v[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        const int j = j0 + e;
        T x = T(0.f);
        if (j < g.N) {
            const int c = j % g.Cin, rs = j / g.Cin;
            const int r = rs / g.S, s = rs - r * g.S;
            const int ih = oh * g.stride + r - g.pad, iw = ow * g.stride + s - g.pad;
            if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W) x = X[((n * g.H + ih) * g.W + iw) * g.Cin + c];
        }
        v[e] = x;
    }
    *reinterpret_cast<uint4 *>(Xcol + pixel * n_pad + j0) = *reinterpret_cast<const uint4 *>(v);
}

// Same unfolding, one block per (output row, example): the R input rows the output row touches are staged in
// shared memory with their zero padding written out (so no window needs a bounds check), then every thread
// assembles 16-byte groups of columns from them through a table  column j -> offset inside the staged rows.
// Within one filter row r the (s, c) columns of a pixel are a contiguous run of the input row.
constexpr int kUnfoldMaxCols = 512;
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
unfold_rows_kernel(const T *__restrict__ X, T *__restrict__ Xcol, const ConvGeom g, int n_pad) {
    extern __shared__ __align__(16) unsigned char unfold_smem[];
    __shared__ __align__(16) short col_off[kUnfoldMaxCols];
    T *rows = reinterpret_cast<T *>(unfold_smem);          // [R][Wp*Cin], Wp = (OW-1)*stride + S padded pixels
    const int oh = blockIdx.x, n = blockIdx.y;
    const int row_p = ((g.OW - 1) * g.stride + g.S) * g.Cin, row_len = g.W * g.Cin, shift = g.pad * g.Cin;
    const int tap_row = g.S * g.Cin;
    for (int j = threadIdx.x; j < n_pad; j += 256) {
        const int r = j / tap_row;
        col_off[j] = (j < g.N) ? (short)(r * row_p + (j - r * tap_row)) : (short)-1;
    }
    for (int r = 0; r < g.R; ++r) {
        const int ih = oh * g.stride + r - g.pad;
        const bool inside = ih >= 0 && ih < g.H;
        const T *src = X + ((long long)n * g.H + (inside ? ih : 0)) * row_len;
        for (int i = threadIdx.x; i < row_p; i += 256) {
            const int col = i - shift;
            rows[r * row_p + i] = (inside && col >= 0 && col < row_len) ? src[col] : T(0.f);
        }
    }
    __syncthreads();
    const int groups = n_pad / VEC, step = g.stride * g.Cin;
    T *dst = Xcol + ((long long)n * g.OH + oh) * g.OW * n_pad;
    for (int chunk = threadIdx.x; chunk < g.OW * groups; chunk += 256) {
        const int ow = chunk / groups;
        const int j0 = (chunk - ow * groups) * VEC;
        const T *win = rows + ow * step;
        __align__(16) short off[VEC];
        if (VEC == 8) *reinterpret_cast<uint4 *>(off) = *reinterpret_cast<const uint4 *>(col_off + j0);
        else *reinterpret_cast<uint2 *>(off) = *reinterpret_cast<const uint2 *>(col_off + j0);
        __align__(16) T v[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) v[e] = off[e] >= 0 ? win[off[e]] : T(0.f);
        *reinterpret_cast<uint4 *>(dst + (long long)chunk * VEC) = *reinterpret_cast<const uint4 *>(v);
    }
}

// Space-to-depth regrouping of a thin strided input (C_in * stride^2 <= 16 channels): pixel (a, b) of the result
// holds the stride x stride block of padded-input pixels (stride*a + dy, stride*b + dx) as channels
// (dy*stride + dx)*C_in + c, zero-filled up to 16.  The strided R x S convolution over the input is then a
// stride-1 convolution with ceil(R/stride) x ceil(S/stride) taps over 16-channel pixels, and the (at most four)
// taps of one filter row are 64 contiguous values: one 128-byte operand row per output pixel, read straight
// from this buffer by a tensor map whose pixel stride (32 bytes) is smaller than its row (128 bytes).
__global__ void __launch_bounds__(256)
space_to_depth_kernel(const __nv_bfloat16 *__restrict__ X, __nv_bfloat16 *__restrict__ Xs, const ConvGeom g, int Hs, int Ws, long long total) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;     // one output pixel each
    if (idx >= total) return;
    const int b = (int)(idx % Ws);
    const long long t = idx / Ws;
    const int a = (int)(t % Hs);
    const long long n = t / Hs;
    __align__(16) __nv_bfloat16 v[16];
#pragma unroll
    for (int ch = 0; ch < 16; ++ch) v[ch] = __float2bfloat16(0.f);
    const int st = g.stride;
    for (int dy = 0; dy < st; ++dy) {
        const int ih = st * a + dy - g.pad;
        if (ih < 0 || ih >= g.H) continue;
        for (int dx = 0; dx < st; ++dx) {
            const int iw = st * b + dx - g.pad;
            if (iw < 0 || iw >= g.W) continue;
            const __nv_bfloat16 *src = X + ((n * g.H + ih) * g.W + iw) * g.Cin;
            for (int c = 0; c < g.Cin; ++c) v[(dy * st + dx) * g.Cin + c] = src[c];
        }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(Xs + idx * 16);
    dst[0] = *reinterpret_cast<const uint4 *>(v);
    dst[1] = *reinterpret_cast<const uint4 *>(v + 8);
}

// ----------------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    });
    return fn;
}

// What the tensor-core kernel is actually given: the layer itself, or its unfolded 1x1 form.
struct TcProblem {
    bool ok, unfold;
    ConvGeom eff;       // geometry the kernel tiles
    int n_pad;          // unfolded row length (columns incl. zero padding)
};

// A 1 x 1 convolution with stride 1 is a plain product over the pixels, whatever their arrangement: its planes are
// flattened to one row of H*W pixels, so that a pixel tile is any run of pixels (no width / height rounding: 14 x 14
// is 208 reduction rows instead of 240) and a TMA box is one long run instead of many short rows.
static void flatten_pointwise(ConvGeom &e) {
    if (e.R == 1 && e.S == 1 && e.stride == 1 && e.pad == 0 && e.H > 1) {
        e.W = e.H * e.W; e.H = 1;
        e.OW = e.OH * e.OW; e.OH = 1;
    }
}

static TcProblem tc_problem(int dtype, const ConvGeom &g) {
    TcProblem pr; pr.ok = false; pr.unfold = false; pr.eff = g; pr.n_pad = g.N;
    const int slab_ch = (dtype == DP_BF16) ? 64 : 32;
    if (g.Kout % slab_ch) return pr;
    if (g.Cin % slab_ch == 0) { pr.ok = true; flatten_pointwise(pr.eff); return pr; }
    // small-channel layers only: the unfolded copy costs N/C_in times the input, which is only worth it for thin inputs
    if (g.Cin > 8 || g.N > 512) return pr;
    pr.unfold = true;
    pr.n_pad = (g.N + slab_ch - 1) / slab_ch * slab_ch;
    ConvGeom e = g;
    e.H = g.OH; e.W = g.OW; e.Cin = pr.n_pad; e.R = 1; e.S = 1; e.stride = 1; e.pad = 0;
    e.N = pr.n_pad;
    flatten_pointwise(e);
    pr.eff = e;
    pr.ok = true;
    return pr;
}

// Cycle model of one MMA step (16 bf16 / 8 tf32 reduction rows) for the tiling search.  Measured on B200: an
// instruction occupies the tensor pipe for N/2 cycles, and shared memory moves 128 B per cycle in total, shared by
// the tensor core's operand reads (always 128 rows of A plus N rows of B, 32 B per row and step), the TMA fill of the
// stage and, for split tf32, the split warps (they read every landed byte once and write the lo copy).
static double step_cycles(int dtype, int n_cols, double a_slabs_loaded, double b_slabs) {
    if (dtype == DP_BF16) {
        const double smem = 4096.0 + 32.0 * n_cols + 2048.0 * (a_slabs_loaded + b_slabs);
        return std::max(n_cols / 2.0, smem / 128.0);
    }
    if (dtype == DP_TF32) {   // one MMA per step of 8 rows
        const double smem = 4096.0 + 32.0 * n_cols + 1024.0 * (a_slabs_loaded + b_slabs);
        return std::max(n_cols / 2.0, smem / 128.0);
    }
    const double smem = 3.0 * (4096.0 + 32.0 * n_cols) + 1024.0 * (a_slabs_loaded + b_slabs) * 3.0;
    return std::max(3.0 * n_cols / 2.0, smem / 128.0);
}

static TcPlan search_plan(int dtype, const ConvGeom &g, int mode);

// Planning on behalf of a batch of layer calls (this thread): launches hold many layers, so every layer is tiled for
// least SM time whatever the SM target is, and a CTA walks through at most this many cycles of one layer.
static thread_local double tl_batch_walk = 0.0;
static thread_local bool tl_beside = false;
BatchPlanning::BatchPlanning(double walk_cycles, bool beside) : saved(tl_batch_walk), saved_beside(tl_beside) { tl_batch_walk = walk_cycles; tl_beside = beside; }
BatchPlanning::~BatchPlanning() { tl_batch_walk = saved; tl_beside = saved_beside; }
static bool side_by_side() { return tl_batch_walk > 0.0 || sm_target_set(); }
// What a block's stages may take, with room left for a block of the normalisation layers' where one runs beside it (the kernels of modes
// 0, 1 and 4 have 16 KB of their own besides).
static int smem_budget(int mode) { return tl_beside ? (mode == 3 ? kBatchSmem : kBatchSmem - 16 * 1024) : kSmemBudget; }
static int launch_sms() { return tl_batch_walk > 0.0 ? sm_count() : sm_target(); }

// single-pass clipped sum: how many clusters share the batch and how many examples each walks through
// scaled-sum product: example ranges per tile.  A launch that already has a CTA for a quarter of the SMs keeps whole
// tiles (no partial sums to fold); fewer tiles are cut up to half of the SMs.
static void ssum_split(int B, int tiles, int &splits, int &per_split) {
    const int sms = launch_sms();
    // (side by side with other calls, under an SM target, a quarter: fewer partial sums to write and fold)
    int want = (tiles * 4 >= sms) ? 1 : (sms / (side_by_side() ? 4 : 2)) / tiles;
    if (want < 1) want = 1;
    if (want > B) want = B;
    per_split = (B + want - 1) / want;
    splits = (B + per_split - 1) / per_split;
}

static int max_active_clusters(int cluster_size);
// K, NT: pixels per example and columns per tile (for a rough time of one example in one CTA)
static void cluster_split(int B, int cluster_size, int K, int NT, int &splits, int &per_split) {
    int want = std::min(launch_sms() / cluster_size, max_active_clusters(cluster_size));
    // A caller that set an SM target runs calls side by side: what counts then is SM time, and a cluster that walks
    // through several examples spends its start-up, its first loads and its final stores once for all of them -- up
    // to thirty-two examples (a whole chunk of the per-layer workload: one example range, nothing to fold), and not
    // beyond some 60 microseconds a launch, so that no call holds its stream up for long.
    if (side_by_side()) {
        const double cycles = (K / 16.0) * std::max(NT / 2.0, 64.0) * 1.5;
        const int per = std::max(1, std::min(kMaxExamplesPerCluster, (int)((tl_batch_walk > 0.0 ? tl_batch_walk : 120000.0) / cycles)));
        want = std::min(want, std::max(1, B / per));
    }
    if (want < 1) want = 1;
    if (want > B) want = B;
    per_split = (B + want - 1) / want;
    splits = (B + per_split - 1) / per_split;
}

// The tiling search is pure; its results are memoised per layer geometry (host side only).
// mode: 0 gradients are stored, 1 norms only, 2 clipped sum (running sum in registers: at most 128 columns per tile)
static TcPlan make_plan(int dtype, const ConvGeom &g, int mode) {
    static std::mutex mu;
    static std::map<std::array<int, 14>, TcPlan> memo;
    const std::array<int, 14> key = {dtype, g.H, g.W, g.Cin, g.Kout, g.R, g.S, g.stride, g.pad, g.B, mode, side_by_side() ? -launch_sms() : launch_sms(), (int)tl_batch_walk, tl_beside};
    std::lock_guard<std::mutex> lock(mu);
    auto it = memo.find(key);
    if (it != memo.end()) return it->second;
    const TcPlan pl = search_plan(dtype, g, mode);
    memo.emplace(key, pl);
    return pl;
}

// max_nt = 128 plans the clipped-sum mode: its running sum lives in registers (128 columns per thread) and the
// work items are (example range, tile) pairs, so the wave count no longer depends on the batch size
// mode 3 plans the single-pass clipped sum: all tiles of an example in one cluster (at most kMaxCluster of them), the
// clusters share the batch, and what is minimised is SM time (clusters x CTAs x time), not the time of one launch
// Rough time of a launch whose items are shared by `by` blocks each: `main` is a block's main loop; loads start from nothing
// (1500 cycles), the tile goes out of tensor memory (8 a column) and through the cluster (every thread's chain of reads), launch
// and two cluster barriers take 2500.
static int max_active_clusters(int cluster_size);
static double split_cycles(int mode, int items, int by, int NT, double main) {
    const double places = std::min((double)max_active_clusters(by) * by, (double)launch_sms());
    const double waves = std::ceil((double)items * by / (std::floor(places / by) * by));
    return (main + 1500.0 + 8.0 * NT + NT * (5.7 / by + 3.6) + (mode == 0 ? 128.0 * NT * 4.0 / by / 16.0 : 0.0) + 2500.0) * waves;
}
// At least a third of an SM's shared memory: two blocks, of 256 columns of tensor memory each, on an SM at most.  A third would wait
// for columns with its cluster waiting for it, and clusters that hold columns might wait for one another.  (Their registers keep a
// third one out as well, as compiled now.)
constexpr size_t kSplitSmemLeast = 77 * 1024;
static size_t split_smem(int a_is_x, int NT) {
    return std::max(kSplitSmemLeast, (a_is_x ? NT * (128 + kSplitPad) : 128 * (NT + kSplitPad)) * sizeof(float) + 1024);
}

static TcPlan search_plan(int dtype, const ConvGeom &g, int mode) {
    const int max_nt = (mode == 2) ? 128 : 256;
    const bool rows_are_inputs = mode == 6 || mode >= 8; // modes 6, 8, 9: modes 3, 0, 1 with the rows of D fixed to the input columns
    const bool any_tiles = mode == 7;                    // mode 7: mode 3 without clusters (factors known): any number of tiles
    if (mode == 6 || mode == 7) mode = 3;
    if (mode >= 8) mode -= 8;
    TcPlan best; best.ok = false;
    const int slab_ch = (dtype == DP_BF16) ? 64 : 32;
    const int krows = (dtype == DP_BF16) ? 16 : 8;
    if (g.Cin % slab_ch || g.Kout % slab_ch) return best;
    if (g.stride > 8 || g.K < 1 || g.OH > 65535) return best;
    const int sms = launch_sms();
    const int a_slabs_tile = 128 / slab_ch;
    const int copies = (dtype == DP_F32) ? 2 : 1;       // split tf32 keeps a hi and a lo copy of every stage
    double best_cost = 1e300, best_main = 0.0, best_epilogue = 0.0, best_waves = 0.0;
    TcPlan shared; shared.ok = false;                    // the best form that shares an item's pixels among a cluster
    double shared_cost = 1e300;
    const bool may_split = dtype == DP_BF16 && mode <= 1 && !side_by_side();
    for (int a_is_x = rows_are_inputs ? 1 : 0; a_is_x < 2; ++a_is_x) {
        const int a_ext = a_is_x ? g.N : g.M, b_ext = a_is_x ? g.M : g.N;
        for (int NT = slab_ch; NT <= max_nt; NT += slab_ch) {
            if (NT != 32 && NT % 64) continue;
            if (NT > b_ext) break;
            const int m_tiles = (a_ext + 127) / 128, n_tiles = (b_ext + NT - 1) / NT;
            const int slabs = a_slabs_tile + NT / slab_ch;
            const long long total_tiles = (long long)g.B * m_tiles * n_tiles;
            if (total_tiles > 0x7fffffffLL) continue;
            if (mode == 3 && !any_tiles && m_tiles * n_tiles > kMaxCluster) continue;
            // (beside normalisation layers, sizes that share no launch with others would be one more to wait for)
            const double apart = mode == 3 && !any_tiles && tl_beside && (m_tiles * n_tiles == 5 || m_tiles * n_tiles == 7) ? 1.1 : 1.0;
            const int y_slabs = (mode == 4) ? (a_is_x ? NT / slab_ch : a_slabs_tile) : 0;     // second (lo) copy of the dY slabs
            // per-CTA share of (example, tile) units: whole waves of tiles, or in clipped-sum mode an even share of the examples
            // (in a batch other layers fill the last wave)
            double waves = (mode != 2 && tl_batch_walk == 0.0) ? (double)((total_tiles + sms - 1) / sms)
                                       : std::max(mode == 2 ? 1.0 : 0.0, (double)total_tiles / sms);
            double sm_share = 1.0;
            if (mode == 4) {
                int splits, per;
                ssum_split(g.B, m_tiles * n_tiles, splits, per);
                waves = per;
                sm_share = (double)std::min(splits * m_tiles * n_tiles, sms);
            }
            if (mode == 3) {
                int splits, per;
                cluster_split(g.B, m_tiles * n_tiles, g.K, NT, splits, per);
                waves = per;                                       // examples a cluster walks through
                sm_share = (double)splits * m_tiles * n_tiles;      // SMs the launch holds meanwhile
            }
            const double a_loaded = (double)(a_ext / slab_ch) / m_tiles, b_loaded = (double)(b_ext / slab_ch) / n_tiles;
            const double step = step_cycles(dtype, NT, a_loaded, b_loaded) * (mode == 4 ? 2.0 : 1.0);
            // the epilogue of a tile overlaps the main loop of the next; what it costs depends on what it does with
            // the 128 x NT accumulator: stores run at about 16 B/clk per SM when lanes write consecutive addresses
            // (rows of D are gradient columns) and about 7 B/clk otherwise; reading TMEM alone is cheap
            const double epilogue = (mode == 0) ? 128.0 * NT * 4.0 / (a_is_x ? 16.0 : 7.0)
                                  : (mode == 1 ? 6.0 * NT : (mode == 2 ? 10.0 * NT : (mode == 4 ? 0.0 : 10.0 * std::min(NT, 128) + 600.0)));
            // a pixel tile may reach past the output plane (its rows there are zero-filled by TMA and add nothing):
            // a 7 x 7 plane is one 8 x 8 tile of 64 reduction rows instead of four 4 x 4 tiles of 16
            const int oh_max = std::min((g.OH + 7) / 8 * 8, 256 / g.stride), ow_max = std::min((g.OW + 15) / 16 * 16, 256 / g.stride);
            for (int OHt = 1; OHt <= oh_max; ++OHt) {
                for (int OWt = 1; OWt <= ow_max; ++OWt) {
                    if (OWt > g.OW && OWt % 8) continue;      // overshoot only to the next multiple of eight
                    if (OHt > g.OH && OHt % 8) continue;
                    const int Kt = OHt * OWt;
                    if (Kt % krows || Kt > 256) continue;
                    const int stage_bytes = (slabs + y_slabs) * Kt * kRowBytes * copies;
                    int stages = smem_budget(mode) / stage_bytes;
                    if (stages < 2) continue;
                    if (stages > kMaxStages) stages = kMaxStages;
                    if (dtype == DP_F32) stages &= ~1;        // each split group has slots of its own (see there)
                    const int tw = (g.OW + OWt - 1) / OWt, th = (g.OH + OHt - 1) / OHt;
                    // a stage: its MMA steps plus the hand-over (barrier wait, commit) of the issuing thread
                    double stage_cost = (double)(Kt / krows) * step + 250.0;
                    // a TMA warp: barrier wait + expect_tx, then one copy per slab it owns (A or B), all latency-bound on that warp
                    stage_cost = std::max(stage_cost, 350.0 + 110.0 * std::max(a_loaded, b_loaded));
                    if (dtype == DP_F32)   // split warps, two groups in turn: a fixed fence/hand-over plus their share of the bytes
                        stage_cost = std::max(stage_cost, 0.5 * (1000.0 + (a_loaded + b_loaded) * Kt * 2.5));
                    double mainloop = stage_cost * tw * th;
                    if (stages < 3) mainloop *= 1.15;
                    auto take = [&](TcPlan &t) {
                        t.ok = true; t.a_is_x = a_is_x; t.a_ext = a_ext; t.b_ext = b_ext;
                        t.m_tiles = m_tiles; t.n_tiles = n_tiles; t.NT = NT;
                        t.OWt = OWt; t.OHt = OHt; t.tiles_w = tw; t.tiles_h = th; t.Kt = Kt;
                        t.k_tiles = tw * th; t.stages = stages; t.stage_bytes = stage_bytes;
                        t.a_bytes = a_slabs_tile * Kt * kRowBytes;
                        t.smem = (size_t)stages * stage_bytes + 1024;
                        t.item_cycles = std::max(mainloop, epilogue) + 300.0;
                        t.split = 1;
                    };
                    for (int by = 2; may_split && by <= std::min(kMaxSplit, tw * th); ++by) {
                        const double c = split_cycles(mode, g.B * m_tiles * n_tiles, by, NT, stage_cost * ((tw * th + by - 1) / by) * (stages < 3 ? 1.15 : 1.0));
                        if (c >= shared_cost) continue;
                        shared_cost = c;
                        take(shared);
                        shared.split = by;
                        shared.smem = std::max(shared.smem, split_smem(a_is_x, NT));
                    }
                    const double cost = ((std::max(mainloop, epilogue) + 300.0) * waves + (mode == 3 ? 4000.0 : (mode == 4 ? 6000.0 : 0.0))) * sm_share * apart;
                    if (cost < best_cost) {
                        best_cost = cost; best_main = mainloop; best_epilogue = epilogue; best_waves = waves;
                        take(best);
                    }
                }
            }
        }
    }
    // (a block's first loads and its last epilogue overlap with nothing; what the memory bounds, two thirds of its rate, stays as it is)
    const double memory = 2.0 * g.B * ((double)g.H * g.W * g.Cin + (double)g.K * g.Kout) / 2250.0;
    if (shared.ok && best.ok && std::max(shared_cost, memory) < 0.85 * ((std::max(best_main, best_epilogue) + 300.0) * best_waves + std::min(best_main, best_epilogue) + 1500.0))
        return shared;
    return best;
}

bool tc_eligible(int dtype, const ConvGeom &g0, int epilogue) {
    const TcProblem pr = tc_problem(dtype, g0);
    if (!pr.ok || !encode_fn() || !make_plan(dtype, pr.eff, epilogue == DP_EPI_STORE_NORM ? 0 : 1).ok) return false;
    return epilogue != DP_EPI_CLIP_ACCUM || make_plan(dtype, pr.eff, 2).ok;
}

// The single-pass kernel's register split only adds up when the launch allocates ClipRegs::kLaunch registers a thread.
static bool clip1_registers_ok() {
    static int ok = -1;
    if (ok < 0) {
        cudaFuncAttributes attr;
        ok = (cudaFuncGetAttributes(&attr, conv_wgrad_clip1_kernel<1>) == cudaSuccess && attr.numRegs == ClipRegs<false>::kLaunch &&
              cudaFuncGetAttributes(&attr, conv_wgrad_clip1_kernel<kTcLayers>) == cudaSuccess && attr.numRegs == ClipRegs<false>::kLaunch &&
              cudaFuncGetAttributes(&attr, conv_wgrad_clip1_kernel<kTcLayers, true>) == cudaSuccess && attr.numRegs == ClipRegs<true>::kLaunch) ? 1 : 0;
        if (!ok) (void)cudaGetLastError();
    }
    return ok == 1;
}

// How many clusters of this size the GPU can hold at once (a cluster needs all its SMs free in one GPC at the same
// time, so this is less than SMs / size); more clusters than that would run as a second wave.  Unknown (no device): no cap.
static int max_active_clusters(int cluster_size) {
    static std::atomic<int> cached[64][kMaxCluster + 1];
    int dev = -1;
    if (cluster_size < 1 || cluster_size > kMaxCluster) return 1 << 30;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { (void)cudaGetLastError(); return 1 << 30; }
    const int known = cached[dev][cluster_size].load(std::memory_order_relaxed);
    if (known) return known;
    int n = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cluster_size * 64)); cfg.blockDim = dim3(kClipThreads); cfg.dynamicSmemBytes = kSmemBudget + 1024;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster_size; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const bool ok = cudaFuncSetAttribute(conv_wgrad_clip1_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget + 2048) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, conv_wgrad_clip1_kernel<1>, &cfg) == cudaSuccess && n > 0;
    if (!ok) { (void)cudaGetLastError(); return 1 << 30; }
    cached[dev][cluster_size].store(n, std::memory_order_relaxed);
    return n;
}

// Thin strided layers (a 7 x 7 stride-2 stem on RGB) in space-to-depth form, see space_to_depth_kernel: the geometry the
// kernel tiles is a stride-1 convolution with ceil(R/stride) x 1 taps of 64 "channels" (one filter row's window).
struct S2dProblem { bool ok; int R2, Hs, Ws; ConvGeom eff; };
static S2dProblem s2d_problem(int dtype, const ConvGeom &g, const TcProblem &pr) {
    S2dProblem sp = {};
    if (dtype != DP_BF16 || !pr.ok || !pr.unfold || g.stride < 2 || g.Cin * g.stride * g.stride > 16 || g.Kout % 64) return sp;
    if ((g.S + g.stride - 1) / g.stride > 4) return sp;
    sp.R2 = (g.R + g.stride - 1) / g.stride;
    sp.Hs = g.OH + sp.R2 - 1; sp.Ws = g.OW + 3;
    if ((size_t)sp.Hs * sp.Ws * 32 > (size_t)g.OH * g.OW * pr.n_pad * 2) return sp;     // lives in the unfolded copy's room
    ConvGeom e = g;
    e.Cin = 64; e.R = sp.R2; e.S = 1; e.stride = 1; e.pad = 0; e.H = sp.Hs; e.W = g.OW;
    e.N = sp.R2 * 64;
    sp.eff = e; sp.ok = true;
    return sp;
}

// The single-pass plan of a layer and the geometry it tiles: bf16 inputs, the example's gradient fits the tensor memory
// of one cluster.  Thin strided layers take the space-to-depth form when that has a plan (rows of D = input columns).
static bool clip1_plan(int dtype, const ConvGeom &g0, const TcProblem &pr, TcPlan &pl, ConvGeom &g, bool &s2d) {
    s2d = false;
    if (dtype != DP_BF16 || !pr.ok) return false;
    const S2dProblem sp = s2d_problem(dtype, g0, pr);
    if (sp.ok) {
        pl = make_plan(dtype, sp.eff, 6);
        if (pl.ok) { g = sp.eff; s2d = true; return true; }
    }
    g = pr.eff;
    pl = make_plan(dtype, pr.eff, 3);
    return pl.ok;
}

// What the store and norm kernels are given: thin strided layers in space-to-depth form as well, where nothing reads an
// unfolded copy later on (32 examples of a 7 x 7 stem on 224 x 224: 69 us for the 154 MB copy, 11 for the regrouping).
struct StoreForm { TcPlan pl; ConvGeom g; bool s2d; };
static StoreForm store_form(int dtype, const ConvGeom &g0, const TcProblem &pr, int epilogue, bool regroup = true) {
    StoreForm f = {};
    const int mode = epilogue == DP_EPI_STORE_NORM ? 0 : 1;
    const S2dProblem sp = regroup && epilogue != DP_EPI_CLIP_ACCUM ? s2d_problem(dtype, g0, pr) : S2dProblem{};
    if (sp.ok) {
        f.pl = make_plan(dtype, sp.eff, mode + 8);
        if (f.pl.ok) { f.g = sp.eff; f.s2d = true; return f; }
    }
    f.g = pr.eff;
    f.pl = make_plan(dtype, pr.eff, mode);
    return f;
}

// clipped-sum mode: how many example ranges each tile is cut into so that every SM has an item
static void clip_split(const ConvGeom &g, const TcPlan &pl, int &splits, int &per_split) {
    const int tiles = pl.m_tiles * pl.n_tiles;
    int want = launch_sms() / tiles;
    if (want < 1) want = 1;
    if (want > g.B) want = g.B;
    per_split = (g.B + want - 1) / want;
    splits = (g.B + per_split - 1) / per_split;
}

// Eight warps read the tiles of a norm pass back where an example has few pixels (32 examples of 3 x 3 512 -> 512 on 7 x 7: 31 us,
// 25; on 14 x 14 the same as four, on 50 x 50 3 us of 47 slower), in a call on its own: a batch's launches hold layers that store, too.
static bool norm_readers(int dtype, int epilogue, const TcPlan &pl) {
    return dtype == DP_BF16 && epilogue != DP_EPI_STORE_NORM && tl_batch_walk == 0.0 && pl.k_tiles * pl.Kt <= 128;
}

int tc_norm_slots(int dtype, const ConvGeom &g0, int epilogue) {
    const TcProblem pr = tc_problem(dtype, g0);
    if (!pr.ok) return 0;
    const TcPlan pl = store_form(dtype, g0, pr, epilogue).pl;
    return pl.ok ? pl.m_tiles * pl.n_tiles * (pl.split > 1 ? pl.split : (norm_readers(dtype, epilogue, pl) ? 8 : 4)) : 0;
}

static size_t unfold_bytes(int dtype, const ConvGeom &g0, const TcProblem &pr) {
    if (!pr.unfold) return 0;
    return round_up((size_t)g0.B * g0.OH * g0.OW * pr.n_pad * (dtype == DP_BF16 ? 2 : 4), 1024);
}

// the row-staging form of the unfolding: its staged rows must fit shared memory and its offsets 16 bits
static size_t unfold_rows_smem(int dtype, const ConvGeom &g) {
    return (size_t)g.R * ((size_t)(g.OW - 1) * g.stride + g.S) * g.Cin * (dtype == DP_BF16 ? 2 : 4);
}
static bool unfold_rows_ok(int dtype, const ConvGeom &g, int n_pad) {
    const size_t bytes = unfold_rows_smem(dtype, g);
    return bytes <= 40 * 1024 && bytes / (dtype == DP_BF16 ? 2 : 4) < 32768 && n_pad <= kUnfoldMaxCols && g.B <= 65535;
}

static size_t ssum_copy_bytes(const ConvGeom &g) { return round_up((size_t)g.B * g.OH * g.OW * g.Kout * 2, 1024); }
bool tc_clip_scaled_sum(int dtype, const ConvGeom &g0);
bool tc_clip_scaled_tiles(int dtype, const ConvGeom &g0);
static void scaled_tiles_split(const ConvGeom &g, const TcPlan &pl, int &splits, int &per);

// layout: [unfolded input, if any][partial sums of the clipped-sum mode, if any], or the scaled copies of dY and partial sums
size_t tc_workspace_bytes(int dtype, const ConvGeom &g0, int epilogue) {
    const TcProblem pr = tc_problem(dtype, g0);
    if (!pr.ok) return 0;
    size_t bytes = unfold_bytes(dtype, g0, pr);
    if (epilogue == DP_EPI_CLIP_ACCUM) {
        const TcPlan pl = make_plan(dtype, pr.eff, 2);
        if (!pl.ok) return 0;
        int splits, per;
        clip_split(pr.eff, pl, splits, per);
        TcPlan one; ConvGeom og; bool s2d;
        if (clip1_plan(dtype, g0, pr, one, og, s2d)) {     // room for either form: the single pass may be unavailable at run time
            int s1, p1;
            cluster_split(og.B, one.m_tiles * one.n_tiles, og.K, one.NT, s1, p1);
            splits = std::max(splits, s1);
        }
        size_t clip_bytes = splits > 1 ? sizeof(float) * (size_t)splits * g0.M * g0.N : 0;
        if (tc_clip_scaled_sum(dtype, g0)) {
            const TcPlan sp = make_plan(dtype, pr.eff, 4);
            int s4, p4;
            ssum_split(pr.eff.B, sp.m_tiles * sp.n_tiles, s4, p4);
            clip_bytes = std::max(clip_bytes, 2 * ssum_copy_bytes(pr.eff) + (s4 > 1 ? sizeof(float) * (size_t)s4 * g0.M * g0.N : 0));
        }
        if (tc_clip_scaled_tiles(dtype, g0)) {
            int s7, p7;
            scaled_tiles_split(pr.eff, make_plan(dtype, pr.eff, 7), s7, p7);
            clip_bytes = std::max(clip_bytes, s7 > 1 ? sizeof(float) * (size_t)s7 * g0.M * g0.N : (size_t)0);
        }
        bytes += clip_bytes;
    }
    return bytes;
}

static int gram_describe(int dtype, const ConvGeom &g0, int *out, int n);
int tc_describe_plan(int dtype, const ConvGeom &g0, int epilogue, int *out, int n) {
    const TcProblem pr = tc_problem(dtype, g0);
    if (!pr.ok) return 0;
    if (epilogue == 5) return gram_describe(dtype, g0, out, n);
    TcPlan pl;
    if (epilogue == 3) {
        ConvGeom g; bool s2d;
        if (!clip1_plan(dtype, g0, pr, pl, g, s2d)) return 0;
    } else {
        pl = epilogue < 2 ? store_form(dtype, g0, pr, epilogue).pl : make_plan(dtype, pr.eff, epilogue);
    }
    if (!pl.ok) return 0;
    const int v[12] = {pl.a_is_x, pl.a_ext, pl.b_ext, pl.m_tiles, pl.n_tiles, pl.NT, pl.OWt, pl.OHt, pl.Kt, pl.k_tiles,
                       pl.stages, pl.stage_bytes};
    for (int i = 0; i < n && i < 12; ++i) out[i] = v[i];
    return 12;
}

// channels-last [B, H, W, C] tensor seen as {slab of channels, W, H, B, slabs}; box = {slab, boxW, boxH, boxN, slabs a copy};
// `step` > 1 walks every step-th pixel (the box then spans boxW*step pixels and delivers boxW of them)
static bool encode_nhwc(CUtensorMap *map, int dtype, const void *base, int C, int W, int H, int Bn, int boxW, int boxH, int step,
                        int boxN = 1, int slabs = 1) {
    const cuuint64_t es = (dtype == DP_BF16) ? 2 : 4, slab_ch = kRowBytes / es;
    const cuuint64_t dims[5] = {slab_ch, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)Bn, (cuuint64_t)C / slab_ch};
    const cuuint64_t strides[4] = {(cuuint64_t)C * es, (cuuint64_t)W * C * es, (cuuint64_t)H * W * C * es, kRowBytes};
    const cuuint32_t box[5] = {(cuuint32_t)slab_ch, (cuuint32_t)(boxW * step), (cuuint32_t)(boxH * step), (cuuint32_t)boxN, (cuuint32_t)slabs};
    const cuuint32_t estr[5] = {1, (cuuint32_t)step, (cuuint32_t)step, 1, 1};
    return encode_fn()(map, dtype == DP_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                             : (dtype == DP_TF32 ? CU_TENSOR_MAP_DATA_TYPE_TFLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32), 5,
                       const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       dtype == DP_BF16 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

typedef TcEntry<TcParams, 2> ConvEntry;
typedef TcEntry<TcParams, 3> SsumEntry;
typedef TcEntry<GramParams, 2> GramEntry;
static_assert(sizeof(TcTable<TcParams, 3, kSsumLayers>) <= 32000 && sizeof(TcTable<TcParams, 2, kTcLayers>) <= 32000, "kernel parameters are limited to 32764 bytes");

// The limit on dynamic shared memory belongs to a function in one context: it is raised for every launch (60 ns), in whichever
// context and on whichever device is current.
template <typename K>
static cudaError_t allow_shared(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget + 2048);
}
template <typename TABLE>
static dp_status launch_table(void (*kernel)(const TABLE), const char *name, const TABLE &tab, int blocks, int threads, size_t smem, cudaStream_t stream) {
    DP_CUDA_TRY(allow_shared(kernel));
    kernel<<<(unsigned)blocks, (unsigned)threads, smem, stream>>>(tab);
    DP_LAUNCH_CHECK(name);
    return DP_OK;
}
template <typename TABLE>
static dp_status launch_table_clusters(void (*kernel)(const TABLE), const char *name, const TABLE &tab, int cluster, int blocks, int threads, size_t smem, cudaStream_t stream) {
    DP_CUDA_TRY(allow_shared(kernel));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const cudaError_t le = cudaLaunchKernelEx(&cfg, kernel, tab);
    if (le != cudaSuccess) return cuda_fail(le, name);
    DP_LAUNCH_CHECK(name);
    return DP_OK;
}

// Slabs one copy brings: neighbours along the channels of one filter tap, a divisor of the tile's and of the tensor's slabs.
static int slab_group(int dtype, const ConvGeom &g, const TcPlan &pl, bool of_a) {
    const int slab_ch = (dtype == DP_BF16) ? 64 : 32;
    const bool is_x = of_a == (pl.a_is_x != 0);
    return std::gcd((is_x ? g.Cin : g.Kout) / slab_ch, (of_a ? 128 : pl.NT) / slab_ch);
}
static int x_group(int dtype, const ConvGeom &g, const TcPlan &pl) { return slab_group(dtype, g, pl, pl.a_is_x != 0); }
static int y_group(int dtype, const ConvGeom &g, const TcPlan &pl) { return slab_group(dtype, g, pl, pl.a_is_x == 0); }

// what the parameters of every kernel take from the layer and its plan
static void fill_common(TcParams &p, int dtype, const ConvGeom &g, int Ng, const TcPlan &pl, int *status) {
    p.B = g.B; p.Kout = g.Kout; p.Ng = Ng; p.Cin = g.Cin; p.S = g.S; p.stride = g.stride; p.pad = g.pad;
    p.n_pad_cols = (g.N != Ng) ? 1 : 0;
    p.slab_ch = (dtype == DP_BF16) ? 64 : 32; p.krows = (dtype == DP_BF16) ? 16 : 8;
    p.a_is_x = pl.a_is_x; p.a_ext = pl.a_ext; p.b_ext = pl.b_ext; p.m_tiles = pl.m_tiles; p.n_tiles = pl.n_tiles; p.NT = pl.NT;
    p.OWt = pl.OWt; p.OHt = pl.OHt; p.tiles_w = pl.tiles_w; p.Kt = pl.Kt; p.k_tiles = pl.k_tiles;
    p.stages = pl.stages; p.stage_bytes = pl.stage_bytes; p.a_bytes = pl.a_bytes;
    p.a_group = slab_group(dtype, g, pl, true); p.b_group = slab_group(dtype, g, pl, false);
    p.status = status;
    p.wait_polls = wait_polls();
}

// Layers with few input channels: the unfolded copy of X in the call's scratch.
static dp_status unfold_input(int dtype, const void *X, const ConvGeom &g0, const TcProblem &pr, void *dst, cudaStream_t stream) {
    const int vec = (dtype == DP_BF16) ? 8 : 4;
    const long long total = (long long)g0.B * g0.OH * g0.OW * (pr.n_pad / vec);
    const unsigned blocks = (unsigned)((total + 255) / 256);
    const size_t row_smem = unfold_rows_smem(dtype, g0);
    if (unfold_rows_ok(dtype, g0, pr.n_pad)) {
        const dim3 grid_rows(g0.OH, g0.B);
        if (dtype == DP_BF16)
            unfold_rows_kernel<__nv_bfloat16, 8><<<grid_rows, 256, row_smem, stream>>>(
                static_cast<const __nv_bfloat16 *>(X), static_cast<__nv_bfloat16 *>(dst), g0, pr.n_pad);
        else
            unfold_rows_kernel<float, 4><<<grid_rows, 256, row_smem, stream>>>(
                static_cast<const float *>(X), static_cast<float *>(dst), g0, pr.n_pad);
    } else if (dtype == DP_BF16)
        unfold_small_channels_kernel<__nv_bfloat16, 8><<<blocks, 256, 0, stream>>>(
            static_cast<const __nv_bfloat16 *>(X), static_cast<__nv_bfloat16 *>(dst), g0, pr.n_pad, total);
    else
        unfold_small_channels_kernel<float, 4><<<blocks, 256, 0, stream>>>(
            static_cast<const float *>(X), static_cast<float *>(dst), g0, pr.n_pad, total);
    DP_LAUNCH_CHECK("unfold_small_channels_kernel");
    return DP_OK;
}

// The input as a kernel reads it: X itself, or its space-to-depth / unfolded copy written to the scratch.
static dp_status prepare_input(int dtype, const void *X, const ConvGeom &g0, const TcProblem &pr, bool s2d, void *tc_workspace,
                               cudaStream_t stream) {
    if (s2d) {
        const S2dProblem sp = s2d_problem(dtype, g0, pr);
        const long long total = (long long)g0.B * sp.Hs * sp.Ws;
        space_to_depth_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(
            static_cast<const __nv_bfloat16 *>(X), static_cast<__nv_bfloat16 *>(tc_workspace), g0, sp.Hs, sp.Ws, total);
        DP_LAUNCH_CHECK("space_to_depth_kernel");
        return DP_OK;
    }
    return pr.unfold ? unfold_input(dtype, X, g0, pr, tc_workspace, stream) : DP_OK;
}

// a space-to-depth copy as the kernels read it: one operand row per output pixel, 64 values from pixel ow on, pixels 16 apart
static bool encode_s2d(CUtensorMap *map, void *base, const S2dProblem &sp, const TcPlan &pl) {
    const ConvGeom &g = sp.eff;
    const cuuint64_t dims[5] = {64, (cuuint64_t)g.OW, (cuuint64_t)sp.Hs, (cuuint64_t)g.B, 1};
    const cuuint64_t strides[4] = {32, (cuuint64_t)sp.Ws * 32, (cuuint64_t)sp.Hs * sp.Ws * 32, (cuuint64_t)g.B * sp.Hs * sp.Ws * 32};
    const cuuint32_t box[5] = {64, (cuuint32_t)pl.OWt, (cuuint32_t)pl.OHt, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
static void fill_s2d(TcParams &p, const ConvGeom &g0) { p.s2d_st = g0.stride; p.s2d_R = g0.R; p.s2d_S = g0.S; p.s2d_Cin = g0.Cin; }

// Parameters of the norm / store / two-pass clipped-sum kernel for one layer; X already regrouped or unfolded where the layer
// needs it.
static dp_status fill_conv_tc(int dtype, int epilogue, const void *X, const void *dY, const ConvGeom &g0, const TcProblem &pr,
                              const ConvGeom &g, const TcPlan &pl, bool s2d, float *G_w, float *partial, int slots, const float *factor, float *acc_w,
                              void *tc_workspace, int *status, const TcPublish *publish, ConvEntry &e) {
    const bool clip = epilogue == DP_EPI_CLIP_ACCUM;
    if (s2d ? !encode_s2d(&e.map[0], const_cast<void *>(X), s2d_problem(dtype, g0, pr), pl)
            : !encode_nhwc(&e.map[0], dtype, X, g.Cin, g.W, g.H, g.B, pl.OWt, pl.OHt, g.stride, 1, x_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(X)");
    if (!encode_nhwc(&e.map[1], dtype, dY, g.Kout, g.OW, g.OH, g.B, pl.OWt, pl.OHt, 1, 1, y_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY)");
    TcParams &p = e.p;
    p = TcParams{};
    fill_common(p, dtype, g, g0.N, pl, status);
    if (s2d) fill_s2d(p, g0);
    p.lo_offset = pl.stage_bytes / 2;
    p.mode = clip ? 2 : (epilogue == DP_EPI_STORE_NORM ? 0 : 1);
    p.G_w = G_w; p.partial = partial; p.slots = slots;
    p.splits = 1; p.per_split = g.B; p.factor = factor; p.sum_out = acc_w;
    if (!clip && publish) {
        p.counters = publish->counters; p.w_slots = publish->w_slots; p.separate = publish->separate; p.fold_slots = slots;
        p.sqnorm = publish->sqnorm; p.sq_stride = publish->sq_stride;
        p.factor_out = publish->factor_out; p.C_l = publish->C_l; p.clip_out = publish->clip_out;
    }
    if (clip) {
        clip_split(g, pl, p.splits, p.per_split);
        if (p.splits > 1) p.sum_out = reinterpret_cast<float *>(static_cast<char *>(tc_workspace) + unfold_bytes(dtype, g0, pr));
        p.total_tiles = p.splits * pl.m_tiles * pl.n_tiles;
    } else {
        p.total_tiles = g.B * pl.m_tiles * pl.n_tiles;
    }
    return DP_OK;
}

dp_status launch_conv_tc(int dtype, int epilogue, const void *X, const void *dY, const ConvGeom &g0, float *G_w,
                         float *partial, int slots, const float *factor, float *acc_w, void *tc_workspace, int *status,
                         cudaStream_t stream, bool second_pass, const TcPublish *publish) {
    const bool clip = epilogue == DP_EPI_CLIP_ACCUM;
    const TcProblem pr = tc_problem(dtype, g0);
    if (!pr.ok || !encode_fn()) return DP_ERR_UNSUPPORTED;
    // (the norm pass of a fused clip call leaves its unfolded copy to the second pass, and a single partial sum a tile)
    const StoreForm form = clip ? StoreForm{make_plan(dtype, pr.eff, 2), pr.eff, false} : store_form(dtype, g0, pr, epilogue, !(publish && publish->factor_out));
    const TcPlan &pl = form.pl;
    if (!pl.ok) return DP_ERR_UNSUPPORTED;
    dp_status rc = DP_OK;
    if (pr.unfold) {
        // in a fused clip call this function runs twice (norm pass, then clipped-sum pass): the unfolded input is
        // rebuilt only by the first of them
        if (!(clip && second_pass) && (rc = prepare_input(dtype, X, g0, pr, form.s2d, tc_workspace, stream)) != DP_OK) return rc;
        X = tc_workspace;
    }
    TcTable<TcParams, 2, 1> tab;
    tab.n = 1; tab.first[0] = 0;
    rc = fill_conv_tc(dtype, epilogue, X, dY, g0, pr, form.g, pl, form.s2d, G_w, partial, slots, factor, acc_w, tc_workspace, status, publish, tab.e[0]);
    if (rc != DP_OK) return rc;
    TcParams &p = tab.e[0].p;
    if (!clip && pl.split > 1) {
        p.splits = pl.split;
        p.blocks = p.total_tiles * pl.split;
        return launch_table_clusters(conv_wgrad_split_kernel, "conv_wgrad_split_kernel", tab, pl.split, p.blocks, 224, pl.smem, stream);
    }
    p.blocks = std::min(p.total_tiles, sm_target());
    auto go = [&](void (*kernel)(const TcTable<TcParams, 2, 1>), int threads) {
        return launch_table(kernel, "conv_wgrad_tc_kernel", tab, p.blocks, threads, pl.smem, stream);
    };
    if (dtype == DP_BF16) {
        if (clip) rc = go(conv_wgrad_tc_kernel<kBf16, true, 1>, 224);
        else if (norm_readers(dtype, epilogue, pl)) rc = go(conv_wgrad_tc_kernel<kBf16, false, 1, true>, 352);
        else rc = go(conv_wgrad_tc_kernel<kBf16, false, 1>, 224);
    } else if (dtype == DP_TF32) {
        rc = clip ? go(conv_wgrad_tc_kernel<kTf32, true, 1>, 224) : go(conv_wgrad_tc_kernel<kTf32, false, 1>, 224);
    } else {
        rc = clip ? go(conv_wgrad_tc_kernel<kSplit, true, 1>, 480) : go(conv_wgrad_tc_kernel<kSplit, false, 1>, 480);
    }
    if (rc != DP_OK) return rc;
    if (clip && p.splits > 1) return launch_fold_partial_sums(p.sum_out, p.splits, (long long)g0.M * g0.N, acc_w, stream);
    return DP_OK;
}

// The fused clipped sum of a bf16 layer that does not fit a cluster: norm pass, then ONE matrix product over all examples.
bool tc_clip_scaled_sum(int dtype, const ConvGeom &g0) {
    const TcProblem pr = tc_problem(dtype, g0);
    return dtype == DP_BF16 && pr.ok && !pr.unfold && encode_fn() && g0.Kout % 8 == 0 && make_plan(dtype, pr.eff, 4).ok;
}

// hi and lo copies of f_n * dY in the call's scratch, partial sums (if any) behind them
static dp_status fill_ssum(int dtype, const void *X, const ConvGeom &g, const TcPlan &pl, float *acc_w, void *tc_workspace,
                           int *status, SsumEntry &e) {
    char *ws_bytes = static_cast<char *>(tc_workspace);
    if (!encode_nhwc(&e.map[0], dtype, X, g.Cin, g.W, g.H, g.B, pl.OWt, pl.OHt, g.stride, 1, x_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(X)");
    if (!encode_nhwc(&e.map[1], dtype, ws_bytes, g.Kout, g.OW, g.OH, g.B, pl.OWt, pl.OHt, 1, 1, y_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY hi)");
    if (!encode_nhwc(&e.map[2], dtype, ws_bytes + ssum_copy_bytes(g), g.Kout, g.OW, g.OH, g.B, pl.OWt, pl.OHt, 1, 1, y_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY lo)");
    TcParams &p = e.p;
    p = TcParams{};
    fill_common(p, dtype, g, g.N, pl, status);
    p.lo_offset = pl.a_bytes + (pl.NT / 64) * pl.Kt * kRowBytes;      // after the A and B slabs
    p.mode = 2;                                                       // items are (example range, tile) pairs
    ssum_split(g.B, pl.m_tiles * pl.n_tiles, p.splits, p.per_split);
    p.sum_out = p.splits > 1 ? reinterpret_cast<float *>(ws_bytes + 2 * ssum_copy_bytes(g)) : acc_w;
    p.total_tiles = p.splits * pl.m_tiles * pl.n_tiles;
    return DP_OK;
}

static SplitSeg split_seg(const void *dY, const float *factor, const ConvGeom &g, void *tc_workspace) {
    SplitSeg s;
    s.y = static_cast<const __nv_bfloat16 *>(dY); s.factor = factor;
    s.per_example = (long long)g.OH * g.OW * g.Kout; s.total8 = s.per_example * g.B / 8;
    s.hi = static_cast<__nv_bfloat16 *>(tc_workspace);
    s.lo = reinterpret_cast<__nv_bfloat16 *>(static_cast<char *>(tc_workspace) + ssum_copy_bytes(g));
    return s;
}

dp_status launch_conv_ssum(int dtype, const void *X, const void *dY, const ConvGeom &g0, const float *factor, float *acc_w,
                           void *tc_workspace, int *status, cudaStream_t stream) {
    if (!tc_clip_scaled_sum(dtype, g0)) return DP_ERR_UNSUPPORTED;
    const TcProblem pr = tc_problem(dtype, g0);
    const ConvGeom &g = pr.eff;
    const TcPlan pl = make_plan(dtype, g, 4);
    dp_status rc = launch_scale_split({split_seg(dY, factor, g, tc_workspace)}, stream);
    if (rc != DP_OK) return rc;
    TcTable<TcParams, 3, 1> tab;
    tab.n = 1; tab.first[0] = 0;
    rc = fill_ssum(dtype, X, g, pl, acc_w, tc_workspace, status, tab.e[0]);
    if (rc != DP_OK) return rc;
    TcParams &p = tab.e[0].p;
    p.blocks = std::min(p.total_tiles, sm_target());
    rc = launch_table(conv_wgrad_ssum_kernel<1>, "conv_wgrad_ssum_kernel", tab, p.blocks, 224, pl.smem, stream);
    if (rc != DP_OK) return rc;
    if (p.splits > 1) return launch_fold_partial_sums(p.sum_out, p.splits, (long long)g.M * g.N, acc_w, stream);
    return DP_OK;
}

// ---- clipped sum with the factors known, per example through tensor memory (the single-pass kernel without its norm
// pass and exchange): one tile per CTA, the CTA walks a range of examples, reads each finished tile once and keeps
// sum_n f_n D_n in registers.  Pays where an example has enough pixels that its MMAs outlast the read-back of the tile
// (some nine steps of 16 pixels); below that the one-product form above is the better one.
constexpr int kScaledTilesMinPixels = 128;
bool tc_clip_scaled_tiles(int dtype, const ConvGeom &g0) {
    const TcProblem pr = tc_problem(dtype, g0);
    return dtype == DP_BF16 && pr.ok && !pr.unfold && encode_fn() && pr.eff.K >= kScaledTilesMinPixels &&
           make_plan(dtype, pr.eff, 7).ok && clip1_registers_ok();
}

static void scaled_tiles_split(const ConvGeom &g, const TcPlan &pl, int &splits, int &per) {
    cluster_split(g.B, pl.m_tiles * pl.n_tiles, g.K, pl.NT, splits, per);
}

static dp_status fill_scaled_tiles(int dtype, const void *X, const void *dY, const ConvGeom &g, const TcPlan &pl,
                                   const float *factor, float *acc_w, void *tc_workspace, int *status, ConvEntry &e) {
    if (!encode_nhwc(&e.map[0], dtype, X, g.Cin, g.W, g.H, g.B, pl.OWt, pl.OHt, g.stride, 1, x_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(X)");
    if (!encode_nhwc(&e.map[1], dtype, dY, g.Kout, g.OW, g.OH, g.B, pl.OWt, pl.OHt, 1, 1, y_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY)");
    TcParams &p = e.p;
    p = TcParams{};
    fill_common(p, dtype, g, g.N, pl, status);
    p.mode = 3; p.factor = factor; p.cluster = 1;
    scaled_tiles_split(g, pl, p.splits, p.per_split);
    p.sum_out = p.splits > 1 ? static_cast<float *>(tc_workspace) : acc_w;
    p.total_tiles = p.blocks = p.splits * pl.m_tiles * pl.n_tiles;
    return DP_OK;
}

dp_status launch_conv_scaled_tiles(int dtype, const void *X, const void *dY, const ConvGeom &g0, const float *factor, float *acc_w,
                                   void *tc_workspace, int *status, cudaStream_t stream) {
    if (!tc_clip_scaled_tiles(dtype, g0)) return DP_ERR_UNSUPPORTED;
    const TcProblem pr = tc_problem(dtype, g0);
    const ConvGeom &g = pr.eff;
    const TcPlan pl = make_plan(dtype, g, 7);
    TcTable<TcParams, 2, 1> tab;
    tab.n = 1; tab.first[0] = 0;
    dp_status rc = fill_scaled_tiles(dtype, X, dY, g, pl, factor, acc_w, tc_workspace, status, tab.e[0]);
    if (rc != DP_OK) return rc;
    const TcParams &p = tab.e[0].p;
    rc = launch_table(conv_wgrad_clip1_kernel<1>, "conv_wgrad_clip1_kernel", tab, p.total_tiles, kClipThreads, pl.smem, stream);
    if (rc != DP_OK) return rc;
    if (p.splits > 1) return launch_fold_partial_sums(p.sum_out, p.splits, (long long)g.M * g.N, acc_w, stream);
    return DP_OK;
}

// ---- norms from Gram matrices (conv_gram_norm_kernel): the whole output plane as one pixel box
struct GramPlan { bool ok; ConvGeom g; int OWb, OHb, rows, pack, m_tiles, stages, stage_bytes; size_t smem; };

static GramPlan gram_plan(int dtype, const ConvGeom &g0) {
    GramPlan gp = {};
    const TcProblem pr = tc_problem(dtype, g0);
    if (dtype != DP_BF16 || !pr.ok || pr.unfold || !encode_fn()) return gp;
    gp.g = pr.eff;
    const ConvGeom &g = gp.g;
    if (g.stride > 8) return gp;
    int best = 1 << 30;
    // the smallest box over the plane whose pixel count is a multiple of 16 (rows past the plane are zero-filled)
    for (int OHb = g.OH; OHb <= g.OH + 15; ++OHb)
        for (int OWb = g.OW; OWb <= g.OW + 15; ++OWb) {
            const int rows = OHb * OWb;
            if (rows % 16 || rows > 256 || OWb * g.stride > 256 || OHb * g.stride > 256 || rows >= best) continue;
            best = rows; gp.OWb = OWb; gp.OHb = OHb;
        }
    if (best > 256) return gp;
    gp.rows = best;
    gp.pack = (best == 64) ? 2 : 1;
    gp.m_tiles = (best + 127) / 128;
    gp.stage_bytes = gp.m_tiles * 128 * kRowBytes;      // a row tile always reads 128 rows, whatever the box holds
    gp.stages = std::min(kMaxStages, smem_budget(3) / gp.stage_bytes);
    gp.smem = (size_t)gp.stages * gp.stage_bytes + 1024;
    gp.ok = true;
    return gp;
}

bool tc_gram_norm(int dtype, const ConvGeom &g0) { return gram_plan(dtype, g0).ok; }

// {1, pixels of the box, same, row tiles, 1, columns of the first row tile, box width, box height, pixels per stage,
//  loads per row tile, stages, bytes per stage}
static int gram_describe(int dtype, const ConvGeom &g0, int *out, int n) {
    const GramPlan gp = gram_plan(dtype, g0);
    if (!gp.ok) return 0;
    const int v[12] = {1, gp.rows, gp.rows, gp.m_tiles, 1, gp.rows, gp.OWb, gp.OHb, gp.rows,
                       gp.g.Kout / 64 + gp.g.R * gp.g.S * (gp.g.Cin / 64), gp.stages, gp.stage_bytes};
    for (int i = 0; i < n && i < 12; ++i) out[i] = v[i];
    return 12;
}

static dp_status fill_gram(int dtype, const void *X, const void *dY, const GramPlan &gp, const TcInlineClip &clipinfo,
                           float *factor_out, int *status, GramEntry &e) {
    const ConvGeom &g = gp.g;
    if (!encode_nhwc(&e.map[0], dtype, X, g.Cin, g.W, g.H, g.B, gp.OWb, gp.OHb, g.stride, gp.pack)) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(X)");
    if (!encode_nhwc(&e.map[1], dtype, dY, g.Kout, g.OW, g.OH, g.B, gp.OWb, gp.OHb, 1, gp.pack)) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY)");
    GramParams &p = e.p;
    p = GramParams{};
    p.B = g.B; p.Cin = g.Cin; p.Kout = g.Kout; p.S = g.S; p.taps = g.R * g.S; p.stride = g.stride; p.pad = g.pad;
    p.rows = gp.rows; p.pack = gp.pack; p.m_tiles = gp.m_tiles; p.stages = gp.stages; p.stage_bytes = gp.stage_bytes;
    p.C_l = clipinfo.C_l; p.sqnorm = clipinfo.sqnorm; p.sq_stride = clipinfo.sq_stride; p.clip_out = clipinfo.clip_out;
    p.factor_out = factor_out; p.status = status;
    p.wait_polls = wait_polls();
    p.blocks = std::min((g.B + gp.pack - 1) / gp.pack, launch_sms());
    return DP_OK;
}

dp_status launch_conv_gram_norm(int dtype, const void *X, const void *dY, const ConvGeom &g0, const TcInlineClip &clipinfo,
                                float *factor_out, int *status, cudaStream_t stream) {
    const GramPlan gp = gram_plan(dtype, g0);
    if (!gp.ok) return DP_ERR_UNSUPPORTED;
    TcTable<GramParams, 2, 1> tab;
    tab.n = 1; tab.first[0] = 0;
    const dp_status rc = fill_gram(dtype, X, dY, gp, clipinfo, factor_out, status, tab.e[0]);
    if (rc != DP_OK) return rc;
    return launch_table(conv_gram_norm_kernel<1>, "conv_gram_norm_kernel", tab, tab.e[0].p.blocks, 192, gp.smem, stream);
}

bool tc_clip_single_pass(int dtype, const ConvGeom &g0) {
    const TcProblem pr = tc_problem(dtype, g0);
    TcPlan pl; ConvGeom g; bool s2d;
    return pr.ok && encode_fn() && clip1_plan(dtype, g0, pr, pl, g, s2d) && clip1_registers_ok();
}

static dp_status fill_clip1(int dtype, const void *X, const void *dY, const ConvGeom &g0, const TcProblem &pr, const ConvGeom &g,
                            const TcPlan &pl, bool s2d, const TcInlineClip &clipinfo, float *acc_w, void *tc_workspace, int *status,
                            ConvEntry &e) {
    char *ws_bytes = static_cast<char *>(tc_workspace);
    if (s2d) {
        if (!encode_s2d(&e.map[0], ws_bytes, s2d_problem(dtype, g0, pr), pl))
            return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(space-to-depth X)");
    } else if (!encode_nhwc(&e.map[0], dtype, pr.unfold ? tc_workspace : X, g.Cin, g.W, g.H, g.B, pl.OWt, pl.OHt, g.stride, 1, x_group(dtype, g, pl))) {
        return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(X)");
    }
    if (!encode_nhwc(&e.map[1], dtype, dY, g.Kout, g.OW, g.OH, g.B, pl.OWt, pl.OHt, 1, 1, y_group(dtype, g, pl))) return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled(dY)");
    TcParams &p = e.p;
    p = TcParams{};
    fill_common(p, dtype, g, g0.N, pl, status);
    p.mode = 3;
    if (s2d) fill_s2d(p, g0);
    p.C_l = clipinfo.C_l; p.sqnorm = clipinfo.sqnorm; p.sq_stride = clipinfo.sq_stride; p.clip_out = clipinfo.clip_out;
    p.cluster = pl.m_tiles * pl.n_tiles;
    cluster_split(g.B, p.cluster, g.K, pl.NT, p.splits, p.per_split);
    p.sum_out = p.splits > 1 ? reinterpret_cast<float *>(ws_bytes + unfold_bytes(dtype, g0, pr)) : acc_w;
    p.total_tiles = p.blocks = p.splits * p.cluster;
    return DP_OK;
}

template <int N, bool BESIDE = false>
static dp_status launch_clip1_table(const TcTable<TcParams, 2, N> &tab, int cluster, int blocks, size_t smem, cudaStream_t stream) {
    return launch_table_clusters(conv_wgrad_clip1_kernel<N, BESIDE>, "conv_wgrad_clip1_kernel", tab, cluster, blocks, kClipThreads, smem, stream);
}

dp_status launch_conv_clip1(int dtype, const void *X, const void *dY, const ConvGeom &g0, const TcInlineClip &clipinfo,
                            float *acc_w, void *tc_workspace, int *status, cudaStream_t stream) {
    const TcProblem pr = tc_problem(dtype, g0);
    TcPlan pl; ConvGeom g; bool s2d;
    if (!pr.ok || !encode_fn() || !clip1_plan(dtype, g0, pr, pl, g, s2d) || !clip1_registers_ok()) return DP_ERR_UNSUPPORTED;
    dp_status rc = prepare_input(dtype, X, g0, pr, s2d, tc_workspace, stream);
    if (rc != DP_OK) return rc;
    TcTable<TcParams, 2, 1> tab;
    tab.n = 1; tab.first[0] = 0;
    rc = fill_clip1(dtype, X, dY, g0, pr, g, pl, s2d, clipinfo, acc_w, tc_workspace, status, tab.e[0]);
    if (rc != DP_OK) return rc;
    const TcParams &p = tab.e[0].p;
    rc = launch_clip1_table<1>(tab, p.cluster, p.blocks, pl.smem, stream);
    if (rc != DP_OK) return rc;
    if (p.splits > 1) return launch_fold_partial_sums(p.sum_out, p.splits, (long long)g0.M * g0.N, acc_w, stream);
    return DP_OK;
}

// ----------------------------------------------------------------------------- batches of layer calls
// Layers of one kind share a launch.  What a layer needs is cut into blocks that each hold an SM for some tens of
// microseconds; the blocks of all layers queue up behind one another, longest first, so that the GPU stays full until
// the last few of them, whatever the size of a single layer.
int conv_batch_kind(int dtype, const ConvGeom &g, int epilogue, bool has_bias) {
    if (epilogue != DP_EPI_CLIP_ACCUM) return kConvTc;
    if (has_bias || !single_pass_enabled()) return kConvSingle;
    if (tc_clip_single_pass(dtype, g)) return kConvClip1;
    if (tc_clip_scaled_sum(dtype, g) && tc_gram_norm(dtype, g)) return tc_clip_scaled_tiles(dtype, g) ? kConvGramTiles : kConvGramSum;
    return kConvSingle;
}

// The longest walk of a block: the GPU's share of all the layers' work in as many rounds of blocks as keep each near 30
// microseconds (a block costs some 4 to start and end; several rounds even out what the estimates get wrong), at most four.
double conv_batch_walk(const std::vector<ConvJob> &jobs, bool beside) {
    BatchPlanning planning(120000.0, beside);
    double cycles = 0.0;
    for (const ConvJob &j : jobs) {
        const TcProblem pr = tc_problem(j.dtype, j.g);
        TcPlan pl; ConvGeom g = pr.eff; bool s2d;
        if (j.kind == kConvTc) pl = store_form(j.dtype, j.g, pr, j.epi).pl;
        else if (j.kind == kConvClip1) clip1_plan(j.dtype, j.g, pr, pl, g, s2d);
        else if (j.kind == kConvGramTiles) pl = make_plan(j.dtype, g, 7);
        else continue;
        cycles += pl.item_cycles * j.g.B * pl.m_tiles * pl.n_tiles;
    }
    const double share = cycles / sm_count();
    const double walk = share / std::max(1.0, std::min(4.0, std::floor(share / 55000.0)));
    return std::max(8000.0, std::min(120000.0, std::ceil(walk / 1000.0) * 1000.0));
}

template <typename P, int MAPS, int MOST>
struct TableQueue {
    // jobs of one kernel: filled entries with the blocks they take, launched longest blocks first, N layers at a time
    struct Job { TcEntry<P, MAPS> e; int blocks; size_t smem; double cost; };
    std::vector<Job> jobs;
    template <int N = MOST, typename F>
    dp_status launch(F &&go) {
        std::stable_sort(jobs.begin(), jobs.end(), [](const Job &a, const Job &b) { return a.cost > b.cost; });
        for (size_t i = 0; i < jobs.size();) {
            std::unique_ptr<TcTable<P, MAPS, N>> tab(new TcTable<P, MAPS, N>);
            int blocks = 0;
            size_t smem = 0;
            for (tab->n = 0; i < jobs.size() && tab->n < N; ++i) {
                tab->first[tab->n] = blocks;
                tab->e[tab->n++] = jobs[i].e;
                blocks += jobs[i].blocks;
                smem = std::max(smem, jobs[i].smem);
            }
            const dp_status rc = go(*tab, blocks, smem);
            if (rc != DP_OK) return rc;
        }
        return DP_OK;
    }
};
typedef TableQueue<TcParams, 2, kTcLayers> ConvQueue;
typedef TableQueue<TcParams, 3, kSsumLayers> SsumQueue;
typedef TableQueue<GramParams, 2, kTcLayers> GramQueue;

// Cluster size of the launch a layer with `tiles` tiles an example joins: sizes that divide one another share one.
static int launch_cluster(int tiles) { return tiles == 1 || tiles == 2 || tiles == 4 ? 4 : (tiles == 3 || tiles == 6 ? 6 : tiles); }

int conv_cluster_stream(int cluster, bool beside) {
    return cluster <= 4 ? BatchStreams::kMain : (beside && cluster <= 6 ? BatchStreams::kClusters6 : BatchStreams::kClusters);
}

int conv_batch_cluster(const ConvJob &j, double walk, bool beside) {
    BatchPlanning planning(walk, beside);
    TcPlan pl; ConvGeom g; bool s2d;
    return j.kind == kConvClip1 && clip1_plan(j.dtype, j.g, tc_problem(j.dtype, j.g), pl, g, s2d) ? launch_cluster(pl.m_tiles * pl.n_tiles) : 0;
}

dp_status launch_conv_batch(const std::vector<ConvJob> &jobs, double walk, bool beside, int *status, const BatchStreams &streams,
                            const std::function<dp_status()> &join) {
    if (jobs.empty()) return join();
    const cudaStream_t stream = streams.s[BatchStreams::kMain], sums = streams.s[BatchStreams::kSums];
    auto cluster_stream = [&](int cluster) { return streams.s[conv_cluster_stream(cluster, beside)]; };
    BatchPlanning planning(walk, beside);
    dp_status rc = DP_OK;
    ConvQueue store[3], clip[kMaxCluster + 1];            // store: by element type; clip: by cluster size of the launch
    GramQueue gram;
    SsumQueue ssum;
    std::vector<SplitSeg> splits;
    std::vector<FoldSeg> folds[BatchStreams::kCount];      // by the stream that leaves the partial sums
    for (const ConvJob &j : jobs) {
        const TcProblem pr = tc_problem(j.dtype, j.g);
        const ConvGeom &g = pr.eff;
        const long long P = (long long)j.g.M * j.g.N;
        if (j.kind == kConvTc) {
            const StoreForm form = store_form(j.dtype, j.g, pr, j.epi);
            const TcPlan &pl = form.pl;
            if (!pl.ok) return DP_ERR_UNSUPPORTED;
            const void *X = j.X;
            if (pr.unfold) {
                rc = prepare_input(j.dtype, X, j.g, pr, form.s2d, j.tc_workspace, stream);
                if (rc != DP_OK) return rc;
                X = j.tc_workspace;
            }
            const TcPublish pub = {j.counter, j.w_slots, j.separate, j.clip.sqnorm, j.clip.sq_stride, nullptr, 0.f, nullptr};
            ConvQueue::Job q;
            rc = fill_conv_tc(j.dtype, j.epi, X, j.dY, j.g, pr, form.g, pl, form.s2d, j.G_w, j.partial, j.slots, nullptr, nullptr, j.tc_workspace, status, &pub, q.e);
            if (rc != DP_OK) return rc;
            TcParams &p = q.e.p;
            if (j.bias_apart) { p.separate = 0; p.fold_slots = j.w_slots; }
            p.run = std::max(1, std::min(p.total_tiles, (int)(walk / pl.item_cycles)));
            p.blocks = q.blocks = (p.total_tiles + p.run - 1) / p.run;
            q.smem = pl.smem; q.cost = p.run * pl.item_cycles;
            store[j.dtype].jobs.push_back(q);
        } else if (j.kind == kConvClip1) {
            TcPlan pl; ConvGeom g1; bool s2d;
            if (!clip1_plan(j.dtype, j.g, pr, pl, g1, s2d)) return DP_ERR_UNSUPPORTED;
            // (small clusters wait for the sums' stream anyway)
            const int of = launch_cluster(pl.m_tiles * pl.n_tiles);
            rc = prepare_input(j.dtype, j.X, j.g, pr, s2d, j.tc_workspace, of > 4 || !streams.gram_done ? cluster_stream(of) : sums);
            if (rc != DP_OK) return rc;
            ConvQueue::Job q;
            rc = fill_clip1(j.dtype, j.X, j.dY, j.g, pr, g1, pl, s2d, j.clip, j.acc_w, j.tc_workspace, status, q.e);
            if (rc != DP_OK) return rc;
            TcParams &p = q.e.p;
            const int tiles = p.cluster, cluster = launch_cluster(tiles), sets = cluster / tiles;
            p.cluster = cluster;
            q.blocks = (p.splits + sets - 1) / sets * cluster;
            q.smem = pl.smem; q.cost = p.per_split * pl.item_cycles;
            if (p.splits > 1) folds[conv_cluster_stream(cluster, beside)].push_back(fold_seg(p.sum_out, p.splits, P, j.acc_w));
            clip[cluster].jobs.push_back(q);
        } else {
            const GramPlan gp = gram_plan(j.dtype, j.g);
            if (!gp.ok) return DP_ERR_UNSUPPORTED;
            GramQueue::Job q;
            rc = fill_gram(j.dtype, j.X, j.dY, gp, j.clip, j.factor, status, q.e);
            if (rc != DP_OK) return rc;
            q.blocks = q.e.p.blocks; q.smem = gp.smem;
            q.cost = (double)(g.Kout / 64 + g.R * g.S * (g.Cin / 64)) * gp.m_tiles * gp.rows;
            gram.jobs.push_back(q);
            if (j.kind == kConvGramTiles) {
                const TcPlan pl = make_plan(j.dtype, g, 7);
                ConvQueue::Job t;
                rc = fill_scaled_tiles(j.dtype, j.X, j.dY, g, pl, j.factor, j.acc_w, j.tc_workspace, status, t.e);
                if (rc != DP_OK) return rc;
                const TcParams &p = t.e.p;
                t.blocks = (p.blocks + 3) / 4 * 4;        // joins the launch of the smallest clusters; blocks past the last have no work
                t.smem = pl.smem; t.cost = p.per_split * pl.item_cycles;
                if (p.splits > 1) folds[BatchStreams::kMain].push_back(fold_seg(p.sum_out, p.splits, P, j.acc_w));
                clip[4].jobs.push_back(t);
            } else {
                const TcPlan pl = make_plan(j.dtype, g, 4);
                splits.push_back(split_seg(j.dY, j.factor, g, j.tc_workspace));
                SsumQueue::Job t;
                rc = fill_ssum(j.dtype, j.X, g, pl, j.acc_w, j.tc_workspace, status, t.e);
                if (rc != DP_OK) return rc;
                TcParams &p = t.e.p;
                t.blocks = p.blocks = p.total_tiles;
                t.smem = pl.smem; t.cost = p.per_split * pl.item_cycles;
                if (p.splits > 1) folds[BatchStreams::kSums].push_back(fold_seg(p.sum_out, p.splits, P, j.acc_w));
                ssum.jobs.push_back(t);
            }
        }
    }
    for (int dtype = 0; dtype < 3; ++dtype) {
        auto go = [&](const auto &tab, int blocks, size_t smem) -> dp_status {
            constexpr int N = std::extent<decltype(tab.first)>::value;
            const auto kernel = dtype == DP_BF16 ? conv_wgrad_tc_kernel<kBf16, false, N> : (dtype == DP_TF32 ? conv_wgrad_tc_kernel<kTf32, false, N> : conv_wgrad_tc_kernel<kSplit, false, N>);
            return launch_table(kernel, "conv_wgrad_tc_kernel", tab, blocks, dtype == DP_F32 ? 480 : 224, smem, stream);
        };
        rc = store[dtype].jobs.size() <= (size_t)kFewLayers ? store[dtype].launch<kFewLayers>(go) : store[dtype].launch<kTcLayers>(go);
        if (rc != DP_OK) return rc;
    }
    // The Gram matrices first: two more launches wait for them.  Larger clusters need all their SMs in one GPC, free at the same
    // time: behind smaller blocks they would be what the chunk ends with, so they come next, each size on a stream of its own.
    auto clip_launch = [&](int c) -> dp_status {
        return clip[c].launch([&](const TcTable<TcParams, 2, kTcLayers> &tab, int blocks, size_t smem) {
            return (beside ? launch_clip1_table<kTcLayers, true> : launch_clip1_table<kTcLayers>)(tab, c, blocks, smem, cluster_stream(c));
        });
    };
    if (rc == DP_OK)
        rc = gram.launch([&](const TcTable<GramParams, 2, kTcLayers> &tab, int blocks, size_t smem) -> dp_status {
            return launch_table(conv_gram_norm_kernel<kTcLayers>, "conv_gram_norm_kernel", tab, blocks, 192, smem, sums);
        });
    for (int c = kMaxCluster; c > 4 && rc == DP_OK; --c) rc = clip_launch(c);
    if (rc == DP_OK && streams.gram_done) {
        DP_CUDA_TRY(cudaEventRecord(streams.gram_done, sums));
        DP_CUDA_TRY(cudaStreamWaitEvent(stream, streams.gram_done, 0));
    }
    for (int c = 4; c >= 1 && rc == DP_OK; --c) rc = clip_launch(c);
    if (rc == DP_OK) rc = launch_scale_split(splits, sums);
    if (rc == DP_OK)
        rc = ssum.launch([&](const TcTable<TcParams, 3, kSsumLayers> &tab, int blocks, size_t smem) -> dp_status {
            return launch_table(conv_wgrad_ssum_kernel<kSsumLayers>, "conv_wgrad_ssum_kernel", tab, blocks, 224, smem, sums);
        });
    // (each stream folds its own: behind the join the fold would be alone on the GPU)
    for (int i = BatchStreams::kCount - 1; i >= 0 && rc == DP_OK; --i) rc = launch_folds(folds[i], streams.s[i]);
    return rc == DP_OK ? join() : rc;
}

}  // namespace dp
