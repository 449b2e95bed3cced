// Norm, clip and accumulate over materialised per-example gradients
// (paper section 2: sum over the batch of clip(g_j, C); section 3.5: per-group threshold C/sqrt(M)).
//
// Three memory-bound stages, all with fixed reduction orders:
//   1. (only when the caller has no norms) per-block partial sums of squares of every example row;
//   2. one small kernel folds the partials, a block per example, and turns squared norms into clip factors;
//   3. every thread owns four parameters, streams the B example rows through registers with 128-bit loads (or 32-bit
//      ones where the rows do not start on 16-byte boundaries), and touches the accumulator once.
// The tensors of a call travel in one table each launch: with 161 tensors in tables of 40 the two passes over 1.6 GB were
// ten launches, each with a last wave of its own, and took 590 us.
#include "common.cuh"
#include "philox.cuh"
#include "clip_rows.cuh"
#include <math.h>
#include <mutex>

namespace dp {

constexpr int kSmallTable = 16, kLargeTable = 512;   // tensors per launch (the table travels as a kernel parameter, 48 bytes each)
constexpr int kNormChunk = 8192;     // floats of one example row reduced by one block (stage 1)
constexpr int kAccCols = 1024;       // parameters per block in stage 3 (256 threads x float4)

template <int N>
struct SegTable {
    const float *G[N];               // [B, P] per tensor
    float *acc[N];                   // [P] per tensor
    long long P[N];
    long long part_start[N];         // first partial slot of each tensor within one example's row of partials
    long long goff[N];               // global index of the tensor's first parameter (per-example noise only)
    int blk_start[N];                // first block of each tensor within this launch
    int col0;                        // index in the [B, L] norm / factor tables of the first of these consecutive tensors
    int nseg;
};

// Per-example noise (the paper's own implementation, section 2, the block after the equation for g_t):
// example e of the step adds sd * z_e(g), sd = sigma*C/sqrt(|B|), to its clipped gradient before the sum.
struct ExampleNoise {
    float sd;
    NoiseStream ns;
    uint32_t example0;               // index within the step of this chunk's first example
};

template <int N>
__device__ __forceinline__ int find_seg(const SegTable<N> &t, int blk) {
    int lo = 0, hi = t.nseg;                                  // the last tensor whose first block is not past blk
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (blk >= t.blk_start[mid]) lo = mid; else hi = mid; }
    return lo;
}

// stage 1: partial[n][part_start[seg] + j] = sum of squares of G_seg[n, j*chunk .. (j+1)*chunk); up to three floats before
// the first 16-byte boundary and after the last one are read alone
template <int AHEAD, int N>
__device__ __forceinline__ void sqnorm_partial(const SegTable<N> &tab, int blk, int n, float *__restrict__ partial, long long parts_per_example) {
    __shared__ float scratch[32];
    const int seg = find_seg(tab, blk);
    const int j = blk - tab.blk_start[seg];
    const long long P = tab.P[seg];
    const long long c0 = (long long)j * kNormChunk;
    const int len = (int)min((long long)kNormChunk, P - c0);
    const float *row = tab.G[seg] + (long long)n * P + c0;
    const int head = min(len, (int)((0u - (unsigned)(reinterpret_cast<uintptr_t>(row) >> 2)) & 3u));
    const float4 *row4 = reinterpret_cast<const float4 *>(row + head);
    const int n4 = (len - head) >> 2, tail = head + 4 * n4;
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    for (int i = threadIdx.x; i < n4; i += 256 * AHEAD) {                    // AHEAD loads in flight a thread
        float4 v[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i + 256 * u < n4) v[u] = __ldg(row4 + i + 256 * u);
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            a0 = fmaf(v[u].x, v[u].x, a0); a1 = fmaf(v[u].y, v[u].y, a1); a2 = fmaf(v[u].z, v[u].z, a2); a3 = fmaf(v[u].w, v[u].w, a3);
        }
    }
    if ((int)threadIdx.x < head) a0 = fmaf(row[threadIdx.x], row[threadIdx.x], a0);
    if (tail + (int)threadIdx.x < len) a1 = fmaf(row[tail + threadIdx.x], row[tail + threadIdx.x], a1);
    const float a = block_sum((a0 + a1) + (a2 + a3), scratch);
    if (threadIdx.x == 0) partial[(long long)n * parts_per_example + tab.part_start[seg] + j] = a;
}

template <int N>
__global__ void __launch_bounds__(256)
sqnorm_partial_kernel(const __grid_constant__ SegTable<N> tab, float *__restrict__ partial, long long parts_per_example) {
    sqnorm_partial<4>(tab, blockIdx.x, blockIdx.y, partial, parts_per_example);
}

// stage 1 for micro-batch clipping: row j of the partials belongs to the MEAN of examples j*micro .. j*micro+micro-1
// (the unit that is clipped), so the rows are added before they are squared.
template <int N>
__global__ void __launch_bounds__(256)
sqnorm_partial_micro_kernel(const __grid_constant__ SegTable<N> tab, float *__restrict__ partial,
                            long long parts_per_example, int micro) {
    __shared__ float scratch[32];
    const int seg = find_seg(tab, blockIdx.x);
    const int j = blockIdx.x - tab.blk_start[seg];
    const long long P = tab.P[seg];
    const long long c0 = (long long)j * kNormChunk;
    const int len = (int)min((long long)kNormChunk, P - c0);
    const float *row = tab.G[seg] + (long long)blockIdx.y * micro * P + c0;
    const float inv = 1.0f / (float)micro;
    // loads of a row side by side, whatever `micro` is: rows at any address word by word (4.4 M parameters, three pairs of
    // examples: 68 us the pass with a word at a time, 21; 25.6 M aligned ones, eight pairs: 313 and 252)
    constexpr int kVecs = 4, kWords = 8;
    float a = 0.f;
    if (((reinterpret_cast<uintptr_t>(row) | (uintptr_t)(P * 4)) & 15) == 0) {
        const int n4 = len >> 2;
        for (int i = threadIdx.x; i < n4; i += 256 * kVecs) {
            float4 v[kVecs];
#pragma unroll
            for (int u = 0; u < kVecs; ++u) v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int r = 0; r < micro; ++r) {
                float4 x[kVecs];
#pragma unroll
                for (int u = 0; u < kVecs; ++u) {
                    x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i + 256 * u < n4) x[u] = __ldg(reinterpret_cast<const float4 *>(row + (long long)r * P) + i + 256 * u);
                }
#pragma unroll
                for (int u = 0; u < kVecs; ++u) { v[u].x += x[u].x; v[u].y += x[u].y; v[u].z += x[u].z; v[u].w += x[u].w; }
            }
#pragma unroll
            for (int u = 0; u < kVecs; ++u) {
                v[u].x *= inv; v[u].y *= inv; v[u].z *= inv; v[u].w *= inv;
                a = fmaf(v[u].x, v[u].x, a); a = fmaf(v[u].y, v[u].y, a); a = fmaf(v[u].z, v[u].z, a); a = fmaf(v[u].w, v[u].w, a);
            }
        }
        for (int i = (n4 << 2) + threadIdx.x; i < len; i += 256) {
            float v = 0.f;
            for (int r = 0; r < micro; ++r) v += row[(long long)r * P + i];
            v *= inv;
            a = fmaf(v, v, a);
        }
    } else {
        for (int i = threadIdx.x; i < len; i += 256 * kWords) {
            float v[kWords];
#pragma unroll
            for (int u = 0; u < kWords; ++u) v[u] = 0.f;
#pragma unroll 2
            for (int r = 0; r < micro; ++r) {
                float x[kWords];
#pragma unroll
                for (int u = 0; u < kWords; ++u) { x[u] = 0.f; if (i + 256 * u < len) x[u] = __ldg(row + (long long)r * P + i + 256 * u); }
#pragma unroll
                for (int u = 0; u < kWords; ++u) v[u] += x[u];
            }
#pragma unroll
            for (int u = 0; u < kWords; ++u) { v[u] *= inv; a = fmaf(v[u], v[u], a); }
        }
    }
    a = block_sum(a, scratch);
    if (threadIdx.x == 0) partial[(long long)blockIdx.y * parts_per_example + tab.part_start[seg] + j] = a;
}

// stage 2.  A block per row (an example, or a micro-batch): folds the partials of this launch's tensors to squared norms,
// in floats that carry their rounding errors along, and after the last table turns the row's norms into factors.  A squared
// norm past the range of float is infinite, and its factor zero.
//   kGlobal   one factor from the sum over the L tensors; the `micro` examples of the row each carry factor / micro, so that
//             stage 3 adds factor * mean
//   kPerLayer one factor per tensor against C/sqrt(L)
//   kGrouped  one factor per group of tensors (section 3.5: M pipeline stages, each clipped to C/sqrt(M))
// A latency chain: many small loads, so they go side by side over a large block, and what every lane reads elsewhere is in
// shared memory (161 tensors of 16 examples in four groups: 30 us with eight warps and the table read from the parameters).
enum { kGlobal = 0, kPerLayer, kGrouped };
constexpr int kFactorThreads = 1024;
constexpr int kPartsPerWarp = 512;                   // tensors with more partials are folded by the whole block
constexpr int kMaxGroupedTensors = 1024;
struct GroupTable {
    int M;
    unsigned short of[kMaxGroupedTensors];   // group of tensor l
};
template <int N, int KIND>
__global__ void __launch_bounds__(kFactorThreads)
norm_factor_kernel(const __grid_constant__ SegTable<N> tab, const float *__restrict__ partial, long long parts_per_row,
                   const float *sq_in, float *sq_ws, int L, int micro, int last, float C, const __grid_constant__ GroupTable gt,
                   float *__restrict__ factor, float *norms_out, float *clip_out) {
    __shared__ double scratch[32];
    __shared__ int large;                                // a tensor of this table is left to the whole block
    __shared__ float f_sh[KIND == kGrouped ? kMaxGroupedTensors : 1];
    __shared__ unsigned short of_sh[KIND == kGrouped ? kMaxGroupedTensors : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long row = blockIdx.x;
    if (KIND == kGrouped) {                              // (read below, behind a barrier)
        for (int l = threadIdx.x; l < L; l += kFactorThreads) of_sh[l] = gt.of[l];
    }
    if (partial) {
        float *out = sq_ws + row * L + tab.col0;
        if (threadIdx.x == 0) large = 0;
        __syncthreads();
        for (int s = w; s < tab.nseg; s += kFactorThreads / 32) {
            const int nparts = (int)((tab.P[s] + kNormChunk - 1) / kNormChunk);
            if (nparts > kPartsPerWarp) { large = 1; continue; }
            const float *p = partial + row * parts_per_row + tab.part_start[s];
            Sum2 a;
#pragma unroll 8
            for (int i = lane; i < nparts; i += 32) a.add(p[i]);
            a = warp_sum(a);
            if (lane == 0) out[s] = (float)a.value();
        }
        __syncthreads();
        for (int s = 0; large && s < tab.nseg; ++s) {
            const int nparts = (int)((tab.P[s] + kNormChunk - 1) / kNormChunk);
            if (nparts <= kPartsPerWarp) continue;
            const float *p = partial + row * parts_per_row + tab.part_start[s];
            Sum2 a;
#pragma unroll 4
            for (int i = threadIdx.x; i < nparts; i += kFactorThreads) a.add(p[i]);
            const double t = block_sum(a.value(), scratch);
            if (threadIdx.x == 0) out[s] = (float)t;
        }
        if (!last) return;
    }
    __syncthreads();                                     // the norms written above are read below, by other threads of the block
    const float *sq = (partial ? sq_ws : sq_in) + row * L;
    if (KIND == kGlobal) {
        double s = 0.0;
        for (int l = threadIdx.x; l < L; l += kFactorThreads) s += (double)sq[l];
        s = block_sum(s, scratch);
        const float f = clip_factor(s, C), each = micro == 1 ? f : f / (float)micro;
        for (int i = threadIdx.x; i < micro; i += kFactorThreads) factor[row * micro + i] = each;
        if (threadIdx.x == 0) {
            if (norms_out) norms_out[row] = (float)sqrt(s);
            if (clip_out) clip_out[row] = f;
        }
    } else if (KIND == kPerLayer) {
        const float thr = (float)((double)C / sqrt((double)L));
        for (int l = threadIdx.x; l < L; l += kFactorThreads) {
            const double s = (double)sq[l];
            const float f = clip_factor(s, thr);
            factor[row * L + l] = f;
            if (norms_out) norms_out[row * L + l] = (float)sqrt(s);
            if (clip_out) clip_out[row * L + l] = f;
        }
    } else {
        const float thr = (float)((double)C / sqrt((double)gt.M));
        for (int m = w; m < gt.M; m += kFactorThreads / 32) {
            Sum2 sum;
            for (int l = lane; l < L; l += 32)
                if (of_sh[l] == m) sum.add(sq[l]);
            sum = warp_sum(sum);                         // (its `hi` is the same in all lanes)
            double s = sum.value();
            if (!sum.fits()) {                           // the tensors' norms fit floats, their sum need not
                s = 0.0;
                for (int l = lane; l < L; l += 32)
                    if (of_sh[l] == m) s += (double)sq[l];
                s = warp_sum(s);
            }
            if (lane == 0) {
                const float f = clip_factor(s, thr);
                f_sh[m] = f;
                if (norms_out) norms_out[row * gt.M + m] = (float)sqrt(s);
                if (clip_out) clip_out[row * gt.M + m] = f;
            }
        }
        __syncthreads();
        for (int l = threadIdx.x; l < L; l += kFactorThreads) factor[row * L + l] = f_sh[of_sh[l]];
    }
}

// stage 2 with the norms given and few of them a row: a thread per example (kGlobal) or per norm (kPerLayer)
constexpr int kFewTensors = 32;
__global__ void clip_factor_kernel(const float *__restrict__ sq, int B, int L, int per_layer, float C,
                                   float *__restrict__ factor, float *norms_out, float *clip_out) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (per_layer ? B * L : B)) return;
    const float thr = per_layer ? (float)((double)C / sqrt((double)L)) : C;
    double s = 0.0;
    if (per_layer) s = (double)sq[idx];
    else
        for (int l = 0; l < L; ++l) s += (double)sq[(long long)idx * L + l];
    const float f = clip_factor(s, thr);
    factor[idx] = f;
    if (norms_out) norms_out[idx] = (float)sqrt(s);
    if (clip_out) clip_out[idx] = f;
}

// Few norms of few examples given: every block of stage 3 works the factors out itself instead of waiting for a launch that
// does (a warp's worth of double divisions and roots, some half a microsecond, against two for a launch).
constexpr int kInlineExamples = 32;
struct InlineFactors {
    const float *sq;                 // [B, L]; null: the factors are given
    float C;
    float *factor, *norms_out, *clip_out;
};
__device__ __forceinline__ void stage_factors(float *f_sh, const float *factor, int n0, int nb, int L, int stride, int off, const InlineFactors &in) {
    const int t = threadIdx.x;
    if (t >= nb) return;
    if (!in.sq) { f_sh[t] = factor[(long long)(n0 + t) * stride + off]; return; }
    double s = 0.0;
    for (int l = 0; l < L; ++l) s += (double)in.sq[(n0 + t) * L + l];
    const float f = clip_factor(s, in.C);
    f_sh[t] = f;
    if (blockIdx.x) return;
    in.factor[n0 + t] = f;
    if (in.norms_out) in.norms_out[n0 + t] = (float)sqrt(s);
    if (in.clip_out) in.clip_out[n0 + t] = f;
}

// stage 3: acc[i] += sum_n factor * G[n, i].  factor index: GLOBAL n, PER_LAYER n*L + col.  Streams B*P floats once; loads
// past the L1 (evict-first: nothing comes back).
template <int N>
__global__ void __launch_bounds__(256)
scale_accumulate_kernel(const __grid_constant__ SegTable<N> tab, const float *__restrict__ factor, int B, int L,
                        int per_layer, const __grid_constant__ InlineFactors in) {
    constexpr int kRows = 8;                                   // rows in flight per thread
    __shared__ float f_sh[256];
    const int seg = find_seg(tab, blockIdx.x);
    const long long P = tab.P[seg];
    const long long c0 = (long long)(blockIdx.x - tab.blk_start[seg]) * kAccCols;
    const float *G = tab.G[seg];
    float *acc = tab.acc[seg];
    const int f_stride = per_layer ? L : 1;
    const int f_off = per_layer ? tab.col0 + seg : 0;
    // vector path needs every row start 16-byte aligned: base aligned and P a multiple of 4
    const bool vec = ((P & 3) == 0) && ((reinterpret_cast<uintptr_t>(G) & 15) == 0) &&
                     ((reinterpret_cast<uintptr_t>(acc) & 15) == 0);
    if (vec) {
        const long long i = c0 + 4 * threadIdx.x;
        const bool live = i < P;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int n0 = 0; n0 < B; n0 += 256) {
            const int nb = min(256, B - n0);
            __syncthreads();
            stage_factors(f_sh, factor, n0, nb, L, f_stride, f_off, in);
            __syncthreads();
            if (live) {
                const float *g = G + (long long)n0 * P + i;
                for (int n = 0; n < nb; n += kRows) {
                    float4 v[kRows];
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (n + u < nb) v[u] = __ldcs(reinterpret_cast<const float4 *>(g + (long long)(n + u) * P));
                    }
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        const float f = n + u < nb ? f_sh[n + u] : 0.f;
                        s.x = fmaf(f, v[u].x, s.x); s.y = fmaf(f, v[u].y, s.y);
                        s.z = fmaf(f, v[u].z, s.z); s.w = fmaf(f, v[u].w, s.w);
                    }
                }
            }
        }
        if (live) {
            float4 a = *reinterpret_cast<const float4 *>(acc + i);
            a.x += s.x; a.y += s.y; a.z += s.z; a.w += s.w;
            *reinterpret_cast<float4 *>(acc + i) = a;
        }
    } else {
        // rows at any address: columns 256 apart, so that the lanes of a load are neighbours wherever the row starts
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const long long left = P - c0 - threadIdx.x;           // column q of this thread exists when 256 q < left
        for (int n0 = 0; n0 < B; n0 += 256) {
            const int nb = min(256, B - n0);
            __syncthreads();
            stage_factors(f_sh, factor, n0, nb, L, f_stride, f_off, in);
            __syncthreads();
            const float *g = G + (long long)n0 * P + c0 + threadIdx.x;
            for (int n = 0; n < nb; n += kRows) {
                float v[kRows][4];
#pragma unroll
                for (int u = 0; u < kRows; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        v[u][q] = 0.f;
                        if (n + u < nb && 256 * q < left) v[u][q] = __ldcs(g + (long long)(n + u) * P + 256 * q);
                    }
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    const float f = n + u < nb ? f_sh[n + u] : 0.f;
#pragma unroll
                    for (int q = 0; q < 4; ++q) s[q] = fmaf(f, v[u][q], s[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (256 * q < left) acc[c0 + threadIdx.x + 256 * q] += s[q];
    }
}

// stage 3 for small models with many examples: too few 1024-parameter blocks exist to fill the GPU, so a block takes
// only 128 parameters and splits the example rows over its eight warps (warp w owns every eighth row), eight rows in
// flight per thread; the eight partial sums are folded in warp order through shared memory.  The blocks are all resident
// or nearly so and walk the examples from the last to the first: stage 1 read those rows last, so that most of a gradient
// up to twice the L2 is still there (256 rows of 175 178 floats, which start at any address: 103 us for the call with four
// words at a time of one row a thread, in ascending order).
constexpr int kSplitCols = 128;
template <int N>
__global__ void __launch_bounds__(256)
scale_accumulate_rowsplit_kernel(const __grid_constant__ SegTable<N> tab, const float *__restrict__ factor, int B, int L,
                                 int per_layer, const __grid_constant__ InlineFactors in) {
    constexpr int kRows = 8;
    __shared__ float f_sh[256];
    __shared__ float part[8][kSplitCols];
    const int seg = find_seg(tab, blockIdx.x);
    const long long P = tab.P[seg];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long c0 = (long long)(blockIdx.x - tab.blk_start[seg]) * kSplitCols;
    const float *G = tab.G[seg];
    float *acc = tab.acc[seg];
    const int f_stride = per_layer ? L : 1;
    const int f_off = per_layer ? tab.col0 + seg : 0;
    const bool vec = ((P & 3) == 0) && ((reinterpret_cast<uintptr_t>(G) & 15) == 0);
    // vec: four neighbouring columns of this lane, all or none; otherwise columns 32 apart
    const long long left = P - c0 - (vec ? 4 * lane : lane);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int n0 = (B - 1) & ~255; n0 >= 0; n0 -= 256) {
        const int nb = min(256, B - n0);
        __syncthreads();
        stage_factors(f_sh, factor, n0, nb, L, f_stride, f_off, in);
        __syncthreads();
        if (left <= 0) continue;
        const float *g = G + (long long)n0 * P + c0 + (vec ? 4 * lane : lane);
        for (int n = nb - 1 - w; n >= 0; n -= 8 * kRows) {
            float v[kRows][4];
            if (vec) {
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (n - 8 * u >= 0) x = __ldcs(reinterpret_cast<const float4 *>(g + (long long)(n - 8 * u) * P));
                    v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
                }
            } else {
#pragma unroll
                for (int u = 0; u < kRows; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        v[u][q] = 0.f;
                        if (n - 8 * u >= 0 && 32 * q < left) v[u][q] = __ldcs(g + (long long)(n - 8 * u) * P + 32 * q);
                    }
            }
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                const float f = n - 8 * u >= 0 ? f_sh[n - 8 * u] : 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) s[q] = fmaf(f, v[u][q], s[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) part[w][vec ? 4 * lane + q : lane + 32 * q] = s[q];
    __syncthreads();
    if (threadIdx.x < kSplitCols && c0 + threadIdx.x < P) {
        float t = part[0][threadIdx.x];
#pragma unroll
        for (int q = 1; q < 8; ++q) t += part[q][threadIdx.x];
        acc[c0 + threadIdx.x] += t;
    }
}

// stage 3 with per-example noise: acc[i] += sum_n ( factor * G[n, i] + sd * z_{example0+n}(goff + i) ).
// Every thread owns the up to four parameters of one Philox block that lie in the tensor, wherever it starts; the rows are
// read 16 bytes at a time where they start on 16-byte boundaries, else word by word.  Bound by the integer and
// transcendental work of B*P normals, not by memory (18.8 M parameters of five examples with rows at any address took
// 673 us with a Philox block for every parameter).
struct PhiloxLane {                          // this thread's parameters [i + k0, i + k1) of the tensor
    long long i;
    int k0, k1;
    uint32_t block;
    __device__ __forceinline__ PhiloxLane(long long tile, long long goff, long long P) {
        i = tile * kAccCols + 4 * threadIdx.x - (goff & 3);
        k0 = i < 0 ? (int)-i : 0;
        k1 = (int)max(0ll, min(4ll, P - i));
        block = (uint32_t)((unsigned long long)(goff + i) >> 2);
    }
    __device__ __forceinline__ bool live() const { return k1 > k0; }
    template <bool VEC>
    __device__ __forceinline__ float4 load(const float *p) const {
        if (VEC) return __ldcs(reinterpret_cast<const float4 *>(p));
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k0 == 0) v.x = __ldcs(p);
        if (k0 <= 1 && k1 > 1) v.y = __ldcs(p + 1);
        if (k0 <= 2 && k1 > 2) v.z = __ldcs(p + 2);
        if (k1 > 3) v.w = __ldcs(p + 3);
        return v;
    }
    __device__ __forceinline__ void add(float *acc, const float4 &s, bool vec) const {
        if (vec) {
            float4 a = *reinterpret_cast<const float4 *>(acc + i);
            a.x += s.x; a.y += s.y; a.z += s.z; a.w += s.w;
            *reinterpret_cast<float4 *>(acc + i) = a;
            return;
        }
        if (k0 == 0) acc[i] += s.x;
        if (k0 <= 1 && k1 > 1) acc[i + 1] += s.y;
        if (k0 <= 2 && k1 > 2) acc[i + 2] += s.z;
        if (k1 > 3) acc[i + 3] += s.w;
    }
};
template <int N>
__device__ __forceinline__ bool noise_vec(const SegTable<N> &tab, int seg) {
    return ((tab.P[seg] & 3) == 0) && ((tab.goff[seg] & 3) == 0) && ((reinterpret_cast<uintptr_t>(tab.G[seg]) & 15) == 0) &&
           ((reinterpret_cast<uintptr_t>(tab.acc[seg]) & 15) == 0);
}
static long long noise_tiles(long long P, long long goff) { return (P + (goff & 3) + kAccCols - 1) / kAccCols; }

__device__ __forceinline__ void noised_row(float4 &s, float f, const float4 &v, const PhiloxLane &me, bool noisy, uint32_t example, const ExampleNoise &nz) {
    if (noisy) {
        float z[4];
        example_normals4(nz.ns, example, me.block, z);
        s.x += fmaf(f, v.x, nz.sd * z[0]); s.y += fmaf(f, v.y, nz.sd * z[1]); s.z += fmaf(f, v.z, nz.sd * z[2]); s.w += fmaf(f, v.w, nz.sd * z[3]);
    } else {
        s.x = fmaf(f, v.x, s.x); s.y = fmaf(f, v.y, s.y); s.z = fmaf(f, v.z, s.z); s.w = fmaf(f, v.w, s.w);
    }
}
// rows n0 .. n0 + nb of one tensor, four at a time (`g`: this thread's place in row n0)
template <bool VEC>
__device__ __forceinline__ void noised_rows(float4 &s, const float *g, const float *f_sh, int n0, int nb, long long P, const PhiloxLane &me,
                                            int odd_only, const ExampleNoise &nz) {
    int n = 0;
    for (; n + 4 <= nb; n += 4) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = me.load<VEC>(g + (long long)(n + u) * P);
#pragma unroll
        for (int u = 0; u < 4; ++u) noised_row(s, f_sh[n + u], v[u], me, (u & 1) || !odd_only, nz.example0 + (uint32_t)(n0 + n + u), nz);
    }
    for (; n < nb; ++n)
        noised_row(s, f_sh[n], me.load<VEC>(g + (long long)n * P), me, (n & 1) || !odd_only, nz.example0 + (uint32_t)(n0 + n), nz);
}

template <int N>
__global__ void __launch_bounds__(256, 6)
scale_accumulate_noised_kernel(const __grid_constant__ SegTable<N> tab, const float *__restrict__ factor, int B, int L,
                               int per_layer, int odd_only, const __grid_constant__ ExampleNoise nz) {
    __shared__ float f_sh[256];
    const int seg = find_seg(tab, blockIdx.x);
    const long long P = tab.P[seg];
    const int f_stride = per_layer ? L : 1;
    const int f_off = per_layer ? tab.col0 + seg : 0;
    const bool vec = noise_vec(tab, seg);
    const PhiloxLane me(blockIdx.x - tab.blk_start[seg], tab.goff[seg], P);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int n0 = 0; n0 < B; n0 += 256) {
        const int nb = min(256, B - n0);
        __syncthreads();
        if (threadIdx.x < nb) f_sh[threadIdx.x] = factor[(long long)(n0 + threadIdx.x) * f_stride + f_off];
        __syncthreads();
        if (!me.live()) continue;
        const float *g = tab.G[seg] + (long long)n0 * P + me.i;
        if (vec) noised_rows<true>(s, g, f_sh, n0, nb, P, me, odd_only, nz);
        else noised_rows<false>(s, g, f_sh, n0, nb, P, me, odd_only, nz);
    }
    if (me.live()) me.add(tab.acc[seg], s, vec);
}

// Stage 1 with half of the per-example noise: the norm pass waits for memory and the noise for the issue slots, and a draw
// does not depend on its example's factor.  So the even examples' draws are added here, acc[i] += sd * sum_n z_n(goff + i),
// by blocks spread evenly among those of the norms (every (ratio + 1)-th), the odd examples' in stage 3 (8 M parameters, 32
// examples: norms 152 us, then all of the draws with the scaled sum 363; this way 255 and 220;
// with the pairs of a draw packed, six blocks an SM in both and eight loads in flight in the blocks of norms, whose few places an SM
// are what the pass waits for, 227 and 196).
template <int N>
struct NoiseStarts { int first[N]; };                          // first noise block of each tensor, tiles of kAccCols parameters
template <int N>
__global__ void __launch_bounds__(256, 6)
sqnorm_noise_kernel(const __grid_constant__ SegTable<N> tab, float *__restrict__ partial, long long parts_per_example, int norm_blocks,
                    int B, int noise_blocks, int ratio, const __grid_constant__ NoiseStarts<N> starts, const __grid_constant__ ExampleNoise nz) {
    const int idx = blockIdx.x, turn = idx / (ratio + 1);
    if (turn >= noise_blocks || idx - turn * (ratio + 1) != ratio) {
        const int blk = idx - min(noise_blocks, turn), n = blk / norm_blocks;
        sqnorm_partial<8>(tab, blk - n * norm_blocks, n, partial, parts_per_example);
        return;
    }
    int lo = 0, hi = tab.nseg;
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (turn >= starts.first[mid]) lo = mid; else hi = mid; }
    const PhiloxLane me(turn - starts.first[lo], tab.goff[lo], tab.P[lo]);
    if (!me.live()) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int n = 0; n < B; n += 2) {
        float z[4];
        example_normals4(nz.ns, nz.example0 + (uint32_t)n, me.block, z);
        s.x = fmaf(nz.sd, z[0], s.x); s.y = fmaf(nz.sd, z[1], s.y); s.z = fmaf(nz.sd, z[2], s.z); s.w = fmaf(nz.sd, z[3], s.w);
    }
    me.add(tab.acc[lo], s, noise_vec(tab, lo));
}

struct ClipPlan {
    size_t partial_off, sq_off, factor_off, total;
    long long parts_per_example;
};

static bool plan(int B, int L, const long long *P_l, ClipPlan &pl) {
    long long parts = 0;
    for (int l = 0; l < L; ++l) {
        if (P_l[l] <= 0) return false;
        parts += (P_l[l] + kNormChunk - 1) / kNormChunk;
    }
    pl.parts_per_example = parts;
    size_t off = 0;
    pl.partial_off = off; off = round_up(off + sizeof(float) * (size_t)parts * B, 256);
    pl.sq_off = off;      off = round_up(off + sizeof(float) * (size_t)B * L, 256);
    pl.factor_off = off;  off = round_up(off + sizeof(float) * (size_t)B * L, 256);
    pl.total = off;
    return true;
}

// One tensor whose rows fit the registers of a cluster goes through them in a single read (clip_rows.cu), where its norms
// are to be computed and the workspace holds the clusters' sums behind the rest.
static bool single_read(int B, int L, const long long *P_l) { return L == 1 && clip_rows_eligible(B, P_l[0]); }

}  // namespace dp

extern "C" size_t dp_clip_workspace_bytes(int B, int L, const long long *P_l) {
    dp::ClipPlan pl;
    if (B <= 0 || L <= 0 || !P_l || !dp::plan(B, L, P_l, pl)) return 0;
    return pl.total + (dp::single_read(B, L, P_l) ? dp::clip_rows_workspace_bytes(B, P_l[0]) : 0);
}

namespace dp {
// What differs from plain dp_clip_accumulate in the other entry points.
struct ClipVariant {
    const ExampleNoise *noise = nullptr;   // stage 3 also adds each example's own noise draw ...
    const long long *goff_l = nullptr;     // ... addressed by the tensors' global offsets
    const GroupTable *groups = nullptr;    // factors per (example, group of tensors) instead of per tensor
    int micro = 1;                         // examples averaged before clipping
    const float *given_factor = nullptr;   // stage 3 only, with the caller's factors ([B] or [B, L]); no workspace
};

struct ClipCall {
    int B, L, per_layer;
    const float *const *G;
    const long long *P_l;
    float *const *acc;
    const float *sq;                       // given squared norms, or null: `partial` and `sq_ws` receive them
    float *partial, *sq_ws, *factor_ws;
    const float *factor;
    float C;
    float *norms_out, *clip_out;
    long long parts_per_example;
};

static dp_status launch_factors(const ClipCall &c, const ClipVariant &var, cudaStream_t stream);

// The launches of one call, its tensors in tables of N.
template <int N>
static dp_status clip_launches(const ClipCall &c, const ClipVariant &var, cudaStream_t stream) {
    const int B = c.B, L = c.L, micro = var.micro;
    // A small model gives few wide blocks, and each thread would walk all B rows alone: with many rows the block narrows
    // to 128 parameters and its warps share the rows (from two rows a warp on where not even two wide blocks an SM exist,
    // from eight on up to a wave of them).
    long long wide_blocks = 0;
    for (int l = 0; l < L; ++l) wide_blocks += (c.P_l[l] + kAccCols - 1) / kAccCols;
    const bool split = !var.noise && ((B >= 64 && wide_blocks < 8 * sm_count()) || (B >= 16 && wide_blocks < 2 * sm_count()));
    const int acc_cols = split ? kSplitCols : kAccCols;

    // half of the noise goes with the norm pass where there is one, with at least a block of norms to each of noise
    const bool halved = var.noise && !c.sq && !var.given_factor && B >= 9 && (wide_blocks + L) * (B + 1) <= 0x7fffffffll;

    SegTable<N> t;
    auto fill = [&](int l0, bool norm_blocks, long long &part_cursor) {
        t.nseg = 0; t.col0 = l0;
        int blk = 0;
        for (int l = l0; l < L && t.nseg < N; ++l) {
            const int s = t.nseg;
            const long long nparts = (c.P_l[l] + kNormChunk - 1) / kNormChunk;
            const long long nb = norm_blocks ? nparts : (var.noise ? noise_tiles(c.P_l[l], var.goff_l[l]) : (c.P_l[l] + acc_cols - 1) / acc_cols);
            if ((long long)blk + nb > 0x7fffffffll) break;
            t.G[s] = c.G[l]; t.acc[s] = c.acc[l]; t.P[s] = c.P_l[l];
            t.goff[s] = var.goff_l ? var.goff_l[l] : 0;
            t.blk_start[s] = blk; t.part_start[s] = part_cursor;
            part_cursor += nparts; blk += (int)nb; ++t.nseg;
        }
        return blk;
    };
    InlineFactors in = {};
    if (!var.given_factor && c.sq && !var.noise && !var.groups && !c.per_layer && B <= kInlineExamples && L <= kFewTensors) {
        in = InlineFactors{c.sq, c.C, c.factor_ws, c.norms_out, c.clip_out};
    } else if (!var.given_factor && c.sq) {
        const dp_status rc = launch_factors(c, var, stream);
        if (rc != DP_OK) return rc;
    } else if (!var.given_factor) {
        long long cursor = 0;
        const unsigned rows = (unsigned)(B / micro);
        for (int l0 = 0; l0 < L; l0 += t.nseg) {
            const int blocks = fill(l0, true, cursor);
            if (t.nseg == 0) return DP_ERR_UNSUPPORTED;
            if (micro > 1) sqnorm_partial_micro_kernel<N><<<dim3((unsigned)blocks, rows), 256, 0, stream>>>(t, c.partial, c.parts_per_example, micro);
            else if (halved) {
                NoiseStarts<N> starts;
                long long tiles = 0;
                for (int s = 0; s < t.nseg; ++s) { starts.first[s] = (int)tiles; tiles += noise_tiles(t.P[s], t.goff[s]); }
                const int ratio = (int)((long long)blocks * B / tiles);       // at least one: a block of norms covers at most nine tiles
                sqnorm_noise_kernel<N><<<(unsigned)((long long)blocks * B + tiles), 256, 0, stream>>>(t, c.partial, c.parts_per_example, blocks, B, (int)tiles, ratio, starts, *var.noise);
            } else sqnorm_partial_kernel<N><<<dim3((unsigned)blocks, rows), 256, 0, stream>>>(t, c.partial, c.parts_per_example);
            DP_LAUNCH_CHECK("sqnorm_partial_kernel");
            const int last = l0 + t.nseg == L;
            static const GroupTable none = {};
            const GroupTable &gt = var.groups ? *var.groups : none;
            if (var.groups)
                norm_factor_kernel<N, kGrouped><<<rows, kFactorThreads, 0, stream>>>(t, c.partial, c.parts_per_example, nullptr, c.sq_ws, L, micro, last, c.C, gt, c.factor_ws, c.norms_out, c.clip_out);
            else if (c.per_layer)
                norm_factor_kernel<N, kPerLayer><<<rows, kFactorThreads, 0, stream>>>(t, c.partial, c.parts_per_example, nullptr, c.sq_ws, L, micro, last, c.C, gt, c.factor_ws, c.norms_out, c.clip_out);
            else
                norm_factor_kernel<N, kGlobal><<<rows, kFactorThreads, 0, stream>>>(t, c.partial, c.parts_per_example, nullptr, c.sq_ws, L, micro, last, c.C, gt, c.factor_ws, c.norms_out, c.clip_out);
            DP_LAUNCH_CHECK("norm_factor_kernel");
        }
    }
    long long cursor = 0;
    for (int l0 = 0; l0 < L; l0 += t.nseg) {
        const int blocks = fill(l0, false, cursor);
        if (t.nseg == 0) return DP_ERR_UNSUPPORTED;
        if (var.noise) scale_accumulate_noised_kernel<N><<<(unsigned)blocks, 256, 0, stream>>>(t, c.factor, B, L, c.per_layer, halved, *var.noise);
        else if (split) scale_accumulate_rowsplit_kernel<N><<<(unsigned)blocks, 256, 0, stream>>>(t, c.factor, B, L, c.per_layer, in);
        else scale_accumulate_kernel<N><<<(unsigned)blocks, 256, 0, stream>>>(t, c.factor, B, L, c.per_layer, in);
        DP_LAUNCH_CHECK("scale_accumulate_kernel");
    }
    return DP_OK;
}

// stage 2 from given squared norms
static dp_status launch_factors(const ClipCall &c, const ClipVariant &var, cudaStream_t stream) {
    const bool few = !var.groups && (c.per_layer || c.L <= kFewTensors);
    if (few) {
        const long long count = c.per_layer ? (long long)c.B * c.L : c.B;
        clip_factor_kernel<<<(unsigned)((count + 127) / 128), 128, 0, stream>>>(c.sq, c.B, c.L, c.per_layer, c.C, c.factor_ws, c.norms_out, c.clip_out);
    } else {
        SegTable<1> t;
        t.nseg = 0; t.col0 = 0;
        static const GroupTable none = {};
        if (var.groups)
            norm_factor_kernel<1, kGrouped><<<(unsigned)c.B, kFactorThreads, 0, stream>>>(t, nullptr, 0, c.sq, nullptr, c.L, 1, 1, c.C, *var.groups, c.factor_ws, c.norms_out, c.clip_out);
        else
            norm_factor_kernel<1, kGlobal><<<(unsigned)c.B, kFactorThreads, 0, stream>>>(t, nullptr, 0, c.sq, nullptr, c.L, 1, 1, c.C, none, c.factor_ws, c.norms_out, c.clip_out);
    }
    DP_LAUNCH_CHECK("clip_factor_kernel");
    return DP_OK;
}

// Host side of dp_clip_accumulate and its variants.
static dp_status clip_accumulate_impl(int mode, int B, int L, const float *const *G, const long long *P_l,
                                      const float *sqnorm, float C, float *const *acc, float *norms_out,
                                      float *clip_out, void *workspace, size_t workspace_bytes, void *cuda_stream,
                                      const ClipVariant &var = ClipVariant()) {
    if (mode != DP_CLIP_GLOBAL && mode != DP_CLIP_PER_LAYER) return DP_ERR_INVALID_ARG;
    if (B <= 0 || L <= 0 || !G || !P_l || !acc || !(C > 0.0f)) return DP_ERR_INVALID_ARG;
    if (B > 65535) return DP_ERR_UNSUPPORTED;
    const bool stage3_only = var.given_factor != nullptr;
    ClipPlan pl;
    if (!plan(B, L, P_l, pl)) return DP_ERR_INVALID_ARG;
    for (int l = 0; l < L; ++l) {
        if (!G[l] || !acc[l] || !aligned(G[l], 4) || !aligned(acc[l], 4)) return DP_ERR_INVALID_ARG;
        if ((P_l[l] + kSplitCols - 1) / kSplitCols > 0x3fffffffll) return DP_ERR_UNSUPPORTED;
    }
    if (sqnorm && !aligned(sqnorm, 4)) return DP_ERR_INVALID_ARG;
    if (!stage3_only && (!workspace || !aligned(workspace, 256) || workspace_bytes < pl.total)) return DP_ERR_WORKSPACE;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    char *ws = static_cast<char *>(workspace);
    if (!stage3_only && !sqnorm && !var.noise && !var.groups && var.micro == 1 && single_read(B, L, P_l) &&
        workspace_bytes >= pl.total + clip_rows_workspace_bytes(B, P_l[0])) {
        const dp_status rc = launch_clip_rows(G[0], B, P_l[0], C, acc[0], norms_out, clip_out, ws + pl.total, stream);
        if (rc != DP_ERR_UNSUPPORTED) return rc;
    }
    ClipCall c = {};
    c.B = B; c.L = L; c.per_layer = mode == DP_CLIP_PER_LAYER;
    c.G = G; c.P_l = P_l; c.acc = acc; c.sq = sqnorm; c.C = C; c.norms_out = norms_out; c.clip_out = clip_out;
    c.parts_per_example = pl.parts_per_example;
    if (stage3_only) {
        c.factor = var.given_factor;
    } else {
        c.partial = reinterpret_cast<float *>(ws + pl.partial_off);
        c.sq_ws = reinterpret_cast<float *>(ws + pl.sq_off);
        c.factor = c.factor_ws = reinterpret_cast<float *>(ws + pl.factor_off);
    }
    return L <= kSmallTable ? clip_launches<kSmallTable>(c, var, stream) : clip_launches<kLargeTable>(c, var, stream);
}
}  // namespace dp

extern "C" dp_status dp_clip_accumulate(int mode, int B, int L, const float *const *G, const long long *P_l,
                                        const float *sqnorm, float C, float *const *acc, float *norms_out,
                                        float *clip_out, void *workspace, size_t workspace_bytes, void *cuda_stream) {
    return dp::clip_accumulate_impl(mode, B, L, G, P_l, sqnorm, C, acc, norms_out, clip_out, workspace, workspace_bytes,
                                    cuda_stream);
}

extern "C" dp_status dp_clip_factors(int mode, int B, int L, const float *sqnorm, float C, float *norms_out,
                                     float *factors_out, void *cuda_stream) {
    if (mode != DP_CLIP_GLOBAL && mode != DP_CLIP_PER_LAYER) return DP_ERR_INVALID_ARG;
    if (B <= 0 || L <= 0 || !sqnorm || !factors_out || !(C > 0.0f)) return DP_ERR_INVALID_ARG;
    if (!dp::aligned(sqnorm, 4) || !dp::aligned(factors_out, 4) || (norms_out && !dp::aligned(norms_out, 4))) return DP_ERR_INVALID_ARG;
    dp::ClipCall c = {};
    c.B = B; c.L = L; c.per_layer = mode == DP_CLIP_PER_LAYER;
    c.sq = sqnorm; c.C = C; c.factor_ws = factors_out; c.norms_out = norms_out;
    return dp::launch_factors(c, dp::ClipVariant(), static_cast<cudaStream_t>(cuda_stream));
}

extern "C" dp_status dp_scale_accumulate(int B, int L, const float *const *G, const long long *P_l, const float *factor,
                                         int per_tensor, float *const *acc, void *cuda_stream) {
    if (!factor || !dp::aligned(factor, 4) || (per_tensor != 0 && per_tensor != 1)) return DP_ERR_INVALID_ARG;
    dp::ClipVariant var;
    var.given_factor = factor;
    return dp::clip_accumulate_impl(per_tensor ? DP_CLIP_PER_LAYER : DP_CLIP_GLOBAL, B, L, G, P_l, nullptr, 1.0f, acc,
                                    nullptr, nullptr, nullptr, 0, cuda_stream, var);
}

extern "C" dp_status dp_clip_accumulate_grouped(int B, int L, int M, const int *group_of, const float *const *G,
                                                const long long *P_l, const float *sqnorm, float C, float *const *acc,
                                                float *norms_out, float *clip_out, void *workspace,
                                                size_t workspace_bytes, void *cuda_stream) {
    if (L <= 0 || M <= 0 || M > L || !group_of) return DP_ERR_INVALID_ARG;
    if (L > dp::kMaxGroupedTensors) return DP_ERR_UNSUPPORTED;
    dp::GroupTable gt;
    gt.M = M;
    unsigned char used[dp::kMaxGroupedTensors] = {0};
    for (int l = 0; l < L; ++l) {
        if (group_of[l] < 0 || group_of[l] >= M) return DP_ERR_INVALID_ARG;
        gt.of[l] = (unsigned short)group_of[l];
        used[group_of[l]] = 1;
    }
    for (int m = 0; m < M; ++m)
        if (!used[m]) return DP_ERR_INVALID_ARG;                 // an empty group would still count in C/sqrt(M)
    dp::ClipVariant var;
    var.groups = &gt;
    return dp::clip_accumulate_impl(DP_CLIP_PER_LAYER, B, L, G, P_l, sqnorm, C, acc, norms_out, clip_out, workspace,
                                    workspace_bytes, cuda_stream, var);
}

extern "C" dp_status dp_clip_accumulate_micro(int B, int L, int micro, const float *const *G, const long long *P_l,
                                              float C, float *const *acc, float *norms_out, float *clip_out,
                                              void *workspace, size_t workspace_bytes, void *cuda_stream) {
    if (micro <= 0 || B <= 0 || B % micro != 0) return DP_ERR_INVALID_ARG;
    dp::ClipVariant var;
    var.micro = micro;
    return dp::clip_accumulate_impl(DP_CLIP_GLOBAL, B, L, G, P_l, nullptr, C, acc, norms_out, clip_out, workspace,
                                    workspace_bytes, cuda_stream, var);
}

extern "C" dp_status dp_clip_accumulate_noised(int mode, int B, int L, const float *const *G, const long long *P_l,
                                               const long long *param_offset_l, const float *sqnorm, float C,
                                               float sigma, long long total_batch, unsigned long long seed,
                                               unsigned long long step, long long example0, float *const *acc,
                                               float *norms_out, float *clip_out, void *workspace,
                                               size_t workspace_bytes, void *cuda_stream) {
    if (!param_offset_l || L <= 0 || B <= 0 || !P_l) return DP_ERR_INVALID_ARG;
    if (!(sigma >= 0.0f) || isinf(sigma) || total_batch <= 0 || example0 < 0) return DP_ERR_INVALID_ARG;
    if (sigma > 0.0f && (isinf(C) || !(C > 0.0f))) return DP_ERR_INVALID_ARG;
    if (example0 + (long long)B > 0x80000000ll) return DP_ERR_INVALID_ARG;
    for (int l = 0; l < L; ++l) {
        if (param_offset_l[l] < 0 || P_l[l] <= 0) return DP_ERR_INVALID_ARG;
        if (((unsigned long long)param_offset_l[l] + (unsigned long long)P_l[l]) > (1ull << 34)) return DP_ERR_UNSUPPORTED;
    }
    if (sigma == 0.0f)
        return dp::clip_accumulate_impl(mode, B, L, G, P_l, sqnorm, C, acc, norms_out, clip_out, workspace,
                                        workspace_bytes, cuda_stream);
    dp::ExampleNoise nz;
    nz.sd = (float)((double)sigma * (double)C / sqrt((double)total_batch));
    nz.ns = dp::noise_stream(seed, step); nz.example0 = (uint32_t)example0;
    dp::ClipVariant var;
    var.noise = &nz;
    var.goff_l = param_offset_l;
    return dp::clip_accumulate_impl(mode, B, L, G, P_l, sqnorm, C, acc, norms_out, clip_out, workspace, workspace_bytes,
                                    cuda_stream, var);
}

// ----------------------------------------------------------------------------------------------------
// Variant of dp_clip_accumulate for callers that cannot supply scratch memory of their own.
// The scratch lives in this file-scope device array, so every GPU that loads the library carries
// kStaticScratchBytes of it until the process exits.
namespace dp {
constexpr size_t kStaticScratchBytes = 2u << 20;   // 2 MiB
static __device__ __align__(256) unsigned char g_clip_scratch[kStaticScratchBytes];

// Device address of g_clip_scratch on the current device.  In host code the array's name is only a
// stand-in for the symbol, never a usable address, so the address is asked for with the caller's
// device current.  It is asked for on every call (after the first one on a device this is a table
// look-up inside the runtime and allocates nothing), so no address outlives a cudaDeviceReset.
static dp_status static_scratch(void **out) {
    void *ptr = nullptr;
    DP_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_clip_scratch));
    if (!ptr) return cuda_fail(cudaErrorInvalidSymbol, "cudaGetSymbolAddress(g_clip_scratch)");
    *out = ptr;
    return DP_OK;
}
}  // namespace dp

extern "C" size_t dp_clip_static_scratch_bytes(void) { return dp::kStaticScratchBytes; }

extern "C" dp_status dp_clip_accumulate_static(int mode, int B, int L, const float *const *G, const long long *P_l,
                                               const float *sqnorm, float C, float *const *acc, float *norms_out,
                                               float *clip_out, void *cuda_stream) {
    if (B <= 0 || L <= 0 || !P_l) return DP_ERR_INVALID_ARG;
    dp::ClipPlan pl;
    if (!dp::plan(B, L, P_l, pl)) return DP_ERR_INVALID_ARG;
    if (pl.total > dp::kStaticScratchBytes) {
        dp::note_error("dp_clip_accumulate_static: this problem needs more scratch than the built-in 2 MiB array; "
                       "use dp_clip_accumulate with a caller-owned workspace");
        return DP_ERR_WORKSPACE;
    }
    void *scratch = nullptr;
    const dp_status rc = dp::static_scratch(&scratch);
    if (rc != DP_OK) return rc;
    // every scratch word the kernels read is written earlier in the same call, so nothing needs clearing
    return dp_clip_accumulate(mode, B, L, G, P_l, sqnorm, C, acc, norms_out, clip_out, scratch, dp::kStaticScratchBytes,
                              cuda_stream);
}
