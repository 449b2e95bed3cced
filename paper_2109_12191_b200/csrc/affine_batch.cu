// Normalisation-affine layers of a whole batch of layer calls: all layers go through three launches together.
//
// One layer of a 32-example chunk is a few microseconds of memory traffic; on its own it then waits for a tail (the
// fold of its pixel chunks, the factors, the clipped sum) that keeps a few blocks busy.  Side by side the layers fill
// the GPU and the tails are one small launch each.  Bound by HBM: 2*2*H*W*C bytes an example in bf16, read once.
// ResNet-50 at 224 x 224, 53 layers: 8 examples 799 us as single calls.
#include "batch.cuh"
#include "affine.cuh"
#include "mbar.cuh"
#include <math.h>

namespace dp {

// The layer that block `blk` of a launch works on (starts ascending, n <= 64): every warp finds it with two compares a lane.
__device__ __forceinline__ int find_layer(const int *starts, int n, int blk) {
    const int lane = threadIdx.x & 31;
    const unsigned lo = __ballot_sync(0xffffffffu, lane < n && blk >= starts[lane]);
    const unsigned hi = __ballot_sync(0xffffffffu, lane + 32 < n && blk >= starts[lane + 32]);
    return __popc(lo) + __popc(hi) - 1;
}

// Launch 1: block = (layer, example, channel block, pixel chunk); thread = (pixel row, vector of channels).
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
affine_batch_partial_kernel(const __grid_constant__ AffineGroup grp) {
    extern __shared__ float red[];                       // [rows][tcv*VEC*2]
    const int li = find_layer(grp.start1, grp.n, blockIdx.x);
    const AffineSeg &sg_ = grp.seg[li];
    const int HW = sg_.HW, C = sg_.C, tcv = sg_.tcv, pix = sg_.pix, chunks = sg_.chunks;
    const T *X = static_cast<const T *>(sg_.X), *dY = static_cast<const T *>(sg_.dY);
    int rest = blockIdx.x - grp.start1[li];
    const int cblocks = (C / VEC + tcv - 1) / tcv;
    const int cb = rest % cblocks; rest /= cblocks;
    const int chunk = rest % chunks, n = rest / chunks;
    const int rows = 256 / tcv;
    const int prow = threadIdx.x / tcv, cvi = threadIdx.x - prow * tcv;
    const int c0 = (cb * tcv + cvi) * VEC;
    const int p_end = min(HW, (chunk + 1) * pix);
    float sg[VEC], sb[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) { sg[v] = 0.f; sb[v] = 0.f; }
    if (prow < rows && c0 < C) affine_pixel_sums<T, VEC>(X, dY, (long long)n * HW, C, c0, chunk * pix + prow, p_end, rows, sg, sb);
    const int half = tcv * VEC, width = half * 2;
    if (prow < rows) affine_stage_sums<VEC>(red, prow, cvi, tcv, sg, sb);
    __syncthreads();
    float *out = grp.partial + sg_.part_off + (((long long)n * chunks + chunk) * 2) * C;
    for (int e = threadIdx.x; e < width; e += 256) {
        const int is_beta = e >= half;
        const int c = cb * half + (is_beta ? e - half : e);
        if (c >= C) continue;
        float a = 0.f;
        for (int rr = 0; rr < rows; ++rr) a += red[rr * width + e];
        out[is_beta ? C + c : c] = a;
    }
}

// Launch 1 beside the tensor-core launches of a batch.  Those take an SM's tensor memory and most of its registers and shared
// memory, so blocks of the kind above only ran where no convolution did, and memory-bound and tensor-bound work took turns.
// This form is one small block an SM that is there first and leaves room for a convolution's: a warp to each quarter of the SM,
// 56 registers a thread, 45 KB.  Bytes are in flight through a ring in shared memory instead of registers; every thread copies
// and reads its own vectors, so that nobody waits for anybody (a warp that filled the ring by bulk copies through barriers
// took 1200 cycles a stage).  Items (an example's pixel chunk, some 130 KB) come from a counter, since SMs stream at the rate
// their convolutions leave them.  What bounds it is the one warp a quarter: 460 us alone for the 53 layers of 32 examples of
// ResNet-50 against 240 in the form above, but the chunk with its convolutions goes from 833 to 759 us.  (At 56 registers the bf16
// form spills six words.)
constexpr int kStreamThreads = 128, kStreamStages = 5;
constexpr int kStreamVecs = 2;                               // vectors of X and of dY that a thread has in a stage, of neighbouring pixel rows
constexpr int kStreamBytes = kStreamVecs * kStreamThreads * 16;
constexpr int kStreamSmem = kStreamStages * 2 * kStreamBytes;

struct StreamItem {
    const AffineSeg *s;
    int n, chunk, c0v, rows, pixels, stages, mine;           // rows: of pixels, kStreamVecs of them a stage; mine: this thread's pixel of a row, or a number past all of them
    __device__ __forceinline__ StreamItem(const AffineGroup &grp, int item, int vec) {
        const int li = find_layer(grp.start1, grp.n, item);
        s = &grp.seg[li];
        const int tcv = s->tcv, cv = s->C / vec, cblocks = (cv + tcv - 1) / tcv;
        int rest = item - grp.start1[li];
        const int cb = rest % cblocks; rest /= cblocks;
        n = rest / s->chunks;
        chunk = rest - n * s->chunks;
        rows = kStreamThreads / tcv;
        pixels = min(s->pix, s->HW - chunk * s->pix);
        // (at least a ring's length, so that the copies are never more than one item ahead)
        stages = max((pixels + kStreamVecs * rows - 1) / (kStreamVecs * rows), kStreamStages - 1);
        const int prow = threadIdx.x / tcv, cvi = threadIdx.x - prow * tcv;
        c0v = cb * tcv + cvi;
        mine = c0v < cv && prow < rows ? prow : 1 << 30;
    }
};
// A thread's copies, one stage a call.
template <typename T>
struct StreamCopies {
    const uint8_t *X;
    long long to_dY;
    int left = 0, pixels_left, step, rows;                   // stages; pixels from this thread's on
    __device__ __forceinline__ void start(const StreamItem &it) {
        const AffineSeg &s = *it.s;
        left = it.stages; rows = it.rows; pixels_left = it.pixels - it.mine;
        X = static_cast<const uint8_t *>(s.X) + (((long long)it.n * s.HW + it.chunk * s.pix + it.mine) * s.C) * (int)sizeof(T) + it.c0v * 16;
        to_dY = static_cast<const uint8_t *>(s.dY) - static_cast<const uint8_t *>(s.X);
        step = it.rows * s.C * (int)sizeof(T);
    }
    __device__ __forceinline__ void copy(uint32_t dst) {
#pragma unroll
        for (int u = 0; u < kStreamVecs; ++u) {
            if (pixels_left > 0) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + u * kStreamThreads * 16), "l"(X) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + u * kStreamThreads * 16 + kStreamBytes), "l"(X + to_dY) : "memory");
            }
            X += step; pixels_left -= rows;
        }
        --left;
    }
};
// Adds the products and the second operands of two vectors, as pairs of channels.
__device__ __forceinline__ void add_vectors(const uint4 &x, const uint4 &g, Float2 (&sg)[4], Float2 (&sb)[4], __nv_bfloat16) {
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, gs[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Float2 gg = pack2(__uint_as_float(gs[i] << 16), __uint_as_float(gs[i] & 0xffff0000u));
        sg[i] = fma2(gg, pack2(__uint_as_float(xs[i] << 16), __uint_as_float(xs[i] & 0xffff0000u)), sg[i]);
        sb[i] = add2(gg, sb[i]);
    }
}
__device__ __forceinline__ void add_vectors(const uint4 &x, const uint4 &g, Float2 (&sg)[2], Float2 (&sb)[2], float) {
    const Float2 g0 = pack2(__uint_as_float(g.x), __uint_as_float(g.y)), g1 = pack2(__uint_as_float(g.z), __uint_as_float(g.w));
    sg[0] = fma2(g0, pack2(__uint_as_float(x.x), __uint_as_float(x.y)), sg[0]);
    sg[1] = fma2(g1, pack2(__uint_as_float(x.z), __uint_as_float(x.w)), sg[1]);
    sb[0] = add2(g0, sb[0]);
    sb[1] = add2(g1, sb[1]);
}

template <typename T>
__global__ void __launch_bounds__(kStreamThreads, 9)
affine_batch_stream_kernel(const __grid_constant__ AffineGroup grp, int items, int *tickets) {
    constexpr int VEC = 16 / sizeof(T);
    extern __shared__ __align__(128) uint8_t ring[];         // [stages][X, dY]
    __shared__ __align__(16) float red[kStreamThreads * VEC];
    __shared__ int ahead[2];                                 // [turn & 1]: item of that turn
    const uint32_t slot0 = smem_u32(ring) + threadIdx.x * 16;
    int item = blockIdx.x, next = item + (int)gridDim.x;
    StreamCopies<T> copies;
    int put = 0, got = 0;                                    // slots of the ring
    auto fill = [&]() {
        if (copies.left == 0 && next < items) {              // (the item after this one: known by now)
            copies.start(StreamItem(grp, next, VEC));
            next = items;
        }
        if (copies.left > 0) {
            copies.copy(slot0 + put * 2 * kStreamBytes);
            if (++put == kStreamStages) put = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    copies.start(StreamItem(grp, item, VEC));
    {
        const int then = next;
        next = items;
        for (int k = 0; k < kStreamStages - 1; ++k) fill();
        next = then;
    }
    for (int turn = 0; item < items; ++turn) {
        const int following = next;
        int later = 0;                                       // item of turn + 2 (back long before it is needed)
        if (threadIdx.x == 0) later = following < items ? 2 * (int)gridDim.x + atomicAdd(tickets, 1) : items;
        const StreamItem it(grp, item, VEC);
        Float2 sg2[VEC / 2], sb2[VEC / 2];
#pragma unroll
        for (int v = 0; v < VEC / 2; ++v) { sg2[v] = pack2(0.f, 0.f); sb2[v] = sg2[v]; }
        int left = it.pixels - it.mine;
        for (int k = 0; k < it.stages; ++k, left -= kStreamVecs * it.rows) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStreamStages - 2) : "memory");
            const uint8_t *at = ring + got * 2 * kStreamBytes + threadIdx.x * 16;
            uint4 x[kStreamVecs], g[kStreamVecs];
#pragma unroll
            for (int u = 0; u < kStreamVecs; ++u) {
                x[u] = *reinterpret_cast<const uint4 *>(at + u * kStreamThreads * 16);
                g[u] = *reinterpret_cast<const uint4 *>(at + u * kStreamThreads * 16 + kStreamBytes);
            }
#pragma unroll
            for (int u = 0; u < kStreamVecs; ++u)
                if (left > u * it.rows) add_vectors(x[u], g[u], sg2, sb2, T());
            if (++got == kStreamStages) got = 0;
            fill();
        }
        float sg[VEC], sb[VEC];
#pragma unroll
        for (int v = 0; v < VEC; v += 2) { unpack2(sg2[v / 2], sg[v], sg[v + 1]); unpack2(sb2[v / 2], sb[v], sb[v + 1]); }
        const AffineSeg &s = *it.s;
        float *out = grp.partial + s.part_off + (((long long)it.n * s.chunks + it.chunk) * 2) * s.C;
        if (it.rows == 1) {
            if (it.mine == 0) {
#pragma unroll
                for (int v = 0; v < VEC; v += 4) {
                    *reinterpret_cast<float4 *>(out + it.c0v * VEC + v) = make_float4(sg[v], sg[v + 1], sg[v + 2], sg[v + 3]);
                    *reinterpret_cast<float4 *>(out + s.C + it.c0v * VEC + v) = make_float4(sb[v], sb[v + 1], sb[v + 2], sb[v + 3]);
                }
            }
        } else {
            const int sums = s.C;                            // (more than one pixel a stage: one channel block)
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                if (which) __syncthreads();                  // the sums of dY * X have been read
#pragma unroll
                for (int v = 0; v < VEC; ++v) red[threadIdx.x * VEC + v] = which ? sb[v] : sg[v];
                __syncthreads();
                for (int e = threadIdx.x; e < sums; e += kStreamThreads) {
                    float a = 0.f;
                    for (int r = 0; r < it.rows; ++r) a += red[r * sums + e];
                    out[which * s.C + e] = a;
                }
            }
        }
        if (threadIdx.x == 0) ahead[turn & 1] = later;
        __syncthreads();                                     // (`red` has been read, too)
        item = following;
        next = ahead[turn & 1];
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(tickets + 1, 1) == (int)gridDim.x - 1) { tickets[0] = 0; tickets[1] = 0; }
    }
}

// Launch 2: block = (layer, example): folds the example's pixel chunks in chunk order, stores its gradients, publishes
// its squared norms and, for the fused clip, its factors.  A chain of L2 round trips: four channels a thread and eight
// chunks in flight, and squares summed in floats that carry their rounding errors along, since the double pipe is what the
// block would wait for (53 layers x 8 examples: 13 us with one channel a thread and double sums).  Where a sum
// leaves the range in which that is exact (squares that overflow or vanish), one warp squares what was stored again, in
// double; looking at the sums of all warps instead of each one's keeps the check off the others (32 examples, 53 layers: 19 us
// without a check, 21 with one a warp).
constexpr float kSmallestSum = 7.9e-31f;                 // some 2^-100: what a square loses to underflow is 2^-50 of it
__global__ void __launch_bounds__(256)
affine_batch_fold_kernel(const __grid_constant__ AffineGroup grp) {
    __shared__ double scratch[2][8];
    const int li = find_layer(grp.start2, grp.n, blockIdx.x);
    const AffineSeg &s = grp.seg[li];
    const int n = blockIdx.x - grp.start2[li], C = s.C, chunks = s.chunks;
    const float *base = grp.partial + s.part_off + (long long)n * chunks * 2 * C;
    float *dgamma = s.dgamma + (long long)n * C, *dbeta = s.dbeta + (long long)n * C;
    Sum2 q[2];
    for (int e = 4 * threadIdx.x; e < 2 * C; e += 1024) {
        const bool beta = e >= C;
        const float4 *p = reinterpret_cast<const float4 *>(base + e);         // [chunk][2][C], C a multiple of four
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < chunks; k += 8) {
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k + u < chunks) x[u] = p[(long long)(k + u) * (C / 2)];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) { a.x += x[u].x; a.y += x[u].y; a.z += x[u].z; a.w += x[u].w; }
        }
        *reinterpret_cast<float4 *>(beta ? dbeta + e - C : dgamma + e) = a;
        Sum2 t;
        t.add_square(a.x); t.add_square(a.y); t.add_square(a.z); t.add_square(a.w);
        if (beta) q[1].add(t); else q[0].add(t);
    }
    const int warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const Sum2 t = warp_sum(q[k]);
        if ((threadIdx.x & 31) == 0) scratch[k][warp] = t.value();
    }
    __syncthreads();
    if (warp != 0) return;
    double qg = 0.0, qb = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { qg += scratch[0][i]; qb += scratch[1][i]; }
    if (!(fmin(qg, qb) >= kSmallestSum && qg + qb < (double)INFINITY)) {
        qg = qb = 0.0;
        for (int e = 4 * threadIdx.x; e < 2 * C; e += 128) {
            const bool beta = e >= C;
            const float4 a = *reinterpret_cast<const float4 *>(beta ? dbeta + e - C : dgamma + e);
            const double s4 = ((double)a.x * a.x + (double)a.y * a.y) + ((double)a.z * a.z + (double)a.w * a.w);
            if (beta) qb += s4; else qg += s4;
        }
        qg = warp_sum(qg); qb = warp_sum(qb);
    }
    if (threadIdx.x != 0) return;
    float f0 = 1.f, f1 = 1.f;
    if (s.separate) {
        s.sqnorm[n * s.sq_stride] = (float)qg; s.sqnorm[n * s.sq_stride + 1] = (float)qb;
        if (s.clip) { f0 = clip_factor(qg, grp.C_l); f1 = clip_factor(qb, grp.C_l); }
        if (s.clip && s.clip_out) { s.clip_out[2 * n] = f0; s.clip_out[2 * n + 1] = f1; }
    } else {
        s.sqnorm[n * s.sq_stride] = (float)(qg + qb);
        if (s.clip) f0 = f1 = clip_factor(qg + qb, grp.C_l);
        if (s.clip && s.clip_out) s.clip_out[n] = f0;
    }
    if (s.clip) { s.factor[2 * n] = f0; s.factor[2 * n + 1] = f1; }
}

// Launch 3 (fused clip): block = (layer, 128 of its 2C sums), four a lane, eight groups of examples folded in group order.
constexpr int kAccumSums = 128;
__global__ void __launch_bounds__(256)
affine_batch_accum_kernel(const __grid_constant__ AffineGroup grp) {
    __shared__ float4 part[8][32];
    const int li = find_layer(grp.start3, grp.n, blockIdx.x);
    const AffineSeg &s = grp.seg[li];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5, C = s.C;
    const int e = (blockIdx.x - grp.start3[li]) * kAccumSums + 4 * lane;
    const int which = e >= C, c = which ? e - C : e;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < 2 * C) {
        const float *v = (which ? s.dbeta : s.dgamma) + c;
#pragma unroll 4
        for (int n = q; n < s.B; n += 8) {
            const float f = s.factor[2 * n + which];
            const float4 x = *reinterpret_cast<const float4 *>(v + (long long)n * C);
            a.x = fmaf(f, x.x, a.x); a.y = fmaf(f, x.y, a.y); a.z = fmaf(f, x.z, a.z); a.w = fmaf(f, x.w, a.w);
        }
    }
    part[q][lane] = a;
    __syncthreads();
    if (q == 0 && e < 2 * C) {
        float4 *dst = reinterpret_cast<float4 *>((which ? s.acc_b : s.acc_w) + c);
        float4 t = part[0][lane], r = *dst;
#pragma unroll
        for (int i = 1; i < 8; ++i) { const float4 x = part[i][lane]; t.x += x.x; t.y += x.y; t.z += x.z; t.w += x.w; }
        r.x += t.x; r.y += t.y; r.z += t.z; r.w += t.w;
        *dst = r;
    }
}

bool affine_batch_eligible(int dtype, int C) { return C % (dtype == DP_F32 ? 4 : 8) == 0; }

void affine_batch_shape(int dtype, int B, int HW, int C, bool beside, AffineSeg &s) {
    const int cv = C / (dtype == DP_F32 ? 4 : 8);
    s.B = B; s.HW = HW; s.C = C;
    // sixteen pixels a thread of 256: four trips, some 130 KB a block, which is long enough to hide the block's own tail and
    // short enough to spread a layer of one example; the same bytes an item where 128 threads add them up
    const int wide = beside ? kStreamThreads : 256;
    s.tcv = cv < wide ? cv : wide;
    const int rows = wide / s.tcv, most = (beside ? 32 : 16) * rows;
    s.chunks = (HW + most - 1) / most;
    s.pix = beside ? ((HW + s.chunks - 1) / s.chunks + rows - 1) / rows * rows : most;
    s.chunks = (HW + s.pix - 1) / s.pix;
}

dp_status launch_affine_batch(int dtype, AffineGroup &grp, int *tickets, cudaEvent_t begun, cudaStream_t st) {
    const int vec = dtype == DP_F32 ? 4 : 8;
    int b1 = 0, b2 = 0, b3 = 0;
    size_t smem = 0;
    for (int i = 0; i < grp.n; ++i) {
        const AffineSeg &s = grp.seg[i];
        grp.start1[i] = b1; grp.start2[i] = b2; grp.start3[i] = b3;
        b1 += s.B * s.chunks * ((s.C / vec + s.tcv - 1) / s.tcv);
        b2 += s.B;
        b3 += s.clip ? (2 * s.C + kAccumSums - 1) / kAccumSums : 0;
        const size_t need = sizeof(float) * (size_t)(256 / s.tcv) * s.tcv * vec * 2;
        if (need > smem) smem = need;
    }
    if (tickets) {
        // the SM's memory is not divided anew while blocks run, and the convolution's needs most of it as shared memory
        const void *kernel = dtype == DP_F32 ? (const void *)affine_batch_stream_kernel<float> : (const void *)affine_batch_stream_kernel<__nv_bfloat16>;
        DP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
        const unsigned grid = (unsigned)(b1 < sm_count() ? b1 : sm_count());
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kStreamThreads); cfg.dynamicSmemBytes = kStreamSmem; cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeLaunchCompletionEvent;
        at[0].val.launchCompletionEvent.event = begun; at[0].val.launchCompletionEvent.flags = 0;
        cfg.attrs = at; cfg.numAttrs = begun ? 1 : 0;
        const cudaError_t le = dtype == DP_F32 ? cudaLaunchKernelEx(&cfg, affine_batch_stream_kernel<float>, grp, b1, tickets)
                                               : cudaLaunchKernelEx(&cfg, affine_batch_stream_kernel<__nv_bfloat16>, grp, b1, tickets);
        if (le != cudaSuccess) return cuda_fail(le, "affine_batch_stream_kernel");
        DP_LAUNCH_CHECK("affine_batch_stream_kernel");
    } else {
        if (dtype == DP_F32) affine_batch_partial_kernel<float, 4><<<(unsigned)b1, 256, smem, st>>>(grp);
        else affine_batch_partial_kernel<__nv_bfloat16, 8><<<(unsigned)b1, 256, smem, st>>>(grp);
        DP_LAUNCH_CHECK("affine_batch_partial_kernel");
    }
    affine_batch_fold_kernel<<<(unsigned)b2, 256, 0, st>>>(grp);
    DP_LAUNCH_CHECK("affine_batch_fold_kernel");
    if (b3 > 0) {
        affine_batch_accum_kernel<<<(unsigned)b3, 256, 0, st>>>(grp);
        DP_LAUNCH_CHECK("affine_batch_accum_kernel");
    }
    return DP_OK;
}

}  // namespace dp
