// Norm, clip and accumulate of one flat [B, P] matrix in a single read (paper section 2: sum over the batch of clip(g_j, C)).
//
// The norm of a row must be known before any of it is scaled, so two passes over memory read every gradient twice.  A row of
// up to some hundred thousand floats fits the registers of a thread-block cluster: a bulk copy brings it to shared
// memory, which is free for another row as soon as it is in registers; it is square-summed there, the cluster's blocks exchange their
// sums through distributed shared memory, and it is scaled into running sums, also in registers, while the next rows arrive.
// Bound by memory where rows are long; the exchange takes some two microseconds, so short rows go several at a time.
// 256 rows of 175 178 floats, rows at any address: 60 us for the three launches that read twice, 45 here (38 for the rows,
// 4.7 TB/s from the 120 SMs that clusters of eight find room on); 600 MB of them 189 and 116.
#include "clip_rows.cuh"
#include "mbar.cuh"
#include <math.h>
#include <algorithm>
#include <atomic>

namespace dp {

constexpr int kRowsThreads = 512, kRowsWarps = kRowsThreads / 32;
constexpr int kRowsValues = 48, kRowsMaxCluster = 8;         // of a row in a thread's registers, at most; blocks
constexpr int kRowsMaxBuffers = 8, kRowsSmem = 216 * 1024;
// A block's part of a row starts at any word: it is copied from the 16-byte boundary before it, to a place as far behind a
// 128-byte boundary.
constexpr int kRowsLine = 128;

// squared norm of the row in a float (infinite past its range) to min(1, C / sqrt(s)), without the double pipe: the reciprocal
// root and what it is off by, worked out with the products' rounding errors.  c2: C * C rounded down.
__device__ __forceinline__ float row_factor(float s, float C, float c2) {
    if (s <= c2) return 1.0f;
    if (s > kFloatMax) return 0.0f;
    const float r = rsqrtf(s);
    const float h = __fmul_rn(s, r), hl = __fmaf_rn(s, r, -h);
    const float e = __fmaf_rn(-hl, r, __fmaf_rn(-h, r, 1.0f));           // 1 - s r^2
    const float f = __fmul_rn(C, r), fl = __fmaf_rn(C, r, -f);
    return f + __fmaf_rn(f, 0.5f * e, fl);
}

struct RowsArgs {
    const float *G;
    long long P;
    int B, clusters, slice;                          // slice: floats of a block, a multiple of 32
    int buffers, stride;                             // rows in shared memory, bytes from one to the next
    float C, c2;
    float *out;                                      // [clusters][P], or the accumulator when there is one cluster
    float *norms_out, *clip_out;
    uint32_t polls;
};

// What the threads of a block wait for.  A thread whose wait gave up runs through to the end and waits for, arms, frees and sends
// nothing more; others miss what it would have sent and give up as well.  What they all compute from then on is thrown away.
// (Leaving the loops instead takes a vote a wait: 54.0 us for 256 rows of 175 178, 52.2 this way.)
__device__ __forceinline__ bool rows_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t polls) {
    return mbar_try_wait(bar, parity) || (!*abort_flag && mbar_wait(bar, parity, abort_flag, polls));
}
__device__ __forceinline__ bool rows_try_peers(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\tselp.b32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(1000u) : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint32_t rows_peer(const void *mine, int block) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(mine)), "r"(block));
    return r;
}

// V values of a row a thread, R rows at a time: V * (R + 1) of its 128 registers.
template <int V, int R>
__global__ void __launch_bounds__(kRowsThreads, 1)
clip_rows_kernel(const RowsArgs a) {
    extern __shared__ __align__(128) uint8_t rows_sh[];
    __shared__ __align__(8) uint64_t full[kRowsMaxBuffers], empty[kRowsMaxBuffers], sums_in[2];
    __shared__ float sums[2][R][kRowsMaxCluster * kRowsWarps];       // [turn & 1][row][warp of the cluster]
    __shared__ int abort_flag;
    const int warp = uniform_warp(), lane = threadIdx.x & 31, t = threadIdx.x;
    volatile int *abort_p = &abort_flag;
    uint32_t rank, blocks;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(blocks));
    const int cluster = blockIdx.x / blocks;
    const long long c0 = min((long long)rank * a.slice, a.P);
    const int len = (int)min((long long)a.slice, a.P - c0);
    if (t == 0) {
        abort_flag = 0;
        for (int s = 0; s < a.buffers; ++s) { mbar_init(smem_u32(&full[s]), 1); mbar_init(smem_u32(&empty[s]), kRowsWarps); }
        for (int s = 0; s < 2; ++s) mbar_init(smem_u32(&sums_in[s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // every block's barriers exist
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

    // the last warp: row n on its way to a buffer
    auto load = [&](int n, int buffer, bool live) {
        const uintptr_t first = (uintptr_t)a.G, end = (uintptr_t)(a.G + (long long)a.B * a.P);
        const uintptr_t lo = (uintptr_t)(a.G + n * a.P + c0), hi = lo + 4 * (uintptr_t)len;
        uint8_t *buf = rows_sh + buffer * a.stride;
        const uintptr_t at = lo & ~(uintptr_t)(kRowsLine - 1);                   // what the buffer's first byte holds
        uintptr_t from = lo & ~(uintptr_t)15, to = (hi + 15) & ~(uintptr_t)15;
        if (from < first || to > end) {                                          // words at the matrix's very ends
            if (from < first) from += 16;
            if (to > end) to -= 16;
            if (live && lo + 4 * lane < min(from, hi)) *reinterpret_cast<float *>(buf + (lo + 4 * lane - at)) = *reinterpret_cast<const float *>(lo + 4 * lane);
            const uintptr_t tail = max(max(to, from), lo);
            if (live && tail + 4 * lane < hi) *reinterpret_cast<float *>(buf + (tail + 4 * lane - at)) = *reinterpret_cast<const float *>(tail + 4 * lane);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");         // before a bulk copy overwrites them one day
            __syncwarp();
        }
        if (lane == 0 && live) {
            const uint32_t bytes = len > 0 && to > from ? (uint32_t)(to - from) : 0u, bar = smem_u32(&full[buffer]);
            mbar_expect_tx(bar, bytes);
            if (bytes)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(smem_u32(buf + (from - at))), "l"(from), "r"(bytes), "r"(bar) : "memory");
        }
        __syncwarp();
    };
    int ahead = cluster, ahead_buffer = 0;           // the next row to load, and where to
    uint32_t ahead_phase = 0;
    if (warp == kRowsWarps - 1)
        for (int s = 0; s < a.buffers && ahead < a.B; ++s, ahead += a.clusters) load(ahead, s, true);

    float acc[V];
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] = 0.f;
    int buffer = 0; uint32_t phase = 0;
    int turn = 0;
    bool live = true;
    for (int n0 = cluster; n0 < a.B; n0 += R * a.clusters, ++turn) {
        const int rows = min(R, (a.B - n0 + a.clusters - 1) / a.clusters), half = turn & 1;
        if (t == 0 && live) mbar_expect_tx(smem_u32(&sums_in[half]), 4u * kRowsWarps * blocks * (uint32_t)rows);
        float v[R][V];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r < rows) {
                live = live && rows_wait(smem_u32(&full[buffer]), phase, abort_p, a.polls);
                const uint32_t shift = (uint32_t)(((uintptr_t)a.G >> 2) + (long long)(n0 + r * a.clusters) * a.P + c0) & (kRowsLine / 4 - 1);
                const float *x = reinterpret_cast<const float *>(rows_sh + buffer * a.stride) + shift + t;
                float sq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < V; ++i) v[r][i] = i * kRowsThreads + t < len ? x[i * kRowsThreads] : 0.f;
#pragma unroll
                for (int i = 0; i < V; ++i) sq[i & 3] = fmaf(v[r][i], v[r][i], sq[i & 3]);
                __syncwarp();
                if (lane == 0 && live) mbar_arrive(smem_u32(&empty[buffer]));
                if (++buffer == a.buffers) { buffer = 0; phase ^= 1u; }
                // every warp's sum goes to all blocks of the cluster by itself: no block adds its own up first
                const float sum = warp_sum((sq[0] + sq[1]) + (sq[2] + sq[3]));
                if (lane < (int)blocks && live)
                    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                                 ::"r"(rows_peer(&sums[half][r][rank * kRowsWarps + warp], lane)), "r"(__float_as_uint(sum)),
                                 "r"(rows_peer(&sums_in[half], lane)) : "memory");
            }
        }
        if (warp == kRowsWarps - 1) {
            for (int r = 0; r < rows && ahead < a.B; ++r, ahead += a.clusters) {
                live = live && rows_wait(smem_u32(&empty[ahead_buffer]), ahead_phase, abort_p, a.polls);
                __syncwarp();
                load(ahead, ahead_buffer, live);
                if (++ahead_buffer == a.buffers) { ahead_buffer = 0; ahead_phase ^= 1u; }
            }
        }
        // (a warp sends the sums of turn j + 2 after it has those of turn j + 1 from all, who send them after reading turn j's)
        bool arrived = false;
        for (uint32_t it = 0; live && it < a.polls && !arrived; ++it) {
            arrived = rows_try_peers(smem_u32(&sums_in[half]), (uint32_t)(turn >> 1) & 1u);
            if ((it & 63u) == 63u && *abort_p) break;
        }
        if (!arrived) { *abort_p = 1; live = false; }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r < rows) {
                Sum2 all;
                for (int i = lane; i < kRowsWarps * (int)blocks; i += 32) all.add(sums[half][r][i]);
                all = warp_sum(all);
                // (`hi` is the same in all lanes, what its rounding lost need not be to the last bit)
                const float s = __shfl_sync(0xffffffffu, all.fits() ? all.hi + all.lo : all.hi, 0);
                const float f = row_factor(s, a.C, a.c2);
                if (rank == 0 && t == 0) {
                    const int n = n0 + r * a.clusters;
                    if (a.norms_out) a.norms_out[n] = __fsqrt_rn(s);
                    if (a.clip_out) a.clip_out[n] = f;
                }
#pragma unroll
                for (int i = 0; i < V; ++i) acc[i] = fmaf(f, v[r][i], acc[i]);
            }
        }
    }
    __syncthreads();
    if (*abort_p) {
        __nanosleep(200000);                         // copies still in flight land before shared memory is released
        if (t < (int)blocks) asm volatile("st.shared::cluster.u32 [%0], 1;" ::"r"(rows_peer(&abort_flag, t)) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // nobody leaves while a peer may still send to it
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const bool failed = *abort_p != 0;               // here or in a peer
    float *out = a.out + (a.clusters > 1 ? cluster * a.P : 0ll) + c0 + t;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        if (i * kRowsThreads + t < len) {
            const float v = failed ? __int_as_float(0x7fffffff) : acc[i];
            if (a.clusters > 1) out[i * kRowsThreads] = v;
            else out[i * kRowsThreads] += v;
        }
    }
    if (failed) {
        for (int n = cluster + t * a.clusters; rank == 0 && n < a.B; n += kRowsThreads * a.clusters) {
            if (a.norms_out) a.norms_out[n] = __int_as_float(0x7fffffff);
            if (a.clip_out) a.clip_out[n] = __int_as_float(0x7fffffff);
        }
        __nanosleep(200000);                         // sums that peers had on their way
    }
}

// acc[i] += the clusters' sums.  A chain of loads: where clusters are few a thread adds those of its column in cluster order, all
// in flight; where they are many a warp takes every eighth of them for 32 columns.
constexpr int kRowsFew = 16;
__global__ void __launch_bounds__(256)
clip_rows_fold_few_kernel(const float *__restrict__ part, int clusters, long long P, float *__restrict__ acc) {
    const long long i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= P) return;
    float v[kRowsFew];
    const float a = acc[i];
#pragma unroll
    for (int c = 0; c < kRowsFew; ++c) { v[c] = 0.f; if (c < clusters) v[c] = __ldcs(part + c * P + i); }
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < kRowsFew; ++c) s += v[c];
    for (int c = kRowsFew; c < clusters; ++c) s += __ldcs(part + c * P + i);
    acc[i] = a + s;
}
__global__ void __launch_bounds__(256)
clip_rows_fold_many_kernel(const float *__restrict__ part, int clusters, long long P, float *__restrict__ acc) {
    __shared__ float sums[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long i = blockIdx.x * 32ll + lane;
    float s = 0.f;
    if (i < P) {
        for (int c = w; c < clusters; c += 64) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) { v[u] = 0.f; if (c + 8 * u < clusters) v[u] = __ldcs(part + (c + 8 * u) * P + i); }
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
    }
    sums[w][lane] = s;
    __syncthreads();
    if (w == 0 && i < P) {
        float a = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) a += sums[k][lane];
        acc[i] += a;
    }
}

typedef void (*RowsKernel)(const RowsArgs);
constexpr int kRowsKernels = 5;
constexpr int kRowsValuesOf[kRowsKernels] = {12, 16, 24, 32, kRowsValues};
static RowsKernel rows_kernel(int i) {
    const RowsKernel all[kRowsKernels] = {clip_rows_kernel<12, 4>, clip_rows_kernel<16, 4>, clip_rows_kernel<24, 3>, clip_rows_kernel<32, 2>, clip_rows_kernel<kRowsValues, 1>};
    return all[i];
}
static int rows_kernel_for(int slice) {
    int i = 0;
    while (kRowsValuesOf[i] * kRowsThreads < slice) ++i;
    return i;
}

struct RowsPlan { int cluster, clusters, slice; };
// The smallest cluster whose registers hold a row, and larger ones while they leave half of the SMs idle.
static RowsPlan rows_plan(int B, long long P) {
    RowsPlan p;
    const int sms = sm_count();
    p.cluster = 1;
    while (p.cluster < kRowsMaxCluster && (P > (long long)p.cluster * kRowsValues * kRowsThreads ||
                                           (B * p.cluster * 2 <= sms && P >= 4096ll * p.cluster)))
        p.cluster *= 2;
    p.clusters = std::max(1, std::min(B, sms / p.cluster));
    p.slice = (int)(((P + p.cluster - 1) / p.cluster + 31) / 32 * 32);
    return p;
}

// Rows up to what the registers of a cluster hold.  In the middle, rows of a few blocks and not many of them, every cluster has
// one or two and the two passes, the second from the L2, are quicker (50 rows of 98 304: 14 us, 21 in a single read; 130 rows: 18
// and 21; 150 rows, 59 MB: 19 and 22; 457 rows: 60 and 45).  On either side of it the single read is, also where the L2 holds
// everything: short rows are too narrow for the passes over columns (12 500 rows of 2001: 293 us, 99 here), long ones fill the GPU
// (38 rows of 131 071: 22 us, 17 here).
constexpr long long kRowsShort = 12288, kRowsLong = 98304, kRowsFewBytes = 6000000, kRowsManyBytes = 60000000;
bool clip_rows_eligible(int B, long long P) {
    const long long bytes = 4ll * B * P;
    return B > 0 && P <= (long long)kRowsMaxCluster * kRowsValues * kRowsThreads &&
           !(P > kRowsShort && P <= kRowsLong && bytes > kRowsFewBytes && bytes < kRowsManyBytes);
}

size_t clip_rows_workspace_bytes(int B, long long P) {
    const RowsPlan p = rows_plan(B, P);
    return p.clusters > 1 ? sizeof(float) * (size_t)p.clusters * (size_t)P : 0;
}

// The limit on dynamic shared memory belongs to a function in one context: it is raised for every launch (60 ns), in whichever
// context and on whichever device is current.
static bool rows_shared(RowsKernel kernel) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmem) == cudaSuccess) return true;
    (void)cudaGetLastError();
    return false;
}

// Clusters of this size that the current device holds at once (one block an SM, all of a cluster in one GPC); 0: none, and the
// caller takes another way.
static int rows_resident(int cluster) {
    static std::atomic<int> cached[64][kRowsMaxCluster + 1];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) { (void)cudaGetLastError(); return 0; }
    if (dev < 64) {
        const int n = cached[dev][cluster].load(std::memory_order_relaxed);
        if (n > 0) return n;
    }
    const RowsKernel kernel = rows_kernel(kRowsKernels - 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cluster * 64)); cfg.blockDim = dim3(kRowsThreads); cfg.dynamicSmemBytes = kRowsSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (!rows_shared(kernel) || cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 0) { (void)cudaGetLastError(); return 0; }
    if (dev < 64) cached[dev][cluster].store(n, std::memory_order_relaxed);
    return n;
}

dp_status launch_clip_rows(const float *G, int B, long long P, float C, float *acc, float *norms_out, float *clip_out,
                           void *workspace, cudaStream_t stream) {
    RowsPlan p = rows_plan(B, P);
    const RowsKernel kernel = rows_kernel(rows_kernel_for(p.slice));
    const int resident = rows_resident(p.cluster);
    if (resident < 1 || !rows_shared(kernel)) return DP_ERR_UNSUPPORTED;
    p.clusters = std::min(p.clusters, resident);
    RowsArgs a = {};
    a.G = G; a.P = P; a.B = B; a.clusters = p.clusters; a.slice = p.slice;
    a.stride = 4 * p.slice + kRowsLine; a.buffers = std::min(kRowsMaxBuffers, kRowsSmem / a.stride);
    a.C = C;
    const double c2 = (double)C * (double)C;
    a.c2 = (float)c2;
    if ((double)a.c2 > c2) a.c2 = nextafterf(a.c2, 0.0f);
    a.out = p.clusters > 1 ? static_cast<float *>(workspace) : acc;
    a.norms_out = norms_out; a.clip_out = clip_out; a.polls = wait_polls();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.clusters * p.cluster)); cfg.blockDim = dim3(kRowsThreads); cfg.dynamicSmemBytes = kRowsSmem; cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)p.cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const cudaError_t le = cudaLaunchKernelEx(&cfg, kernel, a);
    if (le != cudaSuccess) return cuda_fail(le, "clip_rows_kernel");
    DP_LAUNCH_CHECK("clip_rows_kernel");
    if (p.clusters > 1) {
        const float *part = static_cast<const float *>(workspace);
        if (p.clusters <= 2 * kRowsFew) clip_rows_fold_few_kernel<<<(unsigned)((P + 255) / 256), 256, 0, stream>>>(part, p.clusters, P, acc);
        else clip_rows_fold_many_kernel<<<(unsigned)((P + 31) / 32), 256, 0, stream>>>(part, p.clusters, P, acc);
        DP_LAUNCH_CHECK("clip_rows_fold_kernel");
    }
    return DP_OK;
}

}  // namespace dp
