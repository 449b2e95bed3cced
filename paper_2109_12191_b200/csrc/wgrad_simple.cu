// CUDA-core (fp32 FMA) per-example weight gradients: the any-shape path for convolutions, the
// dense outer product, the normalisation-affine reduction, bias sums, and the small kernels that
// fold per-tile squared norms into per-example norms and clip factors.
// Formulas: paper section 2 (per-example gradient, its L2 norm, clip) and section 3.5 (per-layer threshold).
#include "wgrad_simple.cuh"
#include "affine.cuh"
#include <math.h>
#include <algorithm>

namespace dp {

constexpr int TM = kFmaTile, TN = kFmaTile, TK = 16;

// Per-example gradient matrix D_n[m, j] = sum_q A[q, m] * Bm[q, j] with
//   A[q, m]  = dY[n, pix, m]                       q = n*K + pix
//   Bm[q, j] = Xpad[n, oh*st + r - pad, ow*st + s - pad, c],  j = (r*S + s)*Cin + c
// MODE 0/1: the block owns one example (blockIdx.z) and reduces q over that example's pixels.
// MODE 2:   the block owns the tile for a RANGE of examples (blockIdx.z picks the range): q runs over
//           those examples' pixels and A is scaled by the example's clip factor, so the accumulator ends
//           as sum_n f_n D_n[m, j].  With one range the sum is added to acc_w; with several, range z
//           writes its partial sum to sum_ws[z] and a fold kernel adds them in order.
template <typename T, int MODE>
__global__ void __launch_bounds__(256)
conv_wgrad_fma_kernel(const T *__restrict__ X, const T *__restrict__ dY, const ConvGeom g, float *__restrict__ G_w,
                      float *__restrict__ partial, int slots, const float *__restrict__ factor,
                      float *__restrict__ acc_w, int per_split, float *__restrict__ sum_ws) {
    __shared__ __align__(16) float sA[TK][TM];
    __shared__ __align__(16) float sB[TK][TN];
    __shared__ float scratch[32];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * TM, j0 = blockIdx.x * TN;
    const int n_fixed = (MODE == 2) ? 0 : blockIdx.z;
    const long long q_begin = (MODE == 2) ? (long long)blockIdx.z * per_split * g.K : (long long)n_fixed * g.K;
    const long long q_end = (MODE == 2) ? (long long)min(g.B, ((int)blockIdx.z + 1) * per_split) * g.K : q_begin + g.K;
    const bool add_to_acc = (MODE == 2) && gridDim.z == 1;

    // loader role: this thread fills column lm of sA and column lj of sB for rows lp, lp+4, lp+8, lp+12
    const int lcol = tid & 63, lp = tid >> 6;
    const bool a_ok = (m0 + lcol) < g.M;
    const int jj = j0 + lcol;
    const bool b_ok = jj < g.N;
    const int c = b_ok ? jj % g.Cin : 0;
    const int rs = b_ok ? jj / g.Cin : 0;
    const int r = rs / g.S, s = rs % g.S;

    float ra[4], rb[4];
    auto fetch = [&](long long qc) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const long long q = qc + lp + 4 * i;
            ra[i] = 0.f; rb[i] = 0.f;
            if (q < q_end) {
                const int n = (int)(q / g.K);
                const int pix = (int)(q - (long long)n * g.K);
                if (a_ok) {
                    float v = to_float(dY[q * g.Kout + m0 + lcol]);
                    if (MODE == 2) v *= factor[2 * n];
                    ra[i] = v;
                }
                if (b_ok) {
                    const int oh = pix / g.OW, ow = pix - oh * g.OW;
                    const int ih = oh * g.stride + r - g.pad, iw = ow * g.stride + s - g.pad;
                    if (ih >= 0 && ih < g.H && iw >= 0 && iw < g.W)
                        rb[i] = to_float(X[(((long long)n * g.H + ih) * g.W + iw) * g.Cin + c]);
                }
            }
        }
    };

    const int ty = tid >> 4, tx = tid & 15;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][k] = 0.f;

    fetch(q_begin);
    for (long long qc = q_begin; qc < q_end; qc += TK) {
#pragma unroll
        for (int i = 0; i < 4; ++i) { sA[lp + 4 * i][lcol] = ra[i]; sB[lp + 4 * i][lcol] = rb[i]; }
        __syncthreads();
        if (qc + TK < q_end) fetch(qc + TK);
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
            const float4 a = *reinterpret_cast<const float4 *>(&sA[kk][ty * 4]);
            const float4 b = *reinterpret_cast<const float4 *>(&sB[kk][tx * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[i][k] = fmaf(av[i], bv[k], acc[i][k]);
        }
        __syncthreads();
    }

    const int jb = j0 + tx * 4;
    if (MODE == 0 || MODE == 1) {
        float sq = 0.f;   // rows / columns outside the matrix hold exact zeros, no masking needed
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) sq = fmaf(acc[i][k], acc[i][k], sq);
        sq = block_sum(sq, scratch);
        if (tid == 0) partial[(long long)n_fixed * slots + blockIdx.y * gridDim.x + blockIdx.x] = sq;
    }
    if (MODE == 0 || MODE == 2) {
        float *base = (MODE == 0) ? G_w + (long long)n_fixed * g.M * g.N
                                  : (add_to_acc ? acc_w : sum_ws + (long long)blockIdx.z * g.M * g.N);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = m0 + ty * 4 + i;
            if (m >= g.M) continue;
            float *row = base + (long long)m * g.N;
            if ((g.N & 3) == 0) {
                if (jb < g.N) {
                    float4 v = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
                    if (add_to_acc) {
                        const float4 o = *reinterpret_cast<const float4 *>(row + jb);
                        v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
                    }
                    *reinterpret_cast<float4 *>(row + jb) = v;
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (jb + k < g.N) row[jb + k] = add_to_acc ? row[jb + k] + acc[i][k] : acc[i][k];
            }
        }
    }
}

// Thin convolutions (R*S*Cin <= 32 columns, e.g. a 3x3 conv on RGB): one block per example.  The zero-padded
// input of the example sits in shared memory; thread = (pixel group, output channel lane) keeps one gradient row
// (all columns) per owned output channel in registers and walks its share of the pixels, reading dY coalesced and
// the input patch by shared-memory broadcast.  The eight pixel groups are folded in order; the bias gradient and
// both squared norms come out of the same pass.
// RT x SCT > 0 fixes the filter rows and the run length S*Cin at compile time (3 x 9 for a 3x3 conv on RGB), which
// turns every patch read into a shared-memory load with an immediate offset; RT = 0 is the any-shape version.
template <typename T, int KPT, int RT, int SCT>
__global__ void __launch_bounds__(256)
conv_wgrad_thin_kernel(const T *__restrict__ X, const T *__restrict__ dY, const ConvGeom g, float *__restrict__ G_w,
                       float *__restrict__ db, float *__restrict__ partial, int slots, int has_bias) {
    extern __shared__ float thin_smem[];
    __shared__ float scratch[32];
    const int Hp = g.H + 2 * g.pad, Wp = g.W + 2 * g.pad;
    const int xs_count = Hp * Wp * g.Cin;
    float *xs = thin_smem;                                   // [Hp][Wp][Cin], zero border
    float *red = thin_smem + ((xs_count + 3) & ~3);          // [8][Kout*N] then [8][Kout]
    const int n = blockIdx.x, lane = threadIdx.x & 31, pg = threadIdx.x >> 5;
    {
        const int row_in = g.W * g.Cin, row_p = Wp * g.Cin;
        for (int i = threadIdx.x; i < xs_count; i += 256) xs[i] = 0.f;
        __syncthreads();
        const T *Xn = X + (long long)n * g.H * row_in;
        for (int i = threadIdx.x; i < g.H * row_in; i += 256) {
            const int h = i / row_in, rest = i - h * row_in;
            xs[(h + g.pad) * row_p + g.pad * g.Cin + rest] = to_float(Xn[i]);
        }
    }
    int off[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const int jj = j < g.N ? j : 0;
        const int c = jj % g.Cin, rs = jj / g.Cin;
        off[j] = ((rs / g.S) * Wp + rs % g.S) * g.Cin + c;
    }
    float acc[KPT][32], bsum[KPT];
#pragma unroll
    for (int kk = 0; kk < KPT; ++kk) {
        bsum[kk] = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[kk][j] = 0.f;
    }
    __syncthreads();
    int oh = pg / g.OW, ow = pg - oh * g.OW;
    const T *dYn = dY + (long long)n * g.K * g.Kout;
    // U pixels per trip, and the next trip's dY loads are issued before this trip's arithmetic: a warp always has
    // U (then 2U) 128-byte rows in flight, which is what hides the memory latency at one or two blocks per SM.
    constexpr int U = 8;
    float gy[U][KPT], gyn[U][KPT];
    int base[U], basen[U];
    auto load_trip = [&](int pix, float (&y)[U][KPT], int (&b)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int pu = pix + 8 * u;
            b[u] = pu < g.K ? (oh * g.stride * Wp + ow * g.stride) * g.Cin : 0;
#pragma unroll
            for (int kk = 0; kk < KPT; ++kk)
                y[u][kk] = pu < g.K ? to_float(dYn[(long long)pu * g.Kout + lane + 32 * kk]) : 0.f;
            ow += 8;
            while (ow >= g.OW) { ow -= g.OW; ++oh; }
        }
    };
    load_trip(pg, gy, base);
    for (int pix = pg; pix < g.K; pix += 8 * U) {
        if (pix + 8 * U < g.K) load_trip(pix + 8 * U, gyn, basen);
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int kk = 0; kk < KPT; ++kk) bsum[kk] += gy[u][kk];
            if constexpr (RT > 0) {
                const float *patch = xs + base[u];
                const int row_p = Wp * g.Cin;
                // the whole warp reads the same patch (broadcast); 64-bit loads halve the shared-memory instructions,
                // with the pairing chosen by the parity of the patch start (the same for every lane and every row)
                const bool pairs = ((row_p | SCT) & 1) != 0 ? ((row_p & 1) == 0) : true;
                const int lead = (base[u] & 1);          // 1: element 0 is unaligned, pairs start at element 1
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    float x[SCT];
                    const float *row = patch + r * row_p;
                    if (pairs && (row_p & 1) == 0) {
                        if (lead == 0) {
#pragma unroll
                            for (int t = 0; t + 1 < SCT; t += 2) { const float2 v = *reinterpret_cast<const float2 *>(row + t); x[t] = v.x; x[t + 1] = v.y; }
                            if (SCT & 1) x[SCT - 1] = row[SCT - 1];
                        } else {
                            x[0] = row[0];
#pragma unroll
                            for (int t = 1; t + 1 < SCT; t += 2) { const float2 v = *reinterpret_cast<const float2 *>(row + t); x[t] = v.x; x[t + 1] = v.y; }
                            if (!(SCT & 1)) x[SCT - 1] = row[SCT - 1];
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < SCT; ++t) x[t] = row[t];
                    }
#pragma unroll
                    for (int t = 0; t < SCT; ++t) {
#pragma unroll
                        for (int kk = 0; kk < KPT; ++kk) acc[kk][r * SCT + t] = fmaf(gy[u][kk], x[t], acc[kk][r * SCT + t]);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    if (j < g.N) {
                        const float x = xs[base[u] + off[j]];
#pragma unroll
                        for (int kk = 0; kk < KPT; ++kk) acc[kk][j] = fmaf(gy[u][kk], x, acc[kk][j]);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            base[u] = basen[u];
#pragma unroll
            for (int kk = 0; kk < KPT; ++kk) gy[u][kk] = gyn[u][kk];
        }
    }
    const int MN = g.Kout * g.N;
    float *bred = red + 8 * MN;
#pragma unroll
    for (int kk = 0; kk < KPT; ++kk) {
        const int k = lane + 32 * kk;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < g.N) red[pg * MN + k * g.N + j] = acc[kk][j];
        bred[pg * g.Kout + k] = bsum[kk];
    }
    __syncthreads();
    float sq = 0.f, sqb = 0.f;
    for (int t = threadIdx.x; t < MN; t += 256) {
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) v += red[q * MN + t];
        if (G_w) G_w[(long long)n * MN + t] = v;
        sq = fmaf(v, v, sq);
    }
    if (has_bias) {
        for (int k = threadIdx.x; k < g.Kout; k += 256) {
            float v = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) v += bred[q * g.Kout + k];
            db[(long long)n * g.Kout + k] = v;
            sqb = fmaf(v, v, sqb);
        }
    }
    sq = block_sum(sq, scratch);
    sqb = block_sum(sqb, scratch);
    if (threadIdx.x == 0) {
        partial[(long long)n * slots] = sq;
        if (has_bias) partial[(long long)n * slots + 1] = sqb;
    }
}

static size_t thin_smem_bytes(const ConvGeom &g) {
    const size_t xs = ((size_t)(g.H + 2 * g.pad) * (g.W + 2 * g.pad) * g.Cin + 3) & ~(size_t)3;
    return sizeof(float) * (xs + 8 * (size_t)g.Kout * g.N + 8 * (size_t)g.Kout);
}

bool thin_conv_eligible(const ConvGeom &g) {
    return g.N <= 32 && (g.Kout == 32 || g.Kout == 64) && g.K >= 8 && thin_smem_bytes(g) <= 47 * 1024 && g.B <= 0x7fffffff;
}

template <typename T, int KPT>
static void thin_launch_t(const T *X, const T *dY, const ConvGeom &g, float *G_w, float *db, float *partial, int slots,
                          int has_bias, size_t smem, cudaStream_t st) {
    if (g.R == 3 && g.S * g.Cin == 9)
        conv_wgrad_thin_kernel<T, KPT, 3, 9><<<g.B, 256, smem, st>>>(X, dY, g, G_w, db, partial, slots, has_bias);
    else
        conv_wgrad_thin_kernel<T, KPT, 0, 0><<<g.B, 256, smem, st>>>(X, dY, g, G_w, db, partial, slots, has_bias);
}

dp_status launch_conv_thin(int dtype, const void *X, const void *dY, const ConvGeom &g, float *G_w, float *db,
                           float *partial, int slots, int has_bias, cudaStream_t st) {
    const size_t smem = thin_smem_bytes(g);
    if (dtype == DP_F32) {
        if (g.Kout == 32) thin_launch_t<float, 1>(static_cast<const float *>(X), static_cast<const float *>(dY), g, G_w, db, partial, slots, has_bias, smem, st);
        else thin_launch_t<float, 2>(static_cast<const float *>(X), static_cast<const float *>(dY), g, G_w, db, partial, slots, has_bias, smem, st);
    } else {
        if (g.Kout == 32) thin_launch_t<__nv_bfloat16, 1>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), g, G_w, db, partial, slots, has_bias, smem, st);
        else thin_launch_t<__nv_bfloat16, 2>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), g, G_w, db, partial, slots, has_bias, smem, st);
    }
    DP_LAUNCH_CHECK("conv_wgrad_thin_kernel");
    return DP_OK;
}

// 3x3 convolutions on three input channels (image stems), output channels a multiple of 32: a cluster of one to eight
// blocks per example, each with a range of output rows.  The zero-padded input rows a block needs sit in shared memory.
// Lane = output pixel (32 consecutive pixels per trip); warp w owns output channels 8(w%4) .. +7 of the current group of
// 32 and filter row w/4, i.e. an 8 x 9 block of the gradient in registers as 36 pairs of channels, which the packed
// FMA takes two at a time.  What bounds it is shared memory and issue alike: 17 wavefronts and 64 instructions for the
// 72 multiply-adds of a pixel (27 wavefronts, 150 instructions and 16 warps an SM with all 27 columns and four channels
// a thread: 31 us for 256 examples of 32 x 32, and 23 us for 32, which were 32 blocks).  dY streams through a ring of
// kRgbStages stages of 128 pixels x 32 channels, filled by coalesced asynchronous copies two stages ahead of the
// arithmetic, one barrier per stage.  Inside a stage the piece of (pixel l, channel quad c) sits at quad position
// c ^ (l & 7) of its pixel row, so that the lanes of a warp, which read the same quad of 32 pixels, hit different banks.
// The 32 pixel lanes are folded by halving (each step a lane keeps half of its values), the blocks of a cluster add
// their sums through distributed shared memory, in one order; gradient, bias gradient and norms leave from the same pass.
constexpr int kRgbThreads = 384;  // 12 warps: four channel octets x three filter rows
constexpr int kRgbStages = 3;     // stages of dY in the ring
constexpr int kRgbStagePix = 128; // pixels per stage (four trips: a barrier and the copies' addresses every 128 pixels)
constexpr int kRgbStageFloats = kRgbStagePix * 32;   // ring stride in 4-byte words (bf16 stages use half of it)
constexpr int kRgbSums = 32 * 27 + 32;               // sums of a group of 32 channels: gradient rows, then bias

template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(void *smem_dst, const void *src, bool valid) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
    const int n = valid ? BYTES : 0;                          // 0 source bytes: the destination is zero-filled
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src), "n"(BYTES), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void rgb_cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float rgb_peer(const float *mine, unsigned rank) {       // the same word in block `rank` of the cluster
    unsigned addr = (unsigned)__cvta_generic_to_shared(mine);
    float v;
    asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f32 %0, [a];\n\t}" : "=f"(v) : "r"(addr), "r"(rank) : "memory");
    return v;
}
__device__ __forceinline__ double rgb_peer(const double *mine, unsigned rank) {
    unsigned addr = (unsigned)__cvta_generic_to_shared(mine);
    double v;
    asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\tld.shared::cluster.f64 %0, [a];\n\t}" : "=d"(v) : "r"(addr), "r"(rank) : "memory");
    return v;
}

template <typename T>
__global__ void __launch_bounds__(kRgbThreads, 1)
conv_wgrad_rgb3_kernel(const T *__restrict__ X, const T *__restrict__ dY, const ConvGeom g, int cluster, int rows_per,
                       float *__restrict__ G_w, float *__restrict__ db, int has_bias, int separate,
                       float *__restrict__ sqnorm, long long sq_stride) {
    extern __shared__ __align__(16) float rgb_smem[];
    __shared__ double scratch[32];
    __shared__ float sums[kRgbSums];                         // this block's sums of the current 32 channels
    __shared__ double norm2[2];
    constexpr int kQuad = 4 * (int)sizeof(T);                // bytes of four output channels of dY
    const int Wp = g.W + 2 * g.pad, row_p = Wp * 3;
    char *ring = reinterpret_cast<char *>(rgb_smem);         // [kRgbStages][128 pixels][8 quads]
    float *xs = rgb_smem + kRgbStages * kRgbStageFloats;     // [input rows of this block][Wp][3], zero border
    const int n = blockIdx.x / cluster, rank = blockIdx.x - n * cluster;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, oct = w & 3, fr = w >> 2;
    const int oh0 = min(g.OH, rank * rows_per), oh1 = min(g.OH, oh0 + rows_per);
    const int pixels = (oh1 - oh0) * g.OW, rows_in = oh1 > oh0 ? (oh1 - oh0 - 1) * g.stride + 3 : 0;
    {
        const int row_in = g.W * 3, ih0 = oh0 * g.stride - g.pad;
        const T *Xn = X + (long long)n * g.H * row_in;
        for (int i = threadIdx.x; i < rows_in * row_p; i += kRgbThreads) {
            const int r = i / row_p, c = i - r * row_p - g.pad * 3, ih = ih0 + r;
            xs[i] = (ih >= 0 && ih < g.H && c >= 0 && c < row_in) ? to_float(Xn[(long long)ih * row_in + c]) : 0.f;
        }
    }
    const int stages = (pixels + kRgbStagePix - 1) / kRgbStagePix;
    // copies: thread t < 256 brings quad t%8 of pixels t/8, t/8 + 32, ... of a stage; reads: quads 2*oct and 2*oct + 1 of
    // pixel `lane` (+32 on each further trip)
    const int cl = threadIdx.x >> 3, cq = threadIdx.x & 7;
    const int copy_off = cl * 8 * kQuad + ((cq ^ (cl & 7)) * kQuad);        // (cl + 32) & 7 == cl & 7
    const int read0 = lane * 8 * kQuad + (((2 * oct) ^ (lane & 7)) * kQuad), read1 = lane * 8 * kQuad + (((2 * oct + 1) ^ (lane & 7)) * kQuad);
    float sq = 0.f, sqb = 0.f;
    for (int kg = 0; kg < g.Kout / 32; ++kg) {
        const T *dyp = dY + ((long long)n * g.K + (long long)oh0 * g.OW) * g.Kout + kg * 32;
        auto fetch = [&](int stage) {                        // one commit group per stage, also past the end
            if (threadIdx.x < 256) {
                char *dst = ring + (stage % kRgbStages) * (kRgbStageFloats * 4) + copy_off;
#pragma unroll
                for (int h = 0; h < kRgbStagePix / 32; ++h) {
                    const int p = stage * kRgbStagePix + cl + 32 * h;
                    const bool valid = stage < stages && p < pixels;
                    cp_async_zfill<kQuad>(dst + h * 32 * 8 * kQuad, dyp + (long long)(valid ? p : 0) * g.Kout + 4 * cq, valid);
                }
            }
            cp_async_commit();
        };
        unsigned long long acc[4][9], bs[4];                 // pairs of channels x columns of this warp's filter row
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            bs[k] = 0ull;
#pragma unroll
            for (int q = 0; q < 9; ++q) acc[k][q] = 0ull;
        }
        for (int t = 0; t < kRgbStages - 1; ++t) fetch(t);
        int oh = lane / g.OW, ow = lane - oh * g.OW;         // pixel of this lane in the current trip
        const unsigned long long one = pack2(1.f, 1.f);
        for (int st = 0; st < stages; ++st) {
            cp_async_wait<kRgbStages - 2>();                 // this thread's pieces of stage st have landed
            __syncthreads();                                 // ... and everyone's; stage st-1 is no longer read
            fetch(st + kRgbStages - 1);                      // refills the slot of stage st-1
            const char *src = ring + (st % kRgbStages) * (kRgbStageFloats * 4);
#pragma unroll 2
            for (int h = 0; h < kRgbStagePix / 32; ++h) {
                if (st * kRgbStagePix + 32 * h >= pixels) break;
                unsigned long long gy[4];
                if constexpr (sizeof(T) == 4) {
                    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(src + read0 + h * 32 * 8 * kQuad);
                    const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(src + read1 + h * 32 * 8 * kQuad);
                    gy[0] = a.x; gy[1] = a.y; gy[2] = b.x; gy[3] = b.y;
                } else {
                    const uint2 a = *reinterpret_cast<const uint2 *>(src + read0 + h * 32 * 8 * kQuad);
                    const uint2 b = *reinterpret_cast<const uint2 *>(src + read1 + h * 32 * 8 * kQuad);
                    gy[0] = pack2(__uint_as_float(a.x << 16), __uint_as_float(a.x & 0xffff0000u));
                    gy[1] = pack2(__uint_as_float(a.y << 16), __uint_as_float(a.y & 0xffff0000u));
                    gy[2] = pack2(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u));
                    gy[3] = pack2(__uint_as_float(b.y << 16), __uint_as_float(b.y & 0xffff0000u));
                }
                // lanes past the last pixel carry zeros of dY; their patch address is clamped to pixel 0
                const bool live = st * kRgbStagePix + 32 * h + lane < pixels;
                const float *row = xs + fr * row_p + (live ? oh * g.stride * row_p + ow * g.stride * 3 : 0);
                float x[9];
#pragma unroll
                for (int q = 0; q < 9; ++q) x[q] = row[q];
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    const unsigned long long xx = pack2(x[q], x[q]);
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[k][q] = fma2(gy[k], xx, acc[k][q]);
                }
                if (fr == 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) bs[k] = fma2(gy[k], one, bs[k]);
                }
                ow += 32;
                while (ow >= g.OW) { ow -= g.OW; ++oh; }
            }
        }
        cp_async_wait<0>();
        // fold the 32 pixel lanes by halving: 80 values (72 sums, 8 bias sums) -> 5, summed over 16 of the lanes, then the last step
        float v[80];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int q = 0; q < 9; ++q) asm("mov.b64 {%0, %1}, %2;" : "=f"(v[(2 * k) * 9 + q]), "=f"(v[(2 * k + 1) * 9 + q]) : "l"(acc[k][q]));
            asm("mov.b64 {%0, %1}, %2;" : "=f"(v[72 + 2 * k]), "=f"(v[73 + 2 * k]) : "l"(bs[k]));
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int half = 40 >> s, mask = 16 >> s;
            const bool up = (lane & mask) != 0;
#pragma unroll
            for (int i = 0; i < 40; ++i) {
                if (i < half) {
                    const float keep = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
                }
            }
        }
        const int base = ((lane & 16) ? 40 : 0) + ((lane & 8) ? 20 : 0) + ((lane & 4) ? 10 : 0) + ((lane & 2) ? 5 : 0);
        __syncthreads();                                     // sums[] of the previous channels are no longer read
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const float t = v[i] + __shfl_xor_sync(0xffffffffu, v[i], 1);
            const int e = base + i;                          // 0..71: (channel of the octet, column), 72..79: bias
            if (!(lane & 1)) {
                if (e < 72) sums[(8 * oct + e / 9) * 27 + fr * 9 + e % 9] = t;
                else if (fr == 0) sums[32 * 27 + 8 * oct + e - 72] = t;
            }
        }
        if (cluster > 1) rgb_cluster_sync(); else __syncthreads();
        // block `rank` finishes every cluster-th piece of the sums, adding the blocks in one order
        for (int o = rank * kRgbThreads + threadIdx.x; o < kRgbSums; o += cluster * kRgbThreads) {
            float t = sums[o];
            if (cluster > 1) {
                float part[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) { part[c] = 0.f; if (c < cluster) part[c] = rgb_peer(&sums[o], (unsigned)c); }
                t = ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
            }
            if (o < 32 * 27) {
                if (G_w) G_w[(long long)n * g.Kout * 27 + kg * 864 + o] = t;
                sq = fmaf(t, t, sq);
            } else if (has_bias) {
                db[(long long)n * g.Kout + kg * 32 + o - 864] = t;
                sqb = fmaf(t, t, sqb);
            }
        }
        if (cluster > 1 && (kg + 1) * 32 < g.Kout) rgb_cluster_sync();       // nobody overwrites its sums while a peer may read them
    }
    const double mw = block_sum((double)sq, scratch), mb = has_bias ? block_sum((double)sqb, scratch) : 0.0;
    if (threadIdx.x == 0) { norm2[0] = mw; norm2[1] = mb; }
    if (cluster > 1) rgb_cluster_sync(); else __syncthreads();
    if (rank == 0 && threadIdx.x == 0) {
        double sw = norm2[0], sb = norm2[1];
        if (cluster > 1) {
            double pw[8], pb[8];
#pragma unroll
            for (int c = 1; c < 8; ++c) {
                pw[c] = pb[c] = 0.0;
                if (c < cluster) { pw[c] = rgb_peer(&norm2[0], (unsigned)c); pb[c] = rgb_peer(&norm2[1], (unsigned)c); }
            }
#pragma unroll
            for (int c = 1; c < 8; ++c) { sw += pw[c]; sb += pb[c]; }
        }
        if (separate) {
            sqnorm[n * sq_stride] = (float)sw;
            sqnorm[n * sq_stride + 1] = (float)sb;
        } else {
            sqnorm[n * sq_stride] = (float)(sw + sb);
        }
    }
    if (cluster > 1) rgb_cluster_sync();                     // block 0 has read its peers: they may leave
}

// Blocks per example and output rows per block: as many as run side by side (a cluster needs its SMs at the same time: 32
// examples of 1024 pixels took 21 us as clusters of eight, of which 15 fit), as long as each keeps 128 pixels, and at
// least so many that a block's input rows fit beside the ring.
constexpr size_t kRgbSmemMost = 160 * 1024;
static size_t rgb3_smem_bytes(const ConvGeom &g, int rows_per) {
    return sizeof(float) * ((size_t)((rows_per - 1) * g.stride + 3) * (g.W + 2 * g.pad) * 3 + (size_t)kRgbStages * kRgbStageFloats);
}
static int rgb3_side_by_side(int cluster) { return cluster == 1 ? sm_count() : (cluster == 2 ? sm_count() / 2 : sm_count() * 4 / 5 / cluster); }
static bool rgb3_split(const ConvGeom &g, int &cluster, int &rows_per) {
    bool found = false;
    for (int c = 1; c <= 8; c *= 2) {
        const int rows = (g.OH + c - 1) / c;
        if (rgb3_smem_bytes(g, rows) > kRgbSmemMost) continue;
        if (found && (g.B > rgb3_side_by_side(c) || (long long)rows * g.OW < 128)) break;
        cluster = c; rows_per = rows; found = true;
    }
    return found;
}

bool rgb3_conv_eligible(const ConvGeom &g) {
    int cluster, rows_per;
    return g.R == 3 && g.S == 3 && g.Cin == 3 && g.Kout % 32 == 0 && g.Kout <= 256 && g.W <= 512 && g.B <= (1 << 27) && rgb3_split(g, cluster, rows_per);
}

template <typename T>
static dp_status launch_rgb3_t(const T *X, const T *dY, const ConvGeom &g, float *G_w, float *db, int has_bias, int separate,
                               float *sqnorm, long long sq_stride, cudaStream_t st) {
    int cluster, rows_per;
    if (!rgb3_split(g, cluster, rows_per)) return DP_ERR_UNSUPPORTED;
    // (the limit belongs to a function in one context: raised for every launch)
    DP_CUDA_TRY(cudaFuncSetAttribute(conv_wgrad_rgb3_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRgbSmemMost));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.B * cluster)); cfg.blockDim = dim3(kRgbThreads);
    cfg.dynamicSmemBytes = rgb3_smem_bytes(g, rows_per); cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    const cudaError_t le = cudaLaunchKernelEx(&cfg, conv_wgrad_rgb3_kernel<T>, X, dY, g, cluster, rows_per, G_w, db, has_bias, separate, sqnorm, sq_stride);
    if (le != cudaSuccess) return cuda_fail(le, "conv_wgrad_rgb3_kernel");
    DP_LAUNCH_CHECK("conv_wgrad_rgb3_kernel");
    return DP_OK;
}

dp_status launch_conv_rgb3(int dtype, const void *X, const void *dY, const ConvGeom &g, float *G_w, float *db,
                           int has_bias, int separate, float *sqnorm, long long sq_stride,
                           cudaStream_t st) {
    if (dtype == DP_F32) return launch_rgb3_t(static_cast<const float *>(X), static_cast<const float *>(dY), g, G_w, db, has_bias, separate, sqnorm, sq_stride, st);
    return launch_rgb3_t(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), g, G_w, db, has_bias, separate, sqnorm, sq_stride, st);
}

// db[n, k] = sum over pixels of dY[n, pix, k]; 64 channels x 4 pixel lanes per block, lanes folded in order.
template <typename T>
__global__ void __launch_bounds__(256)
bias_kernel(const T *__restrict__ dY, int K, int Kout, float *__restrict__ db, float *__restrict__ partial, int slots,
            int slot0) {
    __shared__ float lanes[4][kBiasCols];
    __shared__ float scratch[32];
    const int n = blockIdx.y, col = threadIdx.x & 63, lane = threadIdx.x >> 6;
    const int k = blockIdx.x * kBiasCols + col;
    float a = 0.f;
    if (k < Kout) {
        const T *p = dY + (long long)n * K * Kout + k;
        for (int pix = lane; pix < K; pix += 4) a += to_float(p[(long long)pix * Kout]);
    }
    lanes[lane][col] = a;
    __syncthreads();
    float sq = 0.f;
    if (lane == 0 && k < Kout) {
        const float v = (lanes[0][col] + lanes[1][col]) + (lanes[2][col] + lanes[3][col]);
        db[(long long)n * Kout + k] = v;
        sq = v * v;
    }
    sq = block_sum(sq, scratch);
    if (threadIdx.x == 0) partial[(long long)n * slots + slot0 + blockIdx.x] = sq;
}

// Vectorised variant for channel counts that are a multiple of one 16-byte vector (and at most 256 vectors):
// one block per example, thread = (pixel row, channel vector), 16-byte loads, pixel rows folded in order.
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
bias_vec_kernel(const T *__restrict__ dY, int K, int Kout, float *__restrict__ db, float *__restrict__ partial, int slots,
                int slot0, int bias_slots, float *__restrict__ sqnorm, long long sq_stride) {
    extern __shared__ float red[];                     // [rows][Kout]
    __shared__ float scratch[32];
    const int n = blockIdx.x;
    const int lanes_k = Kout / VEC, rows = 256 / lanes_k;
    const int prow = threadIdx.x / lanes_k, kv = threadIdx.x - prow * lanes_k;
    float a[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) a[v] = 0.f;
    if (prow < rows) {
        const T *base = dY + (long long)n * K * Kout + kv * VEC;
        // eight pixels per trip, all loads issued before any addition (a block is one example: few threads, so the
        // loads in flight per thread are what hides the memory latency); pixels still add in pixel order
        for (int pix = prow; pix < K; pix += 8 * rows) {
            uint4 g[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (pix + u * rows < K) g[u] = __ldcs(reinterpret_cast<const uint4 *>(base + (long long)(pix + u * rows) * Kout));
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (pix + u * rows < K) {
                    const T *gv = reinterpret_cast<const T *>(&g[u]);
#pragma unroll
                    for (int v = 0; v < VEC; ++v) a[v] += to_float(gv[v]);
                }
            }
        }
#pragma unroll
        for (int v = 0; v < VEC; ++v) red[prow * Kout + kv * VEC + v] = a[v];
    }
    __syncthreads();
    float sq = 0.f;
    for (int k = threadIdx.x; k < Kout; k += 256) {
        float v = 0.f;
        for (int r = 0; r < rows; ++r) v += red[r * Kout + k];
        db[(long long)n * Kout + k] = v;
        sq = fmaf(v, v, sq);
    }
    sq = block_sum(sq, scratch);
    if (threadIdx.x < bias_slots) partial[(long long)n * slots + slot0 + threadIdx.x] = (threadIdx.x == 0) ? sq : 0.f;
    if (sqnorm && threadIdx.x == 0) sqnorm[n * sq_stride] = sq;        // the bias is a group of its own: this is its whole norm
}

// One block per example: weight slots [0, w_slots) and bias slots [w_slots, slots) summed in index order.
__global__ void __launch_bounds__(128)
finalize_norm_kernel(const float *__restrict__ partial, int slots, int w_slots, int separate, float *__restrict__ sqnorm,
                     long long sq_stride, int clip, float C_l, float *__restrict__ factor, float *clip_out) {
    __shared__ double scratch[32];
    const int n = blockIdx.x;
    const float *p = partial + (long long)n * slots;
    double sw = 0.0, sb = 0.0;
    for (int i = threadIdx.x; i < w_slots; i += 128) sw += (double)p[i];
    for (int i = w_slots + threadIdx.x; i < slots; i += 128) sb += (double)p[i];
    sw = block_sum(sw, scratch);
    sb = block_sum(sb, scratch);
    if (threadIdx.x != 0) return;
    if (separate) {
        sqnorm[n * sq_stride] = (float)sw;
        sqnorm[n * sq_stride + 1] = (float)sb;
        if (clip) {
            const float fw = clip_factor(sw, C_l), fb = clip_factor(sb, C_l);
            factor[2 * n] = fw; factor[2 * n + 1] = fb;
            if (clip_out) { clip_out[2 * n] = fw; clip_out[2 * n + 1] = fb; }
        }
    } else {
        const double s = sw + sb;
        sqnorm[n * sq_stride] = (float)s;
        if (clip) {
            const float f = clip_factor(s, C_l);
            factor[2 * n] = f; factor[2 * n + 1] = f;
            if (clip_out) clip_out[n] = f;
        }
    }
}

// acc[k] += sum_n f[n * f_stride] * v[n, k].  Block = 32 channels x 8 example groups (group q owns examples
// q, q+8, ...), groups folded in order.
template <typename T>
__global__ void __launch_bounds__(256)
bias_accum_kernel(const T *__restrict__ db, int B, int Kout, const float *__restrict__ f, long long f_stride,
                  float *__restrict__ acc_b) {
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    float a = 0.f;
    if (k < Kout) {
#pragma unroll 8
        for (int n = q; n < B; n += 8) a = fmaf(f[n * f_stride], to_float(db[(long long)n * Kout + k]), a);
    }
    part[q][lane] = a;
    __syncthreads();
    if (q == 0 && k < Kout) {
        float t = part[0][lane];
#pragma unroll
        for (int i = 1; i < 8; ++i) t += part[i][lane];
        acc_b[k] += t;
    }
}

// Dense layer, clipped sum with known factors: acc[o, i] += sum_n (f_n dY[n, o]) X[n, i], a matrix product with the
// batch as the reduction axis and a tiny output.  Block = 32 input columns x 16 outputs; its eight warps share the
// examples (warp q owns q, q+8, ...), the scaled dY rows sit in shared memory, and the eight partial tiles are folded
// in warp order.  Bound by latency and by the accumulator's read-modify-write, not by arithmetic.
constexpr int kDenseOT = 16;
template <typename T>
__global__ void __launch_bounds__(256)
dense_scaled_sum_kernel(const T *__restrict__ X, const T *__restrict__ dY, const float *__restrict__ factor,
                        long long f_stride, int B, int Cin, int Kout, float *__restrict__ acc,
                        const float *__restrict__ factor_b, long long fb_stride, float *__restrict__ acc_b) {
    __shared__ __align__(16) float fy[256][kDenseOT];
    __shared__ float part[8][kDenseOT][32];
    __shared__ float bsum[16][kDenseOT];
    // the bias gradient of a dense layer is dY itself: the first column block of every output group also adds
    // acc_b[o] += sum_n fb_n dY[n, o] (16 outputs x 16 example groups, groups folded in order), which saves a launch
    if (acc_b && blockIdx.x == 0) {
        const int o = threadIdx.x & (kDenseOT - 1), gq = threadIdx.x >> 4, oo = blockIdx.y * kDenseOT + o;
        float sum = 0.f;
        if (oo < Kout) {
#pragma unroll 8
            for (int n = gq; n < B; n += 16) sum = fmaf(factor_b[n * fb_stride], to_float(dY[(long long)n * Kout + oo]), sum);
        }
        bsum[gq][o] = sum;
        __syncthreads();
        if (threadIdx.x < kDenseOT && blockIdx.y * kDenseOT + threadIdx.x < Kout) {
            float t = bsum[0][threadIdx.x];
#pragma unroll
            for (int g2 = 1; g2 < 16; ++g2) t += bsum[g2][threadIdx.x];
            acc_b[blockIdx.y * kDenseOT + threadIdx.x] += t;
        }
    }
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane, o0 = blockIdx.y * kDenseOT;
    float a[kDenseOT];
#pragma unroll
    for (int o = 0; o < kDenseOT; ++o) a[o] = 0.f;
    for (int n0 = 0; n0 < B; n0 += 256) {
        const int nb = min(256, B - n0);
        __syncthreads();
        for (int t = threadIdx.x; t < nb * kDenseOT; t += 256) {
            const int n = t / kDenseOT, o = t - n * kDenseOT;
            fy[n][o] = (o0 + o < Kout) ? factor[(n0 + n) * f_stride] * to_float(dY[(long long)(n0 + n) * Kout + o0 + o]) : 0.f;
        }
        __syncthreads();
        if (i < Cin) {
#pragma unroll 8
            for (int n = q; n < nb; n += 8) {
                const float x = to_float(X[(long long)(n0 + n) * Cin + i]);
                const float4 *row = reinterpret_cast<const float4 *>(fy[n]);
#pragma unroll
                for (int v = 0; v < kDenseOT / 4; ++v) {
                    const float4 y = row[v];
                    a[4 * v] = fmaf(y.x, x, a[4 * v]); a[4 * v + 1] = fmaf(y.y, x, a[4 * v + 1]);
                    a[4 * v + 2] = fmaf(y.z, x, a[4 * v + 2]); a[4 * v + 3] = fmaf(y.w, x, a[4 * v + 3]);
                }
            }
        }
    }
#pragma unroll
    for (int o = 0; o < kDenseOT; ++o) part[q][o][lane] = a[o];
    __syncthreads();
    // 512 tile entries, two per thread: entry e = (output e / 32, column e % 32)
    for (int e = threadIdx.x; e < kDenseOT * 32; e += 256) {
        const int o = e >> 5, c = e & 31;
        if (o0 + o < Kout && blockIdx.x * 32 + c < Cin) {
            float t = part[0][o][c];
#pragma unroll
            for (int w = 1; w < 8; ++w) t += part[w][o][c];
            acc[(long long)(o0 + o) * Cin + blockIdx.x * 32 + c] += t;
        }
    }
}

// The same for outputs large enough to fill the GPU: block = 128 input columns x 32 outputs, warp = 4 outputs, thread = 4 x 4 of
// the tile, which walks through all examples: 16 FMAs for one load of X (the block's eight warps share it in the L1) and
// one of shared memory, nothing to fold.  Bound by the accumulator's read-modify-write: 2048 x 1000 for 8 examples 19 us
// in blocks of 32 x 16, whose fold through shared memory outweighed the product.
constexpr int kDenseWideCols = 128, kDenseWideOuts = 32;
__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
template <typename T>
__global__ void __launch_bounds__(256)
dense_scaled_sum_wide_kernel(const T *__restrict__ X, const T *__restrict__ dY, const float *__restrict__ factor,
                             long long f_stride, int B, int Cin, int Kout, float *__restrict__ acc,
                             const float *__restrict__ factor_b, long long fb_stride, float *__restrict__ acc_b) {
    __shared__ __align__(16) float fy[128][kDenseWideOuts];
    __shared__ float bsum[8][kDenseWideOuts];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int i = blockIdx.x * kDenseWideCols + 4 * lane, o0 = blockIdx.y * kDenseWideOuts;
    if (acc_b && blockIdx.x == 0) {                          // the bias: outputs by lane, examples by warp
        float sum = 0.f;
        if (o0 + lane < Kout) {
#pragma unroll 4
            for (int n = q; n < B; n += 8) sum = fmaf(factor_b[n * fb_stride], to_float(dY[(long long)n * Kout + o0 + lane]), sum);
        }
        bsum[q][lane] = sum;
        __syncthreads();
        if (q == 0 && o0 + lane < Kout) {
            float t = bsum[0][lane];
#pragma unroll
            for (int g = 1; g < 8; ++g) t += bsum[g][lane];
            acc_b[o0 + lane] += t;
        }
    }
    float4 a[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) a[o] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int n0 = 0; n0 < B; n0 += 128) {
        const int nb = min(128, B - n0);
        __syncthreads();
        for (int n = q; n < nb; n += 8)
            fy[n][lane] = o0 + lane < Kout ? factor[(n0 + n) * f_stride] * to_float(dY[(long long)(n0 + n) * Kout + o0 + lane]) : 0.f;
        __syncthreads();
        if (i >= Cin) continue;
#pragma unroll 8
        for (int n = 0; n < nb; ++n) {
            const float4 x = load4(X + (long long)(n0 + n) * Cin + i), y = *reinterpret_cast<const float4 *>(&fy[n][4 * q]);
            a[0].x = fmaf(y.x, x.x, a[0].x); a[0].y = fmaf(y.x, x.y, a[0].y); a[0].z = fmaf(y.x, x.z, a[0].z); a[0].w = fmaf(y.x, x.w, a[0].w);
            a[1].x = fmaf(y.y, x.x, a[1].x); a[1].y = fmaf(y.y, x.y, a[1].y); a[1].z = fmaf(y.y, x.z, a[1].z); a[1].w = fmaf(y.y, x.w, a[1].w);
            a[2].x = fmaf(y.z, x.x, a[2].x); a[2].y = fmaf(y.z, x.y, a[2].y); a[2].z = fmaf(y.z, x.z, a[2].z); a[2].w = fmaf(y.z, x.w, a[2].w);
            a[3].x = fmaf(y.w, x.x, a[3].x); a[3].y = fmaf(y.w, x.y, a[3].y); a[3].z = fmaf(y.w, x.z, a[3].z); a[3].w = fmaf(y.w, x.w, a[3].w);
        }
    }
    if (i >= Cin) return;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        if (o0 + 4 * q + o >= Kout) continue;
        float4 *dst = reinterpret_cast<float4 *>(acc + (long long)(o0 + 4 * q + o) * Cin + i);
        float4 t = *dst;
        t.x += a[o].x; t.y += a[o].y; t.z += a[o].z; t.w += a[o].w;
        *dst = t;
    }
}

// factor2[n] = (factor_w[n*stride], factor_b[n*stride]): caller-supplied factors in the layout the clipped-sum kernels read
__global__ void expand_factor_kernel(const float *__restrict__ factor_w, const float *__restrict__ factor_b,
                                     long long stride, int B, float *__restrict__ factor2) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= B) return;
    factor2[2 * n] = factor_w[n * stride];
    factor2[2 * n + 1] = factor_b[n * stride];
}

// ------------------------------------------------------------------ dense layer
// Dense layer, everything but the outer-product store, a block for an example: the rank-1 closed form of the squared
// norm (|dY_n^T X_n|_F^2 = |dY_n|^2 |X_n|^2, bias part |dY_n|^2), the bias gradient db_n = dY_n widened to fp32 (when
// a destination is given), and the same publishing of norms / clip factors the convolution paths do in a kernel of its own.
template <typename T>
__device__ __forceinline__ void dense_norm(int n, const T *__restrict__ X, const T *__restrict__ dY, int Cin, int Kout, int has_bias,
                                           float *__restrict__ db, int separate, float *__restrict__ sqnorm, long long sq_stride,
                                           int clip, float C_l, float *__restrict__ factor, float *clip_out) {
    __shared__ double scratch[32];
    double sx = 0.0, sy = 0.0;
    for (int i = threadIdx.x; i < Cin; i += 256) { const double v = to_float(X[(long long)n * Cin + i]); sx += v * v; }
    for (int i = threadIdx.x; i < Kout; i += 256) {
        const float g = to_float(dY[(long long)n * Kout + i]);
        if (db) db[(long long)n * Kout + i] = g;
        sy += (double)g * g;
    }
    sx = block_sum(sx, scratch);
    sy = block_sum(sy, scratch);
    if (threadIdx.x != 0) return;
    const double sw = sx * sy, sb = has_bias ? sy : 0.0;
    if (separate) {
        sqnorm[n * sq_stride] = (float)sw;
        sqnorm[n * sq_stride + 1] = (float)sb;
        if (clip) {
            const float fw = clip_factor(sw, C_l), fb = clip_factor(sb, C_l);
            factor[2 * n] = fw; factor[2 * n + 1] = fb;
            if (clip_out) { clip_out[2 * n] = fw; clip_out[2 * n + 1] = fb; }
        }
    } else {
        sqnorm[n * sq_stride] = (float)(sw + sb);
        if (clip) {
            const float f = clip_factor(sw + sb, C_l);
            factor[2 * n] = f; factor[2 * n + 1] = f;
            if (clip_out) clip_out[n] = f;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
dense_norm_kernel(const T *__restrict__ X, const T *__restrict__ dY, int Cin, int Kout, int has_bias, float *__restrict__ db,
                  int separate, float *__restrict__ sqnorm, long long sq_stride, int clip, float C_l,
                  float *__restrict__ factor, float *clip_out) {
    dense_norm(blockIdx.x, X, dY, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, clip, C_l, factor, clip_out);
}

// Dense layer with its gradients stored, G_w[n, o, :] = dY[n, o] * X[n, :]: the first B blocks are the norms, the others the
// outer product.  Bound by the stores.  A thread keeps VEC columns of X and walks down the outputs, so what a block reads
// is small beside what it writes (a block an output, which reads X again for each, wrote 2048 x 1000 for 16 examples at
// 4.2 TB/s; and small layers are bound by their launches, of which there were two).
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
dense_store_norm_kernel(const T *__restrict__ X, const T *__restrict__ dY, int B, int Cin, int Kout, int tpc, int outs, int col_blocks,
                        int out_blocks, int has_bias, float *__restrict__ db, int separate, float *__restrict__ sqnorm,
                        long long sq_stride, float *__restrict__ G_w) {
    if ((int)blockIdx.x < B) {
        dense_norm(blockIdx.x, X, dY, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, 0, 0.f, (float *)nullptr, (float *)nullptr);
        return;
    }
    const int blk = (int)blockIdx.x - B, cb = blk % col_blocks, rest = blk / col_blocks, ob = rest % out_blocks, n = rest / out_blocks;
    const int teams = 256 / tpc, team = threadIdx.x / tpc, col = (cb * tpc + threadIdx.x - team * tpc) * VEC;
    if (team >= teams || col >= Cin) return;
    const T *x = X + (long long)n * Cin + col, *gy = dY + (long long)n * Kout;
    float xv[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) xv[v] = to_float(x[v]);
    const int o1 = min(Kout, (ob + 1) * outs);
    float *out = G_w + (long long)n * Kout * Cin + col;
#pragma unroll 4
    for (int o = ob * outs + team; o < o1; o += teams) {
        const float g = to_float(gy[o]);
        if constexpr (VEC == 4) __stcs(reinterpret_cast<float4 *>(out + (long long)o * Cin), make_float4(g * xv[0], g * xv[1], g * xv[2], g * xv[3]));
        else out[(long long)o * Cin] = g * xv[0];
    }
}

// ------------------------------------------------------------------ normalisation affine
// What the last thread block to finish an example does in the one-launch form of the layer: fold the example's
// pixel-chunk partial sums in chunk order, publish its squared norms (and clip factors), and -- when it is also the
// last block of the whole call and the batch is small enough to walk alone -- add the clipped sum over the examples
// to the accumulators.  "Last" is found with ticket counters (no block ever waits for another); the arithmetic and
// its order do not depend on which block turns out to be last, so results stay bit-reproducible.
struct AffineTail {
    int *counters;            // [B + 1] tickets: one per example, one for the call; zero on entry, left at zero.  null: off
    int blocks_per_example;
    int B;
    int clip;                 // 1: factors against C_l, clipped sum into acc_w / acc_b;  0: norms only
    int accumulate_here;      // 1: the last block of the call adds the clipped sum itself; 0: a second launch does
    int separate;
    float C_l;
    float *sqnorm; long long sq_stride; float *clip_out;
    float *factor;            // [B][2] scratch: (scale factor, shift factor) per example
    float *dgamma, *dbeta;    // [B][C] finished per-example gradients (scratch, or the caller's G_w / G_b)
    float *acc_w, *acc_b;
};

__device__ __forceinline__ void affine_tail(const AffineTail &t, int n, bool whole, const float *chunk_partial, int chunks,
                                            int C, double qg, double qb, double *scratch) {
    __shared__ int last_flag;
    if (!whole) {
        __threadfence();                                   // this block's chunk partials are visible before its ticket
        __syncthreads();
        if (threadIdx.x == 0) last_flag = (atomicAdd(&t.counters[n], 1) == t.blocks_per_example - 1);
        __syncthreads();
        if (!last_flag) return;
        __threadfence();
        qg = 0.0; qb = 0.0;
        for (int c = threadIdx.x; c < C; c += 256) {
            float a = 0.f, b = 0.f;
            const float *p = chunk_partial + ((long long)n * chunks * 2) * C + c;
            int k = 0;
            for (; k + 8 <= chunks; k += 8) {              // eight chunks' loads in flight, added in chunk order
                float x[8], y[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) { x[u] = __ldcg(p + (long long)(k + u) * 2 * C); y[u] = __ldcg(p + (long long)(k + u) * 2 * C + C); }
#pragma unroll
                for (int u = 0; u < 8; ++u) { a += x[u]; b += y[u]; }
            }
            for (; k < chunks; ++k) { a += __ldcg(p + (long long)k * 2 * C); b += __ldcg(p + (long long)k * 2 * C + C); }
            t.dgamma[(long long)n * C + c] = a;
            t.dbeta[(long long)n * C + c] = b;
            qg += (double)a * a;
            qb += (double)b * b;
        }
        qg = block_sum(qg, scratch);
        qb = block_sum(qb, scratch);
        if (threadIdx.x == 0) t.counters[n] = 0;
    }
    if (threadIdx.x == 0) {
        float f0 = 1.f, f1 = 1.f;
        if (t.separate) {
            t.sqnorm[n * t.sq_stride] = (float)qg; t.sqnorm[n * t.sq_stride + 1] = (float)qb;
            if (t.clip) { f0 = clip_factor(qg, t.C_l); f1 = clip_factor(qb, t.C_l); }
            if (t.clip && t.clip_out) { t.clip_out[2 * n] = f0; t.clip_out[2 * n + 1] = f1; }
        } else {
            t.sqnorm[n * t.sq_stride] = (float)(qg + qb);
            if (t.clip) f0 = f1 = clip_factor(qg + qb, t.C_l);
            if (t.clip && t.clip_out) t.clip_out[n] = f0;
        }
        t.factor[2 * n] = f0; t.factor[2 * n + 1] = f1;
    }
    if (!t.clip || !t.accumulate_here) return;
    __threadfence();                                       // this example's gradients and factors before the call's ticket
    __syncthreads();
    if (threadIdx.x == 0) {
        last_flag = (atomicAdd(&t.counters[t.B], 1) == t.B - 1);
        if (last_flag) t.counters[t.B] = 0;
    }
    __syncthreads();
    if (!last_flag) return;
    __threadfence();
    // thread = (channel, tensor); the factors of up to 256 examples at a time sit in shared memory and eight examples'
    // values are in flight per thread (the walk is latency-bound: everything comes from L2)
    __shared__ float f_sh[2][256];
    for (int c0 = 0; c0 < 2 * C; c0 += 256) {
        const int e = c0 + threadIdx.x;
        const int which = e >= C, c = which ? e - C : e;
        const float *v = (which ? t.dbeta : t.dgamma) + c;
        float a = 0.f;
        for (int m0 = 0; m0 < t.B; m0 += 256) {
            const int mb = min(256, t.B - m0);
            __syncthreads();
            if (threadIdx.x < mb) {
                f_sh[0][threadIdx.x] = __ldcg(t.factor + 2 * (m0 + threadIdx.x));
                f_sh[1][threadIdx.x] = __ldcg(t.factor + 2 * (m0 + threadIdx.x) + 1);
            }
            __syncthreads();
            if (e < 2 * C) {
                int m = 0;
                for (; m + 8 <= mb; m += 8) {
                    float x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) x[u] = __ldcg(v + (long long)(m0 + m + u) * C);
#pragma unroll
                    for (int u = 0; u < 8; ++u) a = fmaf(f_sh[which][m + u], x[u], a);
                }
                for (; m < mb; ++m) a = fmaf(f_sh[which][m], __ldcg(v + (long long)(m0 + m) * C), a);
            }
        }
        if (e < 2 * C) (which ? t.acc_b : t.acc_w)[c] += a;
    }
}

// stage 1: block = (channel-vector block, pixel chunk, example); thread = (pixel row, channel vector).
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
norm_affine_partial_kernel(const T *__restrict__ X, const T *__restrict__ dY, int HW, int C, int tcv, int pix,
                           float *__restrict__ chunk_partial, int chunks, float *__restrict__ dgamma,
                           float *__restrict__ dbeta, float *__restrict__ partial2, const AffineTail tail) {
    extern __shared__ float red[];                       // [rows][tcv*VEC*2]
    const int n = blockIdx.z, chunk = blockIdx.y;
    const int rows = 256 / tcv;
    const int prow = threadIdx.x / tcv, cvi = threadIdx.x - prow * tcv;
    const int c0 = (blockIdx.x * tcv + cvi) * VEC;
    float sg[VEC], sb[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) { sg[v] = 0.f; sb[v] = 0.f; }
    const int p_end = min(HW, (chunk + 1) * pix);
    if (prow < rows && c0 < C) affine_pixel_sums<T, VEC>(X, dY, (long long)n * HW, C, c0, chunk * pix + prow, p_end, rows, sg, sb);
    const int width = tcv * VEC * 2;
    if (prow < rows) affine_stage_sums<VEC>(red, prow, cvi, tcv, sg, sb);
    __syncthreads();
    // every thread folds one output column over the pixel rows, in row order.  When this block holds the whole
    // example (one pixel chunk, all channels) the sums are final: it writes the gradients and both squared norms
    // itself and the separate folding launch is skipped (dgamma != nullptr says so).
    {
        __shared__ double scratch[32];
        const bool whole = dgamma != nullptr;
        float *out = chunk_partial + (((long long)n * chunks + chunk) * 2) * C;
        const int half = tcv * VEC;
        double qg = 0.0, qb = 0.0;
        for (int e = threadIdx.x; e < 2 * half; e += 256) {
            const int is_beta = e >= half;
            const int c = blockIdx.x * half + (is_beta ? e - half : e);
            if (c >= C) continue;
            float a = 0.f;
            for (int rr = 0; rr < rows; ++rr) a += red[rr * width + e];
            if (whole) {
                (is_beta ? dbeta : dgamma)[(long long)n * C + c] = a;
                if (is_beta) qb += (double)a * a; else qg += (double)a * a;
            } else {
                out[is_beta ? C + c : c] = a;
            }
        }
        if (whole) {
            qg = block_sum(qg, scratch);
            qb = block_sum(qb, scratch);
            if (threadIdx.x == 0 && !tail.counters) { partial2[2 * n] = (float)qg; partial2[2 * n + 1] = (float)qb; }
        }
        if (tail.counters) affine_tail(tail, n, whole, chunk_partial, chunks, C, qg, qb, scratch);
    }
}

// stage 2: fold chunks in index order, store dgamma / dbeta, squared norms of both
__global__ void __launch_bounds__(256)
norm_affine_fold_kernel(const float *__restrict__ chunk_partial, int chunks, int C, float *__restrict__ dgamma,
                        float *__restrict__ dbeta, float *__restrict__ partial2) {
    __shared__ double scratch[32];
    const int n = blockIdx.x;
    double qg = 0.0, qb = 0.0;
    for (int c = threadIdx.x; c < C; c += 256) {
        float a = 0.f, b = 0.f;
        for (int k = 0; k < chunks; ++k) {
            const float *p = chunk_partial + (((long long)n * chunks + k) * 2) * C;
            a += p[c];
            b += p[C + c];
        }
        dgamma[(long long)n * C + c] = a;
        dbeta[(long long)n * C + c] = b;
        qg += (double)a * a;
        qb += (double)b * b;
    }
    qg = block_sum(qg, scratch);
    qb = block_sum(qb, scratch);
    if (threadIdx.x == 0) { partial2[2 * n] = (float)qg; partial2[2 * n + 1] = (float)qb; }
}


// Normalisation layers, fused clip: every block works out the factors of all examples from the two squared norms
// (cheap and identical in every block), block 0 publishes norms and factors, then each thread owns one channel and
// adds sum_n f_n dgamma[n, c] / dbeta[n, c] to the accumulators.
__global__ void __launch_bounds__(128)
affine_clip_accum_kernel(const float *__restrict__ partial2, int B, float C_l, int separate, float *__restrict__ sqnorm,
                         long long sq_stride, float *clip_out, const float *__restrict__ dgamma,
                         const float *__restrict__ dbeta, int C, float *__restrict__ acc_w, float *__restrict__ acc_b) {
    __shared__ float fw[512], fb[512];
    const int c = blockIdx.x * 128 + threadIdx.x;
    float a = 0.f, b = 0.f;
    for (int n0 = 0; n0 < B; n0 += 512) {
        const int nb = min(512, B - n0);
        __syncthreads();
        for (int t = threadIdx.x; t < nb; t += 128) {
            const int n = n0 + t;
            const double sw = (double)partial2[2 * n], sb = (double)partial2[2 * n + 1];
            float f0, f1;
            if (separate) { f0 = clip_factor(sw, C_l); f1 = clip_factor(sb, C_l); }
            else { f0 = f1 = clip_factor(sw + sb, C_l); }
            fw[t] = f0; fb[t] = f1;
            if (blockIdx.x == 0) {
                if (separate) {
                    sqnorm[n * sq_stride] = (float)sw; sqnorm[n * sq_stride + 1] = (float)sb;
                    if (clip_out) { clip_out[2 * n] = f0; clip_out[2 * n + 1] = f1; }
                } else {
                    sqnorm[n * sq_stride] = (float)(sw + sb);
                    if (clip_out) clip_out[n] = f0;
                }
            }
        }
        __syncthreads();
        if (c < C) {
            const float *g = dgamma + (long long)n0 * C + c, *h = dbeta + (long long)n0 * C + c;
#pragma unroll 8
            for (int t = 0; t < nb; ++t) {
                a = fmaf(fw[t], g[(long long)t * C], a);
                b = fmaf(fb[t], h[(long long)t * C], b);
            }
        }
    }
    if (c < C) { acc_w[c] += a; acc_b[c] += b; }
}

dp_status launch_affine_clip_accum(const float *partial2, int B, float C_l, int separate, float *sqnorm, long long sq_stride,
                                   float *clip_out, const float *dgamma, const float *dbeta, int C, float *acc_w,
                                   float *acc_b, cudaStream_t st) {
    affine_clip_accum_kernel<<<(C + 127) / 128, 128, 0, st>>>(partial2, B, C_l, separate, sqnorm, sq_stride, clip_out, dgamma,
                                                            dbeta, C, acc_w, acc_b);
    DP_LAUNCH_CHECK("affine_clip_accum_kernel");
    return DP_OK;
}

// ------------------------------------------------------------------ host launchers
int fma_clip_splits(const ConvGeom &g) {
    const int tiles = fma_tiles_m(g) * fma_tiles_n(g);
    int want = (2 * sm_count()) / tiles;
    if (want < 1) want = 1;
    if (want > g.B) want = g.B;
    const int per = (g.B + want - 1) / want;
    return (g.B + per - 1) / per;
}

// acc[i] += sum_s ws[s][i], splits in index order
__global__ void fold_sums_kernel(const float *__restrict__ ws, int splits, long long P, float *__restrict__ acc) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    float a = acc[i];
    for (int s = 0; s < splits; ++s) a += ws[(long long)s * P + i];
    acc[i] = a;
}

template <typename T>
static dp_status conv_fma_t(int mode, const T *X, const T *dY, const ConvGeom &g, float *G_w, float *partial, int slots,
                            const float *factor, float *acc_w, float *sum_ws, cudaStream_t st) {
    const int splits = (mode == 2) ? fma_clip_splits(g) : 1;
    const int per = (g.B + splits - 1) / splits;
    const dim3 grid(fma_tiles_n(g), fma_tiles_m(g), mode == 2 ? splits : g.B);
    if (grid.y > 65535 || grid.z > 65535) return DP_ERR_UNSUPPORTED;
    if (mode == 0) conv_wgrad_fma_kernel<T, 0><<<grid, 256, 0, st>>>(X, dY, g, G_w, partial, slots, factor, acc_w, per, sum_ws);
    else if (mode == 1) conv_wgrad_fma_kernel<T, 1><<<grid, 256, 0, st>>>(X, dY, g, G_w, partial, slots, factor, acc_w, per, sum_ws);
    else conv_wgrad_fma_kernel<T, 2><<<grid, 256, 0, st>>>(X, dY, g, G_w, partial, slots, factor, acc_w, per, sum_ws);
    DP_LAUNCH_CHECK("conv_wgrad_fma_kernel");
    if (mode == 2 && splits > 1) {
        const long long P = (long long)g.M * g.N;
        fold_sums_kernel<<<(unsigned)((P + 255) / 256), 256, 0, st>>>(sum_ws, splits, P, acc_w);
        DP_LAUNCH_CHECK("fold_sums_kernel");
    }
    return DP_OK;
}

dp_status launch_conv_fma(int dtype, int mode, const void *X, const void *dY, const ConvGeom &g, float *G_w,
                          float *partial, int slots, const float *factor, float *acc_w, float *sum_ws, cudaStream_t st) {
    if (dtype == DP_F32)
        return conv_fma_t(mode, static_cast<const float *>(X), static_cast<const float *>(dY), g, G_w, partial, slots, factor, acc_w, sum_ws, st);
    return conv_fma_t(mode, static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), g, G_w, partial, slots, factor, acc_w, sum_ws, st);
}

bool bias_publishes(int dtype, const ConvGeom &g) {
    const int vec = (dtype == DP_F32) ? 4 : 8;
    return g.Kout % vec == 0 && g.Kout / vec <= 256 && bias_blocks(g) <= 256;
}

dp_status launch_bias(int dtype, const void *dY, const ConvGeom &g, float *db, float *partial, int slots, int slot0,
                      cudaStream_t st, float *sqnorm, long long sq_stride) {
    const int vec = (dtype == DP_F32) ? 4 : 8;
    if (bias_publishes(dtype, g)) {
        const size_t smem = sizeof(float) * (size_t)(256 / (g.Kout / vec)) * g.Kout;
        if (dtype == DP_F32)
            bias_vec_kernel<float, 4><<<g.B, 256, smem, st>>>(static_cast<const float *>(dY), g.K, g.Kout, db, partial, slots, slot0, bias_blocks(g), sqnorm, sq_stride);
        else
            bias_vec_kernel<__nv_bfloat16, 8><<<g.B, 256, smem, st>>>(static_cast<const __nv_bfloat16 *>(dY), g.K, g.Kout, db, partial, slots, slot0, bias_blocks(g), sqnorm, sq_stride);
        DP_LAUNCH_CHECK("bias_vec_kernel");
        return DP_OK;
    }
    const dim3 grid(bias_blocks(g), g.B);
    if (grid.y > 65535) return DP_ERR_UNSUPPORTED;
    if (dtype == DP_F32) bias_kernel<<<grid, 256, 0, st>>>(static_cast<const float *>(dY), g.K, g.Kout, db, partial, slots, slot0);
    else bias_kernel<<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(dY), g.K, g.Kout, db, partial, slots, slot0);
    DP_LAUNCH_CHECK("bias_kernel");
    return DP_OK;
}

dp_status launch_finalize(const float *partial, int B, int slots, int w_slots, int separate, float *sqnorm,
                          long long sq_stride, int clip, float C_l, float *factor, float *clip_out, cudaStream_t st) {
    finalize_norm_kernel<<<B, 128, 0, st>>>(partial, slots, w_slots, separate, sqnorm, sq_stride, clip, C_l, factor, clip_out);
    DP_LAUNCH_CHECK("finalize_norm_kernel");
    return DP_OK;
}

dp_status launch_bias_accum(const float *db, int B, int Kout, const float *factor, float *acc_b, cudaStream_t st, int which) {
    bias_accum_kernel<float><<<(Kout + 31) / 32, 256, 0, st>>>(db, B, Kout, factor + which, 2, acc_b);
    DP_LAUNCH_CHECK("bias_accum_kernel");
    return DP_OK;
}

dp_status launch_dense_scaled_sum(int dtype, const void *X, const void *dY, const float *factor, long long f_stride, int B,
                                  int Cin, int Kout, float *acc_w, cudaStream_t st, const float *factor_b, long long fb_stride,
                                  float *acc_b) {
    const long long wide = (long long)((Cin + kDenseWideCols - 1) / kDenseWideCols) * ((Kout + kDenseWideOuts - 1) / kDenseWideOuts);
    // (a classifier of few outputs would leave most of a tile's warps idle: 23232 x 10 for 122 examples 28 us slower)
    if (Cin % 4 == 0 && Kout >= 2 * kDenseWideOuts && aligned(acc_w, 16) && wide >= sm_count() && Kout <= 65535 * kDenseWideOuts) {
        const dim3 g((unsigned)((Cin + kDenseWideCols - 1) / kDenseWideCols), (unsigned)((Kout + kDenseWideOuts - 1) / kDenseWideOuts));
        if (dtype == DP_F32)
            dense_scaled_sum_wide_kernel<float><<<g, 256, 0, st>>>(static_cast<const float *>(X), static_cast<const float *>(dY), factor, f_stride, B, Cin, Kout, acc_w, factor_b, fb_stride, acc_b);
        else
            dense_scaled_sum_wide_kernel<__nv_bfloat16><<<g, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), factor, f_stride, B, Cin, Kout, acc_w, factor_b, fb_stride, acc_b);
        DP_LAUNCH_CHECK("dense_scaled_sum_wide_kernel");
        return DP_OK;
    }
    const dim3 grid((unsigned)((Cin + 31) / 32), (unsigned)((Kout + kDenseOT - 1) / kDenseOT));
    if (grid.y > 65535) return DP_ERR_UNSUPPORTED;
    if (dtype == DP_F32)
        dense_scaled_sum_kernel<float><<<grid, 256, 0, st>>>(static_cast<const float *>(X), static_cast<const float *>(dY), factor, f_stride, B, Cin, Kout, acc_w, factor_b, fb_stride, acc_b);
    else
        dense_scaled_sum_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), factor, f_stride, B, Cin, Kout, acc_w, factor_b, fb_stride, acc_b);
    DP_LAUNCH_CHECK("dense_scaled_sum_kernel");
    return DP_OK;
}

dp_status launch_expand_factor(const float *factor_w, const float *factor_b, long long stride, int B, float *factor2, cudaStream_t st) {
    expand_factor_kernel<<<(B + 127) / 128, 128, 0, st>>>(factor_w, factor_b, stride, B, factor2);
    DP_LAUNCH_CHECK("expand_factor_kernel");
    return DP_OK;
}

template <typename T, int VEC>
static dp_status dense_store_t(const T *X, const T *dY, int B, int Cin, int Kout, int has_bias, float *db, int separate, float *sqnorm,
                               long long sq_stride, float *G_w, cudaStream_t st) {
    const int tpc = std::min(256, (Cin + VEC - 1) / VEC), col_blocks = (Cin + tpc * VEC - 1) / (tpc * VEC), teams = 256 / tpc;
    // outputs a thread walks through: at most sixteen, fewer while that leaves less than eight blocks an SM
    const long long units = (long long)B * col_blocks * ((Kout + teams - 1) / teams);
    const int per = (int)std::max(1ll, std::min(16ll, units / (8ll * sm_count())));
    const int outs = per * teams, out_blocks = (Kout + outs - 1) / outs;
    const long long blocks = B + (long long)B * col_blocks * out_blocks;
    if (blocks > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
    dense_store_norm_kernel<T, VEC><<<(unsigned)blocks, 256, 0, st>>>(X, dY, B, Cin, Kout, tpc, outs, col_blocks, out_blocks, has_bias, db, separate, sqnorm, sq_stride, G_w);
    DP_LAUNCH_CHECK("dense_store_norm_kernel");
    return DP_OK;
}

dp_status launch_dense_store(int dtype, const void *X, const void *dY, int B, int Cin, int Kout, int has_bias, float *db, int separate,
                             float *sqnorm, long long sq_stride, float *G_w, cudaStream_t st) {
    if (dtype == DP_F32) {
        const float *x = static_cast<const float *>(X), *y = static_cast<const float *>(dY);
        return Cin % 4 == 0 ? dense_store_t<float, 4>(x, y, B, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, G_w, st)
                            : dense_store_t<float, 1>(x, y, B, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, G_w, st);
    }
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(X), *y = static_cast<const __nv_bfloat16 *>(dY);
    return Cin % 4 == 0 ? dense_store_t<__nv_bfloat16, 4>(x, y, B, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, G_w, st)
                        : dense_store_t<__nv_bfloat16, 1>(x, y, B, Cin, Kout, has_bias, db, separate, sqnorm, sq_stride, G_w, st);
}

dp_status launch_dense_norm(int dtype, const void *X, const void *dY, int B, int Cin, int Kout, int has_bias, float *db,
                            int separate, float *sqnorm, long long sq_stride, int clip, float C_l, float *factor,
                            float *clip_out, cudaStream_t st) {
    if (dtype == DP_F32)
        dense_norm_kernel<<<B, 256, 0, st>>>(static_cast<const float *>(X), static_cast<const float *>(dY), Cin, Kout, has_bias, db,
                                             separate, sqnorm, sq_stride, clip, C_l, factor, clip_out);
    else
        dense_norm_kernel<<<B, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), Cin, Kout,
                                             has_bias, db, separate, sqnorm, sq_stride, clip, C_l, factor, clip_out);
    DP_LAUNCH_CHECK("dense_norm_kernel");
    return DP_OK;
}

template <typename T, int VEC>
static dp_status norm_affine_t(const T *X, const T *dY, int B, int HW, int C, int tcv, int pix, float *chunk_partial,
                               float *dgamma, float *dbeta, float *partial2, bool &folded, AffineTail tail, cudaStream_t st) {
    const int cv = (C + VEC - 1) / VEC;
    const int chunks = (HW + pix - 1) / pix;
    const dim3 grid((cv + tcv - 1) / tcv, chunks, B);
    if (grid.y > 65535 || grid.z > 65535) return DP_ERR_UNSUPPORTED;
    const size_t smem = sizeof(float) * (size_t)(256 / tcv) * tcv * VEC * 2;
    folded = grid.x == 1 && chunks == 1;      // one block sees the whole example: it finishes the job itself
    tail.blocks_per_example = (int)(grid.x * grid.y);
    norm_affine_partial_kernel<T, VEC><<<grid, 256, smem, st>>>(X, dY, HW, C, tcv, pix, chunk_partial, chunks,
                                                               folded ? dgamma : nullptr, dbeta, partial2, tail);
    DP_LAUNCH_CHECK("norm_affine_partial_kernel");
    return DP_OK;
}

static dp_status norm_affine_dispatch(int dtype, const void *X, const void *dY, int B, int HW, int C, float *chunk_partial,
                                      float *dgamma, float *dbeta, float *partial2, bool &folded, const AffineTail &tail,
                                      cudaStream_t st) {
    int vec, tcv, pix;
    norm_shape(dtype, B, HW, C, vec, tcv, pix);
    if (dtype == DP_F32) {
        if ((C & 3) == 0) return norm_affine_t<float, 4>(static_cast<const float *>(X), static_cast<const float *>(dY), B, HW, C, tcv, pix, chunk_partial, dgamma, dbeta, partial2, folded, tail, st);
        return norm_affine_t<float, 1>(static_cast<const float *>(X), static_cast<const float *>(dY), B, HW, C, tcv, pix, chunk_partial, dgamma, dbeta, partial2, folded, tail, st);
    }
    if ((C & 7) == 0) return norm_affine_t<__nv_bfloat16, 8>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), B, HW, C, tcv, pix, chunk_partial, dgamma, dbeta, partial2, folded, tail, st);
    return norm_affine_t<__nv_bfloat16, 1>(static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(dY), B, HW, C, tcv, pix, chunk_partial, dgamma, dbeta, partial2, folded, tail, st);
}

dp_status launch_norm_affine(int dtype, const void *X, const void *dY, int B, int HW, int C, float *chunk_partial,
                             float *dgamma, float *dbeta, float *partial2, cudaStream_t st) {
    bool folded = false;
    AffineTail off = {};
    const dp_status rc = norm_affine_dispatch(dtype, X, dY, B, HW, C, chunk_partial, dgamma, dbeta, partial2, folded, off, st);
    if (rc != DP_OK || folded) return rc;
    norm_affine_fold_kernel<<<B, 256, 0, st>>>(chunk_partial, norm_chunks(dtype, B, HW, C), C, dgamma, dbeta, partial2);
    DP_LAUNCH_CHECK("norm_affine_fold_kernel");
    return DP_OK;
}

// acc_w[c] += sum_n factor[2n] * dgamma[n, c] and acc_b[c] += sum_n factor[2n + 1] * dbeta[n, c] in one launch
// (blockIdx.y picks the tensor).  Block = 32 channels x 8 example groups, groups folded in order.
__global__ void __launch_bounds__(256)
affine_accum_kernel(const float *__restrict__ dgamma, const float *__restrict__ dbeta, int B, int C,
                    const float *__restrict__ factor, float *__restrict__ acc_w, float *__restrict__ acc_b) {
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5, which = blockIdx.y;
    const float *v = which ? dbeta : dgamma;
    const int c = blockIdx.x * 32 + lane;
    float a = 0.f;
    if (c < C) {
#pragma unroll 8
        for (int n = q; n < B; n += 8) a = fmaf(factor[2 * n + which], v[(long long)n * C + c], a);
    }
    part[q][lane] = a;
    __syncthreads();
    if (q == 0 && c < C) {
        float t = part[0][lane];
#pragma unroll
        for (int i = 1; i < 8; ++i) t += part[i][lane];
        (which ? acc_b : acc_w)[c] += t;
    }
}

bool affine_fused_eligible(int B) { return B + 1 <= kWsCounters - kWsBatchCounters; }

// The whole layer call in one launch (two when the batch times the channel count is large): per-example gradients,
// their squared norms, and for clip != 0 the factors against C_l and the clipped sums.  dgamma / dbeta: [B][C]
// scratch or the caller's outputs; factor: [B][2] scratch; counters: B + 1 cleared tickets.
dp_status launch_norm_affine_fused(int dtype, const void *X, const void *dY, int B, int HW, int C, float *chunk_partial,
                                   float *dgamma, float *dbeta, float *factor, int *counters, int clip, float C_l,
                                   int separate, float *sqnorm, long long sq_stride, float *clip_out, float *acc_w,
                                   float *acc_b, cudaStream_t st) {
    AffineTail t = {};
    t.counters = counters; t.B = B; t.clip = clip; t.separate = separate; t.C_l = C_l;
    t.accumulate_here = clip && (long long)B * C <= 16384;
    t.sqnorm = sqnorm; t.sq_stride = sq_stride; t.clip_out = clip_out; t.factor = factor;
    t.dgamma = dgamma; t.dbeta = dbeta; t.acc_w = acc_w; t.acc_b = acc_b;
    bool folded = false;
    const dp_status rc = norm_affine_dispatch(dtype, X, dY, B, HW, C, chunk_partial, dgamma, dbeta, nullptr, folded, t, st);
    if (rc != DP_OK || !clip || t.accumulate_here) return rc;
    affine_accum_kernel<<<dim3((unsigned)((C + 31) / 32), 2), 256, 0, st>>>(dgamma, dbeta, B, C, factor, acc_w, acc_b);
    DP_LAUNCH_CHECK("affine_accum_kernel");
    return DP_OK;
}


}  // namespace dp
