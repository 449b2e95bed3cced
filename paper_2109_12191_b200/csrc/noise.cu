// Gaussian noise and averaging: out = (acc + sigma*C*z) / |B|  (paper section 2, equation for g_t).
// z comes from Philox4x32-10 (Salmon et al., SC'11) and the Box-Muller transform, addressed by
// (seed, step, global parameter index), so the result does not depend on the launch shape.
#include "common.cuh"
#include "philox.cuh"

namespace dp {

// A thread block covers kNoiseTile parameters, i.e. kNoiseTile/4 Philox blocks from global index 4*(param_offset/4) on;
// local index = global - param_offset.  VEC: param_offset % 4 == 0, so a Philox block is one float4.
// What bounds the kernel is the issue rate (some 35 instructions a normal, of which a third Philox), not the 8 bytes a
// parameter it moves: two blocks a thread halve the index arithmetic and give the ten-round chain a second one to
// overlap with.  25.6 M parameters: 39 us; 42 with one pair of
// words at a time, 62 with one block a thread and the library's logf / sincospif.
constexpr int kNoiseTile = 2048;

template <bool VEC>
__global__ void __launch_bounds__(256)
noise_average_kernel(const float *acc, float *out, long long P,   // out may alias acc
                     unsigned long long param_offset, float noise_std, float inv_batch,
                     const __grid_constant__ NoiseStream ns) {
    const unsigned long long block0 = (param_offset >> 2) + (unsigned long long)blockIdx.x * (kNoiseTile / 4);
    const long long tile0 = (long long)(4ull * block0 - param_offset);       // may be negative for the first tile
    if (VEC && tile0 + kNoiseTile <= P) {
        const float4 *src = reinterpret_cast<const float4 *>(acc + tile0) + threadIdx.x;
        float4 *dst = reinterpret_cast<float4 *>(out + tile0) + threadIdx.x;
        float4 a[2];
        a[0] = __ldcs(src); a[1] = __ldcs(src + 256);                        // on their way while the noise is worked out
        float z[2][4] = {};
        if (noise_std != 0.0f) {
            normals4(ns, block0 + threadIdx.x, z[0]);
            normals4(ns, block0 + threadIdx.x + 256, z[1]);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            float4 r;
            r.x = (a[u].x + noise_std * z[u][0]) * inv_batch;
            r.y = (a[u].y + noise_std * z[u][1]) * inv_batch;
            r.z = (a[u].z + noise_std * z[u][2]) * inv_batch;
            r.w = (a[u].w + noise_std * z[u][3]) * inv_batch;
            __stcs(dst + 256 * u, r);
        }
        return;
    }
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        const long long i0 = tile0 + 4 * (threadIdx.x + 256 * u);
        if (i0 >= P) return;
        float z[4] = {0.f, 0.f, 0.f, 0.f};
        if (noise_std != 0.0f) normals4(ns, block0 + threadIdx.x + 256 * u, z);
#pragma unroll
        for (int lane = 0; lane < 4; ++lane) {
            const long long i = i0 + lane;
            if (i >= 0 && i < P) out[i] = (acc[i] + noise_std * z[lane]) * inv_batch;
        }
    }
}

// Noise, average and the parameter update in one pass: g = (acc + std*z) / |B|;  m <- mu*m + g (when a momentum
// buffer is given);  theta <- theta - lr*m (or - lr*g).  Same thread-to-Philox-block mapping as above.
// VEC: param_offset % 4 == 0 and 16-byte aligned buffers, so the four parameters of a block are one 16-byte access to
// each array (20 bytes a parameter with momentum).
template <bool VEC>
__global__ void __launch_bounds__(256)
noise_average_sgd_kernel(const float *acc, long long P, unsigned long long param_offset, unsigned long long n_blocks,
                         float noise_std, float inv_batch, const __grid_constant__ NoiseStream ns, float lr, float mu,
                         float *theta, float *mom, float *g_out) {
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_blocks) return;
    const unsigned long long block = (param_offset >> 2) + t;
    const long long i0 = (long long)(4ull * block - param_offset);
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (VEC && i0 + 3 < P) {
        // the loads are on their way while the noise is worked out
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(acc + i0));
        float4 th = *reinterpret_cast<const float4 *>(theta + i0);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (mom) v = *reinterpret_cast<const float4 *>(mom + i0);
        if (noise_std != 0.0f) normals4(ns, block, z);
        const float4 g = make_float4((a.x + noise_std * z[0]) * inv_batch, (a.y + noise_std * z[1]) * inv_batch,
                                     (a.z + noise_std * z[2]) * inv_batch, (a.w + noise_std * z[3]) * inv_batch);
        if (mom) {
            v = make_float4(fmaf(mu, v.x, g.x), fmaf(mu, v.y, g.y), fmaf(mu, v.z, g.z), fmaf(mu, v.w, g.w));
            *reinterpret_cast<float4 *>(mom + i0) = v;
        } else {
            v = g;
        }
        th = make_float4(fmaf(-lr, v.x, th.x), fmaf(-lr, v.y, th.y), fmaf(-lr, v.z, th.z), fmaf(-lr, v.w, th.w));
        *reinterpret_cast<float4 *>(theta + i0) = th;
        if (g_out) *reinterpret_cast<float4 *>(g_out + i0) = g;
        return;
    }
    if (noise_std != 0.0f) normals4(ns, block, z);
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
        const long long i = i0 + lane;
        if (i < 0 || i >= P) continue;
        const float g = (acc[i] + noise_std * z[lane]) * inv_batch;
        float v = g;
        if (mom) { v = fmaf(mu, mom[i], g); mom[i] = v; }
        theta[i] = fmaf(-lr, v, theta[i]);
        if (g_out) g_out[i] = g;
    }
}

__global__ void philox_raw_kernel(uint32_t *out4, long long n_blocks, unsigned long long first_block,
                                  const __grid_constant__ NoiseStream ns) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_blocks) return;
    const Words4 w = philox_block(ns, first_block + (unsigned long long)t);
    reinterpret_cast<uint4 *>(out4)[t] = make_uint4(w.w0, w.w1, w.w2, w.w3);
}

__global__ void noise_z_kernel(float *z, long long count, unsigned long long first_index,
                               unsigned long long n_blocks, const __grid_constant__ NoiseStream ns) {
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_blocks) return;
    const unsigned long long block = (first_index >> 2) + t;
    float v[4];
    normals4(ns, block, v);
    const long long i0 = (long long)(4ull * block - first_index);
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
        const long long i = i0 + lane;
        if (i >= 0 && i < count) z[i] = v[lane];
    }
}

// z[t] = normal of example `example`'s stream at global index first_index + t (one thread per Philox block)
__global__ void example_noise_z_kernel(float *z, long long count, unsigned long long first_index,
                                       unsigned long long n_blocks, uint32_t example,
                                       const __grid_constant__ NoiseStream ns) {
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_blocks) return;
    const unsigned long long block = (first_index >> 2) + t;
    float v[4];
    example_normals4(ns, example, (uint32_t)block, v);
    const long long i0 = (long long)(4ull * block - first_index);
#pragma unroll
    for (int lane = 0; lane < 4; ++lane) {
        const long long i = i0 + lane;
        if (i >= 0 && i < count) z[i] = v[lane];
    }
}

}  // namespace dp

extern "C" dp_status dp_noise_average(const float *acc, long long P, long long param_offset, float sigma, float C,
                                      long long total_batch, unsigned long long seed, unsigned long long step,
                                      float *out, void *cuda_stream) {
    if (!acc || !out || P <= 0 || param_offset < 0 || total_batch <= 0) return DP_ERR_INVALID_ARG;
    if (!(sigma >= 0.0f) || !(C > 0.0f)) return DP_ERR_INVALID_ARG;                 // also rejects NaN
    if (sigma > 0.0f && isinf(C)) return DP_ERR_INVALID_ARG;
    if (isinf(sigma)) return DP_ERR_INVALID_ARG;
    if (!dp::aligned(acc, 16) || !dp::aligned(out, 16)) return DP_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const unsigned long long off = (unsigned long long)param_offset;
    const unsigned long long n_blocks = ((off & 3ull) + (unsigned long long)P + 3ull) >> 2;
    const float noise_std = (sigma == 0.0f) ? 0.0f : sigma * C;
    const float inv_batch = 1.0f / (float)total_batch;
    const unsigned long long grid = (n_blocks + dp::kNoiseTile / 4 - 1) / (dp::kNoiseTile / 4);
    if (grid > 0x7fffffffull) return DP_ERR_UNSUPPORTED;
    const dp::NoiseStream ns = dp::noise_stream(seed, step);
    if ((off & 3ull) == 0)
        dp::noise_average_kernel<true><<<(unsigned)grid, 256, 0, stream>>>(acc, out, P, off, noise_std, inv_batch, ns);
    else
        dp::noise_average_kernel<false><<<(unsigned)grid, 256, 0, stream>>>(acc, out, P, off, noise_std, inv_batch, ns);
    DP_LAUNCH_CHECK("noise_average_kernel");
    return DP_OK;
}

extern "C" dp_status dp_noise_average_sgd(const float *acc, long long P, long long param_offset, float sigma, float C,
                                          long long total_batch, unsigned long long seed, unsigned long long step,
                                          float lr, float momentum, float *theta, float *momentum_buf, float *g_out,
                                          void *cuda_stream) {
    if (!acc || !theta || P <= 0 || param_offset < 0 || total_batch <= 0) return DP_ERR_INVALID_ARG;
    if (!(sigma >= 0.0f) || !(C > 0.0f) || isinf(sigma) || (sigma > 0.0f && isinf(C))) return DP_ERR_INVALID_ARG;
    if (!(lr == lr) || isinf(lr) || !(momentum >= 0.0f) || isinf(momentum)) return DP_ERR_INVALID_ARG;
    if (!dp::aligned(acc, 4) || !dp::aligned(theta, 4) || (momentum_buf && !dp::aligned(momentum_buf, 4)) ||
        (g_out && !dp::aligned(g_out, 4)))
        return DP_ERR_INVALID_ARG;
    const unsigned long long off = (unsigned long long)param_offset;
    const unsigned long long n_blocks = ((off & 3ull) + (unsigned long long)P + 3ull) >> 2;
    const unsigned long long grid = (n_blocks + 255) / 256;
    if (grid > 0x7fffffffull) return DP_ERR_UNSUPPORTED;
    const bool vec = (off & 3ull) == 0 && dp::aligned(acc, 16) && dp::aligned(theta, 16) && dp::aligned(momentum_buf, 16) &&
                     dp::aligned(g_out, 16);
    (vec ? dp::noise_average_sgd_kernel<true> : dp::noise_average_sgd_kernel<false>)<<<(unsigned)grid, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        acc, P, off, n_blocks, (sigma == 0.0f) ? 0.0f : sigma * C, 1.0f / (float)total_batch, dp::noise_stream(seed, step), lr, momentum,
        theta, momentum_buf, g_out);
    DP_LAUNCH_CHECK("noise_average_sgd_kernel");
    return DP_OK;
}

extern "C" dp_status dp_debug_philox_raw(unsigned int *out4, long long n_blocks, long long first_block,
                                         unsigned long long seed, unsigned long long step, void *cuda_stream) {
    if (!out4 || n_blocks <= 0 || first_block < 0 || !dp::aligned(out4, 16)) return DP_ERR_INVALID_ARG;
    const long long grid = (n_blocks + 255) / 256;
    if (grid > 0x7fffffffll) return DP_ERR_UNSUPPORTED;
    dp::philox_raw_kernel<<<(unsigned)grid, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        out4, n_blocks, (unsigned long long)first_block, dp::noise_stream(seed, step));
    DP_LAUNCH_CHECK("philox_raw_kernel");
    return DP_OK;
}

extern "C" dp_status dp_debug_noise_z(float *z, long long count, long long first_index, unsigned long long seed,
                                      unsigned long long step, void *cuda_stream) {
    if (!z || count <= 0 || first_index < 0) return DP_ERR_INVALID_ARG;
    const unsigned long long off = (unsigned long long)first_index;
    const unsigned long long n_blocks = ((off & 3ull) + (unsigned long long)count + 3ull) >> 2;
    const unsigned long long grid = (n_blocks + 255) / 256;
    if (grid > 0x7fffffffull) return DP_ERR_UNSUPPORTED;
    dp::noise_z_kernel<<<(unsigned)grid, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(z, count, off, n_blocks,
                                                                                         dp::noise_stream(seed, step));
    DP_LAUNCH_CHECK("noise_z_kernel");
    return DP_OK;
}

extern "C" dp_status dp_debug_example_noise_z(float *z, long long count, long long first_index, long long example,
                                              unsigned long long seed, unsigned long long step, void *cuda_stream) {
    if (!z || count <= 0 || first_index < 0 || example < 0 || example >= 0x80000000ll) return DP_ERR_INVALID_ARG;
    const unsigned long long off = (unsigned long long)first_index;
    if (off + (unsigned long long)count > (1ull << 34)) return DP_ERR_UNSUPPORTED;
    const unsigned long long n_blocks = ((off & 3ull) + (unsigned long long)count + 3ull) >> 2;
    const unsigned long long grid = (n_blocks + 255) / 256;
    if (grid > 0x7fffffffull) return DP_ERR_UNSUPPORTED;
    dp::example_noise_z_kernel<<<(unsigned)grid, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        z, count, off, n_blocks, (uint32_t)example, dp::noise_stream(seed, step));
    DP_LAUNCH_CHECK("example_noise_z_kernel");
    return DP_OK;
}
