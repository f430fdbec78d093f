// a6. L1 rendering losses with the optional filter gate (Sec. 3.3: gate
// G(p) = [D_c(p) > 0][D_g(p) > 0][M_b(p) > gamma] and the joint loss terms
// w2 L_c + w3 L_d; Sec. 3.4: the L1 terms of the mapping loss L_m).
//   L = w_c / (3P) sum_p G(p) |C(p) - C^(p)|_1 + w_d / P sum_p G(p) |D(p) - D^(p)|
// over all P pixels of the batch; writes dL/dC, dL/dD (sign(0) = 0).
#include "chain.cuh"
#include "common.cuh"

namespace gs {

__device__ __forceinline__ float sgn(float x) { return (float)((x > 0.0f) - (x < 0.0f)); }

// Bound by memory (48 B a pixel).  Each addition to the running loss rounds it,
// so the blocks of a cluster add their sums together: 152 additions on large
// images instead of 1,216 (the whole loss of four 641x479 views 85.7 -> 89.8 us
// with the one addition of the SSIM pass; its largest error over 30 runs
// 4.7e-6 -> 9.7e-7).  Blocks of 1,024 threads, 38 additions, were no faster and
// no nearer.
constexpr int kL1Cluster = 8, kL1Threads = 256;

__global__ void __launch_bounds__(kL1Threads) loss_l1_kernel(const float *__restrict__ rgb, const float *__restrict__ depth,
                                                      const float *__restrict__ alpha, const float *__restrict__ trgb,
                                                      const float *__restrict__ tdepth, int64_t P, float kc, float kd,
                                                      int use_gate, float gamma, float *loss, float *d_rgb,
                                                      float *d_depth)
{
    __shared__ float part[kL1Threads / 32];
    __shared__ float block_sum;
    float acc = 0.0f;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P; p += (int64_t)gridDim.x * blockDim.x) {
        const float D = depth[p], Dt = tdepth[p];
        bool gate = true;
        if (use_gate) gate = (Dt > 0.0f) && (D > 0.0f) && (alpha[p] > gamma);
        const float g = gate ? 1.0f : 0.0f;
        float l = 0.0f;
        #pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            const float r = rgb[3 * p + ch] - trgb[3 * p + ch];
            l += kc * fabsf(r);
            d_rgb[3 * p + ch] = g * kc * sgn(r);
        }
        const float r = D - Dt;
        l += kd * fabsf(r);
        d_depth[p] = g * kd * sgn(r);
        acc += g * l;
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        const float s = warp_sum(threadIdx.x < kL1Threads / 32 ? part[threadIdx.x] : 0.0f);
        if (threadIdx.x == 0) block_sum = s;
    }
    cluster_sync();  // every block's sum is written
    if (threadIdx.x == 0 && cluster_rank() == 0 && loss) {
        float s = 0.0f;
        for (int b = 0; b < kL1Cluster; b++) s += ld_cluster(&block_sum, b);
        atomicAdd(loss, s);
    }
    cluster_sync();  // no block ends before its sum is read
}

}  // namespace gs

using namespace gs;

extern "C" gs_status_t gs_loss_l1(const float *rgb, const float *depth, const float *alpha, const float *target_rgb,
                                  const float *target_depth, int64_t n_pixels, float w_c, float w_d,
                                  int32_t use_gate, float gamma, float *loss, float *d_rgb, float *d_depth,
                                  void *stream)
{
    if (n_pixels < 0) return GS_ERR_INVALID_ARG;
    if (n_pixels == 0) return GS_OK;
    if (!rgb || !depth || !target_rgb || !target_depth || !d_rgb || !d_depth || (use_gate && !alpha))
        return GS_ERR_INVALID_ARG;
    const float kc = (float)((double)w_c / (3.0 * (double)n_pixels));
    const float kd = (float)((double)w_d / (double)n_pixels);
    const int sms = num_sms();
    const int64_t want = (n_pixels + kL1Threads - 1) / kL1Threads, most = (int64_t)sms * 8;
    const int64_t blocks = ((want < most ? want : most) + kL1Cluster - 1) / kL1Cluster * kL1Cluster;
    return launch_with(false, kL1Cluster, loss_l1_kernel, (unsigned)blocks, kL1Threads, 0, as_stream(stream), rgb, depth,
                       alpha, target_rgb, target_depth, n_pixels, kc, kd, use_gate, gamma, loss, d_rgb, d_depth);
}
