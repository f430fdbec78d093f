// Keyframe decoding: the RGB-D frames of the experiments (Sec. 4: TUM RGB-D
// sequences, 8-bit colour and 16-bit depth images) arrive from the host in
// their sensor format, five bytes a pixel, and are widened on the device to
// the FP32 targets of the losses: colour c / 255, depth d * depth_scale
// (metres per depth unit; 0 stays 0, the sensor's "no reading").  Both are one
// correctly rounded FP32 operation, so the result equals the same expression
// evaluated in FP32 anywhere.
#include "common.cuh"

namespace gs {

constexpr int kDecodeThreads = 256;
constexpr int kDecodeItems = 4;   // in flight a thread (two or eight: 27.5, 29.0 us)
constexpr int kDecodeBlocks = 8;  // an SM

// c / 255 correctly rounded, for whole c in [0, 255]: the product with the
// rounded reciprocal, corrected by its exact remainder (Markstein 1990); equal
// to the quotient's nearest FP32 number for all 256 values.
__device__ __forceinline__ float over_255(uint32_t c)
{
    constexpr float r = 1.0f / 255.0f;
    const float x = (float)c, q = __fmul_rn(x, r);
    return __fmaf_rn(__fmaf_rn(-255.0f, q, x), r, q);
}

// A frame is two flat arrays: output float4 k of the colours holds the four
// bytes of input word k, whatever pixels they belong to, and output float4 k of
// the depths the four values of input word pair k.  Items are the colour words,
// then the depth word pairs; consecutive threads take consecutive items, so
// every load and store of a warp is one contiguous span.  Bound: HBM.  Four
// pixels a thread, each float4 stored 48 bytes from its neighbour's and twelve
// divisions: 29.0 us for eight 1200x680 frames (28.0 with the stores in order),
// now 24.8 us, 137 MB at 5.5 TB/s.  The last bytes and values beyond whole words
// go one a thread of block 0 (they were a launch of their own).
__global__ void __launch_bounds__(kDecodeThreads) decode_kernel(const uint8_t *__restrict__ rgb8,
                                                                const uint16_t *__restrict__ depth16, int64_t n_pixels,
                                                                float depth_scale, float *__restrict__ rgb,
                                                                float *__restrict__ depth)
{
    const uint32_t *cw = reinterpret_cast<const uint32_t *>(rgb8);
    const uint2 *dw = reinterpret_cast<const uint2 *>(depth16);
    float4 *co = reinterpret_cast<float4 *>(rgb), *po = reinterpret_cast<float4 *>(depth);
    const int64_t colours = 3 * n_pixels / 4, items = colours + n_pixels / 4;
    const int64_t stride = (int64_t)gridDim.x * kDecodeThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kDecodeThreads + threadIdx.x; i0 < items; i0 += kDecodeItems * stride) {
        uint2 w[kDecodeItems];
        #pragma unroll
        for (int k = 0; k < kDecodeItems; k++) {
            const int64_t i = i0 + k * stride;
            w[k] = make_uint2(0u, 0u);
            if (i < colours) w[k].x = __ldcs(cw + i);
            else if (i < items) w[k] = __ldcs(dw + (i - colours));
        }
        #pragma unroll
        for (int k = 0; k < kDecodeItems; k++) {
            const int64_t i = i0 + k * stride;
            if (i < colours) {
                const uint32_t c = w[k].x;
                __stcs(co + i, make_float4(over_255(c & 0xffu), over_255((c >> 8) & 0xffu),
                                           over_255((c >> 16) & 0xffu), over_255(c >> 24)));
            } else if (i < items) {
                const uint2 d = w[k];
                __stcs(po + (i - colours),
                       make_float4(__fmul_rn((float)(d.x & 0xffffu), depth_scale), __fmul_rn((float)(d.x >> 16), depth_scale),
                                   __fmul_rn((float)(d.y & 0xffffu), depth_scale), __fmul_rn((float)(d.y >> 16), depth_scale)));
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < 4) {
        const int64_t c = 4 * colours + threadIdx.x, d = n_pixels / 4 * 4 + threadIdx.x;
        if (c < 3 * n_pixels) rgb[c] = over_255(rgb8[c]);
        if (d < n_pixels) depth[d] = __fmul_rn((float)depth16[d], depth_scale);
    }
}

}  // namespace gs

using namespace gs;

extern "C" gs_status_t gs_decode_keyframes(const uint8_t *rgb8, const uint16_t *depth16, int64_t n_pixels,
                                           float depth_scale, float *rgb, float *depth, void *stream)
{
    if (n_pixels < 0) return GS_ERR_INVALID_ARG;
    if (n_pixels == 0) return GS_OK;
    if (!rgb8 || !depth16 || !rgb || !depth) return GS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(rgb8) & 3) || (reinterpret_cast<uintptr_t>(depth16) & 7) ||
        (reinterpret_cast<uintptr_t>(rgb) & 15) || (reinterpret_cast<uintptr_t>(depth) & 15))
        return GS_ERR_INVALID_ARG;
    cudaStream_t s = as_stream(stream);
    int64_t blocks = (n_pixels + kDecodeThreads - 1) / kDecodeThreads;
    const int64_t cap = (int64_t)num_sms() * kDecodeBlocks;
    if (blocks > cap) blocks = cap;
    decode_kernel<<<(unsigned)blocks, kDecodeThreads, 0, s>>>(rgb8, depth16, n_pixels, depth_scale, rgb, depth);
    return launch_status();
}
