// Host interface of the convolution kernels whose operands the TMA unit
// stages (osog_conv_tma.cu); the C ABI around them is in osog_cnn.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "osog_common.cuh"
#include "osog_device_once.h"

namespace osog {
namespace cnn {

// Launch of a convolution kernel with programmatic stream serialization: it is
// dispatched and sets itself up while the kernel before it finishes.  Such a
// kernel calls pdl_enter() before anything it reads or writes in global memory,
// and after its tensor memory is allocated: the next kernel's CTAs may come as
// soon as every CTA of this one has let them, and one that took the tensor
// memory of an SM before a CTA of this kernel had its own would wait for this
// kernel, which would wait for it.
template <typename... KArgs>
inline cudaError_t launch_conv(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem,
                               cudaStream_t st, const typename KernelArg<KArgs>::type &...args) {
    return launch_pdl(kernel, true, grid, block, smem, st, args...);
}

// Opt-in of a kernel to `bytes` of dynamic shared memory on the current device
// (`once` is the kernel's own).
template <typename... KArgs>
inline cudaError_t opt_in_smem(DeviceOnce &once, void (*kernel)(KArgs...), int bytes) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return once(dev, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

// Most pixels that a filter gradient adds in one accumulator before it sums the
// partial results of its splits.
constexpr int kSplitPixels = 2048;

struct Geo {
    int N, H, W, C, K, R, S, stride, pad, P, Q;
};

// Forward (y = act(conv(x, w) + bias)) and data gradient (dx, times x_act > 0
// when mask is given) on tcgen05; cudaErrorNotSupported when a size is outside
// the kernel's range (see conv_patch_plan; 16-byte aligned operands).
cudaError_t conv_forward_tma(const Geo &g, const uint16_t *x, const uint16_t *w, const float *bias,
                             bool relu, uint16_t *y, float *y32, cudaStream_t st);
cudaError_t conv_dgrad_tma(const Geo &g, const uint16_t *dy, const uint16_t *w,
                           const uint16_t *mask, uint16_t *dx, cudaStream_t st);

// Filter and bias gradients (ws: conv_wgrad_tma_workspace bytes; ws, dw and
// dbias 16-byte aligned); cudaErrorNotSupported as above (workspace 0).
size_t conv_wgrad_tma_workspace(const Geo &g);
cudaError_t conv_wgrad_tma(const Geo &g, const uint16_t *dy, const uint16_t *x, float *dw,
                           float *dbias, float *ws, cudaStream_t st);

// dw, dbias = the sums over the splits of part [splits][K R S C + K], in order
// (all 16-byte aligned).  Split z added the tiles z, z + splits, ... of tile_h x tile_w
// output pixels; ragged_dy: dY when tiles reach past the image, else NULL (see
// k_sum_parts).
cudaError_t conv_sum_parts(const Geo &g, int splits, const float *part, float *dw, float *dbias,
                           const uint16_t *ragged_dy, const uint16_t *x, int tile_h, int tile_w,
                           cudaStream_t st);

// Latched status of the bounded waits (read and cleared), and the
// failure-detection hook (osog_conv_test_wait_limit).
cudaError_t conv_tma_take_status(int *timed_out);
cudaError_t conv_tma_set_probe(int polls);

}  // namespace cnn
}  // namespace osog
