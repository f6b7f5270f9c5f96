// deform.cu -- integer deformable-attention sampling with nearest-neighbour lookup
// (Sec. 3.1.1: bilinear interpolation replaced by the nearest grid point).
//
// One thread owns four channels of one (b, q, h); the L*P sample locations are computed in
// integers (Q16 reference, Q8 offsets, floor to the nearest pixel in the align_corners=False
// convention), each sample gathers 4 bytes with one 32-bit load, accumulation is int32.
#include <cstdint>

#include "ilw_kernels.h"

namespace ilw {
namespace {

__global__ void __launch_bounds__(256) deform_kernel(const DeformParams p, int64_t total) {
    grid_wait();
    int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= total) return;
    const int quads = p.dh >> 2;
    const int dq = (int)(id % quads);
    int64_t bqh = id / quads;
    const int h = (int)(bqh % p.H);
    int64_t bq = bqh / p.H;
    const int b = (int)(bq / p.Q);
    const int64_t rx = p.ref[bq * 2 + 0], ry = p.ref[bq * 2 + 1];
    const int64_t Dm = (int64_t)p.H * p.dh;
    const int LP = p.L * p.P;
    const int32_t *off = p.off + bqh * LP * 2;
    const uint8_t *w = p.w + bqh * LP;
    int32_t acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
    for (int l = 0; l < p.L; ++l) {
        const int64_t Hl = p.lh[l], Wl = p.lw[l];
        const int64_t bx = (rx * Wl) >> 8, by = (ry * Hl) >> 8;  // reference in Q8 pixels
        const int8_t *vl = p.value + ((int64_t)b * p.S_total + p.lstart[l]) * Dm + h * p.dh + 4 * dq;
        for (int pt = 0; pt < p.P; ++pt) {
            const int j = l * p.P + pt;
            const int64_t ix = (bx + off[2 * j]) >> 8, iy = (by + off[2 * j + 1]) >> 8;
            if (ix < 0 || ix >= Wl || iy < 0 || iy >= Hl) continue;
            const int32_t wt = w[j];
            const uint32_t v = *(const uint32_t *)(vl + (iy * Wl + ix) * Dm);
            acc0 += wt * (int32_t)(int8_t)(v & 0xff);
            acc1 += wt * (int32_t)(int8_t)((v >> 8) & 0xff);
            acc2 += wt * (int32_t)(int8_t)((v >> 16) & 0xff);
            acc3 += wt * (int32_t)(int8_t)(v >> 24);
        }
    }
    uint32_t o = (uint32_t)(uint8_t)sat8(rq(acc0, p.m, p.s)) | ((uint32_t)(uint8_t)sat8(rq(acc1, p.m, p.s)) << 8) |
                 ((uint32_t)(uint8_t)sat8(rq(acc2, p.m, p.s)) << 16) |
                 ((uint32_t)(uint8_t)sat8(rq(acc3, p.m, p.s)) << 24);
    *(uint32_t *)(p.out + bq * Dm + h * p.dh + 4 * dq) = o;
}

}  // namespace

cudaError_t launch_deform(const DeformParams &p, cudaStream_t s) {
    int64_t total = (int64_t)p.B * p.Q * p.H * (p.dh / 4);
    if (total == 0) return cudaSuccess;
    launch_after(deform_kernel, (unsigned)((total + 255) / 256), 256, 0, s, p, total);
    return cudaGetLastError();
}

}  // namespace ilw
