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

// Four samples' loads are in flight at a time (one after the other, with a branch around each, 12 samples
// of 300 queries took 10.1 us).  LOGITS: the attention weights' Shiftmax is worked out here, by the dh / 4
// threads of each (b, q, h) from the int16 logits, instead of by three launches (two conversions to int32
// and the row kernel); the weights of the CTA's items stand in shared memory.
template <bool LOGITS>
__global__ void __launch_bounds__(256) deform_kernel(const DeformParams p, int64_t total) {
    grid_wait();
    extern __shared__ uint8_t s_w[];  // LOGITS: [256 / quads, LP]
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int quads = p.dh >> 2, LP = p.L * p.P;
    const bool live = id < total;
    const int dq = (int)(id % quads);
    const int64_t bqh = live ? id / quads : 0;
    const int h = (int)(bqh % p.H);
    const int64_t bq = bqh / p.H;
    const uint8_t *w = p.w + bqh * LP;
    if constexpr (LOGITS) {  // quads is 8 or 16: an item's threads are neighbours in a warp
        const int16_t *x = p.logits + bqh * LP;
        int32_t mx = -32768;
        for (int j = dq; j < LP; j += quads) mx = max(mx, (int32_t)x[j]);
        for (int o = quads >> 1; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        uint64_t sum = 0;
        for (int j = dq; j < LP; j += quads) sum += shift_exp_mag((uint32_t)(mx - x[j]), p.smx.se);
        for (int o = quads >> 1; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const RowNorm rn = shiftmax_norm(sum, p.smx.s_d, p.smx.m_p, p.smx.M_hw, p.smx.k_out);
        uint8_t *sw = s_w + (threadIdx.x / quads) * LP;
        for (int j = dq; j < LP; j += quads) sw[j] = (uint8_t)shiftmax_out(shift_exp_mag((uint32_t)(mx - x[j]), p.smx.se), rn);
        __syncwarp();
        w = sw;
    }
    if (!live) return;
    const int b = (int)(bq / p.Q);
    const int64_t rx = p.ref[bq * 2 + 0], ry = p.ref[bq * 2 + 1];
    const int64_t Dm = (int64_t)p.H * p.dh;
    int32_t acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
    for (int l = 0; l < p.L; ++l) {
        const int64_t Hl = p.lh[l], Wl = p.lw[l];
        const int64_t bx = (rx * Wl) >> 8, by = (ry * Hl) >> 8;  // reference in Q8 pixels
        const int8_t *vl = p.value + ((int64_t)b * p.S_total + p.lstart[l]) * Dm + h * p.dh + 4 * dq;
#pragma unroll 4
        for (int pt = 0; pt < p.P; ++pt) {
            const int j = l * p.P + pt;
            int64_t ox, oy;
            if constexpr (LOGITS) {
                const int16_t *o = p.off16 + (bqh * LP + j) * 2;
                ox = o[0], oy = o[1];
            } else {
                const int32_t *o = p.off + (bqh * LP + j) * 2;
                ox = o[0], oy = o[1];
            }
            const int64_t ix = (bx + ox) >> 8, iy = (by + oy) >> 8;
            const bool in = ix >= 0 && ix < Wl && iy >= 0 && iy < Hl;
            const int32_t wt = w[j];
            const uint32_t v = in ? *(const uint32_t *)(vl + (iy * Wl + ix) * Dm) : 0u;
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
    launch_after(deform_kernel<false>, (unsigned)((total + 255) / 256), 256, 0, s, p, total);
    return cudaGetLastError();
}
// dh of 32 or 64 and L P <= 256 (8 KB of weights a CTA); cudaErrorNotSupported otherwise.
cudaError_t launch_deform_logits(const DeformParams &p, cudaStream_t s) {
    const int LP = p.L * p.P, quads = p.dh / 4;
    if ((p.dh != 32 && p.dh != 64) || LP > 256) return cudaErrorNotSupported;
    const int64_t total = (int64_t)p.B * p.Q * p.H * quads;
    if (total == 0) return cudaSuccess;
    launch_after(deform_kernel<true>, (unsigned)((total + 255) / 256), 256, (size_t)(256 / quads) * LP, s, p, total);
    return cudaGetLastError();
}

}  // namespace ilw
