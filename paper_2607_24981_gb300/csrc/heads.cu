// heads.cu -- the detection head's elementwise and selection kernels: integer sigmoid (the head's
// exponential by ShiftExp, Table 5, in SD-ShiftGELU's sign-dependent sigmoid form, Sec. 3.3.1 and
// Algorithm 1), ReLU on int8, per-row integer top-K (two-stage query selection) and row gather.
#include <climits>
#include <cstdint>

#include "ilw_kernels.h"

namespace ilw {
namespace {

// out = (E F) >> (32 - k_out), E = ShiftExp(min(x, 0)), E' = ShiftExp(-max(x, 0)),
// F = floor((2^31 - 1) / (E + E')).  One of the two ShiftExp inputs is always 0 and ShiftExp(0) =
// I0 2^k, so one ShiftExp of -|x| gives both.  |x| is clamped at 2^30 (past k I0 < 2^20 ShiftExp
// sits in its clamp region, so the clamp changes nothing).
__device__ __forceinline__ int32_t int_sigmoid1(int32_t x, const ShiftExpC &se, int32_t out_sh) {
    const uint32_t a = x < 0 ? 0u - (uint32_t)x : (uint32_t)x;
    const uint32_t e = shift_exp_mag(min(a, 1u << 30), se);
    const uint32_t top = (uint32_t)se.I0 << se.k;
    const uint32_t E = x >= 0 ? top : e;
    const uint32_t F = div_int31(top + e);
    return (int32_t)(((uint64_t)E * F) >> out_sh);
}

__global__ void __launch_bounds__(256) int_sigmoid_kernel(const int32_t *__restrict__ X, int32_t *__restrict__ Y,
                                                          int64_t n, ShiftExpC se, int32_t out_sh) {
    grid_wait();
    const int64_t n4 = n / 4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        const int4 v = ((const int4 *)X)[i];
        ((int4 *)Y)[i] = make_int4(int_sigmoid1(v.x, se, out_sh), int_sigmoid1(v.y, se, out_sh),
                                   int_sigmoid1(v.z, se, out_sh), int_sigmoid1(v.w, se, out_sh));
    }
    for (int64_t i = 4 * n4 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        Y[i] = int_sigmoid1(X[i], se, out_sh);
}

// requant_kernel's formula with the sigmoid of its result, 4 elements a thread: reference logits and boxes
// (4 columns) in one launch instead of two or three.
template <typename TOut>
__global__ void __launch_bounds__(256) requant_sigmoid_kernel(const RequantParams p, int32_t *sig, int64_t ld_sig, ShiftExpC se,
                                                              int32_t out_sh) {
    grid_wait();
    const int32_t cq = p.C >> 2;
    const int64_t total = p.rows * cq;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / cq;
        const int32_t c = (int32_t)(i - r * cq) * 4;
        const int4 x4 = *(const int4 *)((const int32_t *)p.X + r * p.ldx + c);
        const int32_t x[4] = {x4.x, x4.y, x4.z, x4.w};
        const int16_t *z = p.Z ? p.Z + (r % p.z_rows) * p.ldz + c : nullptr;
        int32_t o[4], g[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int64_t v = rq(x[u], p.m1, p.s1);
            if (z) v += rq(z[u], p.m2, p.s2);
            o[u] = sizeof(TOut) == 2 ? sat16(v) : (int32_t)v;
            g[u] = int_sigmoid1(o[u], se, out_sh);
        }
        TOut *y = (TOut *)p.Y + r * p.ldy + c;
        if constexpr (sizeof(TOut) == 2)
            *(uint2 *)y = make_uint2((uint32_t)(uint16_t)o[0] | ((uint32_t)(uint16_t)o[1] << 16),
                                     (uint32_t)(uint16_t)o[2] | ((uint32_t)(uint16_t)o[3] << 16));
        else
            *(int4 *)y = make_int4(o[0], o[1], o[2], o[3]);
        *(int4 *)(sig + r * ld_sig + c) = make_int4(g[0], g[1], g[2], g[3]);
    }
}

// ReLU of int8 values, four per thread step (n4 words), then the tail
__global__ void __launch_bounds__(256) relu_i8_kernel(const int8_t *__restrict__ X, int8_t *__restrict__ Y, int64_t n) {
    grid_wait();
    const int64_t n4 = n / 4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t w = ((const uint32_t *)X)[i];
        // keep the bytes whose sign bit is clear
        const uint32_t neg = (w & 0x80808080u) >> 7;  // 1 in each negative byte's low bit
        ((uint32_t *)Y)[i] = w & ~(neg * 0xFFu);
    }
    for (int64_t i = 4 * n4 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        Y[i] = X[i] < 0 ? (int8_t)0 : X[i];
}

// Per-row top-K, one CTA per row, ties to the lower index.  Bound by latency (a row's 33 KB at 8400
// values are nothing): sorting the whole padded row took 105 steps over 16384 keys, 211 us; selecting
// first leaves K keys to order.  Thread t holds values t VPT .. (VPT of them) in registers.
//   1. the K-th largest value, found bit by bit below the row's maximum: every step counts the values at
//      or above a candidate over the CTA;
//   2. a scan over the threads gives every value above it its place among the selected, and the values
//      equal to it, in index order, the places left;
//   3. the selected keys (value, lower index first) are ordered by counting the larger ones for
//      K <= kRankMax, else by a bitonic sort of the K keys.
// Keys: (value biased to unsigned) << 32 | (2^32 - 1 - index), so one descending order puts larger
// values first and, for equal values, smaller indices first.  Padding keys are 0, below every real key.
constexpr int kTopkThreads = 1024;
constexpr int kRankMax = 512;
template <int VPT>
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(const int32_t *__restrict__ S, int64_t lds, int32_t N,
                                                            int32_t kpad, int32_t K, int32_t *__restrict__ vals,
                                                            int32_t *__restrict__ idx) {
    grid_wait();
    extern __shared__ unsigned long long keys[];  // kpad
    __shared__ uint32_t part[2][32];
    const int32_t *s = S + (int64_t)blockIdx.x * lds;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, i0 = tid * VPT;
    // biased values; past the row 0, which step 2 never selects (it is told apart by its index)
    uint32_t v[VPT];
#pragma unroll
    for (int j = 0; j < VPT; ++j) v[j] = i0 + j < N ? (uint32_t)s[i0 + j] ^ 0x80000000u : 0u;
    // the CTA's sum of one value per thread (alternating buffers: one barrier per call)
    int buf = 0;
    auto cta_sum = [&](uint32_t x) -> uint32_t {
        x = __reduce_add_sync(0xffffffffu, x);
        if (lane == 0) part[buf][warp] = x;
        __syncthreads();
        x = __reduce_add_sync(0xffffffffu, part[buf][lane]);
        buf ^= 1;
        return x;
    };
    // bits above the highest in which the row's values differ are the maximum's
    uint32_t hi = 0, lo = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < VPT; ++j)
        if (i0 + j < N) {
            hi = max(hi, v[j]);
            lo = min(lo, v[j]);
        }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    if (lane == 0) {
        part[0][warp] = hi;
        part[1][warp] = lo;
    }
    __syncthreads();
    hi = __reduce_max_sync(0xffffffffu, part[0][lane]);
    lo = __reduce_min_sync(0xffffffffu, part[1][lane]);
    __syncthreads();
    // thr: the largest value with at least K values at or above it (that many are at or above `lo`)
    const int top = 32 - __clz(hi ^ lo);
    uint32_t thr = top == 32 ? 0u : hi >> top << top;
    for (int bit = top - 1; bit >= 0; --bit) {
        const uint32_t cand = thr | (1u << bit);
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < VPT; ++j) c += (i0 + j < N && v[j] >= cand) ? 1u : 0u;
        if (cta_sum(c) >= (uint32_t)K) thr = cand;
    }
    // places: (values above thr) << 16 | (values equal to it), summed over the threads before this one
    uint32_t c = 0;
#pragma unroll
    for (int j = 0; j < VPT; ++j)
        if (i0 + j < N) c += v[j] > thr ? 1u << 16 : (v[j] == thr ? 1u : 0u);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();
    if (lane == 31) part[0][warp] = incl;
    for (int i = K + tid; i < kpad; i += kTopkThreads) keys[i] = 0ull;
    __syncthreads();
    const uint32_t w = part[0][lane];
    const uint32_t total = __reduce_add_sync(0xffffffffu, w);
    uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + incl - c;
    const uint32_t above = total >> 16;
    uint32_t pg = before >> 16, pe = above + (before & 0xffffu);
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        if (i0 + j >= N || v[j] < thr) continue;
        const uint32_t pos = v[j] > thr ? pg++ : pe++;
        if (pos < (uint32_t)K) keys[pos] = ((unsigned long long)v[j] << 32) | (0xFFFFFFFFu - (uint32_t)(i0 + j));
    }
    __syncthreads();
    auto put = [&](int at, unsigned long long key) {
        vals[(int64_t)blockIdx.x * K + at] = (int32_t)((uint32_t)(key >> 32) ^ 0x80000000u);
        idx[(int64_t)blockIdx.x * K + at] = (int32_t)(0xFFFFFFFFu - (uint32_t)key);
    };
    if (K <= kRankMax) {
        // 2 threads (adjacent lanes) per key, each over half of the keys: its place is the number of larger ones
        const int e = tid >> 1, h = tid & 1;
        if (e - (lane >> 1) < K) {  // the warp has a key
            const unsigned long long key = e < K ? keys[e] : ~0ull;
            const int half = (K + 1) >> 1, b = h * half, n = h ? K - half : half;
            int rank = 0;
#pragma unroll 8
            for (int i = 0; i < n; ++i) rank += keys[b + i] > key ? 1 : 0;
            rank += __shfl_xor_sync(0xffffffffu, rank, 1);
            if (e < K && h == 0) put(rank, key);
        }
        return;
    }
    for (int k = 2; k <= kpad; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < kpad; i += kTopkThreads) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const unsigned long long a = keys[i], b = keys[ixj];
                    if (((i & k) == 0) ? (a < b) : (a > b)) {
                        keys[i] = b;
                        keys[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    for (int i = tid; i < K; i += kTopkThreads) put(i, keys[i]);
}

// K = 1: one warp per row keeps the largest value with the smallest index among its columns, and
// the warp combines the lanes' candidates (larger value, or equal value and smaller index, wins).
__global__ void __launch_bounds__(256) top1_kernel(const int32_t *__restrict__ S, int64_t lds, int32_t rows, int32_t N,
                                                   int32_t *__restrict__ vals, int32_t *__restrict__ idx) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t wpr = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += wpr) {
        const int32_t *s = S + r * lds;
        int32_t bv = INT32_MIN, bi = INT32_MAX;
        for (int j = lane; j < N; j += 32) {
            const int32_t v = s[j];
            if (v > bv || bi == INT32_MAX) {  // columns rise with j, so only a larger value replaces
                bv = v;
                bi = j;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int32_t ov = __shfl_xor_sync(0xffffffffu, bv, o), oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) {
                bv = ov;
                bi = oi;
            }
        }
        if (lane == 0) {
            vals[r] = bv;
            idx[r] = bi;
        }
    }
}

// Row gather in 4-byte words: dst row i = row idx[i] of source i / n (src_rows rows each).  An index
// outside [0, src_rows) gives a zero row and latches kStatusBadIndex in the device status word.
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint32_t *__restrict__ src, int64_t src_ldw,
                                                          int64_t src_rows, const int32_t *__restrict__ idx, int64_t n,
                                                          int64_t batches, int64_t roww, uint32_t *__restrict__ dst,
                                                          int64_t dst_ldw, int *status) {
    grid_wait();
    const int64_t total = n * batches * roww;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / roww, w = t - i * roww;
        const int64_t r = idx[i];
        if (r < 0 || r >= src_rows) {
            dst[i * dst_ldw + w] = 0u;
            if (w == 0 && status) atomicExch(status, kStatusBadIndex);
            continue;
        }
        dst[i * dst_ldw + w] = src[((i / n) * src_rows + r) * src_ldw + w];
    }
}

// I-ViT's ShiftGELU (the baseline of Sec. 3.3.1), one warp per row: M = max(max_row 1.702 x, 0),
// E = ShiftExp(I_p - M), E' = ShiftExp(-M), I_div = (E F) >> out_sh, Y = x I_div.  1.702 x by shifts
// in 64 bits (no int32 overflow for any input); ShiftExp magnitudes clamped at 2^30 (past k I0 the
// result no longer changes).
__device__ __forceinline__ int64_t ip1702(int32_t x) {
    const int64_t v = x;
    return v + (v >> 1) + (v >> 3) + (v >> 4);
}
__global__ void __launch_bounds__(256) ivit_shiftgelu_kernel(const int32_t *__restrict__ X, int64_t ldx, int64_t rows,
                                                             int32_t L, int32_t *__restrict__ Y, int64_t ldy,
                                                             ShiftExpC se, int32_t out_sh) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t wpr = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += wpr) {
        const int32_t *x = X + r * ldx;
        int64_t M = 0;
        for (int c = lane; c < L; c += 32) M = max(M, ip1702(x[c]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = max(M, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)M, o));
        const uint32_t e2 = shift_exp_mag((uint32_t)min(M, (int64_t)1 << 30), se);
        for (int c = lane; c < L; c += 32) {
            const int32_t v = x[c];
            const uint32_t E = shift_exp_mag((uint32_t)min(M - ip1702(v), (int64_t)1 << 30), se);
            const uint32_t F = div_int31(E + e2);
            const int64_t idiv = (int64_t)(((uint64_t)E * F) >> out_sh);
            Y[r * ldy + c] = (int32_t)((int64_t)v * idiv);
        }
    }
}

unsigned grid_for(int64_t work, int per_block) {
    const int64_t g = (work + per_block - 1) / per_block;
    const int64_t cap = (int64_t)sm_count() * 16;  // grid-stride loops: 16 CTAs of 256 threads per SM
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

cudaError_t launch_int_sigmoid(const int32_t *X, int32_t *Y, int64_t n, const ShiftExpC &se, int32_t k_out,
                               cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    launch_after(int_sigmoid_kernel, grid_for((n + 3) / 4, 256), 256, 0, s, X, Y, n, se, 32 - k_out);
    return cudaGetLastError();
}

cudaError_t launch_ivit_shiftgelu(const int32_t *X, int64_t ldx, int64_t rows, int32_t L, int32_t *Y, int64_t ldy,
                                  const GeluC &c, cudaStream_t s) {
    if (rows == 0) return cudaSuccess;
    launch_after(ivit_shiftgelu_kernel, grid_for((rows + 7) / 8, 1), 256, 0, s, X, ldx, rows, L, Y, ldy, c.se, c.out_sh);
    return cudaGetLastError();
}

cudaError_t launch_requant_sigmoid(const RequantParams &p, int32_t *sig, int64_t ld_sig, const ShiftExpC &se, int32_t k_out,
                                   cudaStream_t s) {
    if (p.rows == 0 || p.C == 0) return cudaSuccess;
    const unsigned g = grid_for(p.rows * (p.C / 4), 256);
    if (p.out_bits == 16) launch_after(requant_sigmoid_kernel<int16_t>, g, 256, 0, s, p, sig, ld_sig, se, 32 - k_out);
    else launch_after(requant_sigmoid_kernel<int32_t>, g, 256, 0, s, p, sig, ld_sig, se, 32 - k_out);
    return cudaGetLastError();
}

cudaError_t launch_relu_i8(const int8_t *X, int8_t *Y, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    launch_after(relu_i8_kernel, grid_for((n + 3) / 4, 256), 256, 0, s, X, Y, n);
    return cudaGetLastError();
}

cudaError_t launch_topk(const int32_t *S, int64_t lds, int32_t rows, int32_t N, int32_t K, int32_t *vals,
                        int32_t *idx, cudaStream_t s) {
    if (rows == 0) return cudaSuccess;
    if (K == 1) {
        launch_after(top1_kernel, grid_for(((int64_t)rows + 7) / 8, 1), 256, 0, s, S, lds, rows, N, vals, idx);
        return cudaGetLastError();
    }
    int kpad = 2;
    while (kpad < K) kpad <<= 1;
    const size_t smem = (size_t)kpad * 8;
    auto go = [&](auto kern, SmemLimit &limit) -> cudaError_t {
        const cudaError_t e = raise_smem_limit(limit, (const void *)kern, 16384 * 8);
        if (e != cudaSuccess) return e;
        launch_after(kern, (unsigned)rows, kTopkThreads, smem, s, S, lds, N, kpad, K, vals, idx);
        return cudaGetLastError();
    };
    static SmemLimit l2, l9, l16;
    if (N <= 2 * kTopkThreads) return go(topk_kernel<2>, l2);
    if (N <= 9 * kTopkThreads) return go(topk_kernel<9>, l9);  // the detector's 8400 memory tokens
    return go(topk_kernel<16>, l16);
}

cudaError_t launch_gather_rows(const void *src, int64_t src_ld_bytes, int64_t src_rows, const int32_t *idx, int64_t n,
                               int64_t batches, int64_t row_bytes, void *dst, int64_t dst_ld_bytes, cudaStream_t s) {
    if (n == 0 || batches == 0 || row_bytes == 0) return cudaSuccess;
    launch_after(gather_rows_kernel, grid_for(n * batches * (row_bytes / 4), 256), 256, 0, s, (const uint32_t *)src, src_ld_bytes / 4, src_rows, idx, n, batches, row_bytes / 4, (uint32_t *)dst,
        dst_ld_bytes / 4, status_word_ptr());
    return cudaGetLastError();
}

}  // namespace ilw
