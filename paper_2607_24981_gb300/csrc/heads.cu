// heads.cu -- the detection head's elementwise and selection kernels: integer sigmoid (the head's
// exponential by ShiftExp, Table 5, in SD-ShiftGELU's sign-dependent sigmoid form, Sec. 3.3.1 and
// Algorithm 1), ReLU on int8, per-row integer top-K (two-stage query selection) and row gather.
#include <algorithm>
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

// Per-row top-K, ties to the lower index: T threads (a multiple of 32) work on a row.  Bound by latency (a
// row's 33 KB at 8400 values are nothing) and, for many short rows, by the threads a row holds.  Sorting the
// whole padded row takes 105 steps over 16384 keys, 207 us for 8 rows of 8400; selecting first leaves K keys to
// order, 15 us.  Thread t of a row holds values t VPT .. (VPT of them) in registers.
//   1. the K-th largest value, found bit by bit below the row's maximum: every step counts the values at
//      or above a candidate over the row;
//   2. a scan over the threads gives every value above it its place among the selected, and the values
//      equal to it, in index order, the places left;
//   3. the selected keys (value, lower index first) are ordered by counting the larger ones where that is
//      little work a thread (K <= kRankMax for a whole CTA, else K^2 <= kRankWork T), else by a bitonic sort of the K keys.
// Where K pads to the same power of two as the row does there is nothing to select: topk_sort_kernel.
// A row takes the whole CTA, or a CTA of up to 256 threads takes 256 / T rows.
// Keys: (value biased to unsigned) << 32 | (2^32 - 1 - index), so one descending order puts larger
// values first and, for equal values, smaller indices first.  Padding keys are 0, below every real key.
constexpr int kTopkThreads = 1024;
constexpr int kRankMax = 512;
constexpr int kRankWork = 512;  // (4000 rows: 300 of 2000, T 256, 145 us against 185; 2000 rows: 500 of 2500, T 288, 146 against 107)
enum { kCta = 0, kWarp = 1, kWarps = 2 };  // a row's threads: the whole CTA, a warp, some warps of the CTA
// The T threads of a row meet (kWarps: each of the CTA's rows has a barrier of its own).
template <int ROW>
__device__ __forceinline__ void row_sync(int slot, int T) {
    if (ROW == kCta) __syncthreads();
    else if (ROW == kWarp) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "r"(T) : "memory");
}
__device__ __forceinline__ unsigned long long topk_key(uint32_t biased, int i) {
    return ((unsigned long long)biased << 32) | (0xFFFFFFFFu - (uint32_t)i);
}
// Result `at` of a row from its key
struct TopkOut {
    int32_t *vals, *idx;  // of the row
    __device__ __forceinline__ void put(int at, unsigned long long key) const {
        vals[at] = (int32_t)((uint32_t)(key >> 32) ^ 0x80000000u);
        idx[at] = (int32_t)(0xFFFFFFFFu - (uint32_t)key);
    }
};
// Orders kpad keys by T threads, largest first, and writes the first K
template <int ROW>
__device__ __forceinline__ void topk_sort(unsigned long long *keys, int kpad, int K, int tid, int T, int slot, const TopkOut &out) {
    for (int k = 2; k <= kpad; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < kpad; i += T) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const unsigned long long a = keys[i], b = keys[ixj];
                    if (((i & k) == 0) ? (a < b) : (a > b)) {
                        keys[i] = b;
                        keys[ixj] = a;
                    }
                }
            }
            row_sync<ROW>(slot, T);
        }
    for (int i = tid; i < K; i += T) out.put(i, keys[i]);
}

template <int VPT, int ROW>
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(const int32_t *__restrict__ S, int64_t lds, int32_t rows, int32_t N,
                                                            int32_t threads, int32_t kpad, int32_t K, int32_t *__restrict__ vals,
                                                            int32_t *__restrict__ idx) {
    grid_wait();
    extern __shared__ unsigned long long topk_keys[];  // kpad a row
    __shared__ uint32_t parts[2][32];                  // a value per warp
    const int T = ROW == kCta ? kTopkThreads : (ROW == kWarp ? 32 : threads), slot = ROW == kCta ? 0 : threadIdx.x / T, tid = threadIdx.x - slot * T, W = T >> 5;
    const int64_t row = ROW == kCta ? blockIdx.x : (int64_t)blockIdx.x * (blockDim.x / T) + slot;
    if (row >= rows) return;  // (all of the row's threads)
    const int32_t *s = S + row * lds;
    unsigned long long *keys = topk_keys + slot * kpad;
    uint32_t *part0 = parts[0] + slot * W, *part1 = parts[1] + slot * W;
    const int warp = tid >> 5, lane = tid & 31, i0 = tid * VPT;
    // biased values; past the row 0, which step 2 never selects (it is told apart by its index)
    uint32_t v[VPT];
#pragma unroll
    for (int j = 0; j < VPT; ++j) v[j] = i0 + j < N ? (uint32_t)s[i0 + j] ^ 0x80000000u : 0u;
    // the row's sum of one value per thread (alternating buffers: one barrier per call)
    int buf = 0;
    auto row_sum = [&](uint32_t x) -> uint32_t {
        x = __reduce_add_sync(0xffffffffu, x);
        if (W == 1) return x;
        if (lane == 0) part0[buf + warp] = x;
        row_sync<ROW>(slot, T);
        x = __reduce_add_sync(0xffffffffu, lane < W ? part0[buf + lane] : 0u);
        buf ^= 32;
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
    if (W > 1) {
        if (lane == 0) {
            part0[warp] = hi;
            part1[warp] = lo;
        }
        row_sync<ROW>(slot, T);
        hi = __reduce_max_sync(0xffffffffu, lane < W ? part0[lane] : 0u);
        lo = __reduce_min_sync(0xffffffffu, lane < W ? part1[lane] : 0xffffffffu);
        row_sync<ROW>(slot, T);
    }
    // thr: the largest value with at least K values at or above it (that many are at or above `lo`)
    const int top = 32 - __clz(hi ^ lo);
    uint32_t thr = top == 32 ? 0u : hi >> top << top;
    for (int bit = top - 1; bit >= 0; --bit) {
        const uint32_t cand = thr | (1u << bit);
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < VPT; ++j) c += (i0 + j < N && v[j] >= cand) ? 1u : 0u;
        if (row_sum(c) >= (uint32_t)K) thr = cand;
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
    row_sync<ROW>(slot, T);
    if (lane == 31) part0[warp] = incl;
    for (int i = K + tid; i < kpad; i += T) keys[i] = 0ull;
    row_sync<ROW>(slot, T);
    const uint32_t w = lane < W ? part0[lane] : 0u;
    const uint32_t total = __reduce_add_sync(0xffffffffu, w);
    uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + incl - c;
    const uint32_t above = total >> 16;
    uint32_t pg = before >> 16, pe = above + (before & 0xffffu);
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
        if (i0 + j >= N || v[j] < thr) continue;
        const uint32_t pos = v[j] > thr ? pg++ : pe++;
        if (pos < (uint32_t)K) keys[pos] = topk_key(v[j], i0 + j);
    }
    row_sync<ROW>(slot, T);
    const TopkOut out{vals + row * K, idx + row * K};
    if (ROW == kCta ? K > kRankMax : K * K > kRankWork * T) {
        topk_sort<ROW>(keys, kpad, K, tid, T, slot, out);
        return;
    }
    // 2 threads (adjacent lanes) per key, each over half of the keys: its place is the number of larger ones
    for (int e2 = tid; (e2 - lane) >> 1 < K; e2 += T) {  // while the warp has a key
        const int e = e2 >> 1, h = e2 & 1;
        const unsigned long long key = e < K ? keys[e] : ~0ull;
        const int half = (K + 1) >> 1, b = h * half, n = h ? K - half : half;
        int rank = 0;
#pragma unroll 8
        for (int i = 0; i < n; ++i) rank += keys[b + i] > key ? 1 : 0;
        rank += __shfl_xor_sync(0xffffffffu, rank, 1);
        if (e < K && h == 0) out.put(rank, key);
    }
}

// The same where every value of the (padded) row is ordered.
template <int ROW>
__global__ void __launch_bounds__(kTopkThreads) topk_sort_kernel(const int32_t *__restrict__ S, int64_t lds, int32_t rows, int32_t N,
                                                                 int32_t threads, int32_t kpad, int32_t K, int32_t *__restrict__ vals,
                                                                 int32_t *__restrict__ idx) {
    grid_wait();
    extern __shared__ unsigned long long topk_keys[];
    const int T = ROW == kCta ? blockDim.x : (ROW == kWarp ? 32 : threads), slot = ROW == kCta ? 0 : threadIdx.x / T, tid = threadIdx.x - slot * T;
    const int64_t row = ROW == kCta ? blockIdx.x : (int64_t)blockIdx.x * (blockDim.x / T) + slot;
    if (row >= rows) return;
    const int32_t *s = S + row * lds;
    unsigned long long *keys = topk_keys + slot * kpad;
    for (int i = tid; i < kpad; i += T) keys[i] = i < N ? topk_key((uint32_t)s[i] ^ 0x80000000u, i) : 0ull;
    row_sync<ROW>(slot, T);
    topk_sort<ROW>(keys, kpad, K, tid, T, slot, TopkOut{vals + row * K, idx + row * K});
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

// Row gather in 4-byte words: dst row b n + i = row idx[b n + i] of source b (src_rows rows each); the blocks' y is
// the source.  Bound by the division that finds a word's row (I: 32-bit where the words of a source's rows
// allow it; 134400 rows of 256 bytes 17.9 us, 26.0 with 64 bits, 31.5 with a second one for the source).  An index
// outside [0, src_rows) gives a zero row and latches kStatusBadIndex in the device status word.
template <typename I>
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint32_t *__restrict__ src, int64_t src_ldw,
                                                          int64_t src_rows, const int32_t *__restrict__ idx, int64_t n,
                                                          int64_t batches, I roww, uint32_t *__restrict__ dst,
                                                          int64_t dst_ldw, int *status) {
    grid_wait();
    const I total = (I)n * roww;
    for (int64_t b = blockIdx.y; b < batches; b += gridDim.y) {
        const uint32_t *s = src + b * src_rows * src_ldw;
        const int32_t *ix = idx + b * n;
        uint32_t *d = dst + b * n * dst_ldw;
        for (I t = blockIdx.x * (I)blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
            const I i = t / roww, w = t - i * roww;
            const int64_t r = ix[i];
            if (r < 0 || r >= src_rows) {
                d[i * dst_ldw + w] = 0u;
                if (w == 0 && status) atomicExch(status, kStatusBadIndex);
                continue;
            }
            d[i * dst_ldw + w] = s[r * src_ldw + w];
        }
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
    if (N <= 32)  // too little to select from: 134400 rows, 4 of 16, 65 us, 113 with the selection
        while (kpad < N) kpad <<= 1;
    auto go = [&](auto kern, SmemLimit &limit, int threads, int per) -> cudaError_t {  // per: rows of a CTA
        const cudaError_t e = raise_smem_limit(limit, (const void *)kern, 16384 * 8);
        if (e != cudaSuccess) return e;
        launch_after(kern, (unsigned)(((int64_t)rows + per - 1) / per), per * threads, (size_t)per * kpad * 8, s, S, lds, rows, N,
                     threads, kpad, K, vals, idx);
        return cudaGetLastError();
    };
    static SmemLimit sw, s1, s8, w2, w9, w16, n2, n4, n8;
    if (kpad >= N) {
        const int threads = std::min(std::max(kpad / 2, 32), kTopkThreads);
        if (threads == 32) return go(topk_sort_kernel<kWarp>, sw, 32, 8);
        return threads < 256 ? go(topk_sort_kernel<kWarps>, s8, threads, 256 / threads) : go(topk_sort_kernel<kCta>, s1, threads, 1);
    }
    // A whole CTA per row for long rows (the detector's 8400 memory tokens), and for shorter ones while the chip
    // holds all of them at once; where it does not, and for the shortest always, as few threads as hold the
    // row.  (A CTA per row and this: 134400 rows, 5 of 80, 3926 us and 113; 20000, 100 of 512, 633 and 135; one row of 80
    // 7.4 and 3.5; 8 rows, 100 of 300, 7.9 and 10.4, and 1000 rows, 300 of 8400, 103 and 117, which stay.)
    auto threads = [&](int vpt) { return (N + 32 * vpt - 1) / (32 * vpt) * 32; };
    if (N <= 64) return go(topk_kernel<2, kWarp>, n2, 32, 8);
    if (N <= 128) return go(topk_kernel<4, kWarp>, n4, 32, 8);
    if (N <= 2048 && rows > 2 * sm_count()) return go(topk_kernel<8, kWarps>, n8, threads(8), std::max(256 / threads(8), 1));
    if (N <= 2 * kTopkThreads) return go(topk_kernel<2, kCta>, w2, kTopkThreads, 1);
    if (N <= 9 * kTopkThreads) return go(topk_kernel<9, kCta>, w9, kTopkThreads, 1);
    return go(topk_kernel<16, kCta>, w16, kTopkThreads, 1);
}

cudaError_t launch_gather_rows(const void *src, int64_t src_ld_bytes, int64_t src_rows, const int32_t *idx, int64_t n,
                               int64_t batches, int64_t row_bytes, void *dst, int64_t dst_ld_bytes, cudaStream_t s) {
    if (n == 0 || batches == 0 || row_bytes == 0) return cudaSuccess;
    const dim3 grid(grid_for(n * (row_bytes / 4), 256), (unsigned)std::min<int64_t>(batches, 65535));
    auto go = [&](auto kern, auto roww) {
        launch_after(kern, grid, 256, 0, s, (const uint32_t *)src, src_ld_bytes / 4, src_rows, idx, n, batches, roww,
                     (uint32_t *)dst, dst_ld_bytes / 4, status_word_ptr());
    };
    if (n * (row_bytes / 4) < (1ll << 31)) go(gather_rows_kernel<uint32_t>, (uint32_t)(row_bytes / 4));
    else go(gather_rows_kernel<int64_t>, row_bytes / 4);
    return cudaGetLastError();
}

}  // namespace ilw
