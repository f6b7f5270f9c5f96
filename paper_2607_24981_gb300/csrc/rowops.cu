// rowops.cu -- bandwidth-bound integer nonlinearities: Constrained Shiftmax over rows
// (Algorithm 2), SD-ShiftGELU (Algorithm 1) and I-LayerNorm (Sec. 3.3).
//
// One warp owns one row; the row stays in registers between the two dependent reductions, so
// HBM sees each input byte once.  Rows are read with 128-bit loads when the layout allows.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>

#include "ilw_kernels.h"

namespace ilw {
namespace {

__device__ __forceinline__ int32_t warp_max(int32_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int64_t warp_sum_i64(int64_t v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------------------ Constrained Shiftmax rows
// NCH = 4-element chunks per lane (row length <= 128 * NCH); vector loads need len % 4 == 0
// and 16-byte aligned rows.
template <int LANES>
__device__ __forceinline__ int32_t group_max(int32_t v) {
#pragma unroll
    for (int o = LANES / 2; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o, LANES));
    return v;
}
template <int LANES>
__device__ __forceinline__ uint64_t group_sum_u64(uint64_t v) {
#pragma unroll
    for (int o = LANES / 2; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, LANES);
    return v;
}

// The output floor(e F / 2^sh) as one high-word product: for sh <= 32 and F < 2^sh,
// F 2^(32 - sh) < 2^32 and floor(e F 2^(32 - sh) / 2^32) is the same floor; for sh > 32 the high word
// of e F shifted right by sh - 32 (floors compose).  `ok` is false for the rows neither form covers
// (sh < 32 with F >= 2^sh, i.e. a reduced denominator below 2^(31 - sh)), which take shiftmax_out.
struct RowOut {
    uint32_t Fs;
    uint32_t rs;
    bool ok;
};
__device__ __forceinline__ RowOut row_out(const RowNorm &rn) {
    RowOut o;
    if (rn.sh <= 32) {
        o.ok = rn.sh == 32 || (rn.F >> rn.sh) == 0;
        o.Fs = o.ok ? rn.F << (32 - rn.sh) : 0u;
        o.rs = 0;
    } else {
        o.ok = true;
        o.Fs = rn.F;
        o.rs = (uint32_t)min(rn.sh - 32, 31);
    }
    return o;
}

// LANES lanes own one row (32 / LANES rows per warp); NCH = 4-element chunks per lane (row length
// <= 4 * LANES * NCH).  Vector loads need len % 4 == 0 and 16-byte aligned rows.  All NCH loads of a
// lane are issued before the first use, so each warp keeps 32 * NCH * 16 bytes in flight.
// SUM4: I0 2^k < 2^30, so four ShiftExp values add up in 32 bits (two always do: I0 2^k < 2^31).
template <int NCH, int LANES, bool FASTQ, bool SUM4>
__global__ void __launch_bounds__(256) shiftmax_rows_vec(const int32_t *__restrict__ X, int64_t ldx,
                                                          int64_t rows, int32_t len, const ShiftmaxC c,
                                                          uint8_t *__restrict__ P, int64_t ldp) {
    grid_wait();
    constexpr int RPW = 32 / LANES;
    const int lane = threadIdx.x & 31, sub = lane % LANES;
    const int64_t row = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * RPW + lane / LANES;
    const bool live = row < rows;  // every lane stays for the shuffles
    const int nch = live ? (len >> 2) : 0;
    const int4 *xr = (const int4 *)(X + (live ? row : 0) * ldx);
    int4 v[NCH];
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int ch = sub + LANES * j;
        v[j] = ch < nch ? __ldcs(xr + ch) : make_int4(INT_MIN, INT_MIN, INT_MIN, INT_MIN);
    }
    int32_t mx = INT_MIN;
#pragma unroll
    for (int j = 0; j < NCH; ++j) mx = max(mx, max(max(v[j].x, v[j].y), max(v[j].z, v[j].w)));
    mx = group_max<LANES>(mx);
    // a = mx - x >= 0 as an unsigned difference; magnitudes beyond 2^30 are deep in ShiftExp's
    // clamp region and are replaced by 2^30 (same value).  Padding lanes (INT_MIN) give a >= 2^30
    // and are not summed.
    uint64_t sum = 0;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int ch = sub + LANES * j;
        uint32_t *e = (uint32_t *)&v[j];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t a = min((uint32_t)mx - e[q], 1u << 30);
            e[q] = shift_exp_mag_q<FASTQ>(a, c.se);
        }
        if (ch < nch) {
            if constexpr (SUM4) sum += (uint64_t)(e[0] + e[1] + e[2] + e[3]);
            else sum += (uint64_t)(e[0] + e[1]) + (uint64_t)(e[2] + e[3]);
        }
    }
    sum = group_sum_u64<LANES>(sum);
    if (!live) return;
    const RowNorm rn = shiftmax_norm(sum, c.s_d, c.m_p, c.M_hw, c.k_out);
    const RowOut ro = row_out(rn);
    uint32_t *pr = (uint32_t *)(P + row * ldp);
    // every output is below 2^k_out <= 256: the four bytes of a chunk by two byte permutations
    if (ro.ok && ro.rs == 0) {  // sh <= 32: one high-word product per output
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int ch = sub + LANES * j;
            if (ch < nch) {
                const uint32_t *e = (const uint32_t *)&v[j];
                const uint32_t b01 = __byte_perm(__umulhi(e[0], ro.Fs), __umulhi(e[1], ro.Fs), 0x0040);
                const uint32_t b23 = __byte_perm(__umulhi(e[2], ro.Fs), __umulhi(e[3], ro.Fs), 0x0040);
                __stcs(pr + ch, __byte_perm(b01, b23, 0x5410));
            }
        }
    } else if (ro.ok) {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int ch = sub + LANES * j;
            if (ch < nch) {
                const uint32_t *e = (const uint32_t *)&v[j];
                const uint32_t b01 = __byte_perm(__umulhi(e[0], ro.Fs) >> ro.rs, __umulhi(e[1], ro.Fs) >> ro.rs, 0x0040);
                const uint32_t b23 = __byte_perm(__umulhi(e[2], ro.Fs) >> ro.rs, __umulhi(e[3], ro.Fs) >> ro.rs, 0x0040);
                __stcs(pr + ch, __byte_perm(b01, b23, 0x5410));
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int ch = sub + LANES * j;
            if (ch < nch) {
                const uint32_t *e = (const uint32_t *)&v[j];
                const uint32_t o = shiftmax_out(e[0], rn) | (shiftmax_out(e[1], rn) << 8) |
                                   (shiftmax_out(e[2], rn) << 16) | (shiftmax_out(e[3], rn) << 24);
                __stcs(pr + ch, o);
            }
        }
    }
}

// Any length / alignment: three passes over the row from global memory (L1/L2 resident).
__global__ void __launch_bounds__(256) shiftmax_rows_generic(const int32_t *__restrict__ X, int64_t ldx,
                                                              int64_t rows, int32_t len, const ShiftmaxC c,
                                                              uint8_t *__restrict__ P, int64_t ldp) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int32_t *x = X + row * ldx;
    int32_t mx = INT_MIN;
    for (int i = lane; i < len; i += 32) mx = max(mx, x[i]);
    mx = warp_max(mx);
    const int32_t lowb = mx > INT_MIN + (1 << 30) ? mx - (1 << 30) : INT_MIN;
    uint64_t sum = 0;
    for (int i = lane; i < len; i += 32) {
        uint32_t a = x[i] > lowb ? (uint32_t)(mx - x[i]) : (1u << 30);
        sum += shift_exp_mag(a, c.se);
    }
    sum = warp_sum_u64(sum);
    const RowNorm rn = shiftmax_norm(sum, c.s_d, c.m_p, c.M_hw, c.k_out);
    for (int i = lane; i < len; i += 32) {
        uint32_t a = x[i] > lowb ? (uint32_t)(mx - x[i]) : (1u << 30);
        P[row * ldp + i] = (uint8_t)shiftmax_out(shift_exp_mag(a, c.se), rn);
    }
}

// ------------------------------------------------------------------ SD-ShiftGELU
__device__ __forceinline__ int32_t gelu_one(int32_t x, const GeluC &c) {
    int32_t xc = min(max(x, -(1 << 26)), 1 << 26);  // I_div is constant beyond |x| = 2^19
    return x * gelu_idiv(xc, c);
}

__global__ void __launch_bounds__(256) sdshiftgelu_vec(const int4 *__restrict__ X, int4 *__restrict__ Y,
                                                        int64_t n4, const GeluC c) {
    grid_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        int4 v = __ldcs(X + i);
        int4 o;
        o.x = gelu_one(v.x, c);
        o.y = gelu_one(v.y, c);
        o.z = gelu_one(v.z, c);
        o.w = gelu_one(v.w, c);
        __stcs(Y + i, o);
    }
}
// Table form: I_div depends on x alone and is constant for |x| >= T (both ShiftExp inputs are in
// their clamp regions there), so each CTA tabulates I_div(x) for x in [-T, T] with the same device
// function (exact by construction) and streams the data through lookups.
__global__ void __launch_bounds__(256) sdshiftgelu_table(const int4 *__restrict__ X, int4 *__restrict__ Y, int64_t n4,
                                                          const GeluC c, int32_t T) {
    grid_wait();
    extern __shared__ uint8_t tab[];
    for (int i = threadIdx.x; i <= 2 * T; i += blockDim.x) tab[i] = (uint8_t)gelu_idiv(i - T, c);
    __syncthreads();
    const uint8_t *t0 = tab + T;
    auto f = [&](int32_t x) { return x * (int32_t)t0[min(max(x, -T), T)]; };
    // 4 vectors per thread per step, all loaded before the first lookup (64 bytes in flight)
    constexpr int U = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + (U - 1) * stride < n4; i += U * stride) {
        int4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = __ldcs(X + i + u * stride);
#pragma unroll
        for (int u = 0; u < U; ++u) __stcs(Y + i + u * stride, make_int4(f(v[u].x), f(v[u].y), f(v[u].z), f(v[u].w)));
    }
    for (; i < n4; i += stride) {
        const int4 v = __ldcs(X + i);
        __stcs(Y + i, make_int4(f(v.x), f(v.y), f(v.z), f(v.w)));
    }
}

__global__ void sdshiftgelu_tail(const int32_t *X, int32_t *Y, int64_t start, int64_t n, const GeluC c) {
    grid_wait();
    int64_t i = start + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) Y[i] = gelu_one(X[i], c);
}

// ------------------------------------------------------------------ I-LayerNorm
// Newton's integer square root r <- (r + V / r) >> 1 from r = 2^16, exactly `iters` steps (the loop
// stops at 0, which only V = 0 reaches), cut short once the rest of the sequence is known: a fixed
// point repeats forever, and once r_{i+1} = r_{i-1} the iterates alternate between two values, so
// r_iters is read off the parity of the steps left.  Identical result, fewer 64-bit divisions.
__device__ __noinline__ uint64_t newton_isqrt_early(uint64_t V, int iters) {
    uint64_t r = 1ull << 16, prev = ~0ull;
    for (int it = 0; it < iters; ++it) {
        if (r == 0) break;
        const uint64_t nx = (r + V / r) >> 1;
        if (nx == r) break;
        if (nx == prev) {
            r = ((iters - it - 1) & 1) ? r : nx;
            break;
        }
        prev = r;
        r = nx;
    }
    return r < 1 ? 1 : r;
}

// floor(V / r) for V < 2^48 and 1 <= r < 2^32 with a quotient below 2^26: a float estimate (relative
// error < 2^-20, so absolute error < 2^6), one float refinement from the exact 64-bit remainder
// (error < 1 on a remainder below 2^7 r), and a final +-1 test on the remainder.
// A 64-bit integer of magnitude below 2^62 as a float from its two 32-bit halves (two 32-bit
// conversions and one multiply-add: relative error below 2^-22), instead of a 64-bit conversion.
__device__ __forceinline__ float u64_to_float(uint64_t v) {
    return fmaf(__uint2float_rn((uint32_t)(v >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)v));
}
__device__ __forceinline__ float i64_to_float(int64_t v) {
    return fmaf(__int2float_rn((int32_t)(v >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)v));
}
__device__ __forceinline__ uint32_t div_u48_u32(uint64_t V, uint32_t r) {
    const float rinv = __frcp_rn(__uint2float_rn(r));
    uint32_t q = __float2uint_rz(u64_to_float(V) * rinv);
    int64_t rem = (int64_t)V - (int64_t)q * r;
    const int32_t dq = __float2int_rd(i64_to_float(rem) * rinv);
    q += dq;
    rem -= (int64_t)dq * r;
    if (rem < 0) --q;
    else if (rem >= (int64_t)r) ++q;
    return q;
}
// newton_isqrt_early for V < 2^48: the first step from 2^16 is a shift, and every later divisor r
// is at least isqrt(V) (a floored Newton step from any positive start lands at or above isqrt(V),
// and the iterates then decrease), so r < 2^32 and V / r < isqrt(V) + 3 < 2^25.
__device__ __forceinline__ uint64_t newton_isqrt_fast(uint64_t V, int iters) {
    if (iters <= 0) return 1ull << 16;
    uint64_t r = ((1ull << 16) + (V >> 16)) >> 1, prev = 1ull << 16;
    if (r == prev) return r;
    for (int it = 1; it < iters; ++it) {
        if (r == 0) break;
        const uint64_t nx = (r + div_u48_u32(V, (uint32_t)r)) >> 1;
        if (nx == r) break;
        if (nx == prev) {
            r = ((iters - it - 1) & 1) ? r : nx;
            break;
        }
        prev = r;
        r = nx;
    }
    return r < 1 ? 1 : r;
}

// Output element types of I-LayerNorm: int8, int16, or the int8 values carried in fp16.
template <typename TOut> struct LnOut { static constexpr int bits = 8 * (int)sizeof(TOut); };
template <> struct LnOut<__half> { static constexpr int bits = 8; };
// 4 outputs of one row, stored at y (4-element aligned)
template <typename TOut>
__device__ __forceinline__ void ln_store4(TOut *y, const int32_t (&o)[4]) {
    if constexpr (sizeof(TOut) == 1) {
        *(uint32_t *)y = (uint32_t)(uint8_t)o[0] | ((uint32_t)(uint8_t)o[1] << 8) | ((uint32_t)(uint8_t)o[2] << 16) |
                         ((uint32_t)(uint8_t)o[3] << 24);
    } else if constexpr (LnOut<TOut>::bits == 16) {
        *(uint2 *)y = make_uint2((uint32_t)(uint16_t)o[0] | ((uint32_t)(uint16_t)o[1] << 16),
                                 (uint32_t)(uint16_t)o[2] | ((uint32_t)(uint16_t)o[3] << 16));
    } else {
        // |v| <= 127: the fp16 bits of 1152 + v are 0x6480 + v; one half2 subtract of 1152 leaves v
        const __half2 k1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
        uint32_t w[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            uint32_t x = (uint32_t)(0x6480 + o[2 * j]) | ((uint32_t)(0x6480 + o[2 * j + 1]) << 16);
            __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&x), k1152);
            w[j] = *reinterpret_cast<uint32_t *>(&h);
        }
        *(uint2 *)y = make_uint2(w[0], w[1]);
    }
}

// The same from u = value + 127 (8-bit outputs, in [0, 254]) or value + 32767 (16-bit, in [0, 65534]):
// clamping to u is one add-min-relu, and one add and one exclusive or per word undo the bias (u + 1 never
// carries into the next lane, and flipping the top bit takes 128 or 32768 off).
template <typename TOut> struct LnBias { static constexpr int one = LnOut<TOut>::bits == 8 ? 127 : 32767; };
template <typename TOut>
__device__ __forceinline__ void ln_store4_biased(TOut *y, const int32_t (&u)[4]) {
    const uint32_t a = __byte_perm(u[0], u[1], sizeof(TOut) == 1 ? 0x0040 : 0x5410);
    const uint32_t b = __byte_perm(u[2], u[3], sizeof(TOut) == 1 ? 0x0040 : 0x5410);
    if constexpr (sizeof(TOut) == 1) {
        *(uint32_t *)y = (__byte_perm(a, b, 0x5410) + 0x01010101u) ^ 0x80808080u;
    } else if constexpr (LnOut<TOut>::bits == 16) {
        *(uint2 *)y = make_uint2((a + 0x00010001u) ^ 0x80008000u, (b + 0x00010001u) ^ 0x80008000u);
    } else {
        // the fp16 bits of 1024 + u are 0x6400 + u; one half2 subtract of 1151 leaves the value
        const __half2 k1151 = __half2half2(__ushort_as_half((unsigned short)0x647f));
        uint32_t wa = a | 0x64006400u, wb = b | 0x64006400u;
        __half2 ha = __hsub2(*reinterpret_cast<__half2 *>(&wa), k1151);
        __half2 hb = __hsub2(*reinterpret_cast<__half2 *>(&wb), k1151);
        *(uint2 *)y = make_uint2(*reinterpret_cast<uint32_t *>(&ha), *reinterpret_cast<uint32_t *>(&hb));
    }
}

// The second result of 4 normalised values y of a row.
__device__ __forceinline__ void ln_second4(const LnParams &p, int64_t row, int c, const int32_t (&y)[4]) {
    int64_t z[4] = {0, 0, 0, 0};
    if (p.Z) {
        const uint2 w = *(const uint2 *)(p.Z + row * p.ldz + c);
        z[0] = rq((int16_t)(w.x & 0xFFFFu), p.m2, p.s2);
        z[1] = rq((int16_t)(w.x >> 16), p.m2, p.s2);
        z[2] = rq((int16_t)(w.y & 0xFFFFu), p.m2, p.s2);
        z[3] = rq((int16_t)(w.y >> 16), p.m2, p.s2);
    }
    uint32_t w = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) w |= (uint32_t)(uint8_t)sat8(rq(y[u], p.m1, p.s1) + z[u]) << (8 * u);
    *(uint32_t *)(p.Y2 + row * p.ldy2 + c) = w;
}

// acc += a * b with a 64-bit accumulator in one wide multiply-add
__device__ __forceinline__ void madw(int64_t &acc, int32_t a, int32_t b) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// The normalisation of 4 elements in 64-bit arithmetic, for rows or columns outside the 32-bit
// fast path's conditions (kept out of line so that its registers do not weigh on the fast path).
__device__ __noinline__ void ln_norm4_exact(const int32_t (&x)[4], int64_t mu, int64_t F, const int32_t (&be)[4],
                                            const int32_t (&mm)[4], const int32_t (&ss)[4], int out_bits,
                                            int32_t (&o)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t n = (((int64_t)x[u] - mu) * F) >> 1;
        const int64_t tq = rq(n + be[u], mm[u], ss[u]);
        o[u] = out_bits == 8 ? sat8(tq) : sat16(tq);
    }
}

// A launch's constants: the range of V whose Newton root needs no steps (worked out once per step count),
// 1 / (2 C).
struct LnConst {
    uint64_t lo, hi;
    float inv2c;
};
// isqrt(V) for 4 <= V < 2^48, and rem = V - s^2 in [0, 2 s].  The float root is below 2^-21 relative and 1
// absolute off, 9 at most, so V - s^2 fits 32 bits (and is formed there); one step from it leaves s within 1,
// which the remainder tells.
__device__ __forceinline__ uint32_t isqrt_u48(uint64_t V, uint32_t &rem_out) {
    const float vf = u64_to_float(V), rs = rsqrtf(vf);
    uint32_t s = __float2uint_rz(vf * rs);
    int32_t rem = (int32_t)((uint32_t)V - s * s);
    s += __float2int_rd(__int2float_rn(rem) * (0.5f * rs));
    rem = (int32_t)((uint32_t)V - s * s);
    if (rem < 0) {
        --s;
        rem += 2 * (int32_t)s + 1;
    } else if (rem > 2 * (int32_t)s) {
        rem -= 2 * (int32_t)s + 1;
        ++s;
    }
    rem_out = (uint32_t)rem;
    return s;
}
// floor((2^31 - 1) / s) for 2 <= s < 2^25: the float quotient is below 2^-21 relative and 1 absolute
// off, so the remainder is below 2^10 + s in magnitude and one step from it leaves 1 at most.
__device__ __forceinline__ uint32_t div_int31_u24(uint32_t s) {
    const float rc = __fdividef(1.0f, __uint2float_rn(s));
    uint32_t q = __float2uint_rz(2147483648.0f * rc);
    int32_t rem = (int32_t)(kInt31Max - q * s);
    const int32_t dq = __float2int_rd(__int2float_rn(rem) * rc);
    q += dq;
    rem -= dq * (int32_t)s;
    if (rem < 0) --q;
    else if (rem >= (int32_t)s) ++q;
    return q;
}
// A row's mean, F and whether y F fits 32 bits, from its sums, in full generality.
struct LnRow {
    int64_t mu, F;
    bool fits;
};
// (100000 rows of 256 int32 values past 16 bits to int8: 53.7 us with a 64-bit mean and the steps for every row, 50.8
// so; one thread per row behind two barriers, which 16-bit values are better without, 47.1)
__device__ __noinline__ LnRow ln_row_general(int64_t S, int64_t Q, int32_t C, int32_t iters, uint64_t lo, uint64_t hi) {
    // mu = floor((2S + C) / (2C)); V = Q - 2 mu S + C mu^2 (= sum (x - mu)^2)
    const int64_t num = 2 * S + C, den = 2 * (int64_t)C;
    int64_t mu;
    if (num == (int32_t)num) {
        const int32_t n32 = (int32_t)num, d32 = (int32_t)den, q = n32 / d32;
        mu = q - (n32 < 0 && n32 != q * d32 ? 1 : 0);
    } else {
        mu = num / den;
        if (mu * den != num && num < 0) mu -= 1;
    }
    const uint64_t V = (uint64_t)(Q - 2 * mu * S + (int64_t)C * mu * mu);
    if (V >= lo && V <= hi) {  // the root without the steps, as below
        uint32_t rem;
        const uint32_t s = isqrt_u48(V, rem);
        if (rem != 2 * s) return {mu, (int64_t)div_int31_u24(s), true};
    }
    const uint64_t R = V < (1ull << 48) ? newton_isqrt_fast(V, iters) : newton_isqrt_early(V, iters);
    return {mu, R < (1ull << 32) ? (int64_t)div_int31((uint32_t)R) : 0, iters >= 1 || V < (1ull << 32)};
}

// I-LayerNorm by rows (Sec. 3.3; mean, variance, Newton's integer square root,
// F = floor((2^31 - 1) / R), n = (y F) >> 1, out = sat(rq(n + beta; m, s))).  LPR lanes own one row,
// 32 / LPR rows per warp and step (persistent grid).  A lane reads 16-byte chunks sub, sub + LPR, ... of
// its row (CPL at most, exactly when FULL; the LPR lanes of a row read adjacent chunks, so a warp's load
// covers 32 / LPR row segments of LPR * 16 bytes) and keeps them in registers, sums x and x^2, the LPR lanes
// combine the sums with shuffles, and each works out the row's mean, root and F.  The warps run apart, no
// barrier after the parameters are staged, and a warp's first rows are loaded before that.
// Long inputs are bound by instructions beside the loads, short ones by the chain of one row; so the
// per-row part is kept short: for 16-bit values (a warp's, as almost always) the sums of two products and
// the mean are 32-bit, and the Newton root is taken without its steps.  The iteration, for V in
// [lo, hi], has reached {isqrt(V), isqrt(V) + 1} a step before its last, and from there it stays at
// s = isqrt(V), unless V = s^2 + 2 s, where it alternates between the two.  Those V and V outside the range
// take the steps; wider values sum in 64 bits.
// 2^20 rows of 384 int32 to int8: 302 us, 6.66 TB/s (461 us with the per-row part on one thread per row
// behind two barriers and stepped); with half the values per lane (more lanes repeating the per-row part)
// 10 % slower.
// 32-bit normalisation: after at least one Newton step R >= isqrt(V) >= |y| for every y = x - mu of
// the row (a floored Newton step from any positive start lands at or above isqrt(V)), so
// |y F| <= |y| (2^31 - 1) / R < 2^31 and y F fits int32; with shifts s >= 33 and |beta| <= 2^30 in every
// column the requantisation is the high-word form (with a scalar rounding constant when the shifts are
// the same); otherwise (or for rows with iters = 0 and V >= 2^32) the 64-bit formulas run.
// SECOND: the second result of LnParams.
template <typename TIn, typename TOut, int LPR, int CPL, bool FULL, bool SECOND = false>
__global__ void __launch_bounds__(256, 3) layernorm_rows(const LnParams p, const LnConst lc) {
    grid_wait();
    extern __shared__ __align__(16) int32_t ln_par[];  // beta, mult, shift of CP columns
    constexpr int EB = sizeof(TIn), EPC = 16 / EB;      // elements per 16-byte chunk
    constexpr int RPW = 32 / LPR, CP = LPR * CPL * EPC;
    const int C = p.C;
    int32_t *s_beta = ln_par, *s_mult = ln_par + CP, *s_shift = ln_par + 2 * CP;
    const int lane = threadIdx.x & 31, sub = lane % LPR, rr = lane / LPR;
    const int64_t step = (int64_t)gridDim.x * 8 * RPW;
    int64_t row = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * RPW + rr;
    // the chunks that the lane has of its row: none past the end (every lane stays for the shuffles)
    auto chunks = [&]() { return row < p.rows ? C / EPC - sub : 0; };
    int4 v[CPL];
    auto load = [&]() {
        const int nc = chunks();
        const int4 *xr = (const int4 *)((const uint8_t *)p.X + row * p.ldx * EB) + sub;
#pragma unroll
        for (int i = 0; i < CPL; ++i)
            v[i] = (FULL ? nc > 0 : LPR * i < nc) ? __ldg(xr + LPR * i) : make_int4(0, 0, 0, 0);
    };
    load();
    for (int i = threadIdx.x; i < C / 4; i += blockDim.x) {
        ((int4 *)s_beta)[i] = __ldg((const int4 *)p.beta + i);
        ((int4 *)s_mult)[i] = __ldg((const int4 *)p.mult + i);
        ((int4 *)s_shift)[i] = __ldg((const int4 *)p.shift + i);
    }
    __syncthreads();
    // the fast forms need shifts >= 33 for every column: one for all of them, or each its own
    const int32_t shift0 = s_shift[0];
    bool col_fast = true, col_same = true;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        col_fast &= s_beta[c] >= -(1 << 30) && s_beta[c] <= (1 << 30) && s_shift[c] >= 33;
        col_same &= s_shift[c] == shift0;
    }
    const bool cols_fast = __syncthreads_and(col_fast) != 0, cols_same = __syncthreads_and(col_same) != 0;
    const int32_t rnd = cols_fast ? 1 << (shift0 - 33) : 0, sh = shift0 - 32;

    for (; __any_sync(0xffffffffu, row < p.rows); row += step, load()) {
        bool small = true;
        if constexpr (EB == 4) {
            int32_t mx = 0, mn = 0;
#pragma unroll
            for (int i = 0; i < CPL; ++i) {
                mx = __vimax3_s32(mx, v[i].x, v[i].y);
                mn = __vimin3_s32(mn, v[i].x, v[i].y);
                mx = __vimax3_s32(mx, v[i].z, v[i].w);
                mn = __vimin3_s32(mn, v[i].z, v[i].w);
            }
            small = __all_sync(0xffffffffu, mx < 32768 && mn >= -32768);
        }
        int64_t mu, F;
        bool fits;
        if (small) {
            // |S| <= 2^25, Q <= 2^40: C <= 1024 16-bit values
            int32_t S = 0;
            uint64_t Q = 0;
#pragma unroll
            for (int i = 0; i < CPL; ++i) {
                const int32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
                for (int u = 0; u < 4; u += EB / 2) {
                    const int32_t lo = EB == 2 ? (w[u] << 16) >> 16 : w[u], hi = EB == 2 ? w[u] >> 16 : w[(u + 1) & 3];
                    S += lo + hi;
                    Q += (uint32_t)(lo * lo) + (uint32_t)(hi * hi);  // <= 2^31
                }
            }
#pragma unroll
            for (int o = LPR / 2; o; o >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, o, LPR);
                Q += __shfl_xor_sync(0xffffffffu, Q, o, LPR);
            }
            const int32_t num = 2 * S + C;  // mu = floor((2S + C) / (2C)): a float quotient, at most 1 off
            int32_t m32 = __float2int_rd(__int2float_rn(num) * lc.inv2c);
            const int32_t r = num - 2 * C * m32;
            m32 += r < 0 ? -1 : (r >= 2 * C ? 1 : 0);
            const uint64_t V = Q - (uint64_t)((int64_t)m32 * (2 * S - C * m32));
            bool direct = V >= lc.lo && V <= lc.hi;
            if (direct) {
                uint32_t rem;
                const uint32_t s = isqrt_u48(V, rem);
                direct = rem != 2 * s;
                mu = m32;
                F = div_int31_u24(s);
                fits = true;
            }
            if (!direct) {
                const LnRow lr = ln_row_general(S, (int64_t)Q, C, p.iters, 1, 0);
                mu = lr.mu, F = lr.F, fits = lr.fits;
            }
        } else {
            int64_t S = 0, Q = 0;
            if constexpr (EB == 4) {
#pragma unroll
                for (int i = 0; i < CPL; ++i) {
                    const int32_t e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        madw(S, e[u], 1);
                        madw(Q, e[u], e[u]);
                    }
                }
            }
#pragma unroll
            for (int o = LPR / 2; o; o >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, o, LPR);
                Q += __shfl_xor_sync(0xffffffffu, Q, o, LPR);
            }
            const LnRow lr = ln_row_general(S, Q, C, p.iters, lc.lo, lc.hi);
            mu = lr.mu, F = lr.F, fits = lr.fits;
        }
        const int nc = chunks();
        TOut *yr = (TOut *)p.Y + row * p.ldy + sub * EPC;
        // one chunk's values (4 of them at u4)
        auto values = [&](int i, int u4, int32_t (&x)[4]) {
            const int32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                x[u] = EB == 4 ? w[u] : ((u & 1) ? w[(u4 + u) / 2] >> 16 : (w[(u4 + u) / 2] << 16) >> 16);
        };
        if (cols_fast && __all_sync(0xffffffffu, fits)) {
            const int32_t F32 = (int32_t)F, mF = (int32_t)(0u - (uint32_t)mu * (uint32_t)F);
#pragma unroll
            for (int i = 0; i < CPL; ++i) {
                if (!FULL && LPR * i >= C / EPC) break;
                const int c0 = (sub + LPR * i) * EPC;
#pragma unroll
                for (int u4 = 0; u4 < EPC; u4 += 4) {
                    int32_t x[4], o[4];
                    values(i, u4, x);
                    const int4 b4 = *(const int4 *)(s_beta + c0 + u4), m4 = *(const int4 *)(s_mult + c0 + u4);
                    const int32_t be[4] = {b4.x, b4.y, b4.z, b4.w}, mm[4] = {m4.x, m4.y, m4.z, m4.w};
                    // (x - mu) F = x F + mF in wrapping 32-bit arithmetic (the product fits int32)
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[u] = ((int32_t)((uint32_t)x[u] * (uint32_t)F32 + (uint32_t)mF) >> 1) + be[u];
                    if (cols_same) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) o[u] = rq_hi(o[u], mm[u], rnd, sh);
                    } else {
                        const int4 s4 = *(const int4 *)(s_shift + c0 + u4);
                        const int32_t ss[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u) o[u] = rq_hi1(o[u], mm[u], ss[u] - 33);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[u] = __viaddmin_s32_relu(o[u], LnBias<TOut>::one, 2 * LnBias<TOut>::one);
                    if (FULL ? nc > 0 : LPR * i < nc) {
                        ln_store4_biased<TOut>(yr + LPR * i * EPC + u4, o);
                        if constexpr (SECOND) {
#pragma unroll
                            for (int u = 0; u < 4; ++u) o[u] -= LnBias<TOut>::one;
                            ln_second4(p, row, c0 + u4, o);
                        }
                    }
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < CPL; ++i) {
                if (LPR * i >= nc) break;
                const int c0 = (sub + LPR * i) * EPC;
#pragma unroll
                for (int u4 = 0; u4 < EPC; u4 += 4) {
                    int32_t x[4], be[4], mm[4], ss[4], o[4];
                    values(i, u4, x);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        be[u] = s_beta[c0 + u4 + u];
                        mm[u] = s_mult[c0 + u4 + u];
                        ss[u] = s_shift[c0 + u4 + u];
                    }
                    ln_norm4_exact(x, mu, F, be, mm, ss, LnOut<TOut>::bits, o);
                    ln_store4<TOut>(yr + LPR * i * EPC + u4, o);
                    if constexpr (SECOND) ln_second4(p, row, c0 + u4, o);
                }
            }
        }
    }
}

template <typename TIn, typename TOut, int EPL>
__global__ void __launch_bounds__(256) layernorm_kernel(const LnParams p) {
    grid_wait();
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= p.rows) return;
    const TIn *x = (const TIn *)p.X + row * p.ldx;
    const int C = p.C;
    int32_t v[EPL];
    int64_t s = 0;
#pragma unroll
    for (int j = 0; j < EPL; ++j) {
        int c = lane + 32 * j;
        v[j] = c < C ? (int32_t)x[c] : 0;
        s += v[j];
    }
    s = warp_sum_i64(s);
    // mu = floor((2 sum + C) / (2C))
    const int64_t num = 2 * s + C, den = 2 * (int64_t)C;
    int64_t mu = num / den;
    if ((num % den) != 0 && num < 0) mu -= 1;
    uint64_t V = 0;
#pragma unroll
    for (int j = 0; j < EPL; ++j) {
        int c = lane + 32 * j;
        if (c < C) {
            int64_t y = (int64_t)v[j] - mu;
            V += (uint64_t)(y * y);
        }
    }
    V = warp_sum_u64(V);
    // Newton integer square root from 2^16, `iters` steps (stops at 0 only if V = 0)
    const uint64_t r = newton_isqrt_early(V, p.iters);
    const int64_t F = (int64_t)(0x7fffffffull / r);
    TOut *yo = (TOut *)p.Y + row * p.ldy;
#pragma unroll
    for (int j = 0; j < EPL; ++j) {
        int c = lane + 32 * j;
        if (c < C) {
            int64_t y = (int64_t)v[j] - mu;
            int64_t n = (y * F) >> 1;
            int64_t o = rq(n + p.beta[c], p.mult[c], p.shift[c]);
            const int32_t v = LnOut<TOut>::bits == 8 ? sat8(o) : sat16(o);
            if constexpr (sizeof(TOut) == 2 && LnOut<TOut>::bits == 8) yo[c] = __int2half_rn(v);
            else yo[c] = (TOut)v;
        }
    }
}

// The V for which `iters` Newton steps from 2^16 end at isqrt(V) (or its alternation): from above, the
// integer iteration never exceeds the real one r <- (r + V / r) / 2, so once the latter is within 1 of
// sqrt(V) the former is at isqrt(V) or one above, and one more step settles it.  More steps are needed the
// farther sqrt(V) lies from 2^16 on either side.  (Half of the 1 is left to the rounding of the doubles.)
struct LnRange {
    uint64_t lo, hi;
};
LnRange ln_range(int iters) {
    auto settled = [&](double x) {
        double r = 65536.0;
        for (int j = 1; j < iters; ++j) r = (r + x * x / r) / 2;
        return r - x < 0.5;
    };
    if (iters < 2) return {1, 0};
    double a = 1.0, b = 65536.0;  // the smallest root in reach: settled(b) holds
    if (!settled(a)) {
        for (int i = 0; i < 40; ++i) (settled((a + b) / 2) ? b : a) = (a + b) / 2;
        a = b;
    }
    const double lo = a + 1.0;
    double c = 65536.0, d = 16777215.0;  // the largest
    if (!settled(d)) {
        for (int i = 0; i < 40; ++i) (settled((c + d) / 2) ? c : d) = (c + d) / 2;
        d = c;
    }
    const double hi = d - 1.0;
    return {(uint64_t)(lo * lo), (uint64_t)(hi * hi)};
}
// The range depends on the step count alone (0 .. 64), and its search is two bisections over a chain of
// divisions: once per step count for the process.  (256 rows of 192, 10 steps: 14.5 us of host time a call with
// the search in each, 10.3 without.)
constexpr int kLnMaxIters = 64;
LnConst ln_const(int iters, int C) {
    static std::once_flag once[kLnMaxIters + 1];
    static LnRange range[kLnMaxIters + 1];
    std::call_once(once[iters], [&] { range[iters] = ln_range(iters); });
    return {range[iters].lo, range[iters].hi, 1.0f / (2.0f * (float)C)};
}

template <typename TIn, typename TOut>
cudaError_t ln_dispatch(const LnParams &p, cudaStream_t s, bool &second) {
    const int eb = sizeof(TIn), ob = sizeof(TOut);
    const bool tiled = p.C % 4 == 0 && (p.C * eb) % 16 == 0 && (p.ldx * eb) % 16 == 0 && p.ldy % 4 == 0 &&
                       ((uintptr_t)p.X % 16) == 0 && ((uintptr_t)p.Y % (4 * ob)) == 0 &&
                       (((uintptr_t)p.beta | (uintptr_t)p.mult | (uintptr_t)p.shift) % 16) == 0 && p.C * eb <= 2048;
    if (tiled) {
        const LnConst lc = ln_const(p.iters, p.C);
        const int nch = p.C * eb / 16;
        auto go = [&](auto kern, int lpr, int cpl) -> cudaError_t {
            const size_t smem = (size_t)3 * lpr * cpl * (16 / eb) * sizeof(int32_t);
            int dev = 0, sms = 0, per_sm = 0;
            cudaError_t e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem);
            if (e != cudaSuccess) return e;
            // persistent CTAs of 8 warps, each step of a CTA covering 256 / LPR rows
            const int64_t rpc = 256 / lpr;
            const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)std::max(per_sm, 1) * sms,
                                                                        (p.rows + rpc - 1) / rpc));
            launch_after(kern, (unsigned)grid, 256, smem, s, p, lc);
            return cudaGetLastError();
        };
        // chunks per lane: 6 for int16 rows (8 values each), 12 for int32 rows (4 values each), so a
        // lane holds at most 48 values; lanes per row from the row's chunk count
        constexpr int CPL = sizeof(TIn) == 2 ? 6 : 12;
        // Few int16 rows, a CTA or less per SM: a call is one row's chain, so twice the lanes take half the
        // chunks each.
        // (1600 rows of 192, 25 CTAs of them: 12 such layers 292 and 284 us; a decoder layer of 1200 rows of 256
        // 102.4 and 98.7 us.)
        const bool few = sizeof(TIn) == 2 && p.rows <= (int64_t)sm_count() * (nch <= 4 * CPL ? 64 : 32);
        if constexpr (sizeof(TIn) == 2 && sizeof(TOut) == 2) {
            if (few && !p.Y2) {
                if (nch == 24) return go(layernorm_rows<TIn, TOut, 8, 3, true>, 8, 3);
                if (nch == 48) return go(layernorm_rows<TIn, TOut, 16, 3, true>, 16, 3);
                if (nch <= 48) return go(layernorm_rows<TIn, TOut, 16, 3, false>, 16, 3);
            }
        }
        if constexpr (sizeof(TIn) == 2 && sizeof(TOut) == 2 && LnOut<TOut>::bits == 16) {
            if (p.Y2 && p.ldy2 % 4 == 0 && ((uintptr_t)p.Y2 % 4) == 0 && p.ldz % 4 == 0 && ((uintptr_t)p.Z % 8) == 0 && nch <= 16 * CPL) {
                second = true;
                if (few && nch <= 48) return go(layernorm_rows<TIn, TOut, 16, 3, false, true>, 16, 3);
                if (nch <= 8 * CPL) return go(layernorm_rows<TIn, TOut, 8, CPL, false, true>, 8, CPL);
                return go(layernorm_rows<TIn, TOut, 16, CPL, false, true>, 16, CPL);
            }
        }
        // (rows of 192 and 384 fill their lanes and need no test of a chunk against the row's end)
        if (nch == 4 * CPL) return go(layernorm_rows<TIn, TOut, 4, CPL, true>, 4, CPL);
        if (nch == 8 * CPL) return go(layernorm_rows<TIn, TOut, 8, CPL, true>, 8, CPL);
        if (nch <= 4 * CPL) return go(layernorm_rows<TIn, TOut, 4, CPL, false>, 4, CPL);
        if (nch <= 8 * CPL) return go(layernorm_rows<TIn, TOut, 8, CPL, false>, 8, CPL);
        if (nch <= 16 * CPL) return go(layernorm_rows<TIn, TOut, 16, CPL, false>, 16, CPL);
        if (nch <= 32 * CPL) return go(layernorm_rows<TIn, TOut, 32, CPL, false>, 32, CPL);
    }
    const int rows_per_block = 8;
    dim3 grid((unsigned)((p.rows + rows_per_block - 1) / rows_per_block));
    if (p.C <= 128) launch_after(layernorm_kernel<TIn, TOut, 4>, grid, 256, 0, s, p);
    else if (p.C <= 256) launch_after(layernorm_kernel<TIn, TOut, 8>, grid, 256, 0, s, p);
    else if (p.C <= 384) launch_after(layernorm_kernel<TIn, TOut, 12>, grid, 256, 0, s, p);
    else if (p.C <= 512) launch_after(layernorm_kernel<TIn, TOut, 16>, grid, 256, 0, s, p);
    else if (p.C <= 1024) launch_after(layernorm_kernel<TIn, TOut, 32>, grid, 256, 0, s, p);
    else if (p.C <= 2048) launch_after(layernorm_kernel<TIn, TOut, 64>, grid, 256, 0, s, p);
    else launch_after(layernorm_kernel<TIn, TOut, 128>, grid, 256, 0, s, p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_shiftmax_rows(const int32_t *X, int64_t ldx, int64_t rows, int32_t len,
                                 const ShiftmaxC &c, uint8_t *P, int64_t ldp, cudaStream_t s) {
    if (rows == 0 || len == 0) return cudaSuccess;
    dim3 grid((unsigned)((rows + 7) / 8));
    dim3 grid2((unsigned)((rows + 15) / 16));
    bool vec = (len % 4 == 0) && (ldx % 4 == 0) && (ldp % 4 == 0) && (((uintptr_t)X & 15) == 0) &&
               (((uintptr_t)P & 3) == 0);
    const bool fq = c.se.m32 != 0;
    // rows per CTA: 8 warps x (32 / LANES) rows
    auto g = [&](int lanes) { return dim3((unsigned)((rows + 8 * (32 / lanes) - 1) / (8 * (32 / lanes)))); };
    const bool s4 = ((int64_t)c.se.I0 << c.se.k) < ((int64_t)1 << 30);
#define ILW_SMX(NCH, LANES)                                                                                         \
    (fq ? (s4 ? (launch_after(shiftmax_rows_vec<NCH, LANES, true, true>, g(LANES), 256, 0, s, X, ldx, rows, len, c, P, ldp), 0)  \
              : (launch_after(shiftmax_rows_vec<NCH, LANES, true, false>, g(LANES), 256, 0, s, X, ldx, rows, len, c, P, ldp), 0)) \
        : (s4 ? (launch_after(shiftmax_rows_vec<NCH, LANES, false, true>, g(LANES), 256, 0, s, X, ldx, rows, len, c, P, ldp), 0) \
              : (launch_after(shiftmax_rows_vec<NCH, LANES, false, false>, g(LANES), 256, 0, s, X, ldx, rows, len, c, P, ldp), 0)))
    if (vec && len <= 64) ILW_SMX(4, 4);
    else if (vec && len <= 128) ILW_SMX(4, 8);
    else if (vec && len <= 416) ILW_SMX(13, 8);
    else if (vec && len <= 1024) ILW_SMX(8, 32);
    else if (vec && len <= 1664) ILW_SMX(13, 32);
    else if (vec && len <= 2048) ILW_SMX(16, 32);
#undef ILW_SMX
    else launch_after(shiftmax_rows_generic, grid, 256, 0, s, X, ldx, rows, len, c, P, ldp);
    return cudaGetLastError();
}

cudaError_t launch_sdshiftgelu(const int32_t *X, int32_t *Y, int64_t n, const GeluC &c, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int64_t n4 = 0;
    // the clamp threshold of both ShiftExp inputs: |x| >= ((k I0 + 1)/1.4375 + 3)/1.6875 (< T)
    const double bound = 0.7 * ((double)c.se.kI0 + 1.0) + 8.0;
    if ((((uintptr_t)X | (uintptr_t)Y) & 15) == 0) {
        n4 = n / 4;
        if (n4 && bound <= 32767.0 && n4 >= (1 << 16)) {
            const int32_t T = (int32_t)bound;
            const int smem = 2 * T + 1;
            static SmemLimit limit;
            const cudaError_t e = raise_smem_limit(limit, (const void *)sdshiftgelu_table, 65536);
            if (e != cudaSuccess) return e;
            int64_t blocks = (n4 + 255) / 256;
            if (blocks > 6 * (int64_t)sm_count()) blocks = 6 * (int64_t)sm_count();
            launch_after(sdshiftgelu_table, (unsigned)blocks, 256, smem, s, (const int4 *)X, (int4 *)Y, n4, c, T);
        } else if (n4) {
            int64_t blocks = (n4 + 255) / 256;
            if (blocks > 16 * (int64_t)sm_count()) blocks = 16 * (int64_t)sm_count();
            launch_after(sdshiftgelu_vec, (unsigned)blocks, 256, 0, s, (const int4 *)X, (int4 *)Y, n4, c);
        }
    }
    int64_t start = n4 * 4;
    if (start < n) launch_after(sdshiftgelu_tail, (unsigned)((n - start + 255) / 256), 256, 0, s, X, Y, start, n, c);
    return cudaGetLastError();
}

cudaError_t launch_layernorm(const LnParams &p, cudaStream_t s) {
    if (p.rows == 0) return cudaSuccess;
    bool second = false;  // the launch wrote the second result
    if (p.out_bits == kOutI8InF16)
        return p.in_bits == 16 ? ln_dispatch<int16_t, __half>(p, s, second) : ln_dispatch<int32_t, __half>(p, s, second);
    if (p.in_bits == 16 && p.out_bits == 8) return ln_dispatch<int16_t, int8_t>(p, s, second);
    if (p.in_bits == 32 && p.out_bits == 8) return ln_dispatch<int32_t, int8_t>(p, s, second);
    if (p.in_bits == 32) return ln_dispatch<int32_t, int16_t>(p, s, second);
    const cudaError_t e = ln_dispatch<int16_t, int16_t>(p, s, second);
    if (e != cudaSuccess || !p.Y2 || second) return e;
    RequantParams q{p.Y, 16, p.ldy, p.rows, p.C, p.m1, p.s1, p.Z, p.ldz, p.rows, p.m2, p.s2, 8, p.Y2, p.ldy2};
    return launch_requant(q, s);
}

}  // namespace ilw
