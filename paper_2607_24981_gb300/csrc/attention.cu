// attention.cu -- fused integer attention: scores = q k^T, Constrained Shiftmax (Algorithm 2),
// O = P V, requantisation (Sec. 3.2.1, 3.3.2).
//
// ShiftExp floors its input, so the online rescaling of flash attention is not exact: the row
// maximum must be known before any exponential.  Each CTA therefore streams the keys of its
// attention group three times (they stay in L2): pass 1 takes the exact row max, pass 2 sums
// ShiftExp (int64), which fixes s_d and F, pass 3 forms P (u8) and accumulates P V.
//
// Tensor cores: the int8 q, k, v and the u8 P are carried exactly in fp16 and multiplied with the
// warp-level fp16 MMA (m16n8k16, fp32 accumulation).  Every score |q.k| <= 64 * 127^2 < 2^20 and
// every partial sum of P V (|.| <= 255 * 127 * (sum of P <= 2^8)) is an integer below 2^24, so the
// fp32 accumulation is exact.  (On this GPU the fp16 warp MMA is about 3.8x faster than the int8
// one.)  Q, K, V are read from HBM as int8 and converted while staged into shared memory; the
// score fragments of pass 3 are already laid out as the A operand of P V.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstdlib>

#include "ilw_kernels.h"

namespace ilw {
namespace {

constexpr int QT = 64;   // query rows per CTA (4 warps x 16)
constexpr int KB = 64;   // keys per block
constexpr int THREADS = 128;

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// D = A B + C with a separate C fragment: starts an accumulation from C without initialising D.
// C is a fragment kept for the whole pass ({0,0,0,0} or {c0, c0, c1, c1} for rows g, g + 8).
__device__ __forceinline__ void mma_f16_init(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1,
                                             const float (&c)[4]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

// 16-byte asynchronous global -> shared copy; src_bytes 0 writes zeros (rows past the group)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// two int8 (low bytes of w >> 0 and w >> 8) -> fp16x2, exact: 0x6400 | (b ^ 0x80) is 1152 + b
__device__ __forceinline__ uint32_t i8x2_to_h2(uint32_t w) {
    uint32_t x = __byte_perm(w ^ 0x8080u, 0x64646464u, 0x4140);
    __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&x), __half2half2(__ushort_as_half((unsigned short)0x6480)));
    return *reinterpret_cast<uint32_t *>(&h);
}
// 16 int8 -> 16 fp16 (two uint4)
__device__ __forceinline__ void i8x16_to_h16(const uint4 v, uint4 &lo, uint4 &hi) {
    lo.x = i8x2_to_h2(v.x);
    lo.y = i8x2_to_h2(v.x >> 16);
    lo.z = i8x2_to_h2(v.y);
    lo.w = i8x2_to_h2(v.y >> 16);
    hi.x = i8x2_to_h2(v.z);
    hi.y = i8x2_to_h2(v.z >> 16);
    hi.z = i8x2_to_h2(v.w);
    hi.w = i8x2_to_h2(v.w >> 16);
}
// two integers in [0, 1024) -> fp16x2, exact: 0x6400 | p is 1024 + p
__device__ __forceinline__ uint32_t u10x2_to_h2(uint32_t p0, uint32_t p1) {
    uint32_t x = (0x6400u | p0) | ((0x6400u | p1) << 16);
    __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&x), __half2half2(__ushort_as_half((unsigned short)0x6400)));
    return *reinterpret_cast<uint32_t *>(&h);
}

// Logical right shift whose amount saturates at 32 (PTX shr clamps the shift amount to the
// register width, so any amount >= 32 gives 0).
__device__ __forceinline__ uint32_t shr_sat(uint32_t v, uint32_t n) {
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

// Constrained Shiftmax output straight from ShiftExp's parts.  With e = I_b 2^(k-q) and
// sh = 31 - k_out + 1 + s_d >= k, floor(e F / 2^sh) = floor(I_b F / 2^(sh - k + q)) exactly, and
// I_b F < 2^32 when s_d is chosen per row and m_p <= M_hw - 15 (then F <= 2^(32 + m_p - M_hw), or
// S_R >= I0 2^k when s_d = 0); the host selects this form (DIRECT) only under those conditions.
// b: bits of the fp32 value (max + 2^23) - s, as for shift_exp_bits.
template <bool FASTQ>
__device__ __forceinline__ uint32_t smx_out_direct(uint32_t b, const ShiftExpC &c, uint32_t F, uint32_t sh0) {
    uint32_t n = b + ((b + 1u) >> 1) - ((b + 15u) >> 4) - 1808793600u;
    n = min(n, (uint32_t)c.kI0);
    const uint32_t q = FASTQ ? __umulhi(n, c.m32) : (__umulhi(n, c.m_lo) + n * c.m_hi) >> 8;
    const uint32_t Ib = ((q + 2u) * (uint32_t)c.I0 - n) >> 1;
    return shr_sat(Ib * F, sh0 + q);
}

struct Group {
    int64_t base;  // b * T
    int32_t Tg;
    int32_t nw, ws, gs, wy, wx;
    __device__ __forceinline__ int64_t token(int32_t t) const {
        if (nw <= 1) return base + t;
        return base + (int64_t)(wy * ws + t / ws) * gs + wx * ws + t % ws;
    }
};

// QF16: q, k, v arrive as fp16 (the int8 values, exact) and are copied to shared memory as they
// are; otherwise they arrive as int8 and are converted on the way in.
template <int DH, bool FASTQ, bool QF16, bool DIRECT>
__global__ void __launch_bounds__(THREADS, 4) attn_kernel(const AttnParams p) {
    grid_wait();
    constexpr int LDH = DH * 2 + 16;  // padded fp16 row (bytes): conflict-free ldmatrix
    constexpr int KS = DH / 16;       // k16 steps of q k^T
    constexpr int NT = DH / 8;        // n-tiles of P V
    constexpr int CH = DH / 16;       // 16-byte int8 chunks per row
    constexpr int PER = KB * CH / THREADS;  // 16-byte int8 chunks per thread per key block
    __shared__ __align__(16) uint8_t Ks[2][KB * LDH];
    __shared__ __align__(16) uint8_t Vs[2][KB * LDH];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int h = blockIdx.y;
    Group gr;
    {
        const int G2 = p.nw * p.nw;
        const int z = blockIdx.z;
        const int b = z / G2, w = z % G2;
        gr.base = (int64_t)b * p.T;
        gr.nw = p.nw;
        gr.gs = p.grid_side;
        gr.ws = p.nw > 1 ? p.grid_side / p.nw : 0;
        gr.wy = w / p.nw;
        gr.wx = w % p.nw;
        gr.Tg = p.nw > 1 ? gr.ws * gr.ws : p.T;
    }
    const int Tg = gr.Tg;
    const int q0 = blockIdx.x * QT;
    const int hoff = h * DH;

    // ---- Q rows of this warp -> fp16 A fragments (rows g and g + 8 of the warp's 16)
    uint32_t qa[KS][4];
    if constexpr (QF16) {
        const int r0 = q0 + warp * 16 + g, r1 = r0 + 8;
        const __half *Q0 = r0 < Tg ? (const __half *)p.Q + gr.token(r0) * p.ld_qkv + hoff : nullptr;
        const __half *Q1 = r1 < Tg ? (const __half *)p.Q + gr.token(r1) * p.ld_qkv + hoff : nullptr;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            const int c = ks * 16 + 2 * t;
            qa[ks][0] = Q0 ? *(const uint32_t *)(Q0 + c) : 0u;
            qa[ks][1] = Q1 ? *(const uint32_t *)(Q1 + c) : 0u;
            qa[ks][2] = Q0 ? *(const uint32_t *)(Q0 + c + 8) : 0u;
            qa[ks][3] = Q1 ? *(const uint32_t *)(Q1 + c + 8) : 0u;
        }
    } else {
        const int r0 = q0 + warp * 16 + g, r1 = r0 + 8;
        const int8_t *Q0 = r0 < Tg ? (const int8_t *)p.Q + gr.token(r0) * p.ld_qkv + hoff : nullptr;
        const int8_t *Q1 = r1 < Tg ? (const int8_t *)p.Q + gr.token(r1) * p.ld_qkv + hoff : nullptr;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            const int c = ks * 16 + 2 * t;
            uint32_t w00 = Q0 ? *(const uint16_t *)(Q0 + c) : 0u, w01 = Q0 ? *(const uint16_t *)(Q0 + c + 8) : 0u;
            uint32_t w10 = Q1 ? *(const uint16_t *)(Q1 + c) : 0u, w11 = Q1 ? *(const uint16_t *)(Q1 + c + 8) : 0u;
            qa[ks][0] = i8x2_to_h2(w00);
            qa[ks][1] = i8x2_to_h2(w10);
            qa[ks][2] = i8x2_to_h2(w01);
            qa[ks][3] = i8x2_to_h2(w11);
        }
    }

    // q is negated (exact in fp16), so that the MMAs produce C - s: with C = 0 the row maximum is
    // minus the minimum of pass 1, and with C = max + 2^23 passes 2 and 3 get (max + 2^23) - s directly.
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int i = 0; i < 4; ++i) qa[ks][i] ^= 0x80008000u;

    const int nkb = (Tg + KB - 1) / KB;
    // Key blocks go global (int8) -> registers -> shared (fp16), double buffered: the loads of
    // block kb+1 are in flight while block kb is computed.
    uint4 kreg[PER], vreg[PER];
    auto fetch = [&](int kb, bool with_v) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = tid + i * THREADS;
            const int r = c / CH, ch = c % CH;
            const int key = kb * KB + r;
            kreg[i] = make_uint4(0, 0, 0, 0);
            vreg[i] = make_uint4(0, 0, 0, 0);
            if (key < Tg) {
                const int64_t off = gr.token(key) * p.ld_qkv + hoff + ch * 16;
                kreg[i] = __ldg((const uint4 *)((const int8_t *)p.K + off));
                if (with_v) vreg[i] = __ldg((const uint4 *)((const int8_t *)p.V + off));
            }
        }
    };
    auto commit = [&](int buf, bool with_v) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int c = tid + i * THREADS;
            const int r = c / CH, ch = c % CH;
            uint4 lo, hi;
            i8x16_to_h16(kreg[i], lo, hi);
            *(uint4 *)(Ks[buf] + r * LDH + ch * 32) = lo;
            *(uint4 *)(Ks[buf] + r * LDH + ch * 32 + 16) = hi;
            if (with_v) {
                i8x16_to_h16(vreg[i], lo, hi);
                *(uint4 *)(Vs[buf] + r * LDH + ch * 32) = lo;
                *(uint4 *)(Vs[buf] + r * LDH + ch * 32 + 16) = hi;
            }
        }
    };
    // C - s for this warp's 16 rows x keys 32hf .. 32hf + 31 of buffer `buf` (C from the fragment cq;
    // exact integers in fp32, below 2^24 in magnitude).  A key block is processed in two halves to
    // keep the score fragments at 16 registers.
    auto scores = [&](int buf, int hf, float (&S)[4][4], const float (&cq)[4]) {
        const uint32_t ks_base = (uint32_t)__cvta_generic_to_shared(Ks[buf]) + (uint32_t)(32 * hf * LDH);
#pragma unroll
        for (int np = 0; np < 2; ++np) {      // pairs of n-tiles (16 keys)
#pragma unroll
            for (int kp = 0; kp < KS; kp += 2) {  // pairs of k16 steps (32 dims)
                // matrices: keys [16np + 8(i&1) ...], dims [16kp + 8(i>>1) ...]
                const int i = lane >> 3;
                const uint32_t row = 16 * np + 8 * (i & 1) + (lane & 7);
                const uint32_t addr = ks_base + row * LDH + (16 * kp + 8 * (i >> 1)) * 2;
                uint32_t r0, r1, r2, r3;
                ldsm_x4(addr, r0, r1, r2, r3);  // r0: n-tile 2np, k lo; r1: 2np+1, k lo; r2, r3: k hi
                if (kp == 0) {
                    mma_f16_init(S[2 * np], qa[kp], r0, r2, cq);
                    mma_f16_init(S[2 * np + 1], qa[kp], r1, r3, cq);
                } else {
                    mma_f16(S[2 * np], qa[kp], r0, r2);
                    mma_f16(S[2 * np + 1], qa[kp], r1, r3);
                }
                if (kp + 1 < KS) {
                    ldsm_x4(addr + 16 * 2, r0, r1, r2, r3);  // next k16 step: 16 dims further
                    mma_f16(S[2 * np], qa[kp + 1], r0, r2);
                    mma_f16(S[2 * np + 1], qa[kp + 1], r1, r3);
                }
            }
        }
    };
    // fp16 input: 16-byte asynchronous copies straight into the padded rows
    constexpr int CH16 = DH * 2 / 16;             // 16-byte chunks per fp16 row
    constexpr int PER16 = KB * CH16 / THREADS;    // chunks per thread per key block
    auto issue16 = [&](int kb, int buf, bool with_v) {
#pragma unroll
        for (int i = 0; i < PER16; ++i) {
            const int c = tid + i * THREADS;
            const int r = c / CH16, ch = c % CH16;
            const int key = kb * KB + r;
            const bool ok = key < Tg;
            const int64_t off = gr.token(ok ? key : 0) * p.ld_qkv + hoff + ch * 8;  // elements
            cp_async16((uint32_t)__cvta_generic_to_shared(Ks[buf] + r * LDH + ch * 16), (const __half *)p.K + off,
                       ok ? 16u : 0u);
            if (with_v)
                cp_async16((uint32_t)__cvta_generic_to_shared(Vs[buf] + r * LDH + ch * 16), (const __half *)p.V + off,
                           ok ? 16u : 0u);
        }
        cp_async_commit();
    };
    // A warp whose 16 query rows all lie past the group (the short last tile of a window) only
    // helps stage the key blocks.
    const bool rows_live = q0 + warp * 16 < Tg;
    // One pass over the key blocks: body(kb, buf, full) with block kb staged in buffer buf.  While
    // the last block of a pass is computed, the first block of the next pass (with or without V:
    // next_v) is staged, so only the very first block of the CTA is waited for unhidden.
    bool prestaged = false;
    int pre_buf = 0;
    auto sweep = [&](bool with_v, bool has_next, bool next_v, auto &&body) {
        int b0 = 0;
        if (prestaged) {
            b0 = pre_buf;
        } else {
            if constexpr (QF16) {
                issue16(0, 0, with_v);
                cp_async_wait_all();
            } else {
                fetch(0, with_v);
                commit(0, with_v);
            }
            __syncthreads();
        }
        for (int kb = 0; kb < nkb; ++kb) {
            const int buf = (b0 + kb) & 1;
            const bool more = kb + 1 < nkb, stage = more || has_next;
            const int nkb_ = more ? kb + 1 : 0;
            const bool nv = more ? with_v : next_v;
            // buffer buf^1 was released by the barrier that ended the previous block
            if constexpr (QF16) {
                if (stage) issue16(nkb_, buf ^ 1, nv);
                if (rows_live) body(kb, buf, (kb + 1) * KB <= Tg);
                if (stage) cp_async_wait_all();
            } else {
                if (stage) fetch(nkb_, nv);
                if (rows_live) body(kb, buf, (kb + 1) * KB <= Tg);
                if (stage) commit(buf ^ 1, nv);
            }
            __syncthreads();
        }
        prestaged = has_next;
        pre_buf = (b0 + nkb) & 1;
    };

    // ---- pass 1: exact row maxima (the MMAs give -s; max s = -min)
    float mn0 = 3.0e38f, mn1 = 3.0e38f;
    const float cz[4] = {0.f, 0.f, 0.f, 0.f};
    sweep(false, true, false, [&](int kb, int buf, bool full) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            float S[4][4];
            scores(buf, hf, S, cz);
            if (full) {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    mn0 = fminf(mn0, fminf(S[nt][0], S[nt][1]));
                    mn1 = fminf(mn1, fminf(S[nt][2], S[nt][3]));
                }
            } else {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const int key = kb * KB + 32 * hf + nt * 8 + 2 * t;
                    if (key < Tg) { mn0 = fminf(mn0, S[nt][0]); mn1 = fminf(mn1, S[nt][2]); }
                    if (key + 1 < Tg) { mn0 = fminf(mn0, S[nt][1]); mn1 = fminf(mn1, S[nt][3]); }
                }
            }
        }
    });
    mn0 = fminf(mn0, __shfl_xor_sync(0xffffffffu, mn0, 1));
    mn0 = fminf(mn0, __shfl_xor_sync(0xffffffffu, mn0, 2));
    mn1 = fminf(mn1, __shfl_xor_sync(0xffffffffu, mn1, 1));
    mn1 = fminf(mn1, __shfl_xor_sync(0xffffffffu, mn1, 2));
    // ShiftExp(s - max) is read off the bits of (max + 2^23) - s (exact: integers below 2^23), which
    // the MMAs of passes 2 and 3 produce with C = max + 2^23
    const float mb0 = 8388608.0f - mn0, mb1 = 8388608.0f - mn1;
    const float cmb[4] = {mb0, mb0, mb1, mb1};
    const ShiftExpC se = p.smx.se;
    auto sexp = [&](float d) { return shift_exp_bits<FASTQ>(__float_as_uint(d), se); };

    // ---- pass 2: S_sum = sum ShiftExp(s - max)
    uint64_t sum0 = 0, sum1 = 0;
    sweep(false, true, true, [&](int kb, int buf, bool full) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            float S[4][4];
            scores(buf, hf, S, cmb);
            if (full) {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    sum0 += (uint64_t)sexp(S[nt][0]) + sexp(S[nt][1]);
                    sum1 += (uint64_t)sexp(S[nt][2]) + sexp(S[nt][3]);
                }
            } else {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const int key = kb * KB + 32 * hf + nt * 8 + 2 * t;
                    const bool v0 = key < Tg, v1 = key + 1 < Tg;
                    sum0 += (uint64_t)(v0 ? sexp(S[nt][0]) : 0u) + (v1 ? sexp(S[nt][1]) : 0u);
                    sum1 += (uint64_t)(v0 ? sexp(S[nt][2]) : 0u) + (v1 ? sexp(S[nt][3]) : 0u);
                }
            }
        }
    });
    sum0 += __shfl_xor_sync(0xffffffffu, sum0, 1);
    sum0 += __shfl_xor_sync(0xffffffffu, sum0, 2);
    sum1 += __shfl_xor_sync(0xffffffffu, sum1, 1);
    sum1 += __shfl_xor_sync(0xffffffffu, sum1, 2);
    // rows past Tg see sum >= 1 too (their max is over valid keys); their outputs are not stored
    const RowNorm rn0 = shiftmax_norm(sum0 ? sum0 : 1, p.smx.s_d, p.smx.m_p, p.smx.M_hw, p.smx.k_out);
    const RowNorm rn1 = shiftmax_norm(sum1 ? sum1 : 1, p.smx.s_d, p.smx.m_p, p.smx.M_hw, p.smx.k_out);
    const uint32_t sh00 = (uint32_t)(rn0.sh - se.k), sh01 = (uint32_t)(rn1.sh - se.k);  // >= 8

    // ---- pass 3: P = (I_exp F) >> sh (exact integers < 256), O += P V
    float o[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
    sweep(true, false, false, [&](int kb, int buf, bool full) {
        // P of one score: (I_exp F) >> sh, or its direct form from ShiftExp's parts
        auto pout0 = [&](float d) { return DIRECT ? smx_out_direct<FASTQ>(__float_as_uint(d), se, rn0.F, sh00)
                                                  : shiftmax_out(sexp(d), rn0); };
        auto pout1 = [&](float d) { return DIRECT ? smx_out_direct<FASTQ>(__float_as_uint(d), se, rn1.F, sh01)
                                                  : shiftmax_out(sexp(d), rn1); };
        const uint32_t vs_base = (uint32_t)__cvta_generic_to_shared(Vs[buf]);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            float S[4][4];
            scores(buf, hf, S, cmb);
            uint32_t pa[2][4];  // A fragments of P for the half's 2 k16 steps (16 keys each)
            // n-tile nt covers keys 8nt..8nt+7 of the half = half (nt & 1) of k16 step nt >> 1
            if (full) {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    pa[nt >> 1][(nt & 1) * 2 + 0] = u10x2_to_h2(pout0(S[nt][0]), pout0(S[nt][1]));  // row g
                    pa[nt >> 1][(nt & 1) * 2 + 1] = u10x2_to_h2(pout1(S[nt][2]), pout1(S[nt][3]));  // row g + 8
                }
            } else {
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const int key = kb * KB + 32 * hf + nt * 8 + 2 * t;
                    const bool v0 = key < Tg, v1 = key + 1 < Tg;
                    const uint32_t p0 = v0 ? pout0(S[nt][0]) : 0u;
                    const uint32_t p1 = v1 ? pout0(S[nt][1]) : 0u;
                    const uint32_t p2 = v0 ? pout1(S[nt][2]) : 0u;
                    const uint32_t p3 = v1 ? pout1(S[nt][3]) : 0u;
                    pa[nt >> 1][(nt & 1) * 2 + 0] = u10x2_to_h2(p0, p1);
                    pa[nt >> 1][(nt & 1) * 2 + 1] = u10x2_to_h2(p2, p3);
                }
            }
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
                // A fragment order for m16n8k16: {row g k lo, row g+8 k lo, row g k hi, row g+8 k hi}
                const uint32_t a[4] = {pa[kk][0], pa[kk][1], pa[kk][2], pa[kk][3]};
#pragma unroll
                for (int np = 0; np < NT / 2; ++np) {
                    // V rows = keys 32hf + 16kk.., cols = dims 16np..: transposed 8x8 matrices give B fragments
                    const int i = lane >> 3;
                    const uint32_t row = 32 * hf + 16 * kk + 8 * (i & 1) + (lane & 7);
                    const uint32_t addr = vs_base + row * LDH + (16 * np + 8 * (i >> 1)) * 2;
                    uint32_t r0, r1, r2, r3;
                    ldsm_x4_t(addr, r0, r1, r2, r3);  // r0: k lo, n 16np..; r1: k hi, n 16np..; r2/r3: n 16np+8..
                    mma_f16(o[2 * np], a, r0, r1);
                    mma_f16(o[2 * np + 1], a, r2, r3);
                }
            }
        }
    });

    // ---- epilogue: sat8(rq(O; m_o, s_o)), written back at the tokens' own positions
    const int r0 = q0 + warp * 16 + g, r1 = r0 + 8;
    const bool ok0 = r0 < Tg, ok1 = r1 < Tg;
    const int esz = p.o_f16 ? 2 : 1;
    uint8_t *O0 = ok0 ? (uint8_t *)p.O + (gr.token(r0) * p.ld_o + hoff) * esz : nullptr;
    uint8_t *O1 = ok1 ? (uint8_t *)p.O + (gr.token(r1) * p.ld_o + hoff) * esz : nullptr;
    // two outputs -> int8 pair (16 bits), or the same integers as an fp16 pair: the fp16 bits of
    // 1152 + v are 0x6480 + v (|v| <= 127), and one half2 subtract of 1152 leaves v exactly
    const __half2 k1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
    auto put = [&](uint8_t *dst, int col, int32_t a, int32_t b) {
        if (p.o_f16) {
            uint32_t x = (uint32_t)(0x6480 + a) | ((uint32_t)(0x6480 + b) << 16);
            __half2 h2 = __hsub2(*reinterpret_cast<__half2 *>(&x), k1152);
            *(uint32_t *)(dst + 2 * col) = *reinterpret_cast<uint32_t *>(&h2);
        } else {
            *(uint16_t *)(dst + col) = (uint16_t)((uint8_t)a | ((uint32_t)(uint8_t)b << 8));
        }
    };
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int col = nt * 8 + 2 * t;
        if (ok0)
            put(O0, col, sat8(rq(__float2int_rn(o[nt][0]), p.m_o, p.s_o)), sat8(rq(__float2int_rn(o[nt][1]), p.m_o, p.s_o)));
        if (ok1)
            put(O1, col, sat8(rq(__float2int_rn(o[nt][2]), p.m_o, p.s_o)), sat8(rq(__float2int_rn(o[nt][3]), p.m_o, p.s_o)));
    }
}

}  // namespace

// The tensor-memory kernel is used where it applies unless ILWDETR_ATTENTION_TC=0 is set in the
// environment (read once per process), which selects the warp-MMA kernel for every problem.
static bool attention_tc_enabled() {
    static const bool on = [] {
        const char *v = getenv("ILWDETR_ATTENTION_TC");
        return !(v && v[0] == '0');
    }();
    return on;
}

// The clocks of the other kernels, for the choice of the resident one.  All three were timed by graph replays on
// 1 to 2400 (image, head) units of 1 to 3584 keys, 544 points; with these figures 16 of them take a kernel more than
// 1.5 % slower than the fastest, 7 % at most.  (Before, groups of one key tile went to the resident kernel: 2400 units of
// 64 keys, int8, 64 columns, 79 us against 45, 32 columns 76 against 29; and fp16 with 64 columns to the streaming one:
// 77 us against 42, and 200 keys 336 against 175.)
// Warp-MMA kernel, up to 256 keys: its key tiles of 64 in a CTA alone, or the CTAs of an SM one after another, of which
// the first four overlap.  A last tile that is not whole costs extra.  (In us, int8: a CTA alone 3.5, 6.4 and 9.1 with 1,
// 2 and 3 tiles of 64 columns, 2.1, 4.0 and 5.8 of 32; one of many 2.6, 4.2, 6.4 and 1.7, 3.1, 4.2.)
static int64_t mma_clocks(const AttnParams &p, int Tg, int64_t units) {
    if (Tg > 256) return INT64_MAX;
    const int64_t kt = (Tg + 63) / 64, n = (units * kt + sm_count() - 1) / sm_count();
    const bool ragged = Tg % 64 != 0;
    const int64_t alone = (p.dh == 32 ? 600 + 3700 * kt : 1500 + 5700 * kt) + (ragged ? 3000 : 0);
    const int64_t many = n * ((p.dh == 32 ? 800 + 2600 * kt : 1700 + 3600 * kt) + (ragged ? 600 : 0));
    return std::max(alone, n > 2 && n <= 4 ? many * 7 / 8 : many);
}
// Streaming kernel: waves of two CTAs of 128 queries per SM; a last wave of one per SM takes 3 / 5 of a whole one.  (1600
// keys 99 us a wave, 2300 119 to 122, 3584 165, 400 29.)
static int64_t tc_clocks(const AttnParams &p, int Tg, int64_t units) {
    if (!p.qkv_f16 || p.dh != 64) return INT64_MAX;
    const int64_t sms = sm_count(), jobs = units * ((Tg + 127) / 128), wave = 15000 + 100 * (int64_t)Tg;
    const int64_t last = jobs % (2 * sms);
    return jobs / (2 * sms) * wave + (last == 0 ? 0 : (last <= sms ? wave * 3 / 5 : wave));
}
static int64_t other_clocks(const AttnParams &p) {
    const int G2 = p.nw > 1 ? p.nw * p.nw : 1;
    const int Tg = p.nw > 1 ? (p.grid_side / p.nw) * (p.grid_side / p.nw) : p.T;
    const int64_t units = (int64_t)p.B * p.H * G2;
    return std::min(mma_clocks(p, Tg, units), tc_clocks(p, Tg, units));
}

cudaError_t attention_resident_ctas(const AttnParams &p, int *ctas) {
    *ctas = 0;
    if (!attention_tc_enabled()) return cudaSuccess;
    const cudaError_t e = launch_attention_res(p, nullptr, other_clocks(p), ctas);
    return e == cudaErrorNotSupported ? cudaSuccess : e;
}

cudaError_t launch_attention(const AttnParams &p0, cudaStream_t s) {
    AttnParams p = p0;
    p.status = status_word_ptr();
    const int G2 = p.nw > 1 ? p.nw * p.nw : 1;
    const int Tg = p.nw > 1 ? (p.grid_side / p.nw) * (p.grid_side / p.nw) : p.T;
    if (p.B == 0 || Tg == 0) return cudaSuccess;
    if (attention_tc_enabled()) {
        cudaError_t e = launch_attention_res(p, s, other_clocks(p));
        // (of one key tile the warp-MMA kernel is the faster)
        if (e == cudaErrorNotSupported && (Tg > 64 || p.smx.s_d >= 0)) e = launch_attention_tc(p, s);
        if (e != cudaErrorNotSupported) return e;
    }
    dim3 grid((Tg + QT - 1) / QT, p.H, p.B * G2);
    const bool fastq = p.smx.se.m32 != 0;
    // the direct output form needs per-row s_d and I_b F < 2^32 (m_p <= M_hw - 15), and sh >= k
    const bool direct = p.smx.s_d < 0 && p.smx.m_p + 15 <= p.smx.M_hw && 32 - p.smx.k_out >= p.smx.se.k;
#define ILW_ATTN(DH, QF)                                                                          \
    do {                                                                                          \
        if (fastq && direct) launch_after(attn_kernel<DH, true, QF, true>, grid, THREADS, 0, s, p);         \
        else if (fastq) launch_after(attn_kernel<DH, true, QF, false>, grid, THREADS, 0, s, p);             \
        else if (direct) launch_after(attn_kernel<DH, false, QF, true>, grid, THREADS, 0, s, p);            \
        else launch_after(attn_kernel<DH, false, QF, false>, grid, THREADS, 0, s, p);                       \
    } while (0)
    if (p.qkv_f16) {
        if (p.dh == 64) ILW_ATTN(64, true);
        else ILW_ATTN(32, true);
    } else {
        if (p.dh == 64) ILW_ATTN(64, false);
        else ILW_ATTN(32, false);
    }
#undef ILW_ATTN
    return cudaGetLastError();
}

}  // namespace ilw
