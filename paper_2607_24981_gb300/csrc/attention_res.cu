// attention_res.cu -- fused integer attention whose scores stay in tensor memory: S = q k^T once
// (tcgen05, fp32 accumulators in TMEM), Constrained Shiftmax (Algorithm 2) on the scores where they
// are, O = P V with P read from TMEM as the MMA's A operand, requantisation (Sec. 3.2.1, 3.3.2).
//
// What bounds it: the integer arithmetic per score.  ShiftExp floors its input, so the row maximum
// must be known before any exponential and the row sum before any output; a kernel that streams the
// keys (attention_tc.cu) computes every score three times and every ShiftExp twice.  Here a CTA, or a
// thread-block cluster that shares the keys, holds one attention group's whole score tile in tensor
// memory, at most 128 x 448 per CTA: scores are computed once, ShiftExp runs once per score and its
// value replaces the score, and P replaces that.  The CTAs of a cluster exchange the row maxima, the row
// sums and the partial O through distributed shared memory; all three are exact integers, so the split
// changes nothing in the result.  The K and V rows stay in shared memory for
// all query tiles of a (image, window, head) that the cluster works through.
//
// One CTA = 18 warps, the whole tensor memory of its SM:
//   warps 0-15  softmax: warp w works on TMEM lanes 32 (w % 4) .. + 31 (one query row per thread) and on
//               quarter w / 4 of the CTA's key columns, 16 at a time (five to seven warps per scheduler
//               were 3 to 10 % slower: the arithmetic units, not the waits, set the pace)
//   warp 16     TMEM allocation; MMA issuer: S (4 K steps of 128 x nkp), then O += P V (one MMA
//               128 x 64 x 16 per 16 keys, A in TMEM, v as an N-major operand) as the P of two units of
//               every warp is there; the next job's S while the softmax warps read O
//   warp 17     TMA producer (one thread): the K and V rows of a new unit, the Q tile of every job, ahead
//               of their use (fp16-carried q|k|v with 64-column heads; otherwise the softmax warps load
//               them at the start of a job with plain 16-byte loads, int8 widened to fp16 and 32-column
//               heads to 64: zero columns add nothing)
// One CTA per SM with all 448 columns is faster than two with 208 each (windows of 400 keys, 8 images x
// 6 heads: 58 against 67 us), although those overlap one's waits with the other's arithmetic: a job's
// fixed work (exchanges, normalisation, output) is per CTA.
//
// Measured (8 images x 6 heads x 1600 tokens, dh 64, graph replays): global attention 201 -> 155 us,
// windows of 400 keys 99 -> 51 us; one image x 3 heads: 88 -> 25 and 27 -> 14 us.
// A job is one 128-row query tile of one unit; a cluster takes a contiguous range of the job list
// (units in order, their tiles in order), so K and V are reloaded only when the unit changes.
//
// ShiftExp runs in fp32 on integers, two scores per instruction (shift_exp16): fused multiply-adds
// rounded down take the floors.  Measured on this GPU, per scheduler and score with the row sum and the
// TMEM traffic: 8.2 cycles, against 10.7 for the integer form attention_tc.cu uses (its quotient needs
// a multiply-high, 32 lanes per clock and SM against 128 for packed fp32).
//
// Every mbarrier wait is bounded (about one second); on expiry the kernel latches the device status
// word, every role stops, loads and MMAs in flight are waited for, and all CTAs of the cluster meet at
// the cluster barrier before any exits.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "attn_ptx.cuh"
#include "ilw_kernels.h"

namespace ilw {
namespace {

constexpr int RQ = 128;          // rows of a query tile (MMA M)
constexpr int kResTmem = 512;    // TMEM columns: scores, and O in the last 64
constexpr int kOCol = 448;
constexpr int kMaxKeys = kOCol;  // keys per CTA
constexpr int kCq = 4;           // softmax warps per row
constexpr int kMmaWarp = 4 * kCq, kLoadWarp = kMmaWarp + 1;
constexpr int kResThreads = 32 * (kLoadWarp + 1);

struct ResSmem {
    // from the 1024-aligned base: Q tile, then K and V (nkp rows of 128 bytes each), the O exchange
    // buffer (int16 partial sums), the row exchange buffers, the barriers
    static constexpr int kQ = 0;
    static constexpr int kK = RQ * 128;
    // the row exchange buffers; each has its own space, as the lane quarters work at their own pace
    int v, obuf, rmax, rsum, pmax, psum, fmax, fnorm, bar, bytes;
    __host__ __device__ ResSmem(int nkp, int cs) {
        v = kK + nkp * 128;
        obuf = v + nkp * 128;
        rmax = obuf + (cs > 1 ? RQ * 128 : 0);  // the cluster's row maxima and sums, one per CTA
        rsum = rmax + cs * RQ * 4;
        pmax = rsum + cs * RQ * 8;               // the partial maxima and sums of warps 1 .. of a row
        psum = pmax + (kCq - 1) * RQ * 4;
        fmax = psum + (kCq - 1) * RQ * 8;        // a row's maximum and (F, shift), for the warps of the row
        fnorm = fmax + RQ * 4;
        bar = fnorm + RQ * 8;
        bytes = bar + 8 * 36 + 16;
    }
};
// barrier numbers (from B_PART on: one per lane quarter).  B_PFULL + i: P of units 2 i and 2 i + 1 of every
// softmax warp
constexpr int kStages = ((kMaxKeys / 16 + kCq - 1) / kCq + 1) / 2;
enum { B_QFULL = 0, B_QFREE, B_KFULL, B_KFREE, B_VFULL, B_VFREE, B_SFULL, B_OFREE, B_OFULL, B_DRAIN, B_PFULL,
       B_PART = 16, B_XMAX = 20, B_XSUM = 24, B_ROW = 28, B_XO = 32, B_SLOT = 36 };
static_assert(B_PFULL + kStages <= B_PART, "barriers");

struct ResArgs {
    CUtensorMap qmap, kmap, vmap;  // fp16 q, k, v: 2-D {64 H, B T} or (windows) 3-D {64 H, gs, B gs}; 128-byte swizzle
    AttnParams p;
    int32_t kpc;    // keys per CTA: a multiple of 16 tokens, or rpc whole window rows
    int32_t kbox;   // keys per TMA box (global attention): kpc, or half of it above 256
    int32_t nkp;    // kpc rounded up to 16: rows of K and V in shared memory, score columns
    int32_t rpc;    // window rows per CTA (windows)
    int32_t rqt;    // tokens per query tile: 128, or rqw whole window rows
    int32_t rqw;
    int32_t nq;     // query tiles per unit
    int32_t jobs;   // units x nq
    int32_t tma;    // 1: TMA loads
    int32_t ovec;   // 1: O rows take vector stores
    float rcp;      // 1 / I0 rounded up
    uint32_t ws_rcp;
};

constexpr float kMag = 12582912.0f;  // 1.5 2^23: one unit of the last place is 1 up to 2^24
constexpr float kMag1 = 8388608.0f;  // 2^23

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// Two floats in one 64-bit register: packed arithmetic, one instruction per pair.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 fma2_rd(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 fma2_ru(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// ShiftExp's parameters as floats (integers below 2^24, but for rcp)
struct ExpF {
    float rcp, negI0, kI0, magI0;  // 1 / I0 rounded up, -I0, k I0, 2^23 + I0
};
// ShiftExp(s - max) 2^(16 - k) of N scores in place: Ib 2^(16 - q), whatever k >= q is.  The scores are
// integer-valued floats; with x = s - max and a = -x in [0, 2^21] every step is exact or a floor taken by
// the rounding mode:
//   n = ceil(3a/2) - ceil(a/16) = a + ceil(a/2) - ceil(a/16) = -(I + (I >> 1) - (I >> 4)) for I = -a, at most k I0
//   q = floor(n / I0): n rcp lies above n / I0 by less than n 2^-23 / I0 <= 2^-19 < 1 / I0, and 2^23 + n rcp
//     rounded down has q in its low mantissa bits
//   h = 2^23 + I0 + floor(-r / 2) with r = n - q I0: Ib in its low mantissa bits (Ib <= I0 < 2^15)
// The shift by 16 drops h's exponent bits, and the shift by f takes its low five bits, q <= 16.
// Written stage by stage, so that the N / 2 independent pairs overlap.
template <int N>
__device__ __forceinline__ void shift_exp16(uint32_t (&s)[N], float mx, const ExpF &c) {
    f32x2 v[N / 2], m[N / 2];
#pragma unroll
    for (int i = 0; i < N / 2; ++i) v[i] = add2(pk(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), pk(-mx, -mx));
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        m[i] = fma2_ru(v[i], pk(-1.5f, -1.5f), pk(kMag, kMag));
        v[i] = fma2_rd(v[i], pk(0.0625f, 0.0625f), pk(-kMag, -kMag));
    }
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        float x, y;
        upk(add2(m[i], v[i]), x, y);
        v[i] = pk(fminf(x, c.kI0), fminf(y, c.kI0));
    }
#pragma unroll
    for (int i = 0; i < N / 2; ++i) m[i] = fma2_rd(v[i], pk(c.rcp, c.rcp), pk(kMag1, kMag1));
#pragma unroll
    for (int i = 0; i < N / 2; ++i) v[i] = fma2(add2(m[i], pk(-kMag1, -kMag1)), pk(c.negI0, c.negI0), v[i]);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        float x, y, f, g;
        upk(fma2_rd(v[i], pk(-0.5f, -0.5f), pk(c.magI0, c.magI0)), x, y);
        upk(m[i], f, g);
        s[2 * i] = (__float_as_uint(x) << 16) >> (__float_as_uint(f) & 31u);
        s[2 * i + 1] = (__float_as_uint(y) << 16) >> (__float_as_uint(g) & 31u);
    }
}

__device__ __forceinline__ void tst16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tst8(uint32_t taddr, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void twait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// D += A B with A in TMEM (fp16 pairs: column c holds K elements 2c and 2c + 1 of the lane's row), if `on`: a
// predicate on the instruction, so that every MMA of the issuer stands in the one flat branch of the elected lane.
// A branch of its own around an MMA inside that one (an earlier form of the loop) issued some MMAs with the operands
// of another step.  Why has not been shown; the operands of an MMA are read from uniform registers, which a
// branch within a one-lane branch has to fill again.  (A predicate in place of the elected lane's branch as
// well, as in the GEMM: 8 images of the Medium encoder 1958 us against 1914.)
__device__ __forceinline__ void mma_ts(uint32_t dt, uint32_t at, uint64_t b, uint32_t idesc, uint32_t acc, uint32_t on) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(dt),
        "r"(at), "l"(b), "r"(idesc), "r"(acc), "r"(on)
        : "memory");
}

// ---- thread-block cluster: remote shared memory
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Asynchronous stores to a CTA of the cluster that count their bytes at an mbarrier of the same CTA: the
// sender needs no release (which would wait for its outstanding global stores as well).
__device__ __forceinline__ void sta_b32(uint32_t a, uint32_t v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void sta_b64(uint32_t a, uint64_t v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a), "l"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void sta_v4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(a), "r"(x),
                 "r"(y), "r"(z), "r"(w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool bar_try_cl(uint32_t b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred P;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P, [%1], %2, %3;\n selp.b32 %0, 1, 0, P;\n}\n"
        : "=r"(ok)
        : "r"(b), "r"(parity), "r"(20000)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_wait_cl(uint32_t b, uint32_t parity, volatile int *abort, int *status, int code) {
    if (bar_try_cl(b, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t i = 0;; ++i) {
        if (bar_try_cl(b, parity)) return true;
        if ((i & 63) == 63) {
            if (*abort) return false;
            if (clock64() - t0 > kWaitTc) {
                if (status) atomicExch(status, code);
                *abort = 1;
                return false;
            }
        }
    }
}

// 4 int8 -> 2 words of fp16 pairs, exact (0x6400 | (b ^ 0x80) encodes 1152 + b)
__device__ __forceinline__ void widen4(uint32_t w, uint32_t &lo, uint32_t &hi) {
    const uint32_t x = w ^ 0x80808080u;
    uint32_t a = __byte_perm(x, 0x64646464u, 0x4140), b = __byte_perm(x, 0x64646464u, 0x4342);
    const __half2 k1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
    const __half2 ha = __hsub2(*reinterpret_cast<__half2 *>(&a), k1152), hb = __hsub2(*reinterpret_cast<__half2 *>(&b), k1152);
    lo = *reinterpret_cast<const uint32_t *>(&ha);
    hi = *reinterpret_cast<const uint32_t *>(&hb);
}

// An attention group's tokens: a whole image (ws = 0), or one ws x ws window of a token grid gs wide
struct ResGroup {
    int64_t base;  // the first token
    int32_t ws, gs;
    uint32_t ws_rcp;  // ceil(2^32 / ws): t / ws is one multiply-high (exact for t ws < 2^32)
    __device__ __forceinline__ int64_t token(int32_t t) const {
        if (!ws) return base + t;
        const int32_t y = (int32_t)__umulhi((uint32_t)t, ws_rcp);
        return base + (int64_t)y * gs + (t - y * ws);
    }
};

// `rows` rows of 128 bytes at dst (128-byte swizzle): columns col0 .. col0 + dh - 1 of tokens t0 ..
// t0 + valid - 1 as fp16, zeros elsewhere.  The softmax threads (tid); 16-byte loads.
template <bool I8>
__device__ __forceinline__ void load_rows(uint8_t *dst, const void *src, int64_t ld, int col0, int dh, int rows, int valid,
                                          int t0, const ResGroup &g, int tid) {
    constexpr int CPR = I8 ? 4 : 8, CPC = I8 ? 16 : 8;  // 16-byte source chunks per row, columns per chunk
#pragma unroll 4
    for (int it = tid; it < rows * CPR; it += 128 * kCq) {
        const int r = it / CPR, c = it % CPR;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < valid && c * CPC < dh)
            v = __ldg((const uint4 *)((const char *)src + (g.token(t0 + r) * ld + col0 + c * CPC) * (I8 ? 1 : 2)));
        uint8_t *row = dst + r * 128;
        if constexpr (I8) {
            uint4 lo, hi;
            widen4(v.x, lo.x, lo.y);
            widen4(v.y, lo.z, lo.w);
            widen4(v.z, hi.x, hi.y);
            widen4(v.w, hi.z, hi.w);
            *(uint4 *)(row + (((2 * c) ^ (r & 7)) << 4)) = lo;
            *(uint4 *)(row + (((2 * c + 1) ^ (r & 7)) << 4)) = hi;
        } else {
            *(uint4 *)(row + ((c ^ (r & 7)) << 4)) = v;
        }
    }
}

template <int CS>
__global__ void __launch_bounds__(kResThreads, 1) attn_res_kernel(const __grid_constant__ ResArgs args) {
    const AttnParams &p = args.p;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = su32(sm);
    const ResSmem L(args.nkp, CS);
    auto bar = [&](int i) { return sbase + (uint32_t)L.bar + 8u * (uint32_t)i; };
    uint32_t *tmem_slot = (uint32_t *)(sm + L.bar + 8 * B_SLOT);
    volatile int *abort = (volatile int *)(sm + L.bar + 8 * B_SLOT + 4);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = CS > 1 ? cluster_rank() : 0u;
    const int clusters = (int)gridDim.x / CS, cl = (int)blockIdx.x / CS;
    const int j0 = (int)((int64_t)cl * args.jobs / clusters), j1 = (int)((int64_t)(cl + 1) * args.jobs / clusters);
    const int nkp = args.nkp, G2 = p.nw * p.nw;
    const int ws = p.nw > 1 ? p.grid_side / p.nw : 0;
    const int Tg = p.nw > 1 ? ws * ws : p.T;
    const int nkv = min(args.kpc, Tg - (int)rank * args.kpc);  // this CTA's keys
    auto group = [&](int unit) {
        const int z = unit / p.H;
        const int w = z % G2;
        return ResGroup{(int64_t)(z / G2) * p.T + (int64_t)(w / p.nw) * ws * p.grid_side + (w % p.nw) * ws, ws, p.grid_side, args.ws_rcp};
    };

    if (threadIdx.x == 0) {
        const uint32_t nl = args.tma ? 1u : 4u * kCq;
        bar_init(bar(B_QFULL), nl);
        bar_init(bar(B_KFULL), nl);
        bar_init(bar(B_VFULL), nl);
        bar_init(bar(B_QFREE), 1);
        bar_init(bar(B_KFREE), 1);
        bar_init(bar(B_VFREE), 1);
        bar_init(bar(B_SFULL), 1);
        bar_init(bar(B_OFREE), 4 * kCq);
        for (int i = 0; i < kStages; ++i) bar_init(bar(B_PFULL + i), 4 * kCq);
        bar_init(bar(B_OFULL), 1);
        bar_init(bar(B_DRAIN), 1);
        for (int q = 0; q < 4; ++q) {
            bar_init(bar(B_PART + q), kCq - 1);
            bar_init(bar(B_ROW + q), 1);
            // one arrival (CS > 1: with the bytes expected from the cluster)
            bar_init(bar(B_XMAX + q), 1);
            bar_init(bar(B_XSUM + q), 1);
            bar_init(bar(B_XO + q), 1);
        }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (args.tma) {  // rows that no box writes: finite values for the MMAs (their scores and outputs are not used)
        const int kz = (nkp - args.kpc) * 8, qz = (RQ - args.rqt) * 8;
        for (int i = threadIdx.x; i < kz; i += kResThreads) {
            *(uint4 *)(sm + ResSmem::kK + args.kpc * 128 + i * 16) = make_uint4(0, 0, 0, 0);
            *(uint4 *)(sm + L.v + args.kpc * 128 + i * 16) = make_uint4(0, 0, 0, 0);
        }
        for (int i = threadIdx.x; i < qz; i += kResThreads)
            *(uint4 *)(sm + ResSmem::kQ + args.rqt * 128 + i * 16) = make_uint4(0, 0, 0, 0);
        fence_async_smem();
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)), "n"(kResTmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    grid_wait();
    fence_before();
    __syncthreads();
    fence_after();
    if constexpr (CS > 1) cluster_sync();  // every CTA's barriers exist before any remote arrive
    const uint32_t tmem = *tmem_slot;
    // the score columns: units of 16, split over the kCq softmax warps of a lane quarter (warp c: units
    // ubeg(c) .. ubeg(c + 1) - 1).  A warp's P takes half of its own columns: 8 per unit from its first
    // column on, written in order, so that every column is read before it is overwritten
    const int units = nkp >> 4, stages = ((units + kCq - 1) / kCq + 1) / 2;
    auto ubeg = [&](int c) { return c * (units / kCq) + min(c, units % kCq); };


    if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer
        const bool issue = elect_one();
        auto wait = [&](int b, uint32_t parity, int code) -> bool {
            return __all_sync(0xffffffffu, bar_wait(bar(b), parity, abort, p.status, code));
        };
        const uint32_t id_s = (1u << 4) | ((128u >> 4) << 24);
        const uint32_t id_o = (1u << 4) | (1u << 16) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t dq = desc_sw128(sbase + ResSmem::kQ), dk = desc_sw128(sbase + ResSmem::kK), dv = desc_sw128(sbase + L.v);
        int qt = j0 % args.nq;
        uint32_t ph = 0, kph = 1;  // phases: per job, per unit
        for (int j = j0; j < j1; ++j, ph ^= 1u) {
            const bool fresh = j == j0 || qt == 0, last = j + 1 == j1 || qt + 1 == args.nq;
            qt = qt + 1 == args.nq ? 0 : qt + 1;
            if (fresh) {
                kph ^= 1u;
                if (!wait(B_KFULL, kph, kStatusTimeoutTma)) break;
            }
            if (!wait(B_QFULL, ph, kStatusTimeoutTma)) break;
            // the score columns are free once the previous job's P V has completed
            if (j > j0 && !wait(B_OFULL, ph ^ 1u, kStatusTimeoutMma)) break;
            fence_after();
            // up to 256 keys per MMA
#pragma unroll 1
            for (int c = (nkp - 1) & ~255; c >= 0; c -= 256) {
                const uint32_t id = id_s | ((uint32_t)(min(nkp - c, 256) >> 3) << 17);
                const uint64_t dkc = dk + (uint64_t)(8 * c);
                if (issue) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) mma(tmem + (uint32_t)c, dq + 2 * t, dkc + 2 * t, id, t ? 1u : 0u);
                }
                __syncwarp();
            }
            if (issue) {
                commit(bar(B_SFULL));
                commit(bar(B_QFREE));
                if (last) commit(bar(B_KFREE));
            }
            __syncwarp();
            if (fresh && !wait(B_VFULL, kph, kStatusTimeoutTma)) break;
            // O is free once every softmax warp has read the previous job's
            bool ok = wait(B_OFREE, ph ^ 1u, kStatusTimeoutOperand);
            for (int st = 0; st < stages && ok; ++st) {
                ok = wait(B_PFULL + st, ph, kStatusTimeoutOperand);
                if (!ok) break;
                fence_after();
#pragma unroll 1
                for (int c = 0; c < kCq; ++c) {
                    const int ub = ubeg(c), u = ub + 2 * st, n = ubeg(c + 1) - u;  // this warp's units left: two of them now
                    const uint32_t pc = tmem + (uint32_t)(8 * (u + ub));
                    const uint64_t vd = dv + (uint64_t)(128 * u);
                    if (issue) {
                        mma_ts(tmem + kOCol, pc, vd, id_o, (st | c) ? 1u : 0u, n > 0 ? 1u : 0u);
                        mma_ts(tmem + kOCol, pc + 8u, vd + 128u, id_o, 1u, n > 1 ? 1u : 0u);
                    }
                    __syncwarp();
                }
            }
            if (!ok) break;
            if (issue) {
                commit(bar(B_OFULL));
                if (last) commit(bar(B_VFREE));
            }
            __syncwarp();
        }
        // every MMA issued has completed before the TMEM is released
        if (issue) commit(bar(B_DRAIN));
        const long long t0 = clock64();
        while (!bar_try(bar(B_DRAIN), 0) && clock64() - t0 < kWaitTc) {
        }
        __syncwarp();
    } else if (warp == kLoadWarp) {
        if (args.tma && lane == 0) {
            // -------------------------------------------------------------- TMA producer
            int unit = -1;
            uint32_t ph = 0, kph = 1;
            int nk = 0, nv = 0, nqi = 0;  // loads issued per barrier
            const uint32_t kb = (uint32_t)args.kpc * 128u, qb = (uint32_t)args.rqt * 128u;
            const bool win = p.nw > 1;
            for (int j = j0; j < j1; ++j, ph ^= 1u) {
                const bool fresh = j / args.nq != unit;
                unit = j / args.nq;
                const ResGroup g = group(unit);
                const int head = unit % p.H, qt = j - unit * args.nq;
                // windows: the first token's place in the grid of all images' token rows
                const int wx = win ? (int)(g.base % g.gs) : 0, wy = win ? (int)(g.base / g.gs) : 0;
                if (fresh) {
                    kph ^= 1u;
                    if (!bar_wait(bar(B_KFREE), kph ^ 1u, abort, p.status, kStatusTimeoutFree)) break;
                    bar_expect_tx(bar(B_KFULL), kb);
                    if (win) tma_3d(sbase + ResSmem::kK, &args.kmap, head * 64, wx, wy + (int)rank * args.rpc, bar(B_KFULL));
                    else
                        for (int b = 0; b < args.kpc; b += args.kbox)
                            tma_2d(sbase + ResSmem::kK + 128u * b, &args.kmap, head * 64, (int)g.base + (int)rank * args.kpc + b, bar(B_KFULL));
                    ++nk;
                }
                if (!bar_wait(bar(B_QFREE), ph ^ 1u, abort, p.status, kStatusTimeoutFree)) break;
                bar_expect_tx(bar(B_QFULL), qb);
                if (win) tma_3d(sbase + ResSmem::kQ, &args.qmap, head * 64, wx, wy + qt * args.rqw, bar(B_QFULL));
                else tma_2d(sbase + ResSmem::kQ, &args.qmap, head * 64, (int)g.base + qt * RQ, bar(B_QFULL));
                ++nqi;
                if (fresh) {
                    if (!bar_wait(bar(B_VFREE), kph ^ 1u, abort, p.status, kStatusTimeoutFree)) break;
                    bar_expect_tx(bar(B_VFULL), kb);
                    if (win) tma_3d(sbase + L.v, &args.vmap, head * 64, wx, wy + (int)rank * args.rpc, bar(B_VFULL));
                    else
                        for (int b = 0; b < args.kpc; b += args.kbox)
                            tma_2d(sbase + L.v + 128u * b, &args.vmap, head * 64, (int)g.base + (int)rank * args.kpc + b, bar(B_VFULL));
                    ++nv;
                }
            }
            if (*abort) {  // the loads still in flight land before the CTA exits
                const long long t0 = clock64();
                while (clock64() - t0 < kWaitTc && ((nk && !bar_try(bar(B_KFULL), (nk - 1) & 1)) ||
                                                    (nv && !bar_try(bar(B_VFULL), (nv - 1) & 1)) ||
                                                    (nqi && !bar_try(bar(B_QFULL), (nqi - 1) & 1)))) {
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ softmax, one query row per thread
        const int qw = warp & 3, cq = warp >> 2, row = 32 * qw + lane;
        const int ub = ubeg(cq), nun = ubeg(cq + 1) - ub;                    // this warp's units
        const uint32_t tlane = tmem + ((uint32_t)(32 * qw) << 16), tcol = tlane + (uint32_t)(16 * ub);
        const int nval = min(max(nkv - 16 * ub, 0), 16 * nun);               // and valid columns
        const int nfull = nval >> 4, rem = nval & 15;
        float *rmax = (float *)(sm + L.rmax), *pmax = (float *)(sm + L.pmax), *fmx = (float *)(sm + L.fmax);
        uint64_t *rsum = (uint64_t *)(sm + L.rsum), *psum = (uint64_t *)(sm + L.psum);
        uint2 *frow = (uint2 *)(sm + L.fnorm);
        const ExpF ec{args.rcp, -(float)p.smx.se.I0, (float)p.smx.se.kI0, kMag1 + (float)p.smx.se.I0};
        const bool sum4 = p.smx.se.I0 < (1 << 14);  // four values I0 2^16 add up in 32 bits
        const int k = p.smx.se.k;
        constexpr int NC = CS > 1 ? 8 / CS : 8;  // 8-column chunks of O that belong to this CTA
        const bool owner = CS == 1 || (int)rank * NC * 8 < p.dh;
        uint32_t ph = 0, lph = 0;  // phases: per job, per job in which this quarter has rows
        bool ok = true;
        auto wait_cta = [&](int b, uint32_t parity) -> bool {
            return ok = __all_sync(0xffffffffu, bar_wait(bar(b), parity, abort, p.status, kStatusTimeoutMma));
        };
        auto wait_cl = [&](int b, uint32_t parity) -> bool {
            if constexpr (CS == 1) return ok = __all_sync(0xffffffffu, bar_wait(bar(b), parity, abort, p.status, kStatusTimeoutOperand));
            else return ok = __all_sync(0xffffffffu, bar_wait_cl(bar(b), parity, abort, p.status, kStatusTimeoutOperand));
        };
        // sat8(rq(r; m_o, s_o)) of 8 columns, at element `at` of O
        auto put = [&](int32_t (&r)[8], int64_t at) {
            if (p.s_o >= 33) {
#pragma unroll
                for (int c = 0; c < 8; ++c) r[c] = clamp8(rq_hi(r[c], p.m_o, 1 << (p.s_o - 33), p.s_o - 32));
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) r[c] = sat8(rq(r[c], p.m_o, p.s_o));
            }
            if (p.o_f16) {
                // 1152 + r (|r| <= 127) has the fp16 bits 0x6480 + r; subtracting 1152 leaves r
                const __half2 h1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
                uint32_t hw[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t x = (uint32_t)(0x6480 + r[2 * c]) | ((uint32_t)(0x6480 + r[2 * c + 1]) << 16);
                    const __half2 hh = __hsub2(*reinterpret_cast<__half2 *>(&x), h1152);
                    hw[c] = *reinterpret_cast<const uint32_t *>(&hh);
                }
                __half *dst = (__half *)p.O + at;
                if (args.ovec) {
                    *(uint4 *)dst = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) ((uint16_t *)dst)[c] = (uint16_t)(hw[c >> 1] >> (16 * (c & 1)));
                }
            } else {
                int8_t *dst = (int8_t *)p.O + at;
                if (args.ovec) {
                    uint32_t bw[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        bw[c] = (uint32_t)(uint8_t)r[4 * c] | ((uint32_t)(uint8_t)r[4 * c + 1] << 8) |
                                ((uint32_t)(uint8_t)r[4 * c + 2] << 16) | ((uint32_t)(uint8_t)r[4 * c + 3] << 24);
                    *(uint2 *)dst = make_uint2(bw[0], bw[1]);
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) dst[c] = (int8_t)r[c];
                }
            }
        };
        // CS > 1: one 8-column chunk of a job's output, once every CTA's partial sums are here
        int due = -1;  // the chunk (of this CTA's NC) whose partial sums are on their way; its phase, and its element of O (none: < 0)
        uint32_t dph = 0;
        int64_t dat = -1;
        auto finish = [&]() -> bool {
            if constexpr (CS > 1) {
                if (due < 0) return true;
                const uint8_t *ob = sm + L.obuf + due * 2048 + row * 16;
                due = -1;
                if (!wait_cl(B_XO + qw, dph)) return false;
                int32_t r[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
                for (int d = 0; d < CS; ++d) {
                    const uint4 v = *(const uint4 *)(ob + d * NC * 2048);
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        r[2 * c] += (int32_t)(w[c] << 16) >> 16;
                        r[2 * c + 1] += (int32_t)w[c] >> 16;
                    }
                }
                if (dat >= 0) put(r, dat);
            }
            return true;
        };
        int qt = j0 % args.nq, unit = j0 / args.nq, head = unit % p.H;
        ResGroup g = group(unit);
        for (int j = j0; j < j1; ++j, ph ^= 1u, ++qt) {
            if (qt == args.nq) {
                qt = 0;
                ++unit;
                head = unit % p.H;
                g = group(unit);
            }
            const int t0 = qt * args.rqt, nrow = min(args.rqt, Tg - t0);
            if (!args.tma) {  // the previous job's MMAs have completed (its O has been read): the tiles are free
                auto rows = [&](int off, const void *src, int n, int valid, int tok, int full) {
                    if (p.qkv_f16) load_rows<false>(sm + off, src, p.ld_qkv, head * p.dh, p.dh, n, valid, tok, g, threadIdx.x);
                    else load_rows<true>(sm + off, src, p.ld_qkv, head * p.dh, p.dh, n, valid, tok, g, threadIdx.x);
                    fence_async_smem();  // this warp's stores are visible to the MMAs
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(full));
                };
                const bool fresh = j == j0 || qt == 0;
                if (fresh) rows(ResSmem::kK, p.K, nkp, nkv, (int)rank * args.kpc, B_KFULL);
                rows(ResSmem::kQ, p.Q, RQ, nrow, t0, B_QFULL);
                if (fresh) rows(L.v, p.V, nkp, nkv, (int)rank * args.kpc, B_VFULL);
            }
            const bool live = 32 * qw < nrow;  // some row of this lane quarter is a query (the same in every CTA)
            if (!wait_cta(B_SFULL, ph)) break;
            fence_after();
            if (live) {
                // ---- row maximum
                float mx = -3.0e38f;
                int u = 0;
#pragma unroll 1
                for (; u + 2 <= nfull; u += 2) {
                    uint32_t s[32];
                    tld<32>(tcol + 16u * u, s);
                    twait<32>(s);
                    float m1 = mx;  // two chains
#pragma unroll
                    for (int c = 0; c < 32; c += 4) {
                        mx = max3(mx, __uint_as_float(s[c]), __uint_as_float(s[c + 1]));
                        m1 = max3(m1, __uint_as_float(s[c + 2]), __uint_as_float(s[c + 3]));
                    }
                    mx = fmaxf(mx, m1);
                }
#pragma unroll 1
                for (; 16 * u < nval; ++u) {
                    uint32_t s[16];
                    tld<16>(tcol + 16u * u, s);
                    twait<16>(s);
                    const int v = u < nfull ? 16 : rem;
#pragma unroll
                    for (int c = 0; c < 16; ++c) mx = c < v ? fmaxf(mx, __uint_as_float(s[c])) : mx;
                }
                // the warps of a row meet in the first one, which sends the row's maximum to every CTA of the
                // cluster and hands the cluster's maximum back.  (A later job's values overwrite an exchange
                // buffer only after the exchanges in between, which its readers have passed.)
                if (cq) {
                    pmax[(cq - 1) * RQ + row] = mx;
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(B_PART + qw));
                    if (!finish()) break;  // the previous job's output while the maxima travel
                    if (!wait_cta(B_ROW + qw, 0)) break;
                    mx = fmx[row];
                } else {
                    if (!wait_cta(B_PART + qw, 0)) break;
#pragma unroll
                    for (int c = 0; c < kCq - 1; ++c) mx = fmaxf(mx, pmax[c * RQ + row]);
                    if constexpr (CS > 1) {
                        if (lane == 0) bar_expect_tx(bar(B_XMAX + qw), CS * 32 * 4);
#pragma unroll
                        for (int d = 0; d < CS; ++d)
                            sta_b32(mapa(sbase + (uint32_t)L.rmax + 4u * (rank * RQ + row), (uint32_t)d), __float_as_uint(mx),
                                    mapa(bar(B_XMAX + qw), (uint32_t)d));
                        if (!wait_cl(B_XMAX + qw, lph)) break;
                        mx = rmax[row];
#pragma unroll
                        for (int d = 1; d < CS; ++d) mx = fmaxf(mx, rmax[d * RQ + row]);
                    }
                    fmx[row] = mx;
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(B_ROW + qw));
                    if (!finish()) break;
                }
                // ---- ShiftExp 2^(16 - k) of every score, kept in place of the score, and the row sum
                uint64_t sum = 0;
                auto add = [&](const uint32_t (&s)[16]) {
                    if (sum4) {
#pragma unroll
                        for (int c = 0; c < 16; c += 4) sum += (uint64_t)(s[c] + s[c + 1] + s[c + 2] + s[c + 3]);
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; c += 2) sum += (uint64_t)(s[c] + s[c + 1]);
                    }
                };
#pragma unroll 1
                for (u = 0; u < nfull; ++u) {
                    uint32_t s[16];
                    tld<16>(tcol + 16u * u, s);
                    twait<16>(s);
                    shift_exp16<16>(s, mx, ec);
                    tst16(tcol + 16u * u, s);
                    add(s);
                }
                if (rem) {
                    uint32_t s[16];
                    tld<16>(tcol + 16u * u, s);
                    twait<16>(s);
                    shift_exp16<16>(s, mx, ec);
#pragma unroll
                    for (int c = 0; c < 16; ++c) s[c] = c < rem ? s[c] : 0u;
                    tst16(tcol + 16u * u, s);
                    add(s);
                }
                // the row sum in the same way; its normalisation is worked out once and handed back:
                // P = floor(e F / 2^sh) from e 2^(16 - k)
                uint2 fs;
                if (cq) {
                    psum[(cq - 1) * RQ + row] = sum;
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(B_PART + qw));
                    twait_st();
                    if (!wait_cta(B_ROW + qw, 1)) break;
                    fs = frow[row];
                } else {
                    if (!wait_cta(B_PART + qw, 1)) break;
#pragma unroll
                    for (int c = 0; c < kCq - 1; ++c) sum += psum[c * RQ + row];
                    if constexpr (CS > 1) {
                        if (lane == 0) bar_expect_tx(bar(B_XSUM + qw), CS * 32 * 8);
#pragma unroll
                        for (int d = 0; d < CS; ++d)
                            sta_b64(mapa(sbase + (uint32_t)L.rsum + 8u * (rank * RQ + row), (uint32_t)d), sum,
                                    mapa(bar(B_XSUM + qw), (uint32_t)d));
                        if (!wait_cl(B_XSUM + qw, lph)) break;
                        sum = rsum[row];
#pragma unroll
                        for (int d = 1; d < CS; ++d) sum += rsum[d * RQ + row];
                    }
                    const RowNorm rn = shiftmax_norm(sum >> (16 - k), p.smx.s_d, p.smx.m_p, p.smx.M_hw, p.smx.k_out);
                    fs = make_uint2(rn.F, (uint32_t)(rn.sh + 16 - k));
                    frow[row] = fs;
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(B_ROW + qw));
                    twait_st();
                }
                // ---- P as fp16 operands: P < 256 is written as its own bits, the fp16 subnormal P 2^-24 (exact); O
                // accumulates 2^-24 P V, exact as well.  One high-word product: umulhi(e, F 2^(32 - sh)) for
                // sh <= 32, umulhi(e, F) >> (sh - 32) above; that word is below 2^(8 + rs), so up to rs = 8
                // two outputs share a register before the shift
                const uint32_t F = fs.x, sh = fs.y, G = sh >= 32 ? F : F << (32 - sh), rs = sh > 32 ? min(sh - 32, 31u) : 0u;
                const bool hi_row = sh >= 32 || (F >> sh) == 0u, packed = __all_sync(0xffffffffu, hi_row && rs <= 8u);
                // P of units u and u + 1 complete: their MMAs can start (a warp without these units arrives all the same)
                auto stage = [&](int st) {
                    twait_st();
                    fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar(B_PFULL + st));
                };
                u = 0;
                if (packed) {
#pragma unroll 1
                    for (; u < nfull; ++u) {
                        uint32_t s[16], w[8];
                        tld<16>(tcol + 16u * u, s);
                        twait<16>(s);
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            w[c] = (__byte_perm(__umulhi(s[2 * c], G), __umulhi(s[2 * c + 1], G), 0x5410) >> rs) & 0x00ff00ffu;
                        tst8(tcol + 8u * u, w);
                        if (u & 1) stage(u >> 1);
                    }
                }
#pragma unroll 1
                for (; u < 2 * stages; ++u) {
                    if (u < nun) {
                        uint32_t w[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) w[c] = 0u;
                        if (16 * u < nval) {
                            uint32_t s[16];
                            tld<16>(tcol + 16u * u, s);
                            twait<16>(s);
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const uint32_t p0 = hi_row ? __umulhi(s[2 * c], G) >> rs : (uint32_t)(((uint64_t)s[2 * c] * F) >> sh);
                                const uint32_t p1 = hi_row ? __umulhi(s[2 * c + 1], G) >> rs : (uint32_t)(((uint64_t)s[2 * c + 1] * F) >> sh);
                                w[c] = __byte_perm(p0, p1, 0x5410);
                            }
                            __syncwarp();  // reconverge before the warp-synchronous store
                        }
                        tst8(tcol + 8u * u, w);
                    }
                    if (u & 1) stage(u >> 1);
                }
            } else {
                __syncwarp();
                if (lane == 0)
                    for (int st = 0; st < stages; ++st) bar_arrive(bar(B_PFULL + st));
            }
            // ---- O = P V: sat8(rq(O; m_o, s_o)) at the token's own position
            if (!wait_cta(B_OFULL, ph)) break;
            fence_after();
            uint32_t o[16];  // columns 16 cq .. of the row (the row's first four warps)
            const bool has_o = live && 16 * cq < p.dh;
            if (has_o) {
                tld<16>(tlane + (uint32_t)(kOCol + 16 * cq), o);
                twait<16>(o);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(bar(B_OFREE));
            if (!live) continue;
            // |O| <= 2^8 127: 2^24 O + 1.5 2^23 holds it exactly in the low mantissa bits (two's complement)
            if (has_o)
#pragma unroll
                for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__fmaf_rn(__uint_as_float(o[c]), 16777216.0f, kMag));
            if constexpr (CS == 1) {
                if (has_o && row < nrow) {
                    const int64_t at = g.token(t0 + row) * p.ld_o + head * p.dh + 16 * cq;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        int32_t r[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) r[c] = (int32_t)(o[8 * h + c] - 0x4B400000u);
                        put(r, at + 8 * h);
                    }
                }
            } else {
                // column chunk c (8 columns) belongs to CTA c / NC of the cluster: the partial sums go there as int16
                if (has_o) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t chunk = 2u * cq + h, own = chunk / NC, lc = chunk % NC;
                        sta_v4(mapa(sbase + (uint32_t)L.obuf + (rank * NC + lc) * 2048u + 16u * row, own),
                               __byte_perm(o[8 * h], o[8 * h + 1], 0x5410), __byte_perm(o[8 * h + 2], o[8 * h + 3], 0x5410),
                               __byte_perm(o[8 * h + 4], o[8 * h + 5], 0x5410), __byte_perm(o[8 * h + 6], o[8 * h + 7], 0x5410),
                               mapa(bar(B_XO + qw), own));
                    }
                }
                if (owner) {
                    if (cq == 0 && lane == 0) bar_expect_tx(bar(B_XO + qw), 4096);  // 32 rows of this CTA's columns from every CTA
                    // the row's last NC warps take one chunk each
                    const int mine = cq - (kCq - NC);
                    if (mine >= 0) {
                        due = mine;
                        dph = lph;
                        const int col = ((int)rank * NC + mine) * 8;
                        dat = row < nrow && col < p.dh ? g.token(t0 + row) * p.ld_o + head * p.dh + col : -1;
                    }
                }
            }
            lph ^= 1u;
        }
        if (ok) finish();
    }

    fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        __syncwarp();
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kResTmem) : "memory");
    }
    // no CTA leaves while another of its cluster may still reach into its shared memory: in the normal case
    // each has waited for all that was sent to it; after an abort, stores may still be under way
    if constexpr (CS > 1) {
        __syncwarp();
        cluster_sync();
        if (*abort) {
            const long long t0 = clock64();
            while (clock64() - t0 < 100000) {
            }
        }
        __syncwarp();
        cluster_sync();
    }
}

// Tensor map over the 64 H fp16 columns at `base`: 2-D {64 H, B T} with 64 x rows boxes, or (windows)
// 3-D {64 H, gs, B gs} with 64 x ws x rows boxes; 128-byte swizzle, zero fill.
bool res_map(CUtensorMap *m, const void *base, const AttnParams &p, int ws, int rows) {
    EncodeTiledTc fn = encode_tc();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)p.ld_qkv * 2;
    const bool win = ws > 0;
    const int gs = p.grid_side;
    cuuint64_t dims[3] = {(cuuint64_t)p.H * 64, win ? (cuuint64_t)gs : (cuuint64_t)p.B * p.T, (cuuint64_t)p.B * gs};
    cuuint64_t str[2] = {row, row * (cuuint64_t)gs};
    cuuint32_t box[3] = {64, (cuuint32_t)(win ? ws : rows), (cuuint32_t)rows};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, win ? 3 : 2, const_cast<void *>(base), dims, str, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int res_smem(int nkp, int cs) { return 1024 + ResSmem(nkp, cs).bytes; }

// How a cluster of cs CTAs splits a group of Tg keys (window side ws, 0 for global attention); false
// where a CTA's share exceeds its tensor memory or a CTA would have no key.
bool res_split(int Tg, int ws, int cs, int *kpc, int *rpc) {
    if (ws) {
        *rpc = (ws + cs - 1) / cs;
        *kpc = *rpc * ws;
        return *kpc <= kMaxKeys && (cs - 1) * *rpc < ws;
    }
    *rpc = 0;
    *kpc = ((Tg + cs - 1) / cs + 15) / 16 * 16;
    return *kpc <= kMaxKeys && (cs - 1) * *kpc < Tg;
}

// Clusters of CS CTAs, one per SM, that fit the device at once (asked once per device)
template <int CS>
int active_clusters(cudaError_t *err) {
    static std::mutex mu;
    static int known[kMaxAttrDevices] = {};
    int dev = 0;
    if ((*err = cudaGetDevice(&dev)) != cudaSuccess) return 0;
    if (dev < 0 || dev >= kMaxAttrDevices) {
        *err = cudaErrorInvalidDevice;
        return 0;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (known[dev]) return known[dev];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS);
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = (size_t)res_smem(kMaxKeys, CS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int got = 0;
    if ((*err = cudaOccupancyMaxActiveClusters(&got, attn_res_kernel<CS>, &cfg)) != cudaSuccess) return 0;
    return known[dev] = got;
}

struct ResPlan {
    int cs = 0, kpc = 0, rpc = 0, clusters = 0;
    int64_t cost = 0;
};
template <int CS>
cudaError_t plan_one(int Tg, int ws, int64_t jobs, int job_cost, int key_cost, ResPlan *best) {
    int kpc, rpc;
    if (!res_split(Tg, ws, CS, &kpc, &rpc)) return cudaSuccess;
    const int nkp = (kpc + 15) / 16 * 16;
    static SmemLimit limit;
    cudaError_t e = raise_smem_limit(limit, (const void *)attn_res_kernel<CS>, res_smem(kMaxKeys, CS));
    if (e != cudaSuccess) return e;
    const int nc = active_clusters<CS>(&e);
    if (e != cudaSuccess) return e;
    if (nc < 1) return cudaSuccess;
    // clocks: rounds of jobs x those of one, a part for the exchanges and one that grows with the CTA's keys (more of
    // both where the softmax warps load the rows themselves), and a cluster's launch.  Rounds measured, in us: fp16
    // and 64 columns, one CTA, 64 keys 4.1, 192 5.3, 448 8.7; int8 5.0, 7.5, 10.3 (32 columns 4.8, 6.3); fp16 and 32
    // columns 4.8, 7.6, 10.2; fp16, 64 columns, clusters of 4 with 400 keys a CTA 8.4, of 8 with 448 9.0.  A single
    // job of 64 keys split over 4 CTAs takes 1.2 us longer than one of 48 in one CTA
    const int64_t rounds = (jobs + nc - 1) / nc;
    const int64_t one = job_cost + (CS > 1 ? 300 : 0) + key_cost * (int64_t)nkp;
    const int64_t cost = rounds * one + (CS > 1 ? 2000 : 0);
    if (!best->cs || cost < best->cost) *best = {CS, kpc, rpc, (int)std::min<int64_t>(nc, jobs), cost};
    return cudaSuccess;
}
template <int CS>
cudaError_t launch_res(const ResArgs &a, int clusters, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * CS));
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = (size_t)res_smem(a.nkp, CS);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attn_res_kernel<CS>, a);
}

}  // namespace

// The resident form: per-row s_d, which bounds sum P by 2^k_out and so |O| by 2^15 (with a static s_d
// neither is bounded), scores of at most 64 columns (|s| <= 2^20) and at most 8 x 448 keys per group;
// cudaErrorNotSupported otherwise.
cudaError_t launch_attention_res(const AttnParams &p, cudaStream_t s, int64_t below, int *plan_ctas) {
    const ShiftExpC &se = p.smx.se;
    const bool win = p.nw > 1;
    const int ws = win ? p.grid_side / p.nw : 0, G2 = win ? p.nw * p.nw : 1;
    const int Tg = win ? ws * ws : p.T;
    if (p.smx.s_d >= 0 || se.k > 16 || se.I0 >= (1 << 15) || p.dh > 64 || (win && (ws > RQ || ws * p.nw != p.grid_side)))
        return cudaErrorNotSupported;
    ResArgs a;
    a.p = p;
    a.rqw = win ? std::min(RQ / ws, ws) : 0;
    a.rqt = win ? a.rqw * ws : RQ;
    a.nq = (Tg + a.rqt - 1) / a.rqt;
    const int64_t jobs = (int64_t)p.B * G2 * p.H * a.nq;
    if (jobs > INT32_MAX || (int64_t)p.B * p.T > INT32_MAX) return cudaErrorNotSupported;
    a.jobs = (int32_t)jobs;
    ResPlan plan;
    cudaError_t e;
    a.tma = p.qkv_f16 && p.dh == 64;
    const int jc = a.tma ? 6500 : (p.qkv_f16 ? 8200 : 7800), kc = a.tma ? 24 : (p.qkv_f16 ? 34 : 27);
    if ((e = plan_one<1>(Tg, ws, jobs, jc, kc, &plan)) != cudaSuccess || (e = plan_one<2>(Tg, ws, jobs, jc, kc, &plan)) != cudaSuccess ||
        (e = plan_one<4>(Tg, ws, jobs, jc, kc, &plan)) != cudaSuccess || (e = plan_one<8>(Tg, ws, jobs, jc, kc, &plan)) != cudaSuccess)
        return e;
    if (!plan.cs || plan.cost > below) return cudaErrorNotSupported;
    if (plan_ctas) {
        *plan_ctas = plan.cs;
        return cudaSuccess;
    }
    a.kpc = plan.kpc;
    a.rpc = plan.rpc;
    a.ws_rcp = ws > 1 ? (uint32_t)((((uint64_t)1 << 32) + ws - 1) / ws) : 0u;  // ws = 1: a window is one token
    a.kbox = a.kpc > 256 ? a.kpc / 2 : a.kpc;
    a.nkp = (a.kpc + 15) / 16 * 16;
    a.rcp = 1.0f / (float)se.I0;  // the nearest float, or the next one where that lies below 1 / I0
    if ((double)a.rcp * se.I0 < 1.0) a.rcp = std::nextafter(a.rcp, 2.0f);
    const int esz_o = p.o_f16 ? 2 : 1;
    a.ovec = (p.ld_o * esz_o) % 16 == 0 && ((uintptr_t)p.O % 16) == 0;
    if (a.tma && !(res_map(&a.qmap, p.Q, p, ws, win ? a.rqw : RQ) && res_map(&a.kmap, p.K, p, ws, win ? a.rpc : a.kbox) &&
                   res_map(&a.vmap, p.V, p, ws, win ? a.rpc : a.kbox)))
        return cudaErrorNotSupported;
    switch (plan.cs) {
        case 1: return launch_res<1>(a, plan.clusters, s);
        case 2: return launch_res<2>(a, plan.clusters, s);
        case 4: return launch_res<4>(a, plan.clusters, s);
        default: return launch_res<8>(a, plan.clusters, s);
    }
}

}  // namespace ilw
