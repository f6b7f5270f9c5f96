#pragma once
// gemm_tc.cuh -- exact integer GEMM on the 5th-generation tensor cores (tcgen05.mma, sm_103a)
// with the bias / dyadic requantisation / residual / SD-ShiftGELU / split-convolution epilogues
// fused (Sec. 3.2.1, 3.2.2, 3.3.1).
//
// Exactness.  sm_103a has no int8 tcgen05 MMA, so the int8 values are carried in fp16 (every
// integer of magnitude <= 2048 is exact in fp16) and multiplied by tcgen05.mma.kind::f16 with
// fp32 accumulation in tensor memory.  Each product |a w| <= 127^2 < 2^14 is exact, and every
// partial sum of an accumulator is an integer of magnitude <= 127^2 * 1024 < 2^24, exactly
// representable in fp32, so the accumulation is exact as long as one accumulator never sees more
// than 1024 terms of K.  Longer K is cut into segments of <= 1024, each with its own TMEM
// accumulator; the epilogue converts every segment to int32 (exact) and adds them in integers.
// Split-convolution branches are segments too, each rescaled by its own dyadic (m_b, s_b)
// before the integer sum.
//
// Persistent kernel, one CTA per SM, 128 x BN output tiles, 10 to 18 warps:
//   warp 0      TMA producer: per K stage the activation tile (int8 128 x 64 bytes, or, when A is
//               carried in fp16, the fp16 128 x 64 tile in the MMA's 128-byte swizzled layout) and
//               the fp16 weight tile (BN x 64, 128-byte swizzle); with resident weights the CTA's
//               BN rows of W are loaded once, before its first tile; TMEM allocation
//   warp 1      MMA issuer: 4 x (128 x BN x 16) MMAs per 64-wide K stage
//   warps 2-5   operand converters (int8 A only): int8 activation rows (smem) -> fp16 rows in the
//               same 128-byte swizzled K-major layout TMA produces for the weights
//   the rest    epilogue (from warp 6, or with fp16 A from warp 2): TMEM -> registers -> integer or
//               packed fp32 epilogue -> HBM, one row per thread and a part of the tile's columns per
//               warp (epi_parts)
// Two TMEM accumulator sets (when they fit) let the epilogue of tile i overlap the MMAs of tile
// i+1.  The grid is a multiple of the number of column blocks (with resident weights always, else where
// that costs no round), so every tile of a CTA has the same columns: their parameters are prepared
// once, and resident rows of W leave L2 only the activations to serve.
// Every mbarrier wait is bounded (about one second); on expiry the kernel latches the device
// status word, stops issuing work, drains the loads it issued and frees its TMEM.
#include <cuda.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "ilw_kernels.h"

namespace ilw {
// Host helpers of the tensor-core GEMM shared by its translation units (defined in gemm_tc.cu).
bool gemm_make_map(CUtensorMap *m, const void *base, CUtensorMapDataType dt, int esize, int64_t rows, int64_t cols,
                   int64_t ld, int box_cols, int box_rows, CUtensorMapSwizzle sw);
const uint8_t *gemm_gelu_table(const GeluC &c, int32_t m_g, int32_t s_g, cudaStream_t s, cudaError_t *err);
// The wait bound of the next GEMM launches and the K block whose load the producer skips (-1: none),
// as set by ilwdetr_debug_gemm_wait (defaults: about one second, none).
void gemm_debug_wait(int32_t *skip, long long *cycles);
struct GemmProblem;
struct EpiParams;
// The 64-wide launch shapes (gemm_tc_n64.cu).
template <bool AF16, bool GELU>
cudaError_t run_n64(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s);
cudaError_t run_n64_split(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s);
// The int8-A launch shapes (gemm_tc_i8.cu): run<BN, STAGES, NB, false, false, GELU>.
template <int BN, int STAGES, int NB, bool GELU>
cudaError_t run_i8(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s);
namespace {

constexpr int BM = 128, BK = 64;
constexpr int kMaxSeg = 8;
constexpr int kSegK = 1024;  // max K per accumulator for exact fp32 accumulation
constexpr int kMaxWk = kSegK / 64;  // K blocks of resident weights (one barrier each)
constexpr long long kWaitCycles = 2000000000ll;  // ~1 s at 2 GHz: the default bound of every wait

struct Seg {
    int32_t k0, klen;   // K range of this accumulator (same columns of A and W)
    int32_t map;        // index of the activation / weight tensor maps
    int32_t m_b, s_b;   // split-conv rescale of the branch partial
};

template <int NB>  // NB: tensor-map slots (1 for a plain GEMM, kMaxBranches for split convolution)
struct TcParams {  // CUtensorMap members keep the 64-byte alignment TMA needs
    CUtensorMap amap[NB];
    CUtensorMap wmap[NB];
    Seg seg[kMaxSeg];
    int32_t nseg;
    int32_t branch_rq;
    int32_t M, N;
    int32_t tiles_n, tiles;
    int32_t nbuf;       // TMEM accumulator sets (1 or 2)
    int32_t wres_bytes; // resident weight bytes (WRES), a multiple of 1024
    int32_t tmem_cols;
    int32_t tma_store;  // boxes per epilogue warp (2 or 1) of the outputs' TMA stores through shared memory; 0: plain stores
    int32_t dbg_skip;   // test hook: the producer issues no load for this K-block counter value (-1: none)
    long long wait_cycles;  // the bound of every wait (about one second, shorter for the test hook)
    CUtensorMap cmap;   // C [M, N] with 32 x 32 boxes (2-byte outputs: 64-byte swizzle, 1-byte: 32-byte)
    CUtensorMap rmap;   // the int16 residual in 32 x 32 boxes (res_tma)
    int32_t res_tma;    // 1: each epilogue warp loads its residual box by TMA and writes its results over it
    int32_t stages;     // pipeline stages in use (STAGES at most)
    const uint8_t *gelu_tab;  // SD-ShiftGELU output table in global memory (16-byte aligned, 65536 bytes)
    int *status;
    EpiParams ep;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One try_wait; the waiting thread may be suspended (up to the hint, 20 us) until the phase completes,
// so that waiting roles do not spin on the issue slots the epilogue needs.
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred P;\n mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2, %3;\n selp.b32 %0, 1, 0, P;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000)
        : "memory");
    return ok != 0;
}
// Bounded wait: true when the phase completed; false (after latching `code` in the status word
// and raising the CTA's abort flag) when it ran out, or when another role already aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort, int *status, int code,
                                          long long limit) {
    if (mbar_try(bar, parity)) return true;  // the common case, without reading the clock
    long long t0 = clock64();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255) == 255) {
            if (*abort) return false;
            if (clock64() - t0 > limit) {
                if (status) atomicExch(status, code);
                *abort = 1;
                return false;
            }
        }
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)map) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"((uint64_t)src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int32_t x, int32_t y, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"((uint64_t)map),
                 "r"(x), "r"(y), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void fence_async_smem_g() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;             // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;   // stride byte offset: next 8-row group
    d |= (uint64_t)1 << 46;             // descriptor version
    d |= (uint64_t)2 << 61;             // 128-byte swizzle
    return d;
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_lane() {
    uint32_t p;
    asm volatile("{\n .reg .pred P;\n elect.sync _|P, 0xffffffff;\n selp.b32 %0, 1, 0, P;\n}\n" : "=r"(p));
    return p != 0;
}
// One MMA / commit by the lanes with `issue` set (one of the warp): a predicate, not a branch, so that the
// operands stay in uniform registers.
__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc, uint32_t issue) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(issue)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar, uint32_t issue) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar), "r"(issue)
        : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
}
// Waits for this thread's TMEM loads and marks the 16 destination registers as written by the
// wait, so that no use of them can be scheduled before the data has arrived.
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
}

// TMEM load of 32 consecutive 32-bit columns of this thread's lane, and the matching wait (every
// destination register marked as written by the wait).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_mark32(uint32_t *v) {
    asm volatile(""
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]),
                   "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]),
                   "+r"(v[30]), "+r"(v[31])::"memory");
}
__device__ __forceinline__ void tmem_wait_only() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 4 int8 (one word) -> 2 words of fp16x2, exact: fp16 bits 0x6400 | (b ^ 0x80) encode 1152 + b.
__device__ __forceinline__ void i8x4_to_f16x4(uint32_t w, uint32_t &lo, uint32_t &hi) {
    const uint32_t x = w ^ 0x80808080u;
    uint32_t a = __byte_perm(x, 0x64646464u, 0x4140);
    uint32_t b = __byte_perm(x, 0x64646464u, 0x4342);
    const __half2 k1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
    __half2 ha = __hsub2(*reinterpret_cast<__half2 *>(&a), k1152);
    __half2 hb = __hsub2(*reinterpret_cast<__half2 *>(&b), k1152);
    lo = *reinterpret_cast<uint32_t *>(&ha);
    hi = *reinterpret_cast<uint32_t *>(&hb);
}

// Shared memory per pipeline stage: fp16 A (128 rows x 128 B, swizzled; written by the converter
// warps from the int8 staging rows, or by TMA directly when A arrives as fp16), fp16 W (BN rows x
// 128 B, swizzled by TMA; absent when the CTA's weights are resident), int8 A staging (128 rows x
// 64 B, written by TMA; absent for fp16 A).  Resident weights (WRES) keep every K block of the
// CTA's BN rows of W after the stages.
template <int BN, bool AF16 = false, bool WRES = false>
struct Smem {
    static constexpr int kA16 = BM * 128;
    static constexpr int kW = WRES ? 0 : BN * 128;
    static constexpr int kA8 = AF16 ? 0 : BM * 64;
    static constexpr int kStage = kA16 + kW + kA8;
    static constexpr int kWtile = BN * 128;  // one K block of W
};

// Epilogue parameters in shared memory: four arrays of a column part, per warp or (WRES) per part.
template <int BN, bool WRES>
constexpr int prm_words() { return (WRES ? 4 : 16) * BN; }

// Output kinds: one compact epilogue per kernel instantiation.
// F16OUT: RQ8 values as fp16; GELU_F16: GELU8 values as fp16
enum { KIND_RQ8 = 0, KIND_RQ16 = 1, KIND_RAW32 = 2, KIND_GELU8 = 3, KIND_F16OUT = 4, KIND_GELU_F16 = 5 };
constexpr bool gelu_kind(int kind) { return kind == KIND_GELU8 || kind == KIND_GELU_F16; }

// 16 consecutive int32 of shared memory (16-byte aligned) into registers: four 128-bit loads
__device__ __forceinline__ void lds16(const int32_t *p, int32_t (&o)[16]) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(o[4 * j]), "=r"(o[4 * j + 1]), "=r"(o[4 * j + 2]), "=r"(o[4 * j + 3])
                     : "r"(a + 16 * j));
}

__device__ __forceinline__ void lds8(const int32_t *p, int32_t (&o)[8]) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
#pragma unroll
    for (int j = 0; j < 2; ++j)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(o[4 * j]), "=r"(o[4 * j + 1]), "=r"(o[4 * j + 2]), "=r"(o[4 * j + 3])
                     : "r"(a + 16 * j));
}

enum { FORM_GENERAL = 0, FORM_UNI = 1, FORM_VAR = 2, FORM_FLT = 3 };
// rq(acc + bias; m, s) in 64 bits, clamped to +-2^30, which saturates the same.
__device__ __forceinline__ int32_t rq_clamped(int32_t acc, int32_t bias, int32_t m, int32_t s) {
    const int64_t t = rq((int64_t)acc + bias, m, s);
    return (int32_t)(t < -(1 << 30) ? -(1 << 30) : (t > (1 << 30) ? (1 << 30) : t));
}

// The fused epilogue of 16 consecutive columns of one row, computed stage by stage so that the
// 16 independent elements overlap.  FAST (uniform across the warp, decided per tile) says every
// shift of the warp's columns is >= 33; ss then holds s - 32 and sr 2^(s-33) (rq_hi), else ss
// holds s.  RFAST: the residual's shift s_r is in [17, 46] (2^(s_r - 17) and |x m_r| 2^-16 add up within 32
// bits).  gtab points at entry 0 of the SD-ShiftGELU output table (index -32767 .. 32767).
template <int KIND, bool FAST, bool RFAST>
__device__ __forceinline__ void epi_chunk(const EpiParams &ep, bool has_res, const uint32_t (&rp)[8],
                                          const int32_t (&acc)[16], const int32_t (&sb)[16],
                                          const int32_t (&sm)[16], const int32_t (&ss)[16],
                                          const int32_t (&sr)[16], const uint8_t *gtab, int32_t (&out)[16]) {
    if (KIND == KIND_RAW32) {
#pragma unroll
        for (int i = 0; i < 16; ++i) out[i] = acc[i] + sb[i];
        return;
    }
    int32_t r[16];
    if (FAST) {
#pragma unroll
        for (int i = 0; i < 16; ++i) r[i] = rq_hi(acc[i] + sb[i], sm[i], sr[i], ss[i]);  // |r| < 2^29
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            r[i] = rq_clamped(acc[i], sb[i], sm[i], ss[i]);
        }
    }
    if (KIND == KIND_GELU8 || KIND == KIND_GELU_F16) {
        // g = sat16(r); the table holds sat8(rq(g * I_div(g); m_g, s_g)) for every int16 g
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            out[i] = (int32_t)gtab[clamp16(r[i])] - 128;
        }
        return;
    }
    if (has_res) {
        // rp holds the 16 int16 residuals in pairs; x * 2^16 is the pair word masked or shifted
        // (RFAST: rq(x; m_r, s_r) = rq(x * 2^16; m_r, s_r + 16) with s_r + 16 >= 33; both terms are then below
        // 2^30 or saturate.  Else the sum is formed in 64 bits)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int32_t xs = (i & 1) ? (int32_t)(rp[i >> 1] & 0xFFFF0000u) : (int32_t)(rp[i >> 1] << 16);
            if (RFAST) {
                r[i] += rq_hi(xs, ep.m_r, 1 << (ep.s_r - 17), ep.s_r - 16);
            } else {
                const int64_t t = (FAST ? (int64_t)r[i] : rq((int64_t)acc[i] + sb[i], sm[i], ss[i])) +
                                  rq((int64_t)(xs >> 16), ep.m_r, ep.s_r);
                r[i] = sat16(t);  // (int8 results saturate further below)
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) out[i] = (KIND == KIND_RQ8 || KIND == KIND_F16OUT) ? max(clamp8(r[i]), ep.relu ? 0 : -127) : clamp16(r[i]);
}

// Packed fp32 pairs (two operations an instruction).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair2(uint32_t lo, uint32_t hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ float lo2(f32x2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(f32x2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
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
// max(m, |a|, |b|) in one instruction
__device__ __forceinline__ float max_abs3(float m, float a, float b) {
    asm("max.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(fabsf(a)), "f"(fabsf(b)));
    return m;
}
constexpr uint32_t kMagic = 0x4B400000u;  // 1.5 2^23: adding it to a float rounds it to an integer (ties to even)
__device__ __forceinline__ uint32_t half2_add(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// 8 requantised values of a row, before saturation, as the words of the output type (two fp16 or int16, or
// four int8, a word), w[0] on.  Saturating to [-127, 127] biased by 127 is one add-min-relu; the bias comes off with
// a half2 subtract of 1151 from 1024 + u, or an add and an exclusive or per word (u + 1 never carries into
// the next byte); two int16 are saturated and packed in one instruction, -32768 raised in another.
// lo: the lowest int8 result, -127 or (ReLU) 0.  GELU kinds: sat16 indexes the table of values + 128 (gt points at the entry of -32767).
template <int KIND>
constexpr int out_words() { return KIND == KIND_RQ16 || KIND == KIND_F16OUT || KIND == KIND_GELU_F16 ? 8 : 4; }
template <int KIND>
__device__ __forceinline__ void pack8(const int32_t (&r)[8], const uint8_t *gt, int32_t lo, uint32_t *w) {
    if constexpr (KIND == KIND_RQ16) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            asm("{.reg .b32 t;\n\tcvt.pack.sat.s16.s32 t, %1, %2;\n\tmax.s16x2 %0, t, %3;}"
                : "=r"(w[j]) : "r"(r[2 * j + 1]), "r"(r[2 * j]), "r"(0x80018001u));
    } else {
        uint32_t u[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if constexpr (gelu_kind(KIND)) u[i] = gt[__viaddmin_s32_relu(r[i], 32767, 65534)];
            else u[i] = (uint32_t)__viaddmin_s32_relu(max(r[i], lo), 127, 254);
        }
        if constexpr (out_words<KIND>() == 8) {
            // fp16 1024 + u, less 1151 (u biased by 127) or 1152 (the biased table)
            constexpr uint32_t off = KIND == KIND_F16OUT ? 0xE47FE47Fu : 0xE480E480u;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = half2_add(__byte_perm(u[2 * j], u[2 * j + 1], 0x5410) | 0x64006400u, off);
        } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint32_t x = __byte_perm(__byte_perm(u[4 * j], u[4 * j + 1], 0x0040),
                                               __byte_perm(u[4 * j + 2], u[4 * j + 3], 0x0040), 0x5410);
                w[j] = (KIND == KIND_RQ8 ? x + 0x01010101u : x) ^ 0x80808080u;
            }
        }
    }
}
// The words stored at dst: 16-byte vector stores when vec (16 columns, 16-byte aligned), else element by
// element (ncol columns).
template <int KIND>
__device__ __forceinline__ void store_words(char *dst, const uint32_t (&w)[out_words<KIND>()], int ncol, bool vec) {
    constexpr int NW = out_words<KIND>();
    if (vec) {
#pragma unroll
        for (int j = 0; j < NW / 4; ++j) ((uint4 *)dst)[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    } else if constexpr (NW == 8) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < ncol) ((uint16_t *)dst)[i] = (uint16_t)((i & 1) ? w[i >> 1] >> 16 : w[i >> 1]);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < ncol) ((uint8_t *)dst)[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
    }
}
// A warp's TMA-store box: its 32 rows x 32 columns.  Chunk `half` (0 or 1) of row `lane`: 2-byte outputs
// (fp16-carried int8, int16) as two 16-byte units of a 64-byte row in the 64-byte swizzle the tensor map
// declares (unit j of row r at j ^ ((r >> 1) & 3)), 1-byte outputs as one unit of a 32-byte row in the 32-byte
// swizzle (j ^ ((r >> 2) & 1)): no bank conflicts.  (Boxes of 16 columns fence and store twice as often.)
template <int KIND>
constexpr int box_bytes() { return out_words<KIND>() == 8 ? 2048 : 1024; }
template <int KIND>
__device__ __forceinline__ void box_words(uint8_t *box, int lane, int half, const uint32_t (&w)[out_words<KIND>()]) {
    if constexpr (out_words<KIND>() == 8) {
        const int sw = (lane >> 1) & 3;
        *(uint4 *)(box + lane * 64 + (((2 * half) ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        *(uint4 *)(box + lane * 64 + (((2 * half + 1) ^ sw) << 4)) = make_uint4(w[4], w[5], w[6], w[7]);
    } else {
        *(uint4 *)(box + lane * 32 + ((half ^ ((lane >> 2) & 1)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// The residual pairs (x[2j] | x[2j+1] << 16) of 32 columns of a row starting at rrow + c0 (columns
// at or past ncol read as 0; rvec: 16-byte aligned and all 32 present).
__device__ __forceinline__ void res_group(const int16_t *rrow, int c0, int ncol, bool rvec, uint32_t (&rp)[16]) {
    if (rrow && rvec && c0 + 32 <= ncol) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 a = __ldg((const uint4 *)(rrow + c0) + j);
            rp[4 * j] = a.x; rp[4 * j + 1] = a.y; rp[4 * j + 2] = a.z; rp[4 * j + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int cl = c0 + 2 * j;
            const uint32_t lo = (rrow && cl < ncol) ? (uint16_t)rrow[cl] : 0u;
            const uint32_t hi = (rrow && cl + 1 < ncol) ? (uint16_t)rrow[cl + 1] : 0u;
            rp[j] = lo | (hi << 16);
        }
    }
}

// The epilogue of one warp's part of a tile (its 32 rows x HALF columns) in the common case: a
// plain GEMM whose K is split into NSEG accumulators (compile-time), and requantisations that fit
// 32 bits (the caller checks the part's columns).  FORM_UNI: one dyadic shift s >= 33 for all of them, so
// rq(v; m, s) = mad.hi(v, m, 2^(s-33)) >> (s - 32) with a scalar rounding constant and shift.  FORM_VAR: every
// s >= 29 and |bias| <= 2^26: with k = max(0, 33 - s), rq(v; m, s) = rq(v 2^k; m, s + k) and |v 2^k| < 2^31; the
// four parameters are the bias times 2^k, 2^k, m and s + k - 33.  FORM_FLT: below.  The part's
// accumulators are read from TMEM in 32-column groups (all of them at once for one segment), so the
// accumulator set is released to the MMA warp after the first wait, and the requantisation of the
// 16-column chunks that follows has no TMEM latency left in it.  RES: the two-term residual form
// (17 <= s_r <= 46); rp holds the residual pairs of group 0 (fetched by the caller while the MMAs ran), and
// each later group's pairs are fetched before its TMEM loads.  RES = 1: in registers; RES = 2: the residual is in
// the warp's box already (by TMA, read back as 16 bytes a lane), and the results replace it there.
//
// Bound by instructions (a scheduler owns BM BN / 128 outputs of a tile and has about as long for them as the
// tile's MMAs take); so:
// - Accumulators become integers with one packed add of 1.5 2^23, whose bits are read (float to integer is
//   8 cycles a warp, this 1 a value), for groups whose accumulators are all within 2^22; others convert.
// - int8 results without a residual (FORM_FLT, any shifts) are rounded in packed fp32: y = acc sc + b, sc = m 2^-s and
//   b = bias m 2^-s rounded to float, rr = round(y), d = y - rr exactly.  For |acc sc + b| <= 127.5 and
//   |b| <= 128 the float y is off by at most 256 2^-24 (sc) + 2^-17 (y) + 2^-18 (b) < 2^-15, and with two
//   accumulators by their sum's 256 2^-24 more, < 2^-14; so while |d| <= 1/2 - that, rr is
//   floor(y + 1/2) of the exact y (beyond 127.5 both saturate).  A chunk with any other value (about 3 and
//   6 % of chunks on generic data) is computed again in 64-bit integers.  m 2^-s with fewer than 14 fractional bits
//   would often meet 1/2 exactly, so the caller lets such columns take the integers at once.
// Before (float-to-integer conversions, parameters per tile, 16-column boxes) and now, graph replays on
// 12800 rows: 1152 x 384 to int8 in fp16 21.2 and 17.0 us (a 128 x 192 tile 5750 and 3300 clocks here),
// 384 x 384 with residual 14.6 and 13.0, 1536 x 384 with SD-ShiftGELU 29.5 and 27.0; a 256-token block with
// a shift of its own for every column (the 64-bit form then) 74 and 47.5 us.
//
// box: this warp's one or two TMA-store boxes (nullptr: plain stores at dst), written out at column
// x0 + 32 g, row y0 of cmap by lane 0 once every lane has written its row.
template <int KIND, int BN, int HALF, int NSEG, int RES, int FORM>
__device__ __forceinline__ void epi_fast(const EpiParams &ep, uint32_t tbase, const int32_t *s_bias,
                                         const int32_t *s_mult, const int32_t *s_a, const int32_t *s_b, int n0,
                                         int ncol_all,
                                         int32_t rnd, int32_t sh, uint32_t (&rp)[16],
                                         const int16_t *rrow, bool rvec, char *dst, int ncol_row, bool vec_ok,
                                         const uint8_t *gt, uint32_t empty_bar, int lane, uint8_t *box, int boxes,
                                         const CUtensorMap *cmap, int x0, int y0) {
    static_assert(HALF % 32 == 0, "32-column groups");
    constexpr int NG = HALF / 32;                    // 32-column groups of the part
    // groups read per TMEM pass (32 registers per group and segment): a part of 64 columns at once for one
    // segment without a residual, else one group (three at once spill, and so do the residual's pairs)
    constexpr int GPASS = (NSEG == 1 && RES == 0 && NG <= 2) ? NG : 1;
    static_assert(RES != 2 || (NG == 1 && KIND == KIND_RQ16), "one box holds the residual and the results");
    constexpr int esz = (KIND == KIND_RQ16 || KIND == KIND_F16OUT || KIND == KIND_GELU_F16) ? 2 : (KIND == KIND_RAW32 ? 4 : 1);
    const int32_t lo = RES != 0 ? INT32_MIN : (ep.relu ? 0 : -127);  // of int8 results (a ReLU comes without a residual)
    const uint32_t lo_h = ep.relu ? 0u : 0xD7F0D7F0u;
    const int32_t r_rnd = RES != 0 ? 1 << (ep.s_r - 17) : 0, r_sh = RES != 0 ? ep.s_r - 16 : 0;
#pragma unroll
    for (int g0 = 0; g0 < NG; g0 += GPASS) {
        if constexpr (RES == 1) {  // this group's residual pairs (group 0's came with the call), in flight during the TMEM wait
            if (g0 > 0) res_group(rrow, 32 * g0, ncol_row, rvec, rp);
        }
        uint32_t v[NSEG][GPASS * 32];
#pragma unroll
        for (int gg = 0; gg < GPASS; ++gg)
#pragma unroll
            for (int sg = 0; sg < NSEG; ++sg) tmem_ld32(tbase + (uint32_t)(sg * BN + 32 * (g0 + gg)), v[sg] + 32 * gg);
        tmem_wait_only();
#pragma unroll
        for (int gg = 0; gg < GPASS; ++gg)
#pragma unroll
            for (int sg = 0; sg < NSEG; ++sg) tmem_mark32(v[sg] + 32 * gg);
        if (g0 + GPASS >= NG) {  // every TMEM read of this warp in this accumulator set is done
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(empty_bar);
        }
        // 16 columns out: the chunk's words
        auto emit = [&](int c, const uint32_t (&w)[out_words<KIND>()]) {
            if (box) {
                // chunks 2 g and 2 g + 1 share a box, which an earlier store must have read: with two boxes the
                // store before the last one, but where a part has an odd number of groups, the last one itself
                // used the box of a tile's first group.  (Every group of columns commits, so that the count
                // holds where columns past N store nothing.)
                uint8_t *bx = box + (boxes == 2 ? ((c >> 1) & 1) * box_bytes<KIND>() : 0);
                if ((c & 1) == 0) {
                    if (lane == 0) {
                        if (boxes == 2 && !(NG % 2 != 0 && c == 0)) tma_store_wait_read1();
                        else tma_store_wait_read();
                    }
                    __syncwarp();
                }
                box_words<KIND>(bx, lane, c & 1, w);
                if (c & 1) {
                    fence_async_smem_g();
                    __syncwarp();
                    if (lane == 0) {
                        if (16 * (c - 1) < ncol_row) tma_store_2d(cmap, x0 + 16 * (c - 1), y0, smem_u32(bx));
                        tma_store_commit();
                    }
                }
            } else if (dst) {
                const int ncol = ncol_row - 16 * c;
                if (ncol > 0) store_words<KIND>(dst + 16 * c * esz, w, ncol, vec_ok && ncol >= 16);
            }
        };
        if constexpr (FORM == FORM_FLT) {
            const f32x2 magic = pair2(kMagic, kMagic), nmagic = pair2(kMagic | 0x80000000u, kMagic | 0x80000000u);
#pragma unroll
            for (int cc = 0; cc < GPASS * 2; ++cc) {
                const int c = 2 * g0 + cc;  // 16-column chunk of the part
                int32_t sc[16], bf[16];
                lds16(s_a + 16 * c, sc);
                lds16(s_b + 16 * c, bf);
                uint32_t w[out_words<KIND>()], hw[8];
                float dmax = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = 16 * cc + 2 * j;
                    f32x2 acc = pair2(v[0][i], v[0][i + 1]);
#pragma unroll
                    for (int sg = 1; sg < NSEG; ++sg) acc = add2(acc, pair2(v[sg][i], v[sg][i + 1]));
                    const f32x2 y = fma2(acc, pair2(sc[2 * j], sc[2 * j + 1]), pair2(bf[2 * j], bf[2 * j + 1]));
                    const f32x2 rr = add2(add2(y, magic), nmagic);
                    const f32x2 d = add2(y, rr ^ 0x8000000080000000ull);
                    dmax = max_abs3(dmax, lo2(d), hi2(d));
                    asm("{.reg .b32 t;\n\tcvt.rn.f16x2.f32 t, %1, %2;\n\tmin.f16x2 t, t, %3;\n\tmax.f16x2 %0, t, %4;}"
                        : "=r"(hw[j]) : "f"(hi2(rr)), "f"(lo2(rr)), "r"(0x57F057F0u), "r"(lo_h));  // 127 and lo
                }
                if constexpr (KIND == KIND_F16OUT) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) w[j] = hw[j];
                } else {  // the low byte of the fp16 bits of 1152 + v is 128 + v
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        w[j] = __byte_perm(half2_add(hw[2 * j], 0x64806480u), half2_add(hw[2 * j + 1], 0x64806480u), 0x6420) ^
                               0x80808080u;
                }
                if (__any_sync(0xffffffffu, !(dmax <= 0.5f - (NSEG == 1 ? 0x1p-15f : 0x1p-14f)))) {
#pragma unroll
                    for (int e = 0; e < 16; e += 8) {
                        int32_t cb[8], cm[8], r[8];
                        lds8(s_bias + 16 * c + e, cb);
                        lds8(s_mult + 16 * c + e, cm);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            r[i] = __float2int_rn(__uint_as_float(v[0][16 * cc + e + i]));
#pragma unroll
                            for (int sg = 1; sg < NSEG; ++sg) r[i] += __float2int_rn(__uint_as_float(v[sg][16 * cc + e + i]));
                        }
                        if (rnd) {  // one shift >= 33
#pragma unroll
                            for (int i = 0; i < 8; ++i) r[i] = rq_hi(r[i] + cb[i], cm[i], rnd, sh);
                        } else {
                            const int col = n0 + 16 * c + e;
#pragma unroll
                            for (int i = 0; i < 8; ++i) r[i] = rq_clamped(r[i], cb[i], cm[i], col + i < ncol_all ? __ldg(ep.shift + col + i) : 33);
                        }
                        pack8<KIND>(r, gt, lo, w + e * out_words<KIND>() / 16);
                    }
                }
                emit(c, w);
            }
        } else {
            // the integer accumulators (exact: every partial sum is below 2^24) plus kMagic per segment, in place
            float amax = 0.f;
#pragma unroll
            for (int sg = 0; sg < NSEG; ++sg)
#pragma unroll
                for (int i = 0; i < GPASS * 32; i += 2)
                    amax = max_abs3(amax, __uint_as_float(v[sg][i]), __uint_as_float(v[sg][i + 1]));
            const bool wide = __any_sync(0xffffffffu, amax > 4194304.f);
            if (wide) {
#pragma unroll
                for (int i = 0; i < GPASS * 32; ++i) {
                    uint32_t a = (uint32_t)NSEG * kMagic;
#pragma unroll
                    for (int sg = 0; sg < NSEG; ++sg) a += (uint32_t)__float2int_rn(__uint_as_float(v[sg][i]));
                    v[0][i] = a;
                }
            } else {
#pragma unroll
                for (int i = 0; i < GPASS * 32; i += 2) {
                    f32x2 t = add2(pair2(v[0][i], v[0][i + 1]), pair2(kMagic, kMagic));
                    v[0][i] = (uint32_t)t;
                    v[0][i + 1] = (uint32_t)(t >> 32);
#pragma unroll
                    for (int sg = 1; sg < NSEG; ++sg) {
                        t = add2(pair2(v[sg][i], v[sg][i + 1]), pair2(kMagic, kMagic));
                        v[0][i] += (uint32_t)t;
                        v[0][i + 1] += (uint32_t)(t >> 32);
                    }
                }
            }
#pragma unroll
            for (int cc = 0; cc < GPASS * 2; ++cc) {
                const int c = 2 * g0 + cc;
                uint32_t w[out_words<KIND>()];
#pragma unroll
                for (int e = 0; e < 16; e += 8) {
                    int32_t cb[8], cm[8], r[8];
                    lds8(s_bias + 16 * c + e, cb);  // less the magic numbers
                    lds8(s_mult + 16 * c + e, cm);
                    uint4 *unit = nullptr;
                    uint32_t xr[4];
                    if constexpr (RES == 2) {  // this lane's 8 residuals, in the box its results go to
                        unit = (uint4 *)(box + lane * 64 + (((2 * (c & 1) + e / 8) ^ ((lane >> 1) & 3)) << 4));
                        const uint4 x4 = *unit;
                        xr[0] = x4.x; xr[1] = x4.y; xr[2] = x4.z; xr[3] = x4.w;
                    }
                    if constexpr (FORM == FORM_UNI) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            r[i] = rq_hi((int32_t)(v[0][16 * cc + e + i] + (uint32_t)cb[i]), cm[i], rnd, sh);  // |r| < 2^29
                    } else {
                        int32_t ck[8], cs[8];
                        lds8(s_a + 16 * c + e, ck);
                        lds8(s_b + 16 * c + e, cs);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            r[i] = rq_hi1((int32_t)(v[0][16 * cc + e + i] * (uint32_t)ck[i] + (uint32_t)cb[i]), cm[i], cs[i]);
                    }
                    if constexpr (RES != 0) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const uint32_t x = RES == 1 ? rp[8 * cc + (e + i) / 2] : xr[i / 2];
                            const int32_t xs = (i & 1) ? (int32_t)(x & 0xFFFF0000u) : (int32_t)(x << 16);
                            r[i] += rq_hi(xs, ep.m_r, r_rnd, r_sh);
                        }
                    }
                    pack8<KIND>(r, gt, lo, w + e * out_words<KIND>() / 16);
                    if constexpr (RES == 2) *unit = make_uint4(w[e / 2], w[e / 2 + 1], w[e / 2 + 2], w[e / 2 + 3]);
                }
                if constexpr (RES != 2) emit(c, w);
            }
            if constexpr (RES == 2) {
                fence_async_smem_g();
                __syncwarp();
                if (lane == 0) {
                    if (ncol_row > 0) tma_store_2d(cmap, x0, y0, smem_u32(box));
                    tma_store_commit();
                }
            }
        }
        __syncwarp();  // reconverge before the next warp-synchronous tcgen05 instruction
    }
}

// Epilogue warps: column parts per TMEM lane quarter.  int8 A: two parts next to the four converter warps;
// fp16 A needs no converters, and 128-wide tiles take four parts of 32 columns (a warp's whole residual is
// in registers before the accumulators are ready, and 16 warps hide the chains of their loads; with two
// parts the epilogue of a projection tile took 4900 clocks), 192-wide tiles three of 64.
// EP: that many parts instead (0: these).  128-wide tiles of fp16 A take two where 18 warps have no such loads to hide
// and their 96 registers spill: raw accumulators, and of streamed weights int16 results without a residual box, int8
// results with a residual and more than two accumulators.  (With four parts and with two: 12800 x 1536 x 384 to int16 27.3
// and 21.6 us, 12800 x 2048 x 512 to int8 with a residual 48.8 and 44.6, 12800 x 128 x 4096 to int16 31.8 and 29.1, 51200 x 1100 x
// 256 raw 123.7 and 104.9.)
template <int BN, bool AF16, int EP>
constexpr int epi_parts() { return EP ? EP : (AF16 ? (BN == 192 ? 3 : BN / 32) : 2); }
template <int BN, bool AF16, int EP>
constexpr int epi_warps() { return 4 * epi_parts<BN, AF16, EP>(); }
template <int BN, bool AF16, int EP>
constexpr int tc_threads() { return 32 * ((AF16 ? 2 : 6) + epi_warps<BN, AF16, EP>()); }

template <int V>
using Int = std::integral_constant<int, V>;

template <int BN, int STAGES, int KIND, int NB, bool AF16, bool WRES, int EP>
__global__ void __launch_bounds__(tc_threads<BN, AF16, EP>(), 1) gemm_tc_kernel(const __grid_constant__ TcParams<NB> p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    using SM = Smem<BN, AF16, WRES>;
    constexpr int kStage = SM::kStage;
    constexpr int NP = epi_parts<BN, AF16, EP>(), EPI0 = AF16 ? 2 : 6;  // column parts, first epilogue warp
    constexpr int NWE = 4 * NP;
    const int nst = WRES ? p.stages : STAGES;  // pipeline stages
    uint8_t *wres = smem + nst * kStage;  // resident weights (WRES)
    uint64_t *bars = (uint64_t *)(wres + (WRES ? p.wres_bytes : 0));
    // barriers: full[S], a_ready[S], empty[S], acc_full[2], acc_empty[2], wfull[kMaxWk] (one per K block
    // of the resident weights, so the first MMAs start as soon as their own block has landed)
    uint32_t *tmem_slot = (uint32_t *)(bars + 3 * STAGES + 6 + kMaxWk + NWE);
    volatile int *abort = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto a_ready = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto empty = [&](int s) { return bar0 + 8u * (2 * STAGES + s); };
    auto acc_full = [&](int b) { return bar0 + 8u * (3 * STAGES + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (3 * STAGES + 2 + b); };
    auto wfull = [&](int kk) { return bar0 + 8u * (3 * STAGES + 4 + kk); };
    const uint32_t drain = bar0 + 8u * (3 * STAGES + 4 + kMaxWk);  // every MMA issued has completed
    const uint32_t tab_full = drain + 8u;                          // the GELU table has arrived
    auto res_full = [&](int w) { return tab_full + 8u * (1 + w); };  // an epilogue warp's residual box

    // one barrier a lane: full[S], a_ready[S] (the converter warps), empty[S], acc_full[2], acc_empty[2]
    // (the epilogue warps), wfull, drain, tab_full, res_full
    constexpr int kBars = 3 * STAGES + 6 + kMaxWk + NWE;
    if (warp == 1) {
        for (int i = lane; i < kBars; i += 32)
            mbar_init(bar0 + 8u * i, i >= STAGES && i < 2 * STAGES ? 4 : (i == 3 * STAGES + 2 || i == 3 * STAGES + 3 ? NWE : 1));
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x < NB) {  // the descriptors, ahead of the first loads
        prefetch_map(&p.amap[threadIdx.x]);
        prefetch_map(&p.wmap[threadIdx.x]);
    }
    if (threadIdx.x == 32 && p.tma_store) prefetch_map(&p.cmap);
    if (threadIdx.x == 64 && p.res_tma) prefetch_map(&p.rmap);
    grid_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // the epilogue warps' copies of the tile's per-column parameters: one per warp, or with resident weights,
    // where a CTA's columns never change, one per column part (its warps write the same values)
    int32_t *prm = (int32_t *)(((uintptr_t)(tmem_slot + 4) + 15) & ~(uintptr_t)15);
    // SD-ShiftGELU and its output requantisation depend on the int16 value g alone: the table of
    // sat8(rq(g * I_div(g); m_g, s_g)) + 128 (built once per parameter set by gelu_table_kernel) is copied
    // into shared memory by the producer (one bulk copy behind the first operands; 12 warps copying it
    // themselves held the first tile's epilogue up by 2000 clocks).
    uint8_t *gtab = (uint8_t *)(prm + prm_words<BN, WRES>());
    const int acc_cols = p.nseg * BN;  // columns of one accumulator set
    // the TMA-store boxes (1024-byte aligned, after the parameters and the GELU table)
    uint8_t *stg = (uint8_t *)(((uintptr_t)gtab + (gelu_kind(KIND) ? 65536 : 0) + 1023) & ~(uintptr_t)1023);

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        if (lane == 0) {
            int it = 0, s = 0;  // K blocks issued, ring position
            uint32_t ph = 0;
            int wk = 0;  // K blocks of the resident weights issued
            bool ok = true, tab = gelu_kind(KIND);
            auto load_tab = [&]() {
                mbar_expect_tx(tab_full, 65536);
                bulk_load(smem_u32(gtab), p.gelu_tab, 65536, tab_full);
                tab = false;
            };
            for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x) {
                const int m0 = (t / p.tiles_n) * BM, n0 = (t % p.tiles_n) * BN;
                for (int sg = 0; sg < p.nseg && ok; ++sg) {
                    const Seg &S = p.seg[sg];
                    const int nk = (S.klen + BK - 1) / BK;
                    for (int kk = 0; kk < nk; ++kk, ++it) {
                        if (WRES && t == (int)blockIdx.x && kk < nst) {
                            // the CTA's BN rows of W, resident for all of its tiles (the grid is a
                            // multiple of tiles_n, so every tile of the CTA has the same n block): the
                            // first K blocks travel with the first tile's activations of the same K block,
                            // the rest follow at once (they have shared memory of their own)
                            const int last = kk == (nst < nk ? nst : nk) - 1 ? nk - 1 : kk;
                            for (int j = kk; j <= last; ++j) {
                                mbar_expect_tx(wfull(j), (uint32_t)SM::kWtile);
                                tma_load_2d(smem_u32(wres + j * SM::kWtile), &p.wmap[0], p.seg[0].k0 + j * BK, n0,
                                            wfull(j));
                            }
                            wk = last + 1;
                        }
                        if (it == nst && tab) load_tab();  // behind the first stages, which wait for nothing
                        if (!mbar_wait(empty(s), ph ^ 1, abort, p.status, kStatusTimeoutFree, p.wait_cycles)) {
                            ok = false;
                            break;
                        }
                        uint8_t *st = smem + s * kStage;
                        const uint32_t fb = full(s);
                        if (++s == nst) {
                            s = 0;
                            ph ^= 1u;
                        }
                        if (it == p.dbg_skip) continue;  // test hook: this stage's barrier never completes
                        mbar_expect_tx(fb, (AF16 ? SM::kA16 : SM::kA8) + SM::kW);
                        tma_load_2d(smem_u32(AF16 ? st : st + SM::kA16 + SM::kW), &p.amap[S.map], S.k0 + kk * BK, m0,
                                    fb);
                        if (!WRES) tma_load_2d(smem_u32(st + SM::kA16), &p.wmap[S.map], S.k0 + kk * BK, n0, fb);
                    }
                }
            }
            if (tab) load_tab();  // fewer K blocks than stages
            if (!ok || *abort) {  // drain the loads still in flight (bounded) before the CTA can exit
                long long t0 = clock64();
                while (gelu_kind(KIND) && !mbar_try(tab_full, 0) && clock64() - t0 < p.wait_cycles) {
                }
                for (int kk = 0; kk < wk; ++kk)
                    while (!mbar_try(wfull(kk), 0) && clock64() - t0 < p.wait_cycles) {
                    }
                for (int j = (it > nst ? it - nst : 0); j < it; ++j)
                    while (j != p.dbg_skip && !mbar_try(full(j % nst), (j / nst) & 1) &&
                           clock64() - t0 < p.wait_cycles) {
                    }
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer
        // The whole warp runs the loop and one elected lane issues: the operands then stay in uniform
        // registers.  One thread on its own (`if (lane == 0)`) moves every operand of every MMA over and
        // needs 113 clocks per MMA, above the 64 (N = 128) and 96 (N = 192) the MMA itself takes; this
        // form needs 60 and 86.
        {
            const uint32_t issue = elect_lane() ? 1u : 0u;
            auto wait = [&](uint32_t bar, uint32_t parity, int code) -> bool {
                return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, p.status, code, p.wait_cycles));
            };
            const uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            // operand descriptors from two precomputed bases: a 16-byte step of the address is 1 in
            // the descriptor's low word (shared-memory offsets stay below 256 KB, so nothing carries)
            const uint64_t a_desc0 = sw128_desc(smem_u32(smem)), w_desc0 = sw128_desc(smem_u32(wres));
            int tl = 0, s = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x, ++tl) {
                const int b = p.nbuf == 2 ? tl & 1 : 0;
                const uint32_t use = (uint32_t)(p.nbuf == 2 ? tl >> 1 : tl);
                if (!wait(acc_empty(b), (use & 1) ^ 1, kStatusTimeoutMma)) break;
                tc_fence_after();
                for (int sg = 0; sg < p.nseg && ok; ++sg) {
                    const int nk = (p.seg[sg].klen + BK - 1) / BK;
                    const uint32_t dt = tmem + (uint32_t)(b * acc_cols + sg * BN);
#pragma unroll 1
                    for (int kk = 0; kk < nk; ++kk) {
                        ok = wait(AF16 ? full(s) : a_ready(s), ph, AF16 ? kStatusTimeoutTma : kStatusTimeoutOperand);
                        if (WRES && ok && tl == 0) ok = wait(wfull(kk), 0, kStatusTimeoutTma);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t da = a_desc0 + (uint64_t)((s * kStage) >> 4);
                        const uint64_t dw = WRES ? w_desc0 + (uint64_t)((kk * SM::kWtile) >> 4) : da + (uint64_t)(SM::kA16 >> 4);
#pragma unroll
                        for (int k16 = 0; k16 < BK / 16; ++k16)
                            tc_mma(dt, da + 2 * k16, dw + 2 * k16, idesc, (kk > 0 || k16 > 0) ? 1u : 0u, issue);
                        tc_commit(empty(s), issue);
                        if (++s == nst) {
                            s = 0;
                            ph ^= 1u;
                        }
                    }
                }
                tc_commit(acc_full(b), issue);  // arrives once every MMA of this tile has completed
                __syncwarp();
            }
            // every MMA issued has completed before the CTA can reach the TMEM release (also after an
            // abort, when the epilogue no longer waits for the accumulators)
            tc_commit(drain, issue);
            const long long t0 = clock64();
            while (!mbar_try(drain, 0) && clock64() - t0 < p.wait_cycles) {
            }
            __syncwarp();
        }
    } else if (warp < EPI0) {
        // ---------------------------------------------------------------- operand converters
        if constexpr (!AF16) {  // fp16 A arrives in the MMA's operand layout: nothing to convert
            const int r = (warp - 2) * 32 + lane;  // row of the 128-row A tile
            const int sw = (r >> 1) & 3;           // TMA's 64-byte swizzle of the int8 staging rows
            int it = 0;
            for (int t = blockIdx.x; t < p.tiles; t += gridDim.x) {
                for (int sg = 0; sg < p.nseg; ++sg) {
                    const int nk = (p.seg[sg].klen + BK - 1) / BK;
                    for (int kk = 0; kk < nk; ++kk, ++it) {
                        const int s = it % STAGES;
                        const uint32_t ph = (it / STAGES) & 1;
                        if (!mbar_wait(full(s), ph, abort, p.status, kStatusTimeoutTma, p.wait_cycles)) goto conv_done;
                        uint8_t *st = smem + s * kStage;
                        const uint8_t *a8 = st + SM::kA16 + SM::kW + r * 64;
                        uint8_t *a16 = st + r * 128;
    #pragma unroll
                        for (int j = 0; j < 4; ++j) {  // 16 int8 = K elements 16j .. 16j+15
                            const uint4 v = *(const uint4 *)(a8 + 16 * (j ^ sw));
                            uint4 o0, o1;
                            i8x4_to_f16x4(v.x, o0.x, o0.y);
                            i8x4_to_f16x4(v.y, o0.z, o0.w);
                            i8x4_to_f16x4(v.z, o1.x, o1.y);
                            i8x4_to_f16x4(v.w, o1.z, o1.w);
                            *(uint4 *)(a16 + (((2 * j) ^ (r & 7)) << 4)) = o0;
                            *(uint4 *)(a16 + (((2 * j + 1) ^ (r & 7)) << 4)) = o1;
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(a_ready(s));
                    }
                }
            }
        conv_done:;
        }
    } else {
        // ---------------------------------------------------------------- epilogue
        // NWE warps: warp w reads TMEM lanes 32q..32q+31 (q = w % 4) and owns part h of the columns
        constexpr int HALF = BN / NP;  // columns of this warp in a tile
        const int q = warp & 3, h = (warp - EPI0) >> 2;
        const EpiParams &ep = p.ep;
        int32_t *s_bias = prm + (WRES ? h : warp - EPI0) * 4 * HALF, *s_mult = s_bias + HALF;
        int32_t *s_shift = s_mult + HALF, *s_rnd = s_shift + HALF;  // (or what epi_fast reads there)
        constexpr int bits = (KIND == KIND_RQ16 || KIND == KIND_F16OUT || KIND == KIND_GELU_F16) ? 16
                             : (KIND == KIND_RAW32 ? 32 : 8);
        constexpr int PPL = HALF / 32;  // parameters per lane and per array
        constexpr bool kFastKind = KIND == KIND_RQ8 || KIND == KIND_RQ16 || KIND == KIND_F16OUT || gelu_kind(KIND);
        constexpr bool kResKind = KIND == KIND_RQ8 || KIND == KIND_RQ16;  // kinds with a residual
        const int nseg = p.nseg, nld = (HALF / 16) * nseg;  // TMEM loads per tile
        const bool has_res = ep.res != nullptr, rfast = has_res && ep.s_r >= 17 && ep.s_r <= 46;
        bool fastw = false, one_shift = false;  // every shift >= 33; and the same
        int form = FORM_GENERAL;
        int32_t s_0 = 0;
        // The parameters of this warp's columns into shared memory, and the form they allow.  The launch
        // makes the grid a multiple of the column tiles where it can, so that a CTA stays in its columns
        // and this runs once (per tile it took 1700 of 5800 clocks).
        auto params = [&](int n0) {
            int32_t pb[PPL], pm[PPL], ps[PPL];
            bool ok[PPL];
#pragma unroll
            for (int k = 0; k < PPL; ++k) {
                const int col = n0 + lane + 32 * k;
                ok[k] = col < p.N;
                pb[k] = (ok[k] && ep.bias) ? __ldg(ep.bias + col) : 0;
                pm[k] = (ok[k] && ep.mult) ? __ldg(ep.mult + col) : 0;
                ps[k] = (ok[k] && ep.shift) ? __ldg(ep.shift + col) : 33;
            }
            bool fast_lane = true, same_lane = true, var_lane = true, flt_lane = true;
            s_0 = __shfl_sync(0xffffffffu, ps[0], 0);
            // epi_fast with int8 results in packed fp32: m 2^-s and bias m 2^-s as floats
            constexpr bool kFltKind = KIND == KIND_RQ8 || KIND == KIND_F16OUT;
            float fsc[PPL], fbi[PPL];
#pragma unroll
            for (int k = 0; k < PPL; ++k) {
                fast_lane &= ps[k] >= 33;
                same_lane &= ps[k] == s_0 || !ok[k];
                var_lane &= ps[k] >= 29 && pb[k] >= -(1 << 26) && pb[k] <= (1 << 26);
                if constexpr (kFltKind) {
                    const float two_s = __int_as_float((127 - max(1, min(ps[k], 100))) << 23);
                    fsc[k] = __int2float_rn(pm[k]) * two_s;
                    fbi[k] = __ll2float_rn((int64_t)pb[k] * pm[k]) * two_s;
                    flt_lane &= ps[k] >= 1 && ps[k] <= 100 && fabsf(fbi[k]) <= 128.f && (pm[k] == 0 || ps[k] - (__ffs(pm[k]) - 1) >= 14);
                }
            }
            fastw = __all_sync(0xffffffffu, fast_lane);  // shifts stored as s - 32 if so
            one_shift = fastw && __all_sync(0xffffffffu, same_lane);
            form = FORM_GENERAL;
            if (kFastKind && NB == 1 && !p.branch_rq && p.nseg <= 2 && (!has_res || rfast)) {
                if (kFltKind && !has_res && __all_sync(0xffffffffu, flt_lane)) form = FORM_FLT;
                else if (one_shift) form = FORM_UNI;
                else if (p.nseg == 1 && __all_sync(0xffffffffu, var_lane)) form = FORM_VAR;
            }
            __syncwarp();  // this warp is done with the parameters before
#pragma unroll
            for (int k = 0; k < PPL; ++k) {
                int32_t b = pb[k], sa = fastw ? ps[k] - 32 : ps[k], sb = fastw ? 1 << (ps[k] - 33) : 0;
                const uint32_t off = (uint32_t)p.nseg * kMagic;  // of epi_fast's integers
                if (form == FORM_UNI) b = (int32_t)((uint32_t)b - off);
                if (form == FORM_VAR) {
                    const int kk = max(0, 33 - ps[k]);
                    b = (int32_t)(((uint32_t)b - off) << kk);
                    sa = 1 << kk;
                    sb = max(ps[k], 33) - 33;
                }
                if (kFltKind && form == FORM_FLT) {
                    sa = __float_as_int(fsc[k]);
                    sb = __float_as_int(fbi[k]);
                }
                s_bias[lane + 32 * k] = b;
                s_mult[lane + 32 * k] = pm[k];
                s_shift[lane + 32 * k] = sa;
                s_rnd[lane + 32 * k] = sb;
            }
            __syncwarp();
        };
        // the tile's row block and column tile, advanced without a division
        const int dm = gridDim.x / p.tiles_n, dn = gridDim.x % p.tiles_n;
        int tm = blockIdx.x / p.tiles_n, tn = blockIdx.x % p.tiles_n, cur = -1, tl = 0;
        uint32_t res_ph = 0;   // of the residual box's barrier
        bool res_due = false;  // a residual load is in flight
        const bool tab_ok = !gelu_kind(KIND) || mbar_wait(tab_full, 0, abort, p.status, kStatusTimeoutTma, p.wait_cycles);
        for (int t = blockIdx.x; t < p.tiles && tab_ok; t += gridDim.x, ++tl) {
            const int b = p.nbuf == 2 ? tl & 1 : 0;
            const uint32_t use = (uint32_t)(p.nbuf == 2 ? tl >> 1 : tl);
            const int m0 = tm * BM, n0 = tn * BN + h * HALF;
            if (tn != cur) params(n0);
            cur = tn;
            tm += dm;
            tn += dn;
            if (tn >= p.tiles_n) {
                tn -= p.tiles_n;
                ++tm;
            }
            const int64_t row = (int64_t)m0 + 32 * q + lane;
            const bool row_ok = row < p.M;
            // this row's residual (row modulo res_rows broadcasts a [res_rows, N] table)
            const int16_t *rrow = (ep.res && row_ok) ? ep.res + (row < ep.res_rows ? row : row % ep.res_rows) * ep.ldr + n0 : nullptr;
            const bool rvec = ((uintptr_t)rrow & 15) == 0;
            const uint32_t tbase = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * acc_cols + h * HALF);
            if constexpr (kFastKind && NB == 1) {
                if (form != FORM_GENERAL) {
                    // the residuals (of the first 32 columns) are fetched while the MMAs run
                    constexpr bool kResBox = KIND == KIND_RQ16 && HALF == 32;
                    const bool rbox = kResBox && p.res_tma;
                    uint8_t *box = p.tma_store ? stg + (warp - EPI0) * p.tma_store * box_bytes<KIND>() : nullptr;
                    if (rbox) {
                        if (lane == 0) {
                            tma_store_wait_read();  // the box's last results are on their way
                            const uint32_t y = (uint32_t)(m0 + 32 * q), rows = (uint32_t)ep.res_rows;
                            mbar_expect_tx(res_full(warp - EPI0), 2048);
                            tma_load_2d(smem_u32(box), &p.rmap, n0, (int32_t)(y < rows ? y : y % rows), res_full(warp - EPI0));
                        }
                        __syncwarp();
                        res_due = true;
                    }
                    uint32_t rpa[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) rpa[j] = 0;
                    if (kResKind && has_res && !rbox) res_group(rrow, 0, p.N - n0, rvec, rpa);
                    if (!mbar_wait(acc_full(b), use & 1, abort, p.status, kStatusTimeoutMma, p.wait_cycles)) break;
                    tc_fence_after();
                    char *dst = row_ok ? (char *)ep.C + (row * ep.ldc + n0) * (bits / 8) : nullptr;
                    const bool vec_ok = ((uintptr_t)dst & 15) == 0;
                    const int ncol_row = p.N - n0;
                    const int32_t rnd = one_shift ? 1 << (s_0 - 33) : 0, sh = s_0 - 32;
                    const uint8_t *gt = gtab;  // the entry of -32767
                    const uint32_t eb = acc_empty(b);
                    if (rbox) {
                        if (!mbar_wait(res_full(warp - EPI0), res_ph, abort, p.status, kStatusTimeoutTma, p.wait_cycles)) break;
                        res_ph ^= 1u;
                        res_due = false;
                    }
                    auto epi = [&](auto nseg_c, auto res_c, auto form_c) {
                        constexpr int NS = decltype(nseg_c)::value, RS = decltype(res_c)::value, FM = decltype(form_c)::value;
                        epi_fast<KIND, BN, HALF, NS, RS, FM>(ep, tbase, s_bias, s_mult, s_shift, s_rnd, n0, p.N, rnd, sh, rpa,
                                                             rrow, rvec, dst, ncol_row, vec_ok, gt, eb, lane, box, p.tma_store,
                                                             &p.cmap, n0, m0 + 32 * q);
                    };
                    auto epi_res = [&](auto nseg_c, auto form_c) {
                        if (rbox) epi(nseg_c, Int<kResBox ? 2 : 0>{}, form_c);
                        else if (kResKind && has_res) epi(nseg_c, Int<kResKind ? 1 : 0>{}, form_c);
                        else epi(nseg_c, Int<0>{}, form_c);
                    };
                    constexpr bool kFlt = KIND == KIND_RQ8 || KIND == KIND_F16OUT;
                    if (WRES || p.nseg == 1) {  // (resident weights: K <= 1024)
                        if (kFlt && form == FORM_FLT) epi(Int<1>{}, Int<0>{}, Int<kFlt ? FORM_FLT : FORM_UNI>{});
                        else if (form == FORM_UNI) epi_res(Int<1>{}, Int<FORM_UNI>{});
                        else epi_res(Int<1>{}, Int<FORM_VAR>{});
                    } else {
                        if (kFlt && form == FORM_FLT) epi(Int<2>{}, Int<0>{}, Int<kFlt ? FORM_FLT : FORM_UNI>{});
                        else epi_res(Int<2>{}, Int<FORM_UNI>{});
                    }
                    continue;
                }
            }
            if (!mbar_wait(acc_full(b), use & 1, abort, p.status, kStatusTimeoutMma, p.wait_cycles)) break;
            tc_fence_after();
            uint32_t rp[8];
            // The tile's chunks, with the requantisation forms fixed for the whole tile (a branch per
            // tile instead of both forms predicated per element).  TMEM load i reads segment i % nseg
            // of chunk i / nseg; load i+1 is in flight while the epilogue of load i's chunk runs.
            auto chunks = [&](auto fast_c, auto rfast_c) {
                constexpr bool FAST = decltype(fast_c)::value, RFAST = decltype(rfast_c)::value;
                uint32_t v[16];
                tmem_ld16(tbase, v);
                int32_t acc[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[i] = 0;
                for (int li = 0; li < nld; ++li) {
                    const int c0 = (li / nseg) * 16, sg = li - (li / nseg) * nseg;
                    if (has_res && sg == 0) {  // this chunk's residuals, in flight during the TMEM wait
                        if (rrow && rvec && n0 + c0 + 16 <= p.N) {
                            const uint4 a = __ldg((const uint4 *)(rrow + c0)), b = __ldg((const uint4 *)(rrow + c0) + 1);
                            rp[0] = a.x; rp[1] = a.y; rp[2] = a.z; rp[3] = a.w;
                            rp[4] = b.x; rp[5] = b.y; rp[6] = b.z; rp[7] = b.w;
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int cl = n0 + c0 + 2 * j;
                                const uint32_t lo = (rrow && cl < p.N) ? (uint16_t)rrow[c0 + 2 * j] : 0u;
                                const uint32_t hi = (rrow && cl + 1 < p.N) ? (uint16_t)rrow[c0 + 2 * j + 1] : 0u;
                                rp[j] = lo | (hi << 16);
                            }
                        }
                    }
                    tmem_wait_ld16(v);
                    if (p.branch_rq) {
                        const int32_t mb = p.seg[sg].m_b, sbb = p.seg[sg].s_b;
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[i] += (int32_t)rq(__float2int_rn(__uint_as_float(v[i])), mb, sbb);
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[i] += __float2int_rn(__uint_as_float(v[i]));  // exact: < 2^24
                    }
                    if (li + 1 < nld) {
                        const int c1 = ((li + 1) / nseg) * 16, sg1 = (li + 1) - ((li + 1) / nseg) * nseg;
                        tmem_ld16(tbase + (uint32_t)(sg1 * BN + c1), v);
                    } else {  // every TMEM read of this warp in this accumulator set is done
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acc_empty(b));
                    }
                    if (sg != nseg - 1) continue;
                    int32_t cb[16], cm[16], cs[16], cr[16];  // this chunk's per-column parameters
                    lds16(s_bias + c0, cb);
                    lds16(s_mult + c0, cm);
                    lds16(s_shift + c0, cs);
                    if (FAST) lds16(s_rnd + c0, cr);
                    const int ncol = min(16, p.N - (n0 + c0));
                    if (row_ok && ncol > 0) {
                        int32_t out[16];
                        const uint8_t *gt = gtab + 32767;
                        epi_chunk<KIND, FAST, RFAST>(ep, has_res, rp, acc, cb, cm, cs, cr, gt, out);
                        char *dst = (char *)ep.C + (row * ep.ldc + n0 + c0) * (bits / 8);
                        const bool vec = ncol == 16 && (((uintptr_t)dst & 15) == 0);
                        if constexpr (KIND == KIND_F16OUT || KIND == KIND_GELU_F16) {
                            // |v| <= 127: the fp16 bits of 1152 + v are 0x6480 + v; one half2 subtract of
                            // 1152 leaves v exactly
                            const __half2 k1152 = __half2half2(__ushort_as_half((unsigned short)0x6480));
                            uint32_t hw[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                uint32_t x = (uint32_t)(0x6480 + out[2 * j]) | ((uint32_t)(0x6480 + out[2 * j + 1]) << 16);
                                __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&x), k1152);
                                hw[j] = *reinterpret_cast<uint32_t *>(&h);
                            }
                            if (vec) {
                                ((uint4 *)dst)[0] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                                ((uint4 *)dst)[1] = make_uint4(hw[4], hw[5], hw[6], hw[7]);
                            } else {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (i < ncol) ((uint16_t *)dst)[i] = (uint16_t)((i & 1) ? hw[i >> 1] >> 16 : hw[i >> 1]);
                            }
                        } else if constexpr (bits == 8) {
                            if (vec) {
                                uint32_t w[4];
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    w[u] = (uint32_t)(uint8_t)out[4 * u] | ((uint32_t)(uint8_t)out[4 * u + 1] << 8) |
                                           ((uint32_t)(uint8_t)out[4 * u + 2] << 16) | ((uint32_t)(uint8_t)out[4 * u + 3] << 24);
                                *(uint4 *)dst = make_uint4(w[0], w[1], w[2], w[3]);
                            } else {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (i < ncol) ((int8_t *)dst)[i] = (int8_t)out[i];
                            }
                        } else if constexpr (bits == 16) {
                            if (vec) {
#pragma unroll
                                for (int j = 0; j < 2; ++j) {
                                    uint32_t w[4];
#pragma unroll
                                    for (int u = 0; u < 4; ++u)
                                        w[u] = (uint32_t)(uint16_t)out[8 * j + 2 * u] | ((uint32_t)(uint16_t)out[8 * j + 2 * u + 1] << 16);
                                    ((uint4 *)dst)[j] = make_uint4(w[0], w[1], w[2], w[3]);
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (i < ncol) ((int16_t *)dst)[i] = (int16_t)out[i];
                            }
                        } else {
                            if (vec) {
#pragma unroll
                                for (int j = 0; j < 4; ++j)
                                    ((int4 *)dst)[j] = make_int4(out[4 * j], out[4 * j + 1], out[4 * j + 2], out[4 * j + 3]);
                            } else {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (i < ncol) ((int32_t *)dst)[i] = out[i];
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[i] = 0;
                    __syncwarp();  // reconverge before the next warp-synchronous tcgen05 instruction
                }
            };
            constexpr bool kRes = KIND == KIND_RQ8 || KIND == KIND_RQ16;  // kinds with a residual
            using T_ = std::true_type;
            using F_ = std::false_type;
            using R_ = std::integral_constant<bool, kRes>;
            auto go = [&](auto f, auto r) { chunks(f, r); };
            if (fastw) {
                if (kRes && rfast) go(T_{}, R_{});
                else go(T_{}, F_{});
            } else {
                if (kRes && rfast) go(F_{}, R_{});
                else go(F_{}, F_{});
            }
        }
        if (res_due) {  // after an abort: the load in flight ends (bounded) before the CTA can exit
            const long long t0 = clock64();
            while (!mbar_try(res_full(warp - EPI0), res_ph) && clock64() - t0 < p.wait_cycles) {
            }
        }
        if (p.tma_store && lane == 0) tma_store_wait_all();  // this warp's stores are complete
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
    }
}

inline int num_sms() { return sm_count(); }

// Dynamic shared memory of one instantiation (wres: resident weight bytes).
// stg: the epilogue warps' TMA-store boxes (0 without TMA stores).
template <int BN, int STAGES, int KIND, bool AF16, bool WRES, int EP = 0>
size_t smem_bytes(int wres, int stg = 0, int stages = STAGES) {
    return 1024 + (size_t)stages * Smem<BN, AF16, WRES>::kStage + (WRES ? wres : 0) + 8 * (3 * STAGES + 6 + kMaxWk + epi_warps<BN, AF16, EP>()) +
           32 + 4 * prm_words<BN, WRES>() + (gelu_kind(KIND) ? 65536 : 0) + (stg ? 1024 + stg : 0);
}
constexpr size_t kSmemMax = 227 * 1024;

template <int BN, int STAGES, int KIND, int NB, bool AF16, bool WRES, int EP = 0>
cudaError_t launch_tc(TcParams<NB> &tp, cudaStream_t s) {
    // TMA stores when the output allows them (set up by run) and their boxes fit next to the rest
    constexpr int stg = epi_warps<BN, AF16, EP>() * box_bytes<KIND>();
    tp.stages = STAGES;
    // (a part of one group of columns stores once a tile, long after the last tile's store: one box)
    if (tp.tma_store) tp.tma_store = tp.res_tma || BN == 32 * epi_parts<BN, AF16, EP>() ? 1 : 2;
    auto bytes = [&](int boxes) { return smem_bytes<BN, STAGES, KIND, AF16, WRES, EP>(tp.wres_bytes, boxes * stg, tp.stages); };
    // resident weights: as many stages as fit beside one box a warp (at least 3).  A's blocks come at L2's
    // latency, so the stages in flight set the rate: 12800 x 384 x 384 with 3 stages 600 clocks a K block
    while (WRES && tp.stages > 3 && bytes(tp.tma_store ? 1 : 0) > kSmemMax) --tp.stages;
    while (tp.tma_store && bytes(tp.tma_store) > kSmemMax) --tp.tma_store;
    if (!tp.tma_store) tp.res_tma = 0;
    const size_t smem = bytes(tp.tma_store);
    if (smem > kSmemMax) return cudaErrorInvalidValue;
    static SmemLimit limit;
    const cudaError_t attr_err =
        raise_smem_limit(limit, (const void *)gemm_tc_kernel<BN, STAGES, KIND, NB, AF16, WRES, EP>, (int)kSmemMax);
    if (attr_err != cudaSuccess) return attr_err;
    int grid = tp.tiles < num_sms() ? tp.tiles : num_sms();
    // a multiple of tiles_n: every CTA keeps one n block of W (WRES: always; else where that costs no round, and, for
    // raw accumulators, which have no parameters to keep, where no CTA is left with the narrower last column block:
    // 134400 x 320 x 320 of int8 A 98 us against 108)
    const int tiles_m = tp.tiles / tp.tiles_n;
    int per_n = num_sms() / tp.tiles_n;
    per_n = per_n < 1 ? 1 : (per_n > tiles_m ? tiles_m : per_n);
    const int whole = per_n * tp.tiles_n;
    if (WRES || (whole <= grid && (KIND != KIND_RAW32 || tp.N % BN == 0) && (tp.tiles + whole - 1) / whole == (tp.tiles + grid - 1) / grid)) grid = whole;
    launch_after(gemm_tc_kernel<BN, STAGES, KIND, NB, AF16, WRES, EP>, grid, tc_threads<BN, AF16, EP>(), smem, s, tp);
    return cudaGetLastError();
}

// One launch shape: the tile width, pipeline depth, tensor-map slots, A form and weight residency;
// GELU selects the SD-ShiftGELU output kinds, otherwise the requantising / raw kinds are built.
template <int BN, int STAGES, int NB, bool AF16, bool WRES, bool GELU>
cudaError_t run(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s) {
    if (gp.nb > NB || (ep.kind == EPI_GELU) != GELU) return cudaErrorInvalidValue;
    TcParams<NB> tp;
    memset(&tp, 0, sizeof(tp));
    tp.M = gp.M;
    tp.N = gp.N;
    tp.branch_rq = gp.branch_rq ? 1 : 0;
    tp.ep = ep;
    tp.status = status_word_ptr();
    int nseg = 0;
    for (int b = 0; b < gp.nb; ++b) {
        const GemmBranch &br = gp.br[b];
        const bool amap_ok =
            AF16 ? gemm_make_map(&tp.amap[b], br.A, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, gp.M, br.K, br.lda, BK, BM,
                            CU_TENSOR_MAP_SWIZZLE_128B)
                 : gemm_make_map(&tp.amap[b], br.A, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, gp.M, br.K, br.lda, BK, BM,
                            CU_TENSOR_MAP_SWIZZLE_64B);
        if (!amap_ok ||
            !gemm_make_map(&tp.wmap[b], br.Wp, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, gp.N, br.K, br.K, BK, BN,
                      CU_TENSOR_MAP_SWIZZLE_128B))
            return cudaErrorInvalidValue;
        // cut K into near-equal segments of at most kSegK (multiples of 64)
        const int parts = (br.K + kSegK - 1) / kSegK;
        if (gp.branch_rq && parts != 1) return cudaErrorInvalidValue;
        const int per = ((br.K + parts - 1) / parts + BK - 1) / BK * BK;
        for (int k0 = 0; k0 < br.K; k0 += per) {
            if (nseg >= kMaxSeg) return cudaErrorInvalidValue;
            Seg &S = tp.seg[nseg++];
            S.k0 = k0;
            S.klen = min(per, br.K - k0);
            S.map = b;
            S.m_b = br.m_b;
            S.s_b = br.s_b;
        }
    }
    tp.nseg = nseg;
    tp.tiles_n = (gp.N + BN - 1) / BN;
    tp.tiles = ((gp.M + BM - 1) / BM) * tp.tiles_n;
    const int one = nseg * BN;
    tp.nbuf = 2 * one <= 512 ? 2 : 1;
    int alloc = 32;
    while (alloc < tp.nbuf * one) alloc <<= 1;
    if (alloc > 512) return cudaErrorInvalidValue;
    tp.tmem_cols = alloc;
    gemm_debug_wait(&tp.dbg_skip, &tp.wait_cycles);
    // TMA tensor stores of the outputs: 32 x 32 boxes of C (1-byte outputs: 32-byte rows in the 32-byte
    // swizzle; 2-byte outputs: 64-byte rows in the 64-byte swizzle), for a C whose rows start on 16-byte boundaries
    tp.tma_store = 0;
    if (NB == 1 && ep.out_bits != 32) {
        const int esz = ep.out_bits == 8 ? 1 : 2;  // int8, or int16 / fp16-carried int8
        if (((uintptr_t)ep.C % 16) == 0 && (ep.ldc * esz) % 16 == 0 && gp.N * esz >= 16)
            tp.tma_store = gemm_make_map(&tp.cmap, ep.C, esz == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_UINT16,
                                         esz, gp.M, gp.N, ep.ldc, 32, 32,
                                         esz == 1 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_64B)
                               ? 1
                               : 0;
    }
    // an int16 residual under int16 outputs by TMA, if its rows allow a map and no box wraps around
    tp.res_tma = 0;
    if (tp.tma_store && ep.out_bits == 16 && ep.res && BN == 32 * epi_parts<BN, AF16, 0>() && ((uintptr_t)ep.res % 16) == 0 && ep.ldr % 8 == 0 &&
        ep.res_rows < (1ll << 31) && (ep.res_rows >= gp.M || ep.res_rows % 32 == 0))
        tp.res_tma = gemm_make_map(&tp.rmap, ep.res, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, ep.res_rows, gp.N, ep.ldr, 32, 32,
                                   CU_TENSOR_MAP_SWIZZLE_64B)
                         ? 1
                         : 0;
    if (WRES) {
        if (nseg != 1) return cudaErrorInvalidValue;
        tp.wres_bytes = ((tp.seg[0].klen + BK - 1) / BK) * Smem<BN, AF16, WRES>::kWtile;
    }
    if (ep.kind == EPI_GELU) {
        cudaError_t e = cudaSuccess;
        tp.gelu_tab = gemm_gelu_table(ep.gelu, ep.m_g, ep.s_g, s, &e);
        if (!tp.gelu_tab) return e != cudaSuccess ? e : cudaErrorUnknown;
    }
    if constexpr (GELU) {
        if constexpr (NB == 1)
            return ep.out_bits == kOutI8InF16 ? launch_tc<BN, STAGES, KIND_GELU_F16, NB, AF16, WRES>(tp, s)
                                              : launch_tc<BN, STAGES, KIND_GELU8, NB, AF16, WRES>(tp, s);
        else
            return cudaErrorInvalidValue;  // split convolutions requantise only
    } else {
        if (ep.out_bits == kOutI8InF16) {
            if constexpr (NB == 1) return launch_tc<BN, STAGES, KIND_F16OUT, NB, AF16, WRES>(tp, s);
            else return cudaErrorInvalidValue;
        }
        if constexpr (BN == 128 && NB == 1 && AF16 && !WRES) {  // two column parts: see epi_parts
            if (nseg > 2) tp.res_tma = 0;
            if (ep.out_bits == 8 && (ep.res || nseg > 2)) return launch_tc<BN, STAGES, KIND_RQ8, NB, AF16, WRES, 2>(tp, s);
            if (ep.out_bits == 16 && !tp.res_tma) return launch_tc<BN, STAGES, KIND_RQ16, NB, AF16, WRES, 2>(tp, s);
        }
        if (ep.out_bits == 8) return launch_tc<BN, STAGES, KIND_RQ8, NB, AF16, WRES>(tp, s);
        if (ep.out_bits == 16) return launch_tc<BN, STAGES, KIND_RQ16, NB, AF16, WRES>(tp, s);
        return launch_tc<BN, STAGES, KIND_RAW32, NB, AF16, WRES, BN == 128 && NB == 1 && AF16 ? 2 : 0>(tp, s);  // (two column parts: see epi_parts)
    }
}

}  // namespace
}  // namespace ilw
