// bsm_kernels.cu -- the persistent batched-softmax kernel for sm_103a.
//
// One CTA per SM.  Warp 16 is the producer: one lane pulls the next patch
// (Sec. 4: a block of rows of one slice) from the schedule -- a static list
// for the Sec. 3 baselines, or the CTA's die queue for Cluster Beamforming
// (Sec. 4.1) with stealing after the Sec. 4.2 balance -- and streams the
// patch's contiguous bytes into a ring of shared-memory stages with one 1-D
// TMA bulk copy (cp.async.bulk, completion counted on an mbarrier).  Warps
// 0..15 are consumers: they wait on a stage's "full" barrier, compute the
// softmax of its rows out of shared memory, store y with 128-bit coalesced
// stores, and release the stage on its "empty" barrier.  The patch geometry
// travels with the stage (the "templated kernel fed patch coordinates from a
// queue" of Sec. 5).
//
// Row routine (the arithmetic, identical under every policy): a row is owned
// by a group of T lanes; lane l owns the 16-byte vectors l, l + T, l + 2T, ...
// The maximum is exact; the sum is per vector (a balanced tree), per lane in
// vector order, then a butterfly (xor) shuffle tree over the group.  By row
// length in 16-byte vectors: 1: T = 1, 1 vector per lane; 2: T = 1, 2; <= 4:
// T = 2, 2; <= 8: T = 4, 2; <= 16: T = 8, 2; <= 32: T = 8, 3 or 4; <= 64:
// T = 16, 3 or 4; <= 128: T = 32, 3 or 4 -- all in registers (see
// rows_in_lanes); longer rows: a team of 1 to 16 warps, up to 8 vectors per
// lane in registers (see row_team).  exp(t) is evaluated as 2^(t*log2 e) with
// the exponent formed by one fused multiply-add, v*log2e - offset, and the
// power of two from the PTX ex2.approx instruction; y = p * (1/sum).
//
// Every wait is bounded (2 s of wall time unless the launch asks for less):
// on expiry the CTA
// records BSM_DEV_TIMEOUT in the status word, lets its copies in flight land,
// and returns.

#include <cuda_runtime.h>
#include <cstdint>

#include "bsm_internal.h"

namespace bsm {
namespace {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s
constexpr uint32_t kClaimAhead = 2;                 // rows a group's rank 0 announces ahead
constexpr float kLog2e = 1.4426950408889634f;

// Teams of consumer warps that share a row: 8 of 2 warps, 4 of 4, 2 of 8, or
// all 16 (whose barrier is xwarp).
constexpr int kTeamBars = 14;
constexpr int kTeamVecs = 8;        // 16-byte vectors a lane holds in registers

enum : int32_t { KIND_DATA = 0, KIND_SKIP = 1, KIND_DONE = 2, KIND_LONG = 3, KIND_GROUP = 4 };

struct alignas(16) StageMeta {
    int64_t off;
    int32_t C;          // KIND_LONG: elements of this chunk of the row
    int32_t nrows;
    int32_t row0;
    int32_t kind;
    int32_t R;
    int32_t col0;       // KIND_LONG: column of the chunk's first element
    int32_t pass;       // KIND_LONG: 0 = partial of the segment, 1 = combine and write
    int32_t last;       // KIND_LONG: last chunk of the segment
    int32_t first;      // KIND_LONG: first chunk of the segment
    int32_t part;       // KIND_LONG: the segment's partial slot
    int32_t part_first; // KIND_LONG: the row's first partial slot
    int32_t part_count; // KIND_LONG: the row's number of segments
    int32_t resident;   // KIND_LONG: the whole row stays staged for its second pass
    int32_t pad;
};
static_assert(sizeof(StageMeta) == 64, "StageMeta layout");

struct SmemHeader {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t xwarp;                 // long rows, rows on 16 warps: the warps' partials are in
    union {
        uint64_t team[kTeamBars];   // rows shared by a team of warps: its partials are in
        struct {                    // rows over groups:
            uint64_t xres[2];       // a row's result is in, by row parity
            float2 result[2];       // ... its (offset, sum)
            uint32_t xarrive[2];    // warps whose partial is in, by row parity
            uint32_t xleft;         // consumer warps that have left
        };
    };
    int32_t abort_flag;
    StageMeta meta[kMaxStages];
    float2 partial[2][kConsumerWarps];   // (offset, sum) per warp of a row they share, two rows deep
};
static_assert(sizeof(SmemHeader) <= kSmemHeader, "header too large");

// ---------------------------------------------------------------- PTX helpers

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_timer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t sm_id()
{
    uint32_t s;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(s));
    return s;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// One potentially blocking test of the phase: a waiting thread is suspended
// in hardware (it issues nothing) until the phase completes or kSuspendNs
// pass, so idle warps do not take issue slots from the working ones.
constexpr uint32_t kSuspendNs = 50000;

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}

// Wait until the phase with the given parity of `bar` has completed.  Gives
// up (returns false) when *abort becomes non-zero (if abort != nullptr) or
// after limit_ns.
__device__ __noinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                               const volatile int32_t *abort, uint64_t limit_ns)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 0; it < (1u << 28); ++it) {
        if (mbar_try_wait(bar, parity))
            return true;
        {
            if (abort && *abort)
                return false;
            if (global_timer_ns() - t0 > limit_ns)
                return false;
        }
    }
    return false;
}

// The same wait without the call and without sleeping: for the short waits of
// warps that share a row, which they hold in registers across it (a call
// would spill them).  The clock is read once in 1024 polls.
__device__ __forceinline__ bool mbar_spin_bounded(uint64_t *bar, uint32_t parity, const volatile int32_t *abort,
                                                  uint64_t limit_ns)
{
    uint64_t t0 = 0;
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok)
            return true;
        if ((it & 1023u) == 1023u) {
            const uint64_t t = global_timer_ns();
            t0 = t0 ? t0 : t;
            if (*abort || t - t0 > limit_ns)
                return false;
        }
    }
    return false;
}

// 1-D bulk copy global -> shared, completion counted (bytes) on `bar`.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Stage reads are explicit shared-space accesses (a
// 32-bit shared address), so they are issued as shared loads whatever
// the compiler can infer about the pointer; volatile keeps them on their side
// of the barrier waits.
__device__ __forceinline__ uint4 lds128(const unsigned char *p)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(smem_addr(p)));
    return v;
}

// Output stores: plain 128-bit global stores.
__device__ __forceinline__ void stg128(void *p, uint4 v)
{
    *reinterpret_cast<uint4 *>(p) = v;
}

// ---------------------------------------------------------- self-checks
// The checking instantiation (Checked = true) verifies every shared-memory
// read, global store and bulk copy against the stage and buffer extents; a
// violation is recorded (BSM_DEV_CHECK, plus the first one's details in words
// 1..7 of the status block) and the access is skipped.

struct Bounds {
    const unsigned char *s_lo, *s_hi;   // bytes of the current stage that hold the patch
    const unsigned char *y_lo, *y_hi;   // the output buffer
    uint32_t *status;
};

__device__ __noinline__ void check_fail(uint32_t *status, uint32_t kind, uint64_t a, uint64_t b)
{
    atomicOr(status, BSM_DEV_CHECK);
    if (atomicCAS(&status[1], 0u, kind) == 0u) {
        status[2] = blockIdx.x;
        status[3] = threadIdx.x;
        status[4] = static_cast<uint32_t>(a);
        status[5] = static_cast<uint32_t>(a >> 32);
        status[6] = static_cast<uint32_t>(b);
        status[7] = static_cast<uint32_t>(b >> 32);
    }
}

template <bool Checked>
__device__ __forceinline__ bool load_vec(const unsigned char *p, const Bounds &b, uint4 &out)
{
    if (Checked && (p < b.s_lo || p + 16 > b.s_hi || (reinterpret_cast<uintptr_t>(p) & 15))) {
        check_fail(b.status, 1, static_cast<uint64_t>(p - b.s_lo), static_cast<uint64_t>(b.s_hi - b.s_lo));
        return false;
    }
    out = lds128(p);
    return true;
}

template <bool Checked>
__device__ __forceinline__ void store_vec(unsigned char *p, const Bounds &b, uint4 v)
{
    if (Checked && (p < b.y_lo || p + 16 > b.y_hi || (reinterpret_cast<uintptr_t>(p) & 15))) {
        check_fail(b.status, 2, static_cast<uint64_t>(p - b.y_lo), static_cast<uint64_t>(b.y_hi - b.y_lo));
        return;
    }
    stg128(p, v);
}

__device__ __forceinline__ float ex2(float a)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// ------------------------------------------------------- element-type traits

template <typename Tag> struct Elem;
struct F32 {};
struct BF16 {};

template <> struct Elem<F32> {
    static constexpr int kSize = 4;
    static constexpr int kPerVec = 4;
    __device__ static __forceinline__ void unpack(uint4 r, float (&v)[4])
    {
        v[0] = __uint_as_float(r.x);
        v[1] = __uint_as_float(r.y);
        v[2] = __uint_as_float(r.z);
        v[3] = __uint_as_float(r.w);
    }
    __device__ static __forceinline__ uint4 pack(const float (&v)[4])
    {
        return make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]),
                          __float_as_uint(v[3]));
    }
    // a vector of -inf (stands in for vectors past the end of a row)
    __device__ static __forceinline__ uint4 neg_inf_vec() { return make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u); }
};

template <> struct Elem<BF16> {
    static constexpr int kSize = 2;
    static constexpr int kPerVec = 8;
    __device__ static __forceinline__ void unpack(uint4 r, float (&v)[8])
    {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = __uint_as_float(w[k] << 16);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
    __device__ static __forceinline__ uint4 pack(const float (&v)[8])
    {
        return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                          pack_bf16x2(v[6], v[7]));
    }
    __device__ static __forceinline__ uint4 neg_inf_vec() { return make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u); }
};

// ------------------------------------------------------------- row routines

template <int T> __device__ __forceinline__ float group_max(float m)
{
#pragma unroll
    for (int o = T / 2; o >= 1; o >>= 1)
        m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    return m;
}

template <int T> __device__ __forceinline__ float group_sum(float s)
{
#pragma unroll
    for (int o = T / 2; o >= 1; o >>= 1)
        s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

// Maximum / sum of the N elements of one vector as a balanced tree (fixed
// order: the sum's rounding is the same wherever the row runs).
template <int N> __device__ __forceinline__ float tree_max(const float *v)
{
    if constexpr (N == 1)
        return v[0];
    else
        return fmaxf(tree_max<N / 2>(v), tree_max<N / 2>(v + N / 2));
}

template <int N> __device__ __forceinline__ float tree_sum(const float *v)
{
    if constexpr (N == 1)
        return v[0];
    else
        return tree_sum<N / 2>(v) + tree_sum<N / 2>(v + N / 2);
}

// p = exp(v - m) for one vector, as 2^(v*log2e - m*log2e).  For a vector
// lying wholly above the causal diagonal (v is x, or x + (-inf)) the formula
// gives 0 where x is finite or -inf and NaN where x is NaN or +inf; that is
// computed without the exponential.
template <int EPV>
__device__ __forceinline__ void vec_exp(float (&v)[EPV], float mL, bool masked)
{
    if (masked) {
#pragma unroll
        for (int e = 0; e < EPV; ++e)
            v[e] = v[e] < INFINITY ? 0.0f : __int_as_float(0x7FC00000);
    } else {
#pragma unroll
        for (int e = 0; e < EPV; ++e)
            v[e] = ex2(fmaf(v[e], kLog2e, -mL));
    }
}

// Additive causal mask of one 16-byte vector: element c of the row gets -inf
// when c > row.
template <int EPV>
__device__ __forceinline__ void apply_causal(float (&v)[EPV], int col0, int row)
{
#pragma unroll
    for (int e = 0; e < EPV; ++e)
        v[e] += (col0 + e > row) ? -INFINITY : 0.0f;
}

// ------------------------------------------------ fp32 pair arithmetic
// One instruction, two IEEE operations, each rounded like its scalar form.
// As 64-bit registers (Pair): a constant pair is made once, not at each use.
typedef unsigned long long Pair;

__device__ __forceinline__ Pair pair(float lo, float hi)
{
    Pair d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

__device__ __forceinline__ float2 halves(Pair p)
{
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(p));
    return d;
}

__device__ __forceinline__ Pair pair_fma(Pair a, Pair b, Pair c)
{
    Pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ Pair pair_add(Pair a, Pair b)
{
    Pair d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ Pair pair_mul(Pair a, Pair b)
{
    Pair d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// Element-wise maximum of two bf16 pairs.
__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// p = 2^(v*log2e - mL) for one vector in fp32 pairs (each pair two IEEE
// fmas: the bits of vec_exp), and the vector's sum in tree_sum's order
// ((p0 + p1) + (p2 + p3), and so on).
template <int EPV>
__device__ __forceinline__ float vec_exp_sum_pairs(float (&v)[EPV], float mL)
{
    const float2 l2 = make_float2(kLog2e, kLog2e), nm = make_float2(-mL, -mL);
#pragma unroll
    for (int e = 0; e < EPV; e += 2) {
        const float2 t = fma2(make_float2(v[e], v[e + 1]), l2, nm);
        v[e] = ex2(t.x);
        v[e + 1] = ex2(t.y);
    }
    if constexpr (EPV == 4) {
        const float2 a = add2(make_float2(v[0], v[2]), make_float2(v[1], v[3]));
        return a.x + a.y;
    } else {
        const float2 a = add2(make_float2(v[0], v[4]), make_float2(v[1], v[5]));
        const float2 b = add2(make_float2(v[2], v[6]), make_float2(v[3], v[7]));
        const float2 c = add2(a, b);
        return c.x + c.y;
    }
}

// The additive causal mask on a vector as loaded: x + (-inf) past the
// diagonal (-inf, or NaN where x is NaN or +inf), x + (-0) = x elsewhere --
// exact in the element type, so that what follows needs no mask.
template <typename Tag> __device__ __forceinline__ uint4 mask_vec(uint4 r, int col0, int row);
template <> __device__ __forceinline__ uint4 mask_vec<F32>(uint4 r, int col0, int row)
{
    if (col0 + 3 > row) {
        r.x = __float_as_uint(__uint_as_float(r.x) + (col0 > row ? -INFINITY : -0.0f));
        r.y = __float_as_uint(__uint_as_float(r.y) + (col0 + 1 > row ? -INFINITY : -0.0f));
        r.z = __float_as_uint(__uint_as_float(r.z) + (col0 + 2 > row ? -INFINITY : -0.0f));
        r.w = __float_as_uint(__uint_as_float(r.w) + (col0 + 3 > row ? -INFINITY : -0.0f));
    }
    return r;
}
template <> __device__ __forceinline__ uint4 mask_vec<BF16>(uint4 r, int col0, int row)
{
    if (col0 + 7 > row) {
        uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t add = (col0 + 2 * k > row ? 0xFF80u : 0x8000u) |
                                 (col0 + 2 * k + 1 > row ? 0xFF800000u : 0x80000000u);
            asm("add.rn.bf16x2 %0, %0, %1;" : "+r"(w[k]) : "r"(add));
        }
        r = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return r;
}

// Running maximum of a lane's vectors, NaN operands ignored: bf16 on the
// packed words (exact), two halves; fp32 as a scalar.
template <typename Tag> struct MaxAcc;
template <> struct MaxAcc<F32> {
    float m = -INFINITY;
    __device__ __forceinline__ void add(uint4 r)
    {
        m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(r.x), __uint_as_float(r.y)),
                           fmaxf(__uint_as_float(r.z), __uint_as_float(r.w))));
    }
    __device__ __forceinline__ float get() const { return m; }
};
template <> struct MaxAcc<BF16> {
    uint32_t w = 0xFF80FF80u;
    __device__ __forceinline__ void add(uint4 r) { w = bmax2(w, bmax2(bmax2(r.x, r.y), bmax2(r.z, r.w))); }
    __device__ __forceinline__ float get() const
    {
        return fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
    }
};

// The exponents' offset for a maximum m: m * log2 e rounded down to a whole
// number, no lower than the lowest float.  Whole: then sums taken with
// different offsets are brought together by powers of two, without rounding.
// No lower than the lowest float: there (m = -inf, or a mask of the type's
// lowest value in every element seen) v*log2e - offset is -inf or far below 0
// and adds 0 (NaN for a NaN), where m * log2 e = -inf would give inf - inf.
constexpr float kLowest = -3.402823466e38f;
__device__ __forceinline__ float exp_offset(float m) { return fmaxf(floorf(m * kLog2e), kLowest); }

// Half of a partial's (offset o, sum s) as part of a sum of offset O >= o:
// s/2 2^(o - O); the caller doubles the sum of them (exact).  s can be +inf where
// every value a warp saw is a finite mask such as -1e10: where |m log2 e| is
// 2^31 or more its float is off by up to 2^7 or more, and so is the exponent of
// the largest element.  inf * 2^(o - O) = inf * 0 would be NaN, but floats that
// large lie so far apart that under a higher offset the share is below 2^-127
// whatever the finite s: so s/2 is bounded by the largest float (NaN stays NaN).
// Where o = O the doubled sum is +inf, as it would be without the bound.
// Against a test of s and o per partial: 64 KiB bf16 rows 83.5 us, not 84.0.
__device__ __forceinline__ float half_share(float2 p, float O)
{
    float s;
    asm("min.NaN.f32 %0, %1, 0f7F7FFFFF;" : "=f"(s) : "f"(0.5f * p.y));
    return s * ex2(p.x - O);
}

// Element pair k of a vector as loaded.
template <typename Tag> __device__ __forceinline__ Pair vec_pair(uint4 r, int k);
template <> __device__ __forceinline__ Pair vec_pair<F32>(uint4 r, int k)
{
    return k == 0 ? pair(__uint_as_float(r.x), __uint_as_float(r.y)) : pair(__uint_as_float(r.z), __uint_as_float(r.w));
}
template <> __device__ __forceinline__ Pair vec_pair<BF16>(uint4 r, int k)
{
    const uint32_t w = k == 0 ? r.x : k == 1 ? r.y : k == 2 ? r.z : r.w;
    return pair(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}

__device__ __forceinline__ Pair pair_ex2(Pair t)
{
    const float2 f = halves(t);
    return pair(ex2(f.x), ex2(f.y));
}

// acc + the vector's 2^(v*log2e - mL), pair by pair (nm = -mL twice).
template <typename Tag> __device__ __forceinline__ Pair vec_sum(Pair acc, uint4 r, Pair l2, Pair nm)
{
    constexpr int N = Elem<Tag>::kPerVec / 2;
    Pair p[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        p[k] = pair_ex2(pair_fma(vec_pair<Tag>(r, k), l2, nm));
#pragma unroll
    for (int w = 1; w < N; w *= 2)
#pragma unroll
        for (int k = 0; k < N; k += 2 * w)
            p[k] = pair_add(p[k], p[k + w]);
    return pair_add(acc, p[0]);
}

// A vector of the element type from its element pairs.
template <typename Tag> __device__ __forceinline__ uint4 pack_pairs(const float2 *y)
{
    if constexpr (Elem<Tag>::kSize == 4)
        return make_uint4(__float_as_uint(y[0].x), __float_as_uint(y[0].y), __float_as_uint(y[1].x),
                          __float_as_uint(y[1].y));
    else
        return make_uint4(pack_bf16x2(y[0].x, y[0].y), pack_bf16x2(y[1].x, y[1].y), pack_bf16x2(y[2].x, y[2].y),
                          pack_bf16x2(y[3].x, y[3].y));
}

// 2^(v*log2e - mL) * inv of one vector, packed.
template <typename Tag> __device__ __forceinline__ uint4 vec_softmax(uint4 r, Pair l2, Pair nm, Pair inv2)
{
    constexpr int N = Elem<Tag>::kPerVec / 2;
    float2 y[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        y[k] = halves(pair_mul(pair_ex2(pair_fma(vec_pair<Tag>(r, k), l2, nm)), inv2));
    return pack_pairs<Tag>(y);
}

// Maximum over the warp, in every lane (no operand is NaN: see MaxAcc).
__device__ __forceinline__ float warp_max(float m)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(m));
    return r;
}

// A row shared by a team of W consumer warps (wi = this warp's index in it;
// W = 1, 2, 4, 8 or 16): lane l of warp wi owns the vectors wi*32 + l, + 32 W,
// ..., V of them in registers (the first Full exist in every lane; 8 hold the
// whole row up to W * 4 KiB), further ones (rows of 64 to 113 KiB on 16 warps)
// read again from the stage by each sweep.  W and V are compile-time, so that
// no address outlives its use.  A warp takes its maximum's offset o_w (see
// exp_offset) and s_w, the sum of 2^(v log2 e - o_w); exchange() turns the pair
// into the row's: O = max o_w and S = sum s_w 2^(o_w - O), in a fixed tree, the
// same in every warp; the warp writes 2^(v log2 e - O) / S.  (Exchanging the
// maxima themselves cost accuracy: the rounding of m log2 e then differs from
// warp to warp; 1.0e-7 against 7.2e-8 on a ragged fp32 batch.)  Two
// exponentials per element, one exchange per row.  All in fp32; which warps
// share a row depends on its length only.
//
// release() is called once the warp needs the stage no more; returns false
// when the exchange's wait gave up.
template <typename Tag, bool Checked, int W, int V, int Full, typename Exchange, typename Release>
__device__ __forceinline__ bool row_team(const unsigned char *srow, unsigned char *yrow, int nvec, int row,
                                         bool causal, int col0, int wi, int lane, const Bounds &bd,
                                         Exchange &&exchange, Release &&release)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec;
    constexpr int step = W * 32;
    const int t0 = wi * 32 + lane;
    const bool tail = W == 16 && V == kTeamVecs && nvec > V * step;
    auto fetch = [&](int vi, bool in) -> uint4 {
        uint4 r = E::neg_inf_vec();
        if (in) {
            uint4 u;
            if (load_vec<Checked>(srow + 16 * vi, bd, u))
                r = u;
        }
        return r;
    };
    uint4 r[V];
#pragma unroll
    for (int j = 0; j < V; ++j)
        r[j] = fetch(t0 + j * step, j < Full || t0 + j * step < nvec);
    if (causal) {
#pragma unroll
        for (int j = 0; j < V; ++j)
            r[j] = mask_vec<Tag>(r[j], col0 + (t0 + j * step) * EPV, row);
    }
    auto fetch_tail = [&](int vi) -> uint4 {
        const uint4 u = fetch(vi, true);
        return causal ? mask_vec<Tag>(u, col0 + vi * EPV, row) : u;
    };
    MaxAcc<Tag> mx;
#pragma unroll
    for (int j = 0; j < V; ++j)
        mx.add(r[j]);
    if (tail)
        for (int vi = t0 + V * step; vi < nvec; vi += step)
            mx.add(fetch_tail(vi));
    else
        release();
    const float mL = exp_offset(warp_max(mx.get()));
    const Pair l2 = pair(kLog2e, kLog2e);
    Pair nm = pair(-mL, -mL), acc = pair(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < V; ++j)
        acc = vec_sum<Tag>(acc, r[j], l2, nm);
    if (tail)
        for (int vi = t0 + V * step; vi < nvec; vi += step)
            acc = vec_sum<Tag>(acc, fetch_tail(vi), l2, nm);
    const float2 a2 = halves(acc);
    float2 os = make_float2(mL, group_sum<32>(a2.x + a2.y));
    if (!exchange(os))
        return false;
    nm = pair(-os.x, -os.x);
    const float s = os.y;
    const float inv = __frcp_rn(s);
    const Pair inv2 = pair(inv, inv);
    // the write unpacks the vectors again: kept unpacked from the sum on, they
    // would take twice the registers (bf16) and spill
#pragma unroll
    for (int j = 0; j < V; ++j)
        asm volatile("" : "+r"(r[j].x), "+r"(r[j].y), "+r"(r[j].z), "+r"(r[j].w));
    unsigned char *yp = yrow + 16 * t0;
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (j < Full || t0 + j * step < nvec)
            store_vec<Checked>(yp + 16 * j * step, bd, vec_softmax<Tag>(r[j], l2, nm, inv2));
    }
    if (tail) {
        for (int vi = t0 + V * step; vi < nvec; vi += step)
            store_vec<Checked>(yrow + 16 * vi, bd, vec_softmax<Tag>(fetch_tail(vi), l2, nm, inv2));
        release();
    }
    return true;
}

template <int N> struct Int {
    static constexpr int value = N;
};

// ------------------------------------------------ backward row routines
// dx = y * (dy - <y, dy>) of one row; y and dy sit in the two halves of the
// stage.

// The products of one vector of y and of dy, added to a running pair (as a
// tree first: the running sum is rounded once a vector).
template <typename Tag> __device__ __forceinline__ Pair add_products(Pair acc, uint4 a, uint4 b)
{
    Pair t = pair_fma(vec_pair<Tag>(a, 1), vec_pair<Tag>(b, 1), pair_mul(vec_pair<Tag>(a, 0), vec_pair<Tag>(b, 0)));
    if constexpr (Elem<Tag>::kPerVec == 8)
        t = pair_add(t, pair_fma(vec_pair<Tag>(a, 3), vec_pair<Tag>(b, 3),
                                 pair_mul(vec_pair<Tag>(a, 2), vec_pair<Tag>(b, 2))));
    return pair_add(acc, t);
}

// y * (dy - dot) of one vector (nd = -dot, twice).
template <typename Tag> __device__ __forceinline__ uint4 vec_dx(uint4 a, uint4 b, Pair nd)
{
    constexpr int N = Elem<Tag>::kPerVec / 2;
    float2 o[N];
#pragma unroll
    for (int k = 0; k < N; ++k)
        o[k] = halves(pair_mul(vec_pair<Tag>(a, k), pair_add(vec_pair<Tag>(b, k), nd)));
    return pack_pairs<Tag>(o);
}

// A longer row, shared by a team of W warps as in row_team: the vectors wi*32
// + l, + 32 W, ... of y and of dy, four of each in registers (the last two can
// be missing in some lanes; the whole row up to W * 2 KiB), further ones (rows
// of 32 to 56 KiB on 16 warps, of 2 to 3 KiB on one) read again from the
// stage.  The warps' dot products are exchanged once and added in a fixed tree.
constexpr int kTeamVecsBwd = 4;

template <typename Tag, bool Checked, int W, int Full, typename Exchange, typename Release>
__device__ __forceinline__ bool row_team_bwd(const unsigned char *sy, const unsigned char *sdy, unsigned char *dxrow,
                                             int nvec, int wi, int lane, const Bounds &by, const Bounds &bdy,
                                             Exchange &&exchange, Release &&release)
{
    constexpr int V = kTeamVecsBwd, step = W * 32;
    const int t0 = wi * 32 + lane;
    const bool tail = (W == 1 || W == 16) && nvec > V * step;
    auto fetch = [&](const unsigned char *src, int vi, bool in, const Bounds &b) -> uint4 {
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (in) {
            uint4 u;
            if (load_vec<Checked>(src + 16 * vi, b, u))
                r = u;
        }
        return r;
    };
    uint4 yv[V], dv[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const int vi = t0 + j * step;
        const bool in = j < Full || vi < nvec;
        yv[j] = fetch(sy, vi, in, by);
        dv[j] = fetch(sdy, vi, in, bdy);
    }
    Pair acc = pair(0.0f, 0.0f), acc2 = acc;
#pragma unroll
    for (int j = 0; j < V; j += 2) {
        acc = add_products<Tag>(acc, yv[j], dv[j]);
        acc2 = add_products<Tag>(acc2, yv[j + 1], dv[j + 1]);
    }
    if (tail) {
        for (int vi = t0 + V * step; vi < nvec; vi += step)
            acc = add_products<Tag>(acc, fetch(sy, vi, true, by), fetch(sdy, vi, true, bdy));
    } else {
        release();
    }
    const float2 a2 = halves(pair_add(acc, acc2));
    float dot = group_sum<32>(a2.x + a2.y);
    if (!exchange(dot))
        return false;
    const Pair nd = pair(-dot, -dot);
    // (unpacked again for the write, as in row_team)
#pragma unroll
    for (int j = 0; j < V; ++j) {
        asm volatile("" : "+r"(yv[j].x), "+r"(yv[j].y), "+r"(yv[j].z), "+r"(yv[j].w));
        asm volatile("" : "+r"(dv[j].x), "+r"(dv[j].y), "+r"(dv[j].z), "+r"(dv[j].w));
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
        const int vi = t0 + j * step;
        if (j < Full || vi < nvec)
            store_vec<Checked>(dxrow + 16 * vi, by, vec_dx<Tag>(yv[j], dv[j], nd));
    }
    if (tail) {
        for (int vi = t0 + V * step; vi < nvec; vi += step)
            store_vec<Checked>(dxrow + 16 * vi, by, vec_dx<Tag>(fetch(sy, vi, true, by), fetch(sdy, vi, true, bdy), nd));
        release();
    }
    return true;
}

// Backward rows that one lane group's registers hold, as rows_in_lanes: T
// lanes, V vectors of y and of dy a lane, of which only the last can be
// missing (0: it adds nothing), no other bound.  More than 16 vectors take
// 16 or 32 lanes of two: four of each a lane spill.  GB/s over 512 MiB of y and
// dy, 8 to 32 lanes with a bound on every vector -> this routine: bf16 16 B
// 1845 -> 7092, 32 B 3492 -> 7053, 64 B 6195 -> 7105, 528 B 6833 -> 7054, longer
// ones as before (7.0 to 7.1 TB/s); fp32 16 B 2523 -> 7077, 32 B 4680 -> 7050,
// 48 B 6280 -> 7082.
template <typename Tag, bool Checked, int T, int V>
__device__ __forceinline__ int rows_bwd_in_lanes(const unsigned char *sbuf, int half, const StageMeta &mt,
                                                 unsigned char *ybase, int row_bytes, int nvec, int first,
                                                 int lane, const Bounds &by, const Bounds &bdy)
{
    constexpr int G = 32 / T;
    const int g = lane / T, l = lane % T;
    const bool in_last = (V - 1) * T + l < nvec;
    for (int rb = first * G; rb < mt.nrows; rb += G * kConsumerWarps) {
        const int r = rb + g;
        const bool valid = r < mt.nrows;
        const unsigned char *sy = sbuf + (size_t)(valid ? r : mt.nrows - 1) * row_bytes + 16 * l;
        uint4 yv[V], dv[V];
        Pair acc = pair(0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            yv[j] = dv[j] = make_uint4(0u, 0u, 0u, 0u);
            uint4 a, b;
            if ((j < V - 1 || in_last) && load_vec<Checked>(sy + 16 * j * T, by, a) &&
                load_vec<Checked>(sy + half + 16 * j * T, bdy, b)) {
                yv[j] = a;
                dv[j] = b;
            }
        }
#pragma unroll
        for (int j = 0; j < V; ++j)
            acc = add_products<Tag>(acc, yv[j], dv[j]);
        const float2 a2 = halves(acc);
        const float dot = group_sum<T>(a2.x + a2.y);
        const Pair nd = pair(-dot, -dot);
        // (unpacked again for the write, as in row_team)
#pragma unroll
        for (int j = 0; j < V; ++j) {
            asm volatile("" : "+r"(yv[j].x), "+r"(yv[j].y), "+r"(yv[j].z), "+r"(yv[j].w));
            asm volatile("" : "+r"(dv[j].x), "+r"(dv[j].y), "+r"(dv[j].z), "+r"(dv[j].w));
        }
        unsigned char *dx = ybase + (size_t)r * row_bytes + 16 * l;
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (valid && (j < V - 1 || in_last))
                store_vec<Checked>(dx + 16 * j * T, by, vec_dx<Tag>(yv[j], dv[j], nd));
    }
    return (mt.nrows + G - 1) / G;
}

template <typename Tag, bool Checked>
__device__ __forceinline__ int consume_stage_bwd(const unsigned char *sbuf, int half, const StageMeta &mt,
                                                 unsigned char *y, int first, int lane, Bounds by)
{
    using E = Elem<Tag>;
    const int row_bytes = mt.C * E::kSize;
    const int nvec = row_bytes >> 4;
    unsigned char *ybase = y + mt.off * E::kSize;
    by.s_lo = sbuf;
    by.s_hi = sbuf + (size_t)mt.nrows * row_bytes;
    Bounds bdy = by;
    bdy.s_lo = sbuf + half;
    bdy.s_hi = sbuf + half + (size_t)mt.nrows * row_bytes;
    auto rows = [&](auto t, auto v) {
        return rows_bwd_in_lanes<Tag, Checked, decltype(t)::value, decltype(v)::value>(
            sbuf, half, mt, ybase, row_bytes, nvec, first, lane, by, bdy);
    };
    if (nvec <= 8)
        return nvec > 4    ? rows(Int<4>{}, Int<2>{})
               : nvec > 2  ? rows(Int<2>{}, Int<2>{})
               : nvec == 2 ? rows(Int<1>{}, Int<2>{})
                           : rows(Int<1>{}, Int<1>{});
    if (nvec <= 32)
        return nvec > 16 ? rows(Int<16>{}, Int<2>{}) : rows(Int<8>{}, Int<2>{});
    if (E::kSize == 2 || nvec <= 64)   // (bf16 rows of more than 64 vectors go to teams)
        return rows(Int<32>{}, Int<2>{});
    return nvec > 96 ? rows(Int<32>{}, Int<4>{}) : rows(Int<32>{}, Int<3>{});
}

// ------------------------------------------------------------ long rows
// A row longer than a stage is streamed through the stages twice, in
// chunks of equal length; all consumer warps share every chunk (warp w takes
// the vectors w*32 + lane, + 512, ...).  Pass 0 keeps a running (max m, sum s
// of exp(v - m)) per lane -- when the max grows, s is rescaled by exp(m_old -
// m_new) -- then the lanes, the warps (through shared memory) combine their
// pairs in a fixed order; pass 1 writes exp(v - m) / s.  For a whole row in
// one launch, pass 1 starts on the last chunk, still in its stage, and takes
// the others in reverse order.

// The exponents' offset of the streamed rows: m * log2 e itself, no lower than the
// lowest float (see exp_offset; for a mask of the type's lowest value it would be
// -inf, and a -inf beside it NaN).
__device__ __forceinline__ float long_offset(float m) { return fmaxf(m * kLog2e, kLowest); }

// A sum s of 2^((v - m) log2 e) once a value above m is the maximum: one that
// overflowed counts nothing.  It does where m is a finite mask such as -1e10 (see
// half_share), and inf * 2^(far below 0) would be NaN.
__device__ __forceinline__ float finite_or_none(float s) { return s == INFINITY ? 0.0f : s; }

// A sum s of maximum m as part of one of maximum M >= m.
__device__ __forceinline__ float ms_share(float m, float s, float M)
{
    return m == M ? s : finite_or_none(s) * ex2((m - M) * kLog2e);
}

// The (maximum, sum) of one pair per lane (-inf, 0 adds nothing), in every lane:
// a fixed tree.
__device__ __forceinline__ float2 lanes_ms(float m, float s)
{
    const float M = warp_max(m);
    return make_float2(M, group_sum<32>(ms_share(m, s, M)));
}

template <typename Tag, bool Checked>
__device__ __forceinline__ void long_chunk(const unsigned char *sbuf, const StageMeta &mt, unsigned char *y,
                                           bool causal, int warp, int lane, Bounds bd, float &m_l,
                                           float &s_l, float mL, float inv)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec;
    const int nvec = (mt.C * E::kSize) >> 4;
    bd.s_lo = sbuf;
    bd.s_hi = sbuf + (size_t)mt.C * E::kSize;
    unsigned char *ybase = y + mt.off * E::kSize;
    const int row = mt.row0;
    for (int vi = warp * 32 + lane; vi < nvec; vi += kConsumerWarps * 32) {
        uint4 raw;
        if (!load_vec<Checked>(sbuf + 16 * vi, bd, raw))
            continue;
        float v[EPV];
        E::unpack(raw, v);
        const int col = mt.col0 + vi * EPV;
        const bool masked = causal && col > row;
        if (causal && !masked && col + EPV - 1 > row)
            apply_causal<EPV>(v, col, row);
        if (mt.pass == 0) {
            if (!masked) {
                const float vm = tree_max<EPV>(v);
                if (vm > m_l) {
                    s_l = finite_or_none(s_l) * ex2((m_l - vm) * kLog2e);
                    m_l = vm;
                }
            }
            // the exponentials in fp32 pairs (the same bits as one at a time);
            // while the running max is still -inf every value seen is -inf (or
            // NaN) and adds 0 (NaN), as a masked vector does
            if (masked) {
                vec_exp<EPV>(v, 0.0f, true);
                s_l += tree_sum<EPV>(v);
            } else {
                s_l += vec_exp_sum_pairs<EPV>(v, long_offset(m_l));
            }
        } else {
            vec_exp<EPV>(v, mL, masked);
#pragma unroll
            for (int e = 0; e < EPV; ++e)
                v[e] *= inv;
            store_vec<Checked>(ybase + 16 * vi, bd, E::pack(v));
        }
    }
}

// Backward long rows: y and dy of a chunk sit in the two halves of a stage.
// Pass 0 adds this lane's y*dy products to dot_l (its vectors in order, chunk
// after chunk); pass 1 writes dx = y * (dy - dot).
template <typename Tag, bool Checked>
__device__ __forceinline__ void long_chunk_bwd(const unsigned char *sbuf, int half, const StageMeta &mt,
                                               unsigned char *dx, int warp, int lane, Bounds by, float &dot_l,
                                               float dot)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec;
    const int nvec = (mt.C * E::kSize) >> 4;
    by.s_lo = sbuf;
    by.s_hi = sbuf + (size_t)mt.C * E::kSize;
    Bounds bdy = by;
    bdy.s_lo = sbuf + half;
    bdy.s_hi = sbuf + half + (size_t)mt.C * E::kSize;
    unsigned char *base = dx + mt.off * E::kSize;
    for (int vi = warp * 32 + lane; vi < nvec; vi += kConsumerWarps * 32) {
        uint4 ry, rd;
        if (!load_vec<Checked>(sbuf + 16 * vi, by, ry) || !load_vec<Checked>(sbuf + half + 16 * vi, bdy, rd))
            continue;
        float yv[EPV], dv[EPV];
        E::unpack(ry, yv);
        E::unpack(rd, dv);
        if (mt.pass == 0) {
#pragma unroll
            for (int e = 0; e < EPV; ++e)
                yv[e] *= dv[e];
            dot_l += tree_sum<EPV>(yv);
        } else {
#pragma unroll
            for (int e = 0; e < EPV; ++e)
                yv[e] = yv[e] * (dv[e] - dot);
            store_vec<Checked>(base + 16 * vi, by, E::pack(yv));
        }
    }
}

// Warps that share a row: the fewest whose registers hold it.
__device__ __forceinline__ int team_warps(int nvec)
{
    return nvec <= 256 ? 1 : nvec <= 512 ? 2 : nvec <= 1024 ? 4 : nvec <= 2048 ? 8 : 16;
}

// Backward: half as many vectors of each of y and dy fit, but a warp by itself
// takes rows of up to 192 vectors (64 of them read from the stage twice: bf16
// rows of 2064 bytes 7080 GB/s, on two warps 6634).
__device__ __forceinline__ int team_warps_bwd(int nvec) { return nvec <= 192 ? 1 : team_warps(2 * nvec); }

// The barrier of a team (teams of one warp use none).
__device__ __forceinline__ uint64_t *team_bar(SmemHeader &h, int W, int team)
{
    return W == 16 ? &h.xwarp : &h.team[(W == 8 ? 12 : W == 4 ? 8 : 0) + (W == 1 ? 0 : team)];
}

// A consumer warp's view of the exchanges it took part in: bit W (2, 4, 8, 16)
// is the phase of its team of W (16: xwarp, long rows too), which is also
// the half of SmemHeader::partial that the next one uses; the bits from
// kTeamLast on hold the W of the last one.
constexpr uint32_t kTeamLast = 8;

// Rows of different team sizes share the partials' slots: before the size
// changes, all consumer warps meet, so that none still reads the other
// size's.  (Every warp sees the same stages, hence the same changes.)
__device__ __forceinline__ bool team_switch(SmemHeader &h, uint32_t W, int lane, uint64_t limit_ns, uint32_t &xs)
{
    const uint32_t was = xs >> kTeamLast;
    if (was == W)
        return true;
    xs = (xs & 0xFFu) | (W << kTeamLast);
    if (was == 0)
        return true;
    __syncwarp();
    if (lane == 0)
        mbar_arrive(&h.xwarp);
    const bool ok = mbar_spin_bounded(&h.xwarp, (xs >> 4) & 1u, &h.abort_flag, limit_ns);
    xs ^= 16u;
    return __all_sync(0xFFFFFFFFu, ok);
}

// The rows of one stage that teams of W warps share (see row_team), those of
// this warp, dealt to the teams round robin after the `seen` warps' worth of
// rows before.  Returns false when a wait gave up; release() is called
// exactly once otherwise.
template <typename Tag, bool Checked, int W, int V, typename Release>
__device__ __forceinline__ bool rows_team(SmemHeader &h, const unsigned char *sbuf, const StageMeta &mt,
                                          unsigned char *ybase, int row_bytes, int nvec, bool causal, uint32_t seen,
                                          int warp, int lane, const Bounds &bd, uint64_t limit_ns,
                                          uint32_t &xs, Release &&release)
{
    constexpr int teams = kConsumerWarps / W;
    const int team = warp / W;
    uint64_t *bar = team_bar(h, W, team);
    int r = static_cast<int>((team + teams - (seen / W) % teams) % teams);
    int q = 0, qstep = 0;
    if (causal) {
        q = (mt.row0 + r) % mt.R;
        qstep = teams % mt.R;
    }
    if (r >= mt.nrows)
        release();
    for (; r < mt.nrows; r += teams) {
        const uint32_t par = (xs & W) ? 1u : 0u;
        const bool last = r + teams >= mt.nrows;
        float2 *part = &h.partial[par][team * W];
        auto exchange = [&](float2 &os) -> bool {
            if (W == 1)
                return true;
            if (lane == 0) {
                part[warp % W] = os;
                mbar_arrive(bar);
            }
            if (!__all_sync(0xFFFFFFFFu, mbar_spin_bounded(bar, par, &h.abort_flag, limit_ns)))
                return false;
            const int k = lane & 15;
            const float2 pw = k < W ? part[k] : make_float2(-INFINITY, 0.0f);
            os.x = warp_max(pw.x);
            os.y = 2.0f * group_sum<16>(half_share(pw, os.x));
            return true;
        };
        if (!row_team<Tag, Checked, W, V, V - 2>(sbuf + (size_t)r * row_bytes, ybase + (size_t)r * row_bytes, nvec, q,
                                                 causal, 0, warp % W, lane, bd, exchange, [&]() {
                                                     if (last)
                                                         release();
                                                 }))
            return false;
        if (W > 1)
            xs ^= W;
        q += qstep;
        if (q >= mt.R)
            q -= mt.R;
    }
    return true;
}

template <typename Tag, bool Checked, typename Release>
__device__ __forceinline__ bool consume_stage_team(SmemHeader &h, const unsigned char *sbuf, const StageMeta &mt,
                                                   unsigned char *y, bool causal, uint32_t seen, int warp, int lane,
                                                   Bounds bd, uint64_t limit_ns, uint32_t &xs, Release &&release)
{
    const int row_bytes = mt.C * Elem<Tag>::kSize;
    const int nvec = row_bytes >> 4;
    unsigned char *yb = y + mt.off * Elem<Tag>::kSize;
    bd.s_lo = sbuf;
    bd.s_hi = sbuf + (size_t)mt.nrows * row_bytes;
    const int W = team_warps(nvec);
    if (W > 1 && !team_switch(h, W, lane, limit_ns, xs))
        return false;
    auto go = [&](auto w) {
        constexpr int w_ = decltype(w)::value;
        if (nvec <= 6 * 32 * w_)
            return rows_team<Tag, Checked, w_, 6>(h, sbuf, mt, yb, row_bytes, nvec, causal, seen, warp, lane, bd,
                                                  limit_ns, xs, release);
        return rows_team<Tag, Checked, w_, kTeamVecs>(h, sbuf, mt, yb, row_bytes, nvec, causal, seen, warp, lane, bd,
                                                      limit_ns, xs, release);
    };
    return W == 1 ? go(Int<1>{}) : W == 2 ? go(Int<2>{}) : W == 4 ? go(Int<4>{}) : W == 8 ? go(Int<8>{}) : go(Int<16>{});
}

// The backward pass's rows of one stage that teams share; as rows_team.
template <typename Tag, bool Checked, int W, typename Release>
__device__ __forceinline__ bool rows_team_bwd(SmemHeader &h, const unsigned char *sbuf, int half, const StageMeta &mt,
                                              unsigned char *ybase, int row_bytes, int nvec, uint32_t seen, int warp,
                                              int lane, const Bounds &by, const Bounds &bdy, uint64_t limit_ns,
                                              uint32_t &xs, Release &&release)
{
    constexpr int teams = kConsumerWarps / W;
    const int team = warp / W;
    uint64_t *bar = team_bar(h, W, team);
    int r = static_cast<int>((team + teams - (seen / W) % teams) % teams);
    if (r >= mt.nrows)
        release();
    for (; r < mt.nrows; r += teams) {
        const uint32_t par = (xs & W) ? 1u : 0u;
        const bool last = r + teams >= mt.nrows;
        const size_t o = (size_t)r * row_bytes;
        float2 *part = &h.partial[par][team * W];
        auto exchange = [&](float &dot) -> bool {
            if (W == 1)
                return true;
            if (lane == 0) {
                part[warp % W] = make_float2(dot, 0.0f);
                mbar_arrive(bar);
            }
            if (!__all_sync(0xFFFFFFFFu, mbar_spin_bounded(bar, par, &h.abort_flag, limit_ns)))
                return false;
            const int k = lane & 15;
            dot = group_sum<16>(k < W ? part[k].x : 0.0f);
            return true;
        };
        if (!row_team_bwd<Tag, Checked, W, kTeamVecsBwd - 2>(sbuf + o, sbuf + half + o, ybase + o, nvec, warp % W, lane,
                                                             by, bdy, exchange, [&]() {
                                                                 if (last)
                                                                     release();
                                                             }))
            return false;
        if (W > 1)
            xs ^= W;
    }
    return true;
}

template <typename Tag, bool Checked, typename Release>
__device__ __forceinline__ bool consume_stage_team_bwd(SmemHeader &h, const unsigned char *sbuf, int half,
                                                       const StageMeta &mt, unsigned char *y, uint32_t seen, int warp,
                                                       int lane, Bounds by, uint64_t limit_ns, uint32_t &xs,
                                                       Release &&release)
{
    const int row_bytes = mt.C * Elem<Tag>::kSize;
    const int nvec = row_bytes >> 4;
    unsigned char *yb = y + mt.off * Elem<Tag>::kSize;
    by.s_lo = sbuf;
    by.s_hi = sbuf + (size_t)mt.nrows * row_bytes;
    Bounds bdy = by;
    bdy.s_lo = sbuf + half;
    bdy.s_hi = sbuf + half + (size_t)mt.nrows * row_bytes;
    const int W = team_warps_bwd(nvec);
    if (W > 1 && !team_switch(h, W, lane, limit_ns, xs))
        return false;
    auto go = [&](auto w) {
        return rows_team_bwd<Tag, Checked, decltype(w)::value>(h, sbuf, half, mt, yb, row_bytes, nvec, seen, warp, lane,
                                                               by, bdy, limit_ns, xs, release);
    };
    return W == 1 ? go(Int<1>{}) : W == 2 ? go(Int<2>{}) : W == 4 ? go(Int<4>{}) : W == 8 ? go(Int<8>{}) : go(Int<16>{});
}

// Rows that one lane group's registers hold: T lanes, V vectors a lane (vector
// j of lane l is vector j*T + l), of which only the last can be missing
// ((V-1) * T <= nvec, see consume_stage).  Issue bounds these rows (shared
// memory and the copies are ahead of it), so a group has no more lanes than
// two to four vectors a lane leave: fewer steps of the two butterflies a row,
// and no vector slot that is empty in every lane.  The mask is added to the
// vectors as loaded, a missing vector is -inf, and nothing else has a bound;
// rows past the patch repeat its last row and are not stored.  Maximum, offset
// and 2^(v log2 e - offset) as in row_team; the exponentials stay in registers,
// one per element.  Up to four vectors the offset is m log2 e itself: there the
// largest element carries the sum, and 2^0 has no error (rounded down, the
// error at unit variance is 8 % larger at 4 elements, 1 % at 16; at larger
// variances and lengths rounding down has the smaller error).
// GB/s over 256 MiB, bf16, groups of 8, 16 or 32 lanes with a bound on every
// vector -> this routine: 16 B 828 -> 6728, 64 B 3020 -> 6821, 112 B 4821 ->
// 6607, 192 B 5308 -> 6300, 256 B 6703 -> 6740, 528 B 4287 -> 6466, 1024 B
// 6649 -> 6795, 1040 B 4233 -> 6327, 1232 B 4888 -> 6617; fp32: 16 B 888 ->
// 6840, 64 B 3267 -> 6841, 528 B 5620 -> 6726, 2048 B 6799 -> 6848.
template <typename Tag, bool Checked, int T, int V>
__device__ __forceinline__ int rows_in_lanes(const unsigned char *sbuf, const StageMeta &mt, unsigned char *ybase,
                                             int row_bytes, int nvec, bool causal, int first, int lane,
                                             const Bounds &bd)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec, N = EPV / 2, G = 32 / T, step = G * kConsumerWarps;
    const int g = lane / T, l = lane % T;
    const Pair l2 = pair(kLog2e, kLog2e);
    const bool in_last = (V - 1) * T + l < nvec;
    int q = 0, qstep = 0;
    if (causal) {
        q = (mt.row0 + first * G + g) % mt.R;
        qstep = step % mt.R;
    }
    for (int rb = first * G; rb < mt.nrows; rb += step) {
        const int r = rb + g;
        const bool valid = r < mt.nrows;
        const unsigned char *sp = sbuf + (size_t)(valid ? r : mt.nrows - 1) * row_bytes + 16 * l;
        uint4 raw[V];
        MaxAcc<Tag> mx;
#pragma unroll
        for (int j = 0; j < V; ++j) {
            raw[j] = E::neg_inf_vec();
            if (j < V - 1 || in_last) {
                uint4 u;
                if (load_vec<Checked>(sp + 16 * j * T, bd, u))
                    raw[j] = causal ? mask_vec<Tag>(u, (j * T + l) * EPV, q) : u;
            }
            mx.add(raw[j]);
        }
        const float m = group_max<T>(mx.get());
        const float o = T > 2 ? exp_offset(m) : fmaxf(m * kLog2e, kLowest);
        const Pair nm = pair(-o, -o);
        Pair p[V][N], acc = pair(0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j < V; ++j) {
#pragma unroll
            for (int k = 0; k < N; ++k)
                p[j][k] = pair_ex2(pair_fma(vec_pair<Tag>(raw[j], k), l2, nm));
            if constexpr (N == 4)
                acc = pair_add(acc, pair_add(pair_add(p[j][0], p[j][1]), pair_add(p[j][2], p[j][3])));
            else
                acc = pair_add(acc, pair_add(p[j][0], p[j][1]));
        }
        const float2 a2 = halves(acc);
        const float inv = __frcp_rn(group_sum<T>(a2.x + a2.y));
        const Pair inv2 = pair(inv, inv);
        unsigned char *yp = ybase + (size_t)r * row_bytes + 16 * l;
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (valid && (j < V - 1 || in_last)) {
                float2 y2[N];
#pragma unroll
                for (int k = 0; k < N; ++k)
                    y2[k] = halves(pair_mul(p[j][k], inv2));
                store_vec<Checked>(yp + 16 * j * T, bd, pack_pairs<Tag>(y2));
            }
        q += qstep;
        if (q >= mt.R)
            q -= mt.R;
    }
    return (mt.nrows + G - 1) / G;
}

// All rows of one stage that belong to this consumer warp, for rows that one
// lane group's registers hold.  The routine depends on the row length only.
// Two vectors a lane up to 16: 128-byte bf16 rows on 8 lanes of one 5905 GB/s,
// on 4 of two 6788; 64-byte rows on 4 of one 5918, on 2 of two 6821.  Three
// instead of four where three hold the row.  Row groups are dealt round robin
// over the consumer warps starting at warp `first`; the caller advances
// `first` by the returned group count, so a stage with fewer groups than warps
// does not always land on the same warps.
template <typename Tag, bool Checked>
__device__ __forceinline__ int consume_stage(const unsigned char *sbuf, const StageMeta &mt, unsigned char *y,
                                             bool causal, int first, int lane, Bounds bd)
{
    using E = Elem<Tag>;
    // the lane's place in each class's group is not worth registers held across
    // the stages (and the teams' rows): opaque, so derived where it is used.
    // Spills 8 bytes -> none, fp32 96 -> 68 registers; 64 KiB bf16 rows in the
    // teams' instance 6330 -> 6432 GB/s
    asm volatile("" : "+r"(lane));
    const int row_bytes = mt.C * E::kSize;
    const int nvec = row_bytes >> 4;
    unsigned char *ybase = y + mt.off * E::kSize;
    bd.s_lo = sbuf;
    bd.s_hi = sbuf + (size_t)mt.nrows * row_bytes;
    auto rows = [&](auto t, auto v) {
        return rows_in_lanes<Tag, Checked, decltype(t)::value, decltype(v)::value>(sbuf, mt, ybase, row_bytes, nvec,
                                                                                   causal, first, lane, bd);
    };
    if (nvec <= 8)
        return nvec > 4    ? rows(Int<4>{}, Int<2>{})
               : nvec > 2  ? rows(Int<2>{}, Int<2>{})
               : nvec == 2 ? rows(Int<1>{}, Int<2>{})
                           : rows(Int<1>{}, Int<1>{});
    if (nvec <= 32)
        return nvec > 24   ? rows(Int<8>{}, Int<4>{})
               : nvec > 16 ? rows(Int<8>{}, Int<3>{})
                           : rows(Int<8>{}, Int<2>{});
    if (nvec <= 64)
        return nvec > 48 ? rows(Int<16>{}, Int<4>{}) : rows(Int<16>{}, Int<3>{});
    return nvec > 96 ? rows(Int<32>{}, Int<4>{}) : rows(Int<32>{}, Int<3>{});
}

// -------------------------------------------------------------- the schedule

// The pulling unit is a CTA, or for rows split over groups of CTAs a whole
// group (unit = group index, n_units = groups): the static and round-robin
// deals and the tail rule count units, not CTAs.
struct Puller {
    const KernelArgs &a;
    int32_t unit, n_units;
    int32_t k = 0;           // PULL_STATIC: patches taken so far
    int32_t slice = -1;      // PULL_RR_SLICE
    int32_t cur = 0, end = 0;
    int32_t q = 0;           // PULL_QUEUE: index into the try order
    int32_t die = 0;
    uint32_t fetch = kFetch; // PULL_QUEUE: patches per claim (1 near the end of a queue)

    __device__ explicit Puller(const KernelArgs &args)
        : Puller(args, static_cast<int32_t>(blockIdx.x), static_cast<int32_t>(gridDim.x))
    {
    }

    __device__ Puller(const KernelArgs &args, int32_t unit_, int32_t n_units_)
        : a(args), unit(unit_), n_units(n_units_)
    {
        if (a.mode == PULL_QUEUE && a.sm_die) {
            int d = a.sm_die[sm_id() & (BSM_MAX_SM - 1)];
            die = (d >= 0 && d < a.n_queues) ? d : 0;
        }
        // a short queue (small batch: about a patch per SM) is claimed one
        // patch at a time from the first claim on, so every SM gets one
        if (a.mode == PULL_QUEUE && static_cast<uint32_t>(a.queue_len[die]) < 2u * kFetch * static_cast<uint32_t>(n_units))
            fetch = 1;
        if (a.mode == PULL_RR_SLICE)
            slice = unit - n_units;
    }

    // Positions in a.items of this CTA's next patches (up to `most`, at most
    // kFetch); returns how many (0 when the CTA has no more work).
    __device__ int next_batch(int32_t (&pos)[kFetch], int most = kFetch)
    {
        int n = 0;
        if (a.mode == PULL_STATIC) {
#pragma unroll
            for (int j = 0; j < kFetch; ++j) {
                const int64_t idx = (int64_t)a.item_begin + unit + (int64_t)(k + j) * n_units;
                if (j < most && idx < a.item_end)
                    pos[n++] = static_cast<int32_t>(idx);
            }
            k += most;
            return n;
        }
        if (a.mode == PULL_RR_SLICE) {
            while (cur >= end) {
                slice += n_units;
                if (slice >= a.n_slices)
                    return 0;
                cur = a.slice_first_item[slice];
                end = a.slice_first_item[slice + 1];
            }
#pragma unroll
            for (int j = 0; j < kFetch; ++j)
                if (j < most && cur < end)
                    pos[n++] = cur++;
            return n;
        }
        // PULL_QUEUE: claim kFetch consecutive slots of the own die's queue,
        // then (steal) of the other dies' queues in order.
        const int tries = a.steal ? a.n_queues : 1;
        while (q < tries) {
            const int qq = (die + q) % a.n_queues;
            const uint32_t take = fetch < static_cast<uint32_t>(most) ? fetch : static_cast<uint32_t>(most);
            const uint32_t t = atomicAdd(&a.heads[qq], take);
            const uint32_t len = static_cast<uint32_t>(a.queue_len[qq]);
            if (t < len) {
#pragma unroll
                for (int j = 0; j < kFetch; ++j)
                    if (static_cast<uint32_t>(j) < take && t + j < len)
                        pos[n++] = a.queue_begin[qq] + static_cast<int32_t>(t + j);
                // near the end of the queue, claim one patch at a time so the
                // last patches spread over the SMs instead of queueing in fours
                if (len - t < 2u * kFetch * static_cast<uint32_t>(n_units))
                    fetch = 1;
                return n;
            }
            ++q;
        }
        return 0;
    }
};

// Warm L2 with the patches this CTA most likely copies first, before the
// wait on the previous kernel: the first kPrefetch slots of its first batch
// (the static deal's and round robin's exactly; under a queue, slots
// r*kFetch .. of queue u mod n_queues for CTA u = r*n_queues + (u mod
// n_queues), so that the CTAs together cover the first claims).  Two patches
// (19.5 MB over 152 SMs at 64 KiB) measured best: 1, 3 and 4 gave 0.4-0.7 %
// less on 384 x 512 x 512 rows, a second batch 2-5 % less (the prefetches
// then slow the previous kernel's last wave).  A prefetch into L2 carries no data to
// the SM and has no effect on what any load returns (L2 is the point of
// coherence), so it may run while the previous kernel still writes; what it
// buys is that DRAM serves these lines during that kernel's last wave
// instead of after it.  Records are checked like the producer checks them;
// one that fails is skipped.
constexpr int kPrefetch = 2;

__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <int ES>
__device__ __forceinline__ void prefetch_first_batch(const KernelArgs &a, bool two_inputs)
{
    int64_t first = 0, end = 0, step = 1;
    const int64_t u = blockIdx.x;
    if (a.mode == PULL_STATIC) {
        first = a.item_begin + u;
        end = a.item_end;
        step = gridDim.x;
    } else if (a.mode == PULL_RR_SLICE) {
        if (u >= a.n_slices)
            return;
        first = a.slice_first_item[u];
        end = a.slice_first_item[u + 1];
    } else {
        const int nq = a.n_queues > 0 ? a.n_queues : 1;
        const int q = static_cast<int>(u % nq);
        first = a.queue_begin[q] + (u / nq) * kFetch;
        end = (int64_t)a.queue_begin[q] + a.queue_len[q];
    }
    if (end > a.n_items)
        end = a.n_items;
    const int64_t cap = two_inputs ? a.stage_bytes / 2 : a.stage_bytes;
    for (int j = 0; j < kPrefetch; ++j) {
        const int64_t idx = first + j * step;
        if (idx < 0 || idx >= end)
            break;
        const Item it = a.items[idx];
        const int64_t ne = (int64_t)it.nrows * it.C;
        const int64_t nbytes = ne * ES;
        if (it.off < 0 || it.C <= 0 || it.nrows <= 0 || it.off + ne > a.total_elems || nbytes > cap ||
            (nbytes & 15) != 0 || ((it.off * ES) & 15) != 0)
            continue;
        prefetch_l2(static_cast<const unsigned char *>(a.x) + it.off * ES, static_cast<uint32_t>(nbytes));
        if (two_inputs)
            prefetch_l2(static_cast<const unsigned char *>(a.x2) + it.off * ES, static_cast<uint32_t>(nbytes));
    }
}

template <typename Tag, int Op, bool Checked>
__global__ void __launch_bounds__(kThreads, 1) softmax_persistent(const KernelArgs a)
{
    using E = Elem<Tag>;
    // the long-row machinery is compiled into its own instance, so plans
    // without long rows do not pay its registers
    constexpr bool kLong = Op == OP_FORWARD_LONG || Op == OP_BACKWARD_LONG;
    constexpr bool kBwd = Op == OP_BACKWARD || Op == OP_BACKWARD_LONG || Op == OP_BACKWARD_TEAM;
    // likewise the rows that teams of warps share
    constexpr bool kTeam = kLong || Op == OP_FORWARD_TEAM || Op == OP_BACKWARD_TEAM;
    constexpr int kLaneVecs = (kBwd ? kLaneRowBytesBwd<E::kSize> : kLaneRowBytes) / 16;
    extern __shared__ __align__(1024) unsigned char smem[];
    SmemHeader &h = *reinterpret_cast<SmemHeader *>(smem);
    unsigned char *stages = smem + kSmemHeader;
    // (broadcast for the teams: the compiler then knows that a warp's lanes agree)
    const int warp = kTeam ? __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0) : threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int S = a.n_stages;
    const uint64_t wait_limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&h.full[s], 1);
            mbar_init(&h.empty[s], kConsumerWarps);
        }
        mbar_init(&h.xwarp, kConsumerWarps);
        for (int t = 0; t < kTeamBars; ++t)
            mbar_init(&h.team[t], t < 8 ? 2 : t < 12 ? 4 : 8);
        h.abort_flag = 0;
        mbar_init_fence();
    }
    __syncthreads();
    // rows that fit a stage: the first batch's bytes are prefetched into L2
    // (a hint: it reads nothing into this CTA and writes nothing)
    if (!kLong && warp == kConsumerWarps && lane == 0)
        prefetch_first_batch<E::kSize>(a, kBwd);
    // Programmatic dependent launch: this kernel may have started while the
    // previous kernel of the stream was finishing.  No role loads data,
    // stores or starts a bounded wait before that kernel is done (a no-op
    // without such a predecessor); then the next kernel may begin its own
    // launch.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == kConsumerWarps) {
        // ------------------------------------------------------- producer
        if (lane == 0) {
            Puller pull(a);
            uint32_t issued_phase[kMaxStages];
            bool issued[kMaxStages];
            for (int s = 0; s < kMaxStages; ++s)
                issued[s] = false;
            bool aborted = false, done = false;
            uint32_t it = 0;
            // take the next stage of the ring once the consumers released it
            auto next_stage = [&](int &s, uint32_t &ph) -> bool {
                s = static_cast<int>(it % S);
                ph = (it / S) & 1u;
                if (!mbar_wait_bounded(&h.empty[s], ph ^ 1u, &h.abort_flag, wait_limit)) {
                    aborted = true;
                    return false;
                }
                issued[s] = false;
                ++it;
                return true;
            };
            // Long-row instances claim one patch at a time, and the next one
            // while a row streams: the queue atomic and the record loads
            // behind it are round trips of microseconds under full load,
            // which would otherwise stall the ring at every row start.
            int nx_n = -1;              // patches claimed ahead (-1: none)
            int32_t nx_pos = 0;
            Item nx_item{0, 0, 0, 0, 0};
            LongSeg nx_seg{0, 0, 0, 0};
            auto claim_ahead = [&]() {
                int32_t p1[kFetch];
                nx_n = pull.next_batch(p1, 1);
                nx_pos = p1[0];
                if (nx_n > 0 && nx_pos >= 0 && nx_pos < a.n_items) {
                    nx_item = a.items[nx_pos];
                    nx_seg = a.segs ? a.segs[nx_pos] : LongSeg{0, 0, 0, 0};
                }
            };
            while (!done && !aborted) {
                // the next patches: their records load in parallel
                int32_t pos[kFetch];
                Item batch[kFetch];
                LongSeg lseg[kFetch];   // long-row instances: the segment records
                int n = 0;
                if (kLong && nx_n >= 0) {
                    n = nx_n;
                    pos[0] = nx_pos;
                    batch[0] = nx_item;
                    lseg[0] = nx_seg;
                    nx_n = -1;
                } else {
                    n = pull.next_batch(pos, kLong ? 1 : kFetch);
#pragma unroll
                    for (int j = 0; j < kFetch; ++j)
                        if (j < n && pos[j] >= 0 && pos[j] < a.n_items) {
                            batch[j] = a.items[pos[j]];
                            if (kLong && a.segs)
                                lseg[j] = a.segs[pos[j]];
                        }
                }
                if (n == 0) {
                    // no more work: tell the consumers through the next stage
                    int s = 0;
                    uint32_t ph = 0;
                    if (!next_stage(s, ph))
                        break;
                    h.meta[s].kind = KIND_DONE;
                    mbar_arrive(&h.full[s]);
                    done = true;
                    break;
                }
                for (int j = 0; j < n && !aborted; ++j) {
                    // long-row instances check the patch (and cut a long one
                    // into chunks) before the wait for its stage, the others
                    // after it
                    int s = 0;
                    uint32_t ph = 0;
                    if (!kLong && !next_stage(s, ph))
                        break;
                    const Item item = batch[j];
                    const int64_t ne = (int64_t)item.nrows * item.C;
                    const int64_t nbytes = ne * E::kSize;
                    const int64_t cap = kBwd ? a.stage_bytes / 2 : a.stage_bytes;
                    LongSeg sg{0, 0, 0, 0};
                    if (kLong && a.segs && pos[j] >= 0 && pos[j] < a.n_items)
                        sg = lseg[j];
                    const bool is_long = kLong && sg.part_count > 0;
                    const bool ok = pos[j] >= 0 && pos[j] < a.n_items && item.off >= 0 && item.C > 0 &&
                                    item.nrows > 0 && item.R > 0 && item.row0 >= 0 &&
                                    item.row0 < item.R && item.off + ne <= a.total_elems &&
                                    (nbytes <= cap || is_long) && (nbytes & 15) == 0 &&
                                    ((item.off * E::kSize) & 15) == 0 && (!is_long || item.nrows == 1) &&
                                    (!is_long || (sg.part >= sg.part_first &&
                                                  sg.part < sg.part_first + sg.part_count && sg.part_first >= 0));
                    // a long segment: chunks of equal length in whole 16-byte
                    // vectors (no short last chunk leaves the consumers waiting
                    // on the next copy), every one non-empty; 32-bit arithmetic
                    // (C < 2^31, a stage < 2^18 bytes)
                    int64_t chunk = 1, nch = 0;
                    if (kLong && is_long && ok) {
                        const uint32_t cl = static_cast<uint32_t>(item.C);
                        const uint32_t cmax = static_cast<uint32_t>(cap / E::kSize);
                        const uint32_t n_min = (cl + cmax - 1) / cmax;
                        const uint32_t c = ((cl + n_min - 1) / n_min + E::kPerVec - 1) & ~uint32_t(E::kPerVec - 1);
                        chunk = c;
                        nch = (cl + c - 1) / c;
                    }
                    if (kLong && !next_stage(s, ph))
                        break;
                    StageMeta &mt = h.meta[s];
                    if ((a.debug & KDEBUG_WITHHOLD_STAGE0) && it == 1)
                        continue;                      // test hook: stage 0 is never filled
                    if (!ok) {
                        atomicOr(a.status, BSM_DEV_BOUNDS);
                        mt.kind = KIND_SKIP;
                        mbar_arrive(&h.full[s]);
                        continue;
                    }
                    if (kLong && is_long) {
                        // the segment in chunks of one stage: a whole row (one
                        // segment) streams twice in this launch; a segment of a
                        // longer row streams once, for this launch's phase
                        // a whole row with fewer chunks than stages stays staged:
                        // its second pass needs no copies
                        const bool resident = sg.part_count == 1 && nch < S;
                        const int p_lo = sg.part_count == 1 ? 0 : a.phase;
                        const int p_hi = sg.part_count == 1 && !resident ? 1 : a.phase;
                        bool first_stage = true;
                        for (int pass = p_lo; pass <= p_hi && !aborted; ++pass) {
                        // a whole row's second pass runs backwards from its
                        // last chunk, which the consumers keep in its stage
                        // and finish first (no copy); the others follow, the
                        // most recently read (most likely still in L2) first
                        const bool rev = pass == 1 && sg.part_count == 1;
                        for (int64_t kk = 0; kk < (rev ? nch - 1 : nch) && !aborted; ++kk) {
                            const int64_t k = rev ? nch - 2 - kk : kk;
                            if (!first_stage && !next_stage(s, ph))
                                break;
                            first_stage = false;
                            StageMeta &lm = h.meta[s];
                            const int64_t c0 = k * chunk;
                            const int64_t cn = item.C - c0 < chunk ? item.C - c0 : chunk;
                            lm.off = item.off + c0;
                            lm.C = static_cast<int32_t>(cn);
                            lm.nrows = 1;
                            lm.row0 = item.row0;
                            lm.R = item.R;
                            lm.col0 = static_cast<int32_t>(sg.col0 + c0);
                            lm.pass = pass;
                            lm.last = rev ? k == 0 : k == nch - 1;
                            lm.first = rev ? kk == 0 : k == 0;
                            lm.part = sg.part;
                            lm.part_first = sg.part_first;
                            lm.part_count = sg.part_count;
                            lm.resident = resident;
                            lm.kind = KIND_LONG;
                            const uint32_t cb = static_cast<uint32_t>(cn * E::kSize);
                            unsigned char *ldst = stages + (size_t)s * a.stage_bytes;
                            mbar_arrive_expect_tx(&h.full[s], kBwd ? 2 * cb : cb);
                            bulk_load(ldst,
                                      static_cast<const unsigned char *>(a.x) + (item.off + c0) * E::kSize,
                                      cb, &h.full[s]);
                            if (kBwd)   // dy's chunk into the second half
                                bulk_load(ldst + a.stage_bytes / 2,
                                          static_cast<const unsigned char *>(a.x2) + (item.off + c0) * E::kSize,
                                          cb, &h.full[s]);
                            issued[s] = true;
                            issued_phase[s] = ph;
                            // the row's second chunk is on its way (or its only
                            // one): claim the next patch now
                            if (nx_n < 0 && j == n - 1 && pass == p_lo && (kk == 1 || nch == 1))
                                claim_ahead();
                        }
                        }
                        continue;
                    }
                    mt.off = item.off;
                    mt.C = item.C;
                    mt.nrows = item.nrows;
                    mt.row0 = item.row0;
                    mt.R = item.R;
                    mt.kind = KIND_DATA;
                    const uint32_t bytes = static_cast<uint32_t>(nbytes);
                    unsigned char *dst = stages + (size_t)s * a.stage_bytes;
                    const unsigned char *src = static_cast<const unsigned char *>(a.x) + item.off * E::kSize;
                    const int half = a.stage_bytes / 2;
                    const unsigned char *src2 =
                        kBwd ? static_cast<const unsigned char *>(a.x2) + item.off * E::kSize : nullptr;
                    if (Checked) {
                        const unsigned char *x0 = static_cast<const unsigned char *>(a.x);
                        bool bad = s < 0 || s >= S || S > kMaxStages ||
                                   src < x0 || src + bytes > x0 + a.total_elems * E::kSize ||
                                   (reinterpret_cast<uintptr_t>(src) & 15) ||
                                   (smem_addr(dst) & 15) || (bytes & 15) || bytes == 0 ||
                                   dst + bytes > smem + kSmemHeader + (size_t)S * a.stage_bytes;
                        if (kBwd) {
                            const unsigned char *g0 = static_cast<const unsigned char *>(a.x2);
                            bad = bad || bytes > (uint32_t)half || src2 < g0 ||
                                  src2 + bytes > g0 + a.total_elems * E::kSize ||
                                  (reinterpret_cast<uintptr_t>(src2) & 15) || (half & 15);
                        }
                        if (bad) {
                            check_fail(a.status, 3, static_cast<uint64_t>(pos[j]), bytes);
                            mt.kind = KIND_SKIP;
                            mbar_arrive(&h.full[s]);
                            continue;
                        }
                    }
                    if (kBwd) {
                        mbar_arrive_expect_tx(&h.full[s], 2 * bytes);
                        bulk_load(dst, src, bytes, &h.full[s]);
                        bulk_load(dst + half, src2, bytes, &h.full[s]);
                    } else {
                        mbar_arrive_expect_tx(&h.full[s], bytes);
                        bulk_load(dst, src, bytes, &h.full[s]);
                    }
                    issued[s] = true;
                    issued_phase[s] = ph;
                }
            }
            if (aborted) {
                atomicOr(a.status, BSM_DEV_TIMEOUT);
                h.abort_flag = 1;
            }
            // every copy this lane issued has landed before it leaves (normally
            // they have: the consumers waited for them; after an abort they may not)
            for (int s = 0; s < S; ++s)
                if (issued[s])
                    mbar_wait_bounded(&h.full[s], issued_phase[s], nullptr, wait_limit);
            if (a.mode == PULL_QUEUE) {
                // the last CTA to finish pulling rewinds the queue heads
                __threadfence();
                const uint32_t prev = atomicAdd(&a.heads[BSM_MAX_DIES], 1u);
                if (prev == gridDim.x - 1) {
                    for (int d = 0; d < BSM_MAX_DIES; ++d)
                        atomicExch(&a.heads[d], 0u);
                    atomicExch(&a.heads[BSM_MAX_DIES], 0u);
                }
            }
        }
        return;
    }

    // ----------------------------------------------------------- consumers
    const bool causal = (a.flags & BSM_FLAG_CAUSAL) != 0;
    unsigned char *y = static_cast<unsigned char *>(a.y);
    uint32_t groups_seen = 0;   // warps' worth of rows dealt so far (the same count in every warp)
    uint32_t xs = 0;            // the exchanges between warps so far (see kTeamLast)
    // long rows: this lane's running (max, sum); the row's final exponent
    // offset and reciprocal; which partial buffer and barrier phase is next
    float m_l = -INFINITY, s_l = 0.0f, long_mL = 0.0f, long_inv = 0.0f;
    uint32_t long_first_it = 0;  // stage iteration of the current row's first chunk
    (void)m_l, (void)s_l, (void)long_mL, (void)long_inv, (void)xs;
    for (uint32_t it = 0;; ++it) {
        const int s = it % S;
        const uint32_t ph = (it / S) & 1u;
        if (!mbar_wait_bounded(&h.full[s], ph, &h.abort_flag, wait_limit)) {
            if (lane == 0) {
                atomicOr(a.status, BSM_DEV_TIMEOUT);
                h.abort_flag = 1;
            }
            break;
        }
        const StageMeta mt = h.meta[s];
        if (mt.kind == KIND_DONE)
            break;
        if (kLong && mt.kind == KIND_LONG) {
            Bounds bd{nullptr, nullptr, y, y + a.total_elems * E::kSize, a.status};
            if (mt.pass == 1 && mt.first && mt.part_count > 1) {
                // the row's partials, left by phase 0: dot products added in slot
                // order, (maximum, sum) pairs over the lanes and a fixed tree
                // (every segment of the row, on any SM, gets the same result).
                // One pair after another by every thread took 20 of 92 us on 8
                // fp32 rows of 16 MiB (109 segments each)
                const float *pp = a.partials + 2 * static_cast<int64_t>(mt.part_first);
                if constexpr (kBwd) {
                    float dot = 0.0f;
                    for (int k = 0; k < mt.part_count; ++k)
                        dot += pp[2 * k];
                    long_mL = dot;
                } else {
                    float m = -INFINITY, sum = 0.0f;
                    for (int k = lane; k < mt.part_count; k += 32)
                        m = fmaxf(m, pp[2 * k]);
                    m = warp_max(m);
                    for (int k = lane; k < mt.part_count; k += 32)
                        sum += ms_share(pp[2 * k], pp[2 * k + 1], m);
                    long_mL = long_offset(m);
                    long_inv = __frcp_rn(group_sum<32>(sum));
                }
            }
            if constexpr (kBwd)
                long_chunk_bwd<Tag, Checked>(stages + (size_t)s * a.stage_bytes, a.stage_bytes / 2, mt, y, warp,
                                             lane, bd, s_l, long_mL);
            else
                long_chunk<Tag, Checked>(stages + (size_t)s * a.stage_bytes, mt, y, causal, warp, lane, bd, m_l,
                                         s_l, long_mL, long_inv);
            __syncwarp();
            if (mt.pass == 0 && mt.first)
                long_first_it = it;
            // a whole row keeps its last chunk (a resident row: every chunk)
            // staged for the second pass
            const bool keep = mt.resident || (mt.pass == 0 && mt.last && mt.part_count == 1);
            if (lane == 0 && !keep)
                mbar_arrive(&h.empty[s]);
            if (mt.pass == 0 && mt.last) {
                // the segment's partial: lanes, then warps in a fixed order
                if constexpr (kBwd) {
#pragma unroll
                    for (int o = 16; o >= 1; o >>= 1)
                        s_l += __shfl_xor_sync(0xFFFFFFFFu, s_l, o);
                } else {
                    const float2 all = lanes_ms(m_l, s_l);
                    m_l = all.x;
                    s_l = all.y;
                }
                if constexpr (kTeam) {
                    if (!team_switch(h, 16, lane, wait_limit, xs)) {
                        if (lane == 0) {
                            atomicOr(a.status, BSM_DEV_TIMEOUT);
                            h.abort_flag = 1;
                        }
                        break;
                    }
                }
                const int par = (xs >> 4) & 1;
                if (lane == 0) {
                    h.partial[par][warp] = make_float2(kBwd ? s_l : m_l, kBwd ? 0.0f : s_l);
                    mbar_arrive(&h.xwarp);
                }
                if (!mbar_wait_bounded(&h.xwarp, par, &h.abort_flag, wait_limit)) {
                    if (lane == 0) {
                        atomicOr(a.status, BSM_DEV_TIMEOUT);
                        h.abort_flag = 1;
                    }
                    break;
                }
                float m = 0.0f, sum = 0.0f;
                if constexpr (kBwd) {
                    for (int w = 0; w < kConsumerWarps; ++w) {
                        const float2 pw = h.partial[par][w];
                        m = w == 0 ? pw.x : m + pw.x;
                    }
                } else {
                    const float2 pw = lane < kConsumerWarps ? h.partial[par][lane] : make_float2(-INFINITY, 0.0f);
                    const float2 all = lanes_ms(pw.x, pw.y);
                    m = all.x;
                    sum = all.y;
                }
                if (mt.part_count == 1) {
                    // the whole row: its second pass follows in this launch,
                    // starting on the chunk still in this stage
                    if constexpr (kBwd) {
                        long_mL = m;
                    } else {
                        long_mL = long_offset(m);
                        long_inv = __frcp_rn(sum);
                    }
                    if (!mt.resident) {
                        StageMeta m1 = mt;
                        m1.pass = 1;
                        if constexpr (kBwd)
                            long_chunk_bwd<Tag, Checked>(stages + (size_t)s * a.stage_bytes, a.stage_bytes / 2, m1,
                                                         y, warp, lane, bd, s_l, long_mL);
                        else
                            long_chunk<Tag, Checked>(stages + (size_t)s * a.stage_bytes, m1, y, causal, warp, lane,
                                                     bd, m_l, s_l, long_mL, long_inv);
                        __syncwarp();
                        if (lane == 0)
                            mbar_arrive(&h.empty[s]);
                    } else {
                        // a resident row: every chunk, from the first one's stage
                        for (uint32_t j = long_first_it; j <= it; ++j) {
                            const int sj = static_cast<int>(j % S);
                            StageMeta m1 = h.meta[sj];
                            m1.pass = 1;
                            if constexpr (kBwd)
                                long_chunk_bwd<Tag, Checked>(stages + (size_t)sj * a.stage_bytes,
                                                             a.stage_bytes / 2, m1, y, warp, lane, bd, s_l, long_mL);
                            else
                                long_chunk<Tag, Checked>(stages + (size_t)sj * a.stage_bytes, m1, y, causal, warp,
                                                         lane, bd, m_l, s_l, long_mL, long_inv);
                        }
                        __syncwarp();
                        if (lane == 0)
                            for (uint32_t j = long_first_it; j <= it; ++j)
                                mbar_arrive(&h.empty[j % S]);
                    }
                } else if (warp == 0 && lane == 0) {
                    a.partials[2 * static_cast<int64_t>(mt.part)] = m;
                    a.partials[2 * static_cast<int64_t>(mt.part) + 1] = sum;
                }
                m_l = -INFINITY;
                s_l = 0.0f;
                xs ^= 16u;
            }
            continue;
        }
        if (mt.kind == KIND_DATA) {
            Bounds bd{nullptr, nullptr, y, y + a.total_elems * E::kSize, a.status};
            const int64_t cap = kBwd ? a.stage_bytes / 2 : a.stage_bytes;
            const int nvec = (mt.C * E::kSize) >> 4;
            if (Checked && (mt.nrows <= 0 || mt.C <= 0 || (int64_t)mt.nrows * mt.C * E::kSize > cap)) {
                if (lane == 0)
                    check_fail(a.status, 4, static_cast<uint64_t>(mt.nrows), static_cast<uint64_t>(mt.C));
            } else if (kTeam && nvec > kLaneVecs) {
                auto release = [&]() {
                    __syncwarp();
                    if (lane == 0)
                        mbar_arrive(&h.empty[s]);
                };
                bool ok;
                if constexpr (kBwd)
                    ok = consume_stage_team_bwd<Tag, Checked>(h, stages + (size_t)s * a.stage_bytes, a.stage_bytes / 2,
                                                              mt, y, groups_seen, warp, lane, bd, wait_limit, xs,
                                                              release);
                else
                    ok = consume_stage_team<Tag, Checked>(h, stages + (size_t)s * a.stage_bytes, mt, y, causal,
                                                          groups_seen, warp, lane, bd, wait_limit, xs, release);
                if (!ok) {
                    if (lane == 0) {
                        atomicOr(a.status, BSM_DEV_TIMEOUT);
                        h.abort_flag = 1;
                    }
                    break;
                }
                groups_seen +=
                    static_cast<uint32_t>(mt.nrows) * (kBwd ? team_warps_bwd(nvec) : team_warps(nvec));
                continue;                  // the stage is released
            } else {
                const int first = static_cast<int>((warp + kConsumerWarps - groups_seen % kConsumerWarps) %
                                                   kConsumerWarps);
                if constexpr (kBwd)
                    groups_seen += consume_stage_bwd<Tag, Checked>(stages + (size_t)s * a.stage_bytes,
                                                                   a.stage_bytes / 2, mt, y, first, lane, bd);
                else
                    groups_seen += consume_stage<Tag, Checked>(stages + (size_t)s * a.stage_bytes, mt, y, causal,
                                                               first, lane, bd);
            }
        }
        __syncwarp();
        if (lane == 0)
            mbar_arrive(&h.empty[s]);
    }
}


// ------------------------------------------------ rows over groups of CTAs
// A row too long for one SM's shared memory is cut into K parts of equal
// length (whole 16-byte vectors; the last may be shorter or empty), and the K
// CTAs of a group each stage one part in one stage: every element is read
// from memory once.  Each CTA takes its part's (offset, sum) -- warps, then
// the CTA in a fixed tree, the offset as in row_team
// -- and publishes it in global memory as two words tagged with the row's
// sequence number; every member then reads the K partials (one per lane)
// until all carry the tag, combines them in the same fixed tree, and writes
// its part of y.  An exchange warp of its own does that, and the consumers
// work one row ahead: they take the next row's partial (from its stage) before
// writing the previous row (held in registers), so the exchange overlaps
// work.  fp32 1 MiB rows (K = 16) ran at 4811 GB/s when every consumer warp
// polled for itself, with a running maximum rescaled per chunk and the
// producer's chain of round trips (see there), and run at 5496; bf16 4137 and
// 5212.  On the way, without the row between, 4180; with the exchange warp
// publishing as well (so behind its polling), 4830.  The group's rank-0 CTA
// claims the rows (any policy's puller, with the group as the
// unit) and announces them to its members through a ring of claim words.
// The launch is cooperative, so every member of a group is resident and each
// wait ends; every wait is bounded all the same.

__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Wait until the claim word at p carries sequence number seq (bounded).
__device__ __noinline__ bool wait_claim(const unsigned long long *p, uint32_t seq, const volatile int32_t *abort,
                                        uint64_t limit_ns, unsigned long long &word)
{
    word = ld_relaxed_u64(p);
    if (static_cast<uint32_t>(word >> 32) == seq)
        return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 0; it < (1u << 26); ++it) {
        __nanosleep(32);
        word = ld_relaxed_u64(p);
        if (static_cast<uint32_t>(word >> 32) == seq)
            return true;
        if ((abort && *abort) || global_timer_ns() - t0 > limit_ns)
            return false;
    }
    return false;
}

// A member's part of a group row held in registers: consumer thread t (of
// the kConsumerWarps * 32) holds the part's 16-byte vectors t, t + 512, ...
constexpr int kConsumerThreads = kConsumerWarps * 32;

// Vector vi of the part in the stage; -inf past its end.
template <typename Tag, bool Checked>
__device__ __forceinline__ uint4 group_vec(const unsigned char *sbuf, int vi, int nvec, const Bounds &bd)
{
    uint4 r = Elem<Tag>::neg_inf_vec();
    if (vi < nvec) {
        uint4 t;
        if (load_vec<Checked>(sbuf + 16 * vi, bd, t))
            r = t;
    }
    return r;
}

// A member's two exchange words in one access (each word is validated by its
// own tag, so nothing depends on the two being one).
__device__ __forceinline__ void st_words(unsigned long long *p, unsigned long long w0, unsigned long long w1)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
}

__device__ __forceinline__ void ld_words(const unsigned long long *p, unsigned long long &w0, unsigned long long &w1)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
}

// The (offset, sum) of up to 32 partials, one per lane (-inf, 0 in the others),
// in every lane: a fixed tree.
__device__ __forceinline__ float2 combine_lanes(float2 p)
{
    const float o = warp_max(p.x);
    return make_float2(o, 2.0f * group_sum<32>(half_share(p, o)));
}

template <typename Tag, bool Checked>
__global__ void __launch_bounds__(kGroupThreads, 1) softmax_group(const KernelArgs a)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec;
    extern __shared__ __align__(1024) unsigned char smem[];
    SmemHeader &h = *reinterpret_cast<SmemHeader *>(smem);
    unsigned char *stages = smem + kSmemHeader;
    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int S = a.n_stages;
    const int K = a.group_k;
    const int grp = static_cast<int>(blockIdx.x) / K, rank = static_cast<int>(blockIdx.x) % K;
    const uint64_t wait_limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;
    unsigned long long *ring = a.ring + static_cast<size_t>(grp) * kGroupRing;
    unsigned long long *xch = a.xch + 2 * static_cast<size_t>(grp) * kGroupSlots * K;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&h.full[s], 1);
            mbar_init(&h.empty[s], kConsumerWarps);
        }
        mbar_init(&h.xres[0], 1);
        mbar_init(&h.xres[1], 1);
        h.xarrive[0] = h.xarrive[1] = h.xleft = 0u;
        h.abort_flag = 0;
        mbar_init_fence();
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == kConsumerWarps) {
        // ------------------------------------------------------- producer
        if (lane == 0) {
            Puller pull(a, grp, a.n_groups);
            uint32_t issued_phase[kMaxStages];
            bool issued[kMaxStages];
            for (int s = 0; s < kMaxStages; ++s)
                issued[s] = false;
            bool aborted = false;
            uint32_t it = 0;
            // Rank 0 announces rows up to kClaimAhead + 1 beyond the current
            // one; the claim after the last one announced is under way.  Every
            // member reads a row's claim word and record while the copy of the
            // row before is under way.  (One after the other at each row,
            // atomic, release store, acquire load, record load and copy were a
            // chain of about 4 us of round trips, which set the pace: fp32
            // 768 KiB rows 4780 GB/s against 5440.)  The words carry all that their readers use, so
            // relaxed accesses do.
            uint32_t posted = 0, claim = 0xFFFFFFFFu;
            bool post_done = false;
            auto claim_next = [&]() {
                int32_t p1[kFetch];
                claim = pull.next_batch(p1, 1) > 0 ? static_cast<uint32_t>(p1[0]) : 0xFFFFFFFFu;
            };
            auto post = [&](uint32_t upto) {
                while (rank == 0 && !post_done && posted <= upto) {
                    st_relaxed_u64(&ring[posted % kGroupRing],
                                   (static_cast<unsigned long long>(posted + 1) << 32) | claim);
                    ++posted;
                    post_done = claim == 0xFFFFFFFFu;
                    if (!post_done)
                        claim_next();
                }
            };
            uint32_t next_pos = 0xFFFFFFFFu;
            Item next_item{-1, 0, 0, 0, 0};
            auto fetch = [&](uint32_t t) -> bool {
                unsigned long long word = 0;
                if (!wait_claim(&ring[t % kGroupRing], t + 1, &h.abort_flag, wait_limit, word))
                    return false;
                next_pos = static_cast<uint32_t>(word);
                if (next_pos < static_cast<uint32_t>(a.n_items))
                    next_item = a.items[next_pos];
                return true;
            };
            if (rank == 0)
                claim_next();
            post(kClaimAhead);
            aborted = !fetch(0);
            for (uint32_t t = 0; !aborted; ++t) {
                if (t > 0 && !fetch(t)) {
                    aborted = true;
                    break;
                }
                const uint32_t pos = next_pos;
                const Item item = next_item;
                post(t + 1 + kClaimAhead);
                const int s = static_cast<int>(it % S);
                const uint32_t ph = (it / S) & 1u;
                if (!mbar_wait_bounded(&h.empty[s], ph ^ 1u, &h.abort_flag, wait_limit)) {
                    aborted = true;
                    break;
                }
                issued[s] = false;
                ++it;
                StageMeta &mt = h.meta[s];
                if (pos == 0xFFFFFFFFu) {
                    mt.kind = KIND_DONE;
                    mbar_arrive(&h.full[s]);
                    break;
                }
                if ((a.debug & KDEBUG_WITHHOLD_STAGE0) && it == 1)
                    continue;                      // test hook: stage 0 is never filled
                const bool in = pos < static_cast<uint32_t>(a.n_items);
                // this member's part (the same cut in every member)
                const int64_t part = ((int64_t(item.C) + K - 1) / K + EPV - 1) / EPV * EPV;
                const int64_t c0 = part * rank;
                const int64_t cn = item.C - c0 < 0 ? 0 : (item.C - c0 < part ? item.C - c0 : part);
                const bool ok = in && item.off >= 0 && item.C > 0 && item.nrows == 1 && item.R > 0 &&
                                item.row0 >= 0 && item.row0 < item.R && item.off + item.C <= a.total_elems &&
                                ((item.off * E::kSize) & 15) == 0 && ((int64_t(item.C) * E::kSize) & 15) == 0 &&
                                part * E::kSize <= a.stage_bytes &&
                                part * E::kSize <= int64_t(kGroupVecs) * 16 * kConsumerThreads;
                if (!ok) {
                    // every member sees the same record and skips the row alike
                    atomicOr(a.status, BSM_DEV_BOUNDS);
                    mt.kind = KIND_SKIP;
                    mbar_arrive(&h.full[s]);
                    continue;
                }
                mt.off = item.off + c0;
                mt.C = static_cast<int32_t>(cn);
                mt.nrows = 1;
                mt.row0 = item.row0;
                mt.R = item.R;
                mt.col0 = static_cast<int32_t>(c0);
                mt.pass = 0;
                mt.kind = KIND_GROUP;
                if (cn == 0) {
                    mbar_arrive(&h.full[s]);
                    continue;
                }
                const uint32_t bytes = static_cast<uint32_t>(cn * E::kSize);
                unsigned char *dst = stages + static_cast<size_t>(s) * a.stage_bytes;
                const unsigned char *src = static_cast<const unsigned char *>(a.x) + (item.off + c0) * E::kSize;
                if (Checked) {
                    const unsigned char *x0 = static_cast<const unsigned char *>(a.x);
                    if (src < x0 || src + bytes > x0 + a.total_elems * E::kSize ||
                        (reinterpret_cast<uintptr_t>(src) & 15) || (smem_addr(dst) & 15) ||
                        bytes > static_cast<uint32_t>(a.stage_bytes) ||
                        dst + bytes > smem + kSmemHeader + static_cast<size_t>(S) * a.stage_bytes) {
                        check_fail(a.status, 3, pos, bytes);
                        mt.kind = KIND_SKIP;       // the group's other members time out
                        mbar_arrive(&h.full[s]);
                        continue;
                    }
                }
                mbar_arrive_expect_tx(&h.full[s], bytes);
                bulk_load(dst, src, bytes, &h.full[s]);
                issued[s] = true;
                issued_phase[s] = ph;
            }
            if (aborted) {
                atomicOr(a.status, BSM_DEV_TIMEOUT);
                h.abort_flag = 1;
            }
            for (int s = 0; s < S; ++s)
                if (issued[s])
                    mbar_wait_bounded(&h.full[s], issued_phase[s], nullptr, wait_limit);
        }
        __syncwarp();
    } else if (warp == kConsumerWarps + 1) {
        // ------------------------------------------------------- exchange
        // For every row: the group's words read until all are in, combined,
        // and handed to the consumers through shared memory.  One warp a CTA
        // polls (16 polling the same few lines held the stores up), and the
        // consumers never wait on global memory.  Barrier and result alternate
        // by row: row t + 1's result can be in before a consumer warp has
        // tested row t's (all partials of t + 1 are out by then, that warp's
        // too), row t + 2's cannot (that warp's partial follows its test).
        uint64_t t0 = 0;
        uint32_t xt = 0;
        for (uint32_t tries = 0; tries < (1u << 30); ++tries) {
            const unsigned long long *xs = &xch[2 * static_cast<size_t>(xt & (kGroupSlots - 1)) * K];
            const uint32_t tag = xt + 1;
            float2 pw = make_float2(-INFINITY, 0.0f);
            bool all = true;
            if (lane < K) {
                unsigned long long w0, w1;
                ld_words(&xs[2 * lane], w0, w1);
                all = static_cast<uint32_t>(w0 >> 32) == tag && static_cast<uint32_t>(w1 >> 32) == tag;
                pw = make_float2(__uint_as_float(static_cast<uint32_t>(w0)),
                                 __uint_as_float(static_cast<uint32_t>(w1)));
            }
            if (__all_sync(0xFFFFFFFFu, all)) {
                pw = combine_lanes(pw);
                if (lane == 0) {
                    h.result[xt & 1] = pw;
                    mbar_arrive(&h.xres[xt & 1]);
                }
                __syncwarp();
                ++xt;
                t0 = 0;
                continue;
            }
            // (a consumer that waits for a result gives up by itself; this
            // warp, idle between rows, only after a long while)
            const uint32_t left = *const_cast<volatile uint32_t *>(&h.xleft);
            const uint64_t now = (tries & 63u) == 63u ? global_timer_ns() : 0;
            t0 = t0 ? t0 : now;
            if (__any_sync(0xFFFFFFFFu, left == kConsumerWarps || *const_cast<volatile int32_t *>(&h.abort_flag) ||
                                            (now && now - t0 > 8 * wait_limit)))
                break;
            __nanosleep(20);
        }
    } else {
        // ----------------------------------------------------------- consumers
        // Thread t of the 512 consumer threads owns the part's vectors t, t +
        // 512, ... (at most kGroupVecs).  A row's partial is taken from its
        // stage (read twice, for the maximum and for the sum); then the row
        // before -- held in registers, its exchange under way meanwhile -- is
        // written, and this row moves from the stage into the registers.  One
        // stage is held at a time; the others are in flight.
        const bool causal = (a.flags & BSM_FLAG_CAUSAL) != 0;
        unsigned char *y = static_cast<unsigned char *>(a.y);
        const Bounds bdy{nullptr, nullptr, y, y + a.total_elems * E::kSize, a.status};
        const int tid = warp * 32 + lane;
        const Pair l2 = pair(kLog2e, kLog2e);
        uint32_t xt = 0;            // group rows this CTA took part in (the exchange sequence)
        uint4 rr[kGroupVecs];       // the row one behind: its partial is out, it is not yet written
        int rvec = 0;               // ... its vectors, and where they go
        unsigned char *ry = nullptr;
        // the row held in rr, once its group's result is in; false when that wait gave up
        auto finish = [&]() -> bool {
            const uint32_t par = (xt - 1) & 1u;
            if (!__all_sync(0xFFFFFFFFu,
                            mbar_spin_bounded(&h.xres[par], ((xt - 1) >> 1) & 1u, &h.abort_flag, wait_limit))) {
                if (lane == 0) {
                    atomicOr(a.status, BSM_DEV_TIMEOUT);
                    h.abort_flag = 1;
                }
                return false;
            }
            const float2 t = h.result[par];
            const float inv = __frcp_rn(t.y);
            const Pair nm = pair(-t.x, -t.x), inv2 = pair(inv, inv);
            if (rvec >= (kGroupVecs - 2) * kConsumerThreads) {
                // (the usual part: only the last two vectors can be missing)
#pragma unroll
                for (int j = 0; j < kGroupVecs; ++j)
                    if (j < kGroupVecs - 2 || tid + j * kConsumerThreads < rvec)
                        store_vec<Checked>(ry + 16 * j * kConsumerThreads, bdy, vec_softmax<Tag>(rr[j], l2, nm, inv2));
            } else {
#pragma unroll
                for (int j = 0; j < kGroupVecs; ++j)
                    if (tid + j * kConsumerThreads < rvec)
                        store_vec<Checked>(ry + 16 * j * kConsumerThreads, bdy, vec_softmax<Tag>(rr[j], l2, nm, inv2));
            }
            return true;
        };
        int s = 0;
        uint32_t ph = 0;            // the ring's stage and phase
        bool held = false;
        for (;;) {
            // the whole warp gives up together (the shuffles need all lanes)
            if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(&h.full[s], ph, &h.abort_flag, wait_limit))) {
                if (lane == 0) {
                    atomicOr(a.status, BSM_DEV_TIMEOUT);
                    h.abort_flag = 1;
                }
                held = false;
                break;
            }
            const int32_t kind = h.meta[s].kind;
            if (kind == KIND_DONE)
                break;
            if (kind == KIND_GROUP) {
                const int C = h.meta[s].C, row = h.meta[s].row0, col0 = h.meta[s].col0;
                const int nvec = (C * E::kSize) >> 4;
                const unsigned char *sbuf = stages + static_cast<size_t>(s) * a.stage_bytes;
                Bounds bs = bdy;
                bs.s_lo = sbuf;
                bs.s_hi = sbuf + static_cast<size_t>(C) * E::kSize;
                auto part = [&](auto full) -> float2 {
                    // vector j of this thread (only the last two can be missing in a full part)
                    auto vec = [&](int j) {
                        const int vi = tid + j * kConsumerThreads;
                        const uint4 v = group_vec<Tag, Checked>(
                            sbuf, vi, decltype(full)::value && j < kGroupVecs - 2 ? INT32_MAX : nvec, bs);
                        return causal ? mask_vec<Tag>(v, col0 + vi * EPV, row) : v;
                    };
                    MaxAcc<Tag> mx;
#pragma unroll
                    for (int j = 0; j < kGroupVecs; ++j)
                        mx.add(vec(j));
                    const float o = exp_offset(warp_max(mx.get()));
                    const Pair nm = pair(-o, -o);
                    Pair acc = pair(0.0f, 0.0f);
#pragma unroll
                    for (int j = 0; j < kGroupVecs; ++j)
                        acc = vec_sum<Tag>(acc, vec(j), l2, nm);
                    const float2 a2 = halves(acc);
                    return make_float2(o, group_sum<32>(a2.x + a2.y));
                };
                const bool full = nvec >= (kGroupVecs - 2) * kConsumerThreads;
                const float2 mine = full ? part(Int<1>{}) : part(Int<0>{});
                // the last warp to bring its partial combines the warps' (a fixed
                // tree over 16 lanes) and publishes the CTA's.  (A warp's partial
                // of row t + 2 comes after it has seen row t's result, i.e. after
                // row t's publication: two slots by row parity.)
                const int par = xt & 1;
                int last = 0;
                if (lane == 0) {
                    h.partial[par][warp] = mine;
                    __threadfence_block();
                    last = atomicAdd(&h.xarrive[par], 1u) == static_cast<uint32_t>(kConsumerWarps - 1) ? 1 : 0;
                    if (last) {
                        __threadfence_block();
                        h.xarrive[par] = 0u;
                    }
                }
                if (__shfl_sync(0xFFFFFFFFu, last, 0)) {
                    __syncwarp();
                    const float2 pw =
                        combine_lanes(lane < kConsumerWarps ? h.partial[par][lane] : make_float2(-INFINITY, 0.0f));
                    // two self-validating words (value, row tag): a reader that
                    // sees the tag sees the value written with it
                    if (lane == 0) {
                        const unsigned long long tag = static_cast<unsigned long long>(xt + 1) << 32;
                        st_words(&xch[2 * (static_cast<size_t>(xt & (kGroupSlots - 1)) * K + rank)],
                                 tag | __float_as_uint(pw.x), tag | __float_as_uint(pw.y));
                    }
                }
                if (Checked && (a.debug & KDEBUG_LAG_WARP) && warp == 5)
                    for (int i = 0; i < 50; ++i)     // test hook: the row before's result is read late
                        __nanosleep(1000);
                if (held && !finish()) {
                    held = false;
                    break;
                }
                // this row into the registers; the stage is free
#pragma unroll
                for (int j = 0; j < kGroupVecs; ++j) {
                    const int vi = tid + j * kConsumerThreads;
                    const uint4 v = group_vec<Tag, Checked>(sbuf, vi, nvec, bs);
                    rr[j] = causal ? mask_vec<Tag>(v, col0 + vi * EPV, row) : v;
                }
                rvec = nvec;
                ry = y + h.meta[s].off * E::kSize + 16 * tid;
                held = true;
                ++xt;
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&h.empty[s]);
            if (++s == S) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (held)
            finish();
        // the exchange warp leaves too
        if (lane == 0)
            atomicAdd(&h.xleft, 1u);
        __syncwarp();
    }
    // the last CTA out resets the queue heads, the claim rings and the
    // exchange counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const uint32_t prev = atomicAdd(&a.heads[BSM_MAX_DIES], 1u);
        if (prev == gridDim.x - 1) {
            __threadfence();
            for (int d = 0; d < BSM_MAX_DIES; ++d)
                atomicExch(&a.heads[d], 0u);
            for (int i = 0; i < a.n_groups * kGroupRing; ++i)
                a.ring[i] = 0ull;
            for (int i = 0; i < 2 * a.n_groups * kGroupSlots * a.group_k; ++i)
                a.xch[i] = 0ull;
            __threadfence();
            atomicExch(&a.heads[BSM_MAX_DIES], 0u);
        }
    }
}

// ------------------------------------------------ rows over clusters of CTAs
// Batches of rows too long for one stage, enough of them to fill the SMs: a
// cluster of K = 2, 4, 8 or 16 CTAs shares a row, a part of it in one stage of each
// (the parts of a row of 64 to 113 KiB are what a team of 16 warps takes
// alone), so every element is read once.  The row routines are the teams',
// W = 16; the exchange goes over the cluster: every warp sends its (offset, sum)
// (backward: its dot product) to all K CTAs' shared memory with an
// asynchronous store that counts on the receiver's barrier, and every warp of
// the cluster combines the 16 K of them in the same fixed tree.  The first
// CTA claims the rows (any policy's puller, with the cluster as the unit) and
// posts them to the others' rings of claim words.
//
// What bounded these rows: one CTA streamed a row twice, its second read from
// L2 while the first of the next row waited for a stage.  GB/s over 256 MiB,
// one CTA a row -> clusters: forward fp32 128 KiB rows 5463 -> 6495, 256 KiB
// (K = 4, 36 clusters: 144 SMs) 5056 -> 6532; bf16 128 KiB 4592 -> 6356, 224 KiB
// 4620 -> 6313, 256 KiB 4407 -> 6373; backward (512 MiB of y and dy) fp32 64 KiB
// 6182 -> 6950, 128 KiB (K = 4) 5887 -> 6981, bf16 5916 -> 6845.
struct ClusterMeta {
    int64_t off;
    int32_t C, row0, col0, kind;
};

constexpr int kClusterRing = 16;

struct ClusterSmem {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t xbar[2];                   // a row's partials are in, by row parity
    unsigned long long ring[kClusterRing];
    ClusterMeta meta[kMaxStages];
    int32_t abort_flag;
};
static_assert(sizeof(ClusterSmem) <= kClusterHeader, "cluster header too large");

__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Wait (without sleeping, bounded; `abort` may be null) for a phase that other
// CTAs of the cluster complete.
__device__ __forceinline__ bool cluster_spin_bounded(uint64_t *bar, uint32_t parity, const volatile int32_t *abort,
                                                     uint64_t limit_ns)
{
    uint64_t t0 = 0;
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(parity)
            : "memory");
        if (ok)
            return true;
        if ((it & 1023u) == 1023u) {
            const uint64_t t = global_timer_ns();
            t0 = t0 ? t0 : t;
            if ((abort && *abort) || t - t0 > limit_ns)
                return false;
        }
    }
    return false;
}

// The row's (offset, sum) or dot product from 32 P pairs in shared memory, P a
// lane: fixed trees, the loads and exponentials of a lane independent of one
// another (a loop over them cost 12 % on bf16 256 KiB rows).
template <int P> __device__ __forceinline__ float2 lanes_pairs(const float2 *in, int lane)
{
    float2 p[P];
    float o[P], t[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        p[j] = in[lane + 32 * j];
        o[j] = p[j].x;
    }
    const float O = warp_max(tree_max<P>(o));
#pragma unroll
    for (int j = 0; j < P; ++j)
        t[j] = half_share(p[j], O);
    return make_float2(O, 2.0f * group_sum<32>(tree_sum<P>(t)));
}

template <int P> __device__ __forceinline__ float lanes_dot(const float2 *in, int lane)
{
    float t[P];
#pragma unroll
    for (int j = 0; j < P; ++j)
        t[j] = in[lane + 32 * j].x;
    return group_sum<32>(tree_sum<P>(t));
}

template <typename Tag, bool Bwd, bool Checked>
__global__ void __launch_bounds__(kThreads, 1) softmax_cluster(const KernelArgs a)
{
    using E = Elem<Tag>;
    constexpr int EPV = E::kPerVec, kArrays = Bwd ? 2 : 1;
    extern __shared__ __align__(1024) unsigned char smem[];
    ClusterSmem &h = *reinterpret_cast<ClusterSmem *>(smem);
    float2 *parts = reinterpret_cast<float2 *>(smem + kClusterHeader);     // [2][K * 16], by row parity
    unsigned char *stages = smem + cluster_header(a.group_k);
    const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int S = a.n_stages, K = a.group_k, half = a.stage_bytes / 2;
    const int unit = static_cast<int>(blockIdx.x) / K, n_units = static_cast<int>(gridDim.x) / K;
    const int rank = static_cast<int>(blockIdx.x) % K;          // = the CTA's rank in its cluster
    const uint64_t wait_limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;
    // this CTA's part of a row of C elements: whole vectors
    auto part_of = [&](int32_t C, int64_t &c0, int64_t &cn, int64_t &bytes) {
        const int64_t nv = (int64_t(C) * E::kSize) >> 4, pv = (nv + K - 1) / K;
        const int64_t v0 = pv * rank, vn = nv - v0 < 0 ? 0 : (nv - v0 < pv ? nv - v0 : pv);
        c0 = v0 * EPV;
        cn = vn * EPV;
        bytes = pv * 16;                                        // the longest part
    };
    auto item_ok = [&](const Item &it, int64_t part_bytes) {
        return it.off >= 0 && it.C > 0 && it.nrows == 1 && it.R > 0 && it.row0 >= 0 && it.row0 < it.R &&
               it.off + it.C <= a.total_elems && ((it.off * E::kSize) & 15) == 0 &&
               ((int64_t(it.C) * E::kSize) & 15) == 0 && part_bytes <= (Bwd ? half : a.stage_bytes);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&h.full[s], 1);
            mbar_init(&h.empty[s], kConsumerWarps);
        }
        mbar_init(&h.xbar[0], 1);
        mbar_init(&h.xbar[1], 1);
        for (int i = 0; i < kClusterRing; ++i)
            h.ring[i] = 0ull;
        h.abort_flag = 0;
        mbar_init_fence();
    }
    __syncthreads();
    cluster_barrier();
    // the cluster's likely first row into L2 (a hint, as prefetch_first_batch)
    if (warp == kConsumerWarps && lane == 0 && a.mode == PULL_QUEUE) {
        const int q = unit % (a.n_queues > 0 ? a.n_queues : 1), k = unit / (a.n_queues > 0 ? a.n_queues : 1);
        const int64_t idx = int64_t(a.queue_begin[q]) + k;
        if (k < a.queue_len[q] && idx >= 0 && idx < a.n_items) {
            const Item it = a.items[idx];
            int64_t c0, cn, pb;
            part_of(it.C, c0, cn, pb);
            if (item_ok(it, pb) && cn > 0) {
                prefetch_l2(static_cast<const unsigned char *>(a.x) + (it.off + c0) * E::kSize,
                            static_cast<uint32_t>(cn * E::kSize));
                if (Bwd)
                    prefetch_l2(static_cast<const unsigned char *>(a.x2) + (it.off + c0) * E::kSize,
                                static_cast<uint32_t>(cn * E::kSize));
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == kConsumerWarps) {
        // ------------------------------------------------------- producer
        if (lane == 0) {
            Puller pull(a, unit, n_units);
            bool aborted = false, post_done = false;
            uint32_t posted = 0, claim = 0xFFFFFFFFu;
            auto claim_next = [&]() {
                int32_t p1[kFetch];
                claim = pull.next_batch(p1, 1) > 0 ? static_cast<uint32_t>(p1[0]) : 0xFFFFFFFFu;
            };
            // rows are announced two ahead, the claim after them under way; a
            // word carries all that its reader uses.  No word is overwritten
            // unread: a producer is at most S stages and one row ahead of the
            // slowest.
            auto post = [&](uint32_t upto) {
                while (rank == 0 && !post_done && posted <= upto) {
                    const unsigned long long w = (static_cast<unsigned long long>(posted + 1) << 32) | claim;
                    for (int r = 0; r < K; ++r)
                        asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(
                                         cluster_addr(&h.ring[posted % kClusterRing], r)),
                                     "l"(w)
                                     : "memory");
                    ++posted;
                    post_done = claim == 0xFFFFFFFFu;
                    if (!post_done)
                        claim_next();
                }
            };
            auto ring_word = [&](uint32_t t, uint32_t &pos) -> bool {
                const uint32_t addr = smem_addr(&h.ring[t % kClusterRing]);
                uint64_t t0 = 0;
                for (uint32_t it = 0; it < (1u << 28); ++it) {
                    unsigned long long w;
                    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w) : "r"(addr) : "memory");
                    if (static_cast<uint32_t>(w >> 32) == t + 1) {
                        pos = static_cast<uint32_t>(w);
                        return true;
                    }
                    if ((it & 15u) == 15u) {
                        const uint64_t now = global_timer_ns();
                        t0 = t0 ? t0 : now;
                        if (h.abort_flag || now - t0 > wait_limit)
                            return false;
                        __nanosleep(64);
                    }
                }
                return false;
            };
            if (rank == 0)
                claim_next();
            post(1);
            int s = 0;
            uint32_t ph = 0;
            uint32_t issued = 0, issued_phase = 0;      // by stage: a copy issued, its phase
            bool first = true;
            for (uint32_t t = 0; !aborted; ++t) {
                uint32_t pos = 0;
                if (!ring_word(t, pos)) {
                    aborted = true;
                    break;
                }
                const bool in = pos < static_cast<uint32_t>(a.n_items);
                Item item{-1, 0, 0, 0, 0};
                if (in)
                    item = a.items[pos];        // on its way while the stage is waited for
                post(t + 2);
                if (!mbar_wait_bounded(&h.empty[s], ph ^ 1u, &h.abort_flag, wait_limit)) {
                    aborted = true;
                    break;
                }
                ClusterMeta &mt = h.meta[s];
                uint64_t *full = &h.full[s];
                unsigned char *dst = stages + static_cast<size_t>(s) * a.stage_bytes;
                const uint32_t bit = 1u << s, phase_bit = ph << s;
                issued &= ~bit;
                if (++s == S) {
                    s = 0;
                    ph ^= 1u;
                }
                if (pos == 0xFFFFFFFFu) {
                    mt.kind = KIND_DONE;
                    mbar_arrive(full);
                    break;
                }
                if ((a.debug & KDEBUG_WITHHOLD_STAGE0) && first) {
                    first = false;
                    continue;                      // test hook: the first stage is never filled
                }
                first = false;
                int64_t c0, cn, pb;
                part_of(item.C, c0, cn, pb);
                if (!in || !item_ok(item, pb)) {
                    // every CTA of the cluster sees the same record and skips the row alike
                    atomicOr(a.status, BSM_DEV_BOUNDS);
                    mt.kind = KIND_SKIP;
                    mbar_arrive(full);
                    continue;
                }
                mt.off = item.off + c0;
                mt.C = static_cast<int32_t>(cn);
                mt.row0 = item.row0;
                mt.col0 = static_cast<int32_t>(c0);
                mt.kind = KIND_DATA;
                if (cn == 0) {
                    mbar_arrive(full);
                    continue;
                }
                const uint32_t bytes = static_cast<uint32_t>(cn * E::kSize);
                const unsigned char *src = static_cast<const unsigned char *>(a.x) + (item.off + c0) * E::kSize;
                const unsigned char *src2 = Bwd ? static_cast<const unsigned char *>(a.x2) + (item.off + c0) * E::kSize
                                                : nullptr;
                if (Checked) {
                    const unsigned char *x0 = static_cast<const unsigned char *>(a.x);
                    const unsigned char *g0 = static_cast<const unsigned char *>(a.x2);
                    const int64_t all = a.total_elems * E::kSize;
                    if (src < x0 || src + bytes > x0 + all || (reinterpret_cast<uintptr_t>(src) & 15) ||
                        (Bwd && (src2 < g0 || src2 + bytes > g0 + all || (reinterpret_cast<uintptr_t>(src2) & 15))) ||
                        (smem_addr(dst) & 15) || (half & 15) || bytes > static_cast<uint32_t>(Bwd ? half : a.stage_bytes) ||
                        dst + a.stage_bytes > stages + static_cast<size_t>(S) * a.stage_bytes) {
                        check_fail(a.status, 3, pos, bytes);
                        mt.kind = KIND_SKIP;       // the cluster's other CTAs time out
                        mbar_arrive(full);
                        continue;
                    }
                }
                mbar_arrive_expect_tx(full, kArrays * bytes);
                bulk_load(dst, src, bytes, full);
                if (Bwd)
                    bulk_load(dst + half, src2, bytes, full);
                issued |= bit;
                issued_phase = (issued_phase & ~bit) | phase_bit;
            }
            if (aborted) {
                atomicOr(a.status, BSM_DEV_TIMEOUT);
                h.abort_flag = 1;
            }
            // every copy issued has landed before the CTA leaves, whoever gave
            // up (normally they have: the consumers waited for them)
            for (int j = 0; j < S; ++j)
                if (issued >> j & 1u)
                    mbar_wait_bounded(&h.full[j], issued_phase >> j & 1u, nullptr, wait_limit);
            if (rank == 0 && a.mode == PULL_QUEUE) {
                // the last cluster to finish pulling rewinds the queue heads
                __threadfence();
                const uint32_t prev = atomicAdd(&a.heads[BSM_MAX_DIES], 1u);
                if (prev == static_cast<uint32_t>(n_units - 1)) {
                    for (int d = 0; d < BSM_MAX_DIES; ++d)
                        atomicExch(&a.heads[d], 0u);
                    atomicExch(&a.heads[BSM_MAX_DIES], 0u);
                }
            }
        }
        __syncwarp();
    } else {
        // ----------------------------------------------------------- consumers
        const bool causal = (a.flags & BSM_FLAG_CAUSAL) != 0;
        unsigned char *y = static_cast<unsigned char *>(a.y);
        uint32_t x = 0;             // rows exchanged
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        // this warp's pair to every CTA of the cluster; true once all the
        // cluster's are in, at parts_in.  Barrier and slots alternate by row:
        // a warp sends row t + 2's after it has row t + 1's pairs, which every
        // warp sent after it had taken row t's.
        const int n_pairs = K * kConsumerWarps;
        const float2 *parts_in = nullptr;
        auto gather = [&](float2 mine) -> bool {
            const uint32_t par = x & 1u;
            float2 *in = parts + par * n_pairs;
            if (warp == 0 && lane == 0)
                mbar_arrive_expect_tx(&h.xbar[par], static_cast<uint32_t>(n_pairs * sizeof(float2)));
            __syncwarp();
            if (lane < K) {
                unsigned long long w;
                asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "f"(mine.x), "f"(mine.y));
                asm volatile(
                    "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(
                        cluster_addr(&in[rank * kConsumerWarps + warp], lane)),
                    "l"(w), "r"(cluster_addr(&h.xbar[par], lane))
                    : "memory");
            }
            if (!__all_sync(0xFFFFFFFFu, cluster_spin_bounded(&h.xbar[par], (x >> 1) & 1u, &h.abort_flag, wait_limit)))
                return false;
            ++x;
            parts_in = in;
            return true;
        };
        for (;;) {
            ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&h.full[s], ph, &h.abort_flag, wait_limit));
            if (!ok)
                break;
            const int32_t kind = h.meta[s].kind;
            if (kind == KIND_DONE)
                break;
            const int s0 = s;
            auto release = [&]() {
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&h.empty[s0]);
            };
            if (++s == S) {
                s = 0;
                ph ^= 1u;
            }
            if (kind != KIND_DATA) {
                release();
                continue;
            }
            const unsigned char *sbuf = stages + static_cast<size_t>(s0) * a.stage_bytes;
            const int bytes = h.meta[s0].C * E::kSize, nvec = bytes >> 4;
            unsigned char *yp = y + h.meta[s0].off * E::kSize;
            const Bounds bd{sbuf, sbuf + bytes, y, y + a.total_elems * E::kSize, a.status};
            if constexpr (Bwd) {
                auto exchange = [&](float &dot) -> bool {
                    if (!gather(make_float2(dot, 0.0f)))
                        return false;
                    dot = K == 2   ? lanes_dot<1>(parts_in, lane)
                          : K == 4 ? lanes_dot<2>(parts_in, lane)
                          : K == 8 ? lanes_dot<4>(parts_in, lane)
                                   : lanes_dot<8>(parts_in, lane);
                    return true;
                };
                const Bounds bdy{sbuf + half, sbuf + half + bytes, y, y + a.total_elems * E::kSize, a.status};
                if (nvec >= 2 * kConsumerWarps * 32)
                    ok = row_team_bwd<Tag, Checked, 16, kTeamVecsBwd - 2>(sbuf, sbuf + half, yp, nvec, warp, lane, bd, bdy,
                                                                          exchange, release);
                else
                    ok = row_team_bwd<Tag, Checked, 16, 0>(sbuf, sbuf + half, yp, nvec, warp, lane, bd, bdy, exchange,
                                                           release);
            } else {
                const int row = h.meta[s0].row0, col0 = h.meta[s0].col0;
                auto exchange = [&](float2 &os) -> bool {
                    if (!gather(os))
                        return false;
                    os = K == 2   ? lanes_pairs<1>(parts_in, lane)
                         : K == 4 ? lanes_pairs<2>(parts_in, lane)
                         : K == 8 ? lanes_pairs<4>(parts_in, lane)
                                  : lanes_pairs<8>(parts_in, lane);
                    return true;
                };
                if (nvec >= (kTeamVecs - 2) * kConsumerWarps * 32)
                    ok = row_team<Tag, Checked, 16, kTeamVecs, kTeamVecs - 2>(sbuf, yp, nvec, row, causal, col0, warp,
                                                                             lane, bd, exchange, release);
                else
                    ok = row_team<Tag, Checked, 16, kTeamVecs, 0>(sbuf, yp, nvec, row, causal, col0, warp, lane, bd,
                                                                 exchange, release);
            }
            if (!ok)
                break;
        }
        if (!ok && lane == 0) {
            atomicOr(a.status, BSM_DEV_TIMEOUT);
            h.abort_flag = 1;
            // pairs of the row given up may still be on their way here: they
            // are in, or a wait limit has passed, before this CTA leaves
            cluster_spin_bounded(&h.xbar[x & 1u], (x >> 1) & 1u, nullptr, wait_limit);
        }
        __syncwarp();
    }
    // no CTA leaves while another of its cluster may still write to it
    cluster_barrier();
}

}  // namespace

int kernel_set_smem_limit(int bytes)
{
    const void *fns[] = {
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD_TEAM, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD_TEAM, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD, true>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD_TEAM, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD_TEAM, true>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD_TEAM, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD_TEAM, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD, true>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD_TEAM, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD_TEAM, true>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD_LONG, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD_LONG, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_FORWARD_LONG, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_FORWARD_LONG, true>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD_LONG, false>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD_LONG, false>),
        reinterpret_cast<const void *>(softmax_persistent<F32, OP_BACKWARD_LONG, true>),
        reinterpret_cast<const void *>(softmax_persistent<BF16, OP_BACKWARD_LONG, true>),
        reinterpret_cast<const void *>(softmax_cluster<F32, false, false>),
        reinterpret_cast<const void *>(softmax_cluster<F32, false, true>),
        reinterpret_cast<const void *>(softmax_cluster<F32, true, false>),
        reinterpret_cast<const void *>(softmax_cluster<F32, true, true>),
        reinterpret_cast<const void *>(softmax_cluster<BF16, false, false>),
        reinterpret_cast<const void *>(softmax_cluster<BF16, false, true>),
        reinterpret_cast<const void *>(softmax_cluster<BF16, true, false>),
        reinterpret_cast<const void *>(softmax_cluster<BF16, true, true>),
        reinterpret_cast<const void *>(softmax_group<F32, false>),
        reinterpret_cast<const void *>(softmax_group<BF16, false>),
        reinterpret_cast<const void *>(softmax_group<F32, true>),
        reinterpret_cast<const void *>(softmax_group<BF16, true>)};
    for (const void *f : fns) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess)
            return static_cast<int>(e);
    }
    return 0;
}

namespace {
template <typename Tag, int Op>
void launch_one(const KernelArgs &a, int grid, size_t smem, cudaStream_t st, bool checked)
{
    // launched with programmatic stream serialisation: the kernel's prologue
    // overlaps the tail of the previous kernel (see griddepcontrol.wait)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
#ifdef BSM_NO_PDL
    cfg.numAttrs = 0;
#endif
    if (checked)
        cudaLaunchKernelEx(&cfg, softmax_persistent<Tag, Op, true>, a);
    else
        cudaLaunchKernelEx(&cfg, softmax_persistent<Tag, Op, false>, a);
}

// Rows over groups of CTAs: a cooperative launch (every CTA resident at once,
// so the members of a group can wait on one another), without the
// programmatic overlap with the previous kernel.
template <typename Tag>
void launch_group(const KernelArgs &a, int grid, size_t smem, cudaStream_t st, bool checked)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kGroupThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (checked)
        cudaLaunchKernelEx(&cfg, softmax_group<Tag, true>, a);
    else
        cudaLaunchKernelEx(&cfg, softmax_group<Tag, false>, a);
}
// Rows over clusters of CTAs: clusters of a.group_k, with the programmatic
// overlap of launch_one.
template <typename Tag, bool Bwd>
cudaError_t cluster_launch(const KernelArgs *a, int K, int grid, size_t smem, cudaStream_t st, bool checked, int *units)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(K);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = units ? 1 : 2;
#ifdef BSM_NO_PDL
    cfg.numAttrs = 1;
#endif
    if (units) {
        // clusters of 16 are past the portable size: allowed once, before the
        // first plan that uses them
        for (const void *f : {reinterpret_cast<const void *>(softmax_cluster<Tag, Bwd, false>),
                              reinterpret_cast<const void *>(softmax_cluster<Tag, Bwd, true>)})
            if (cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1))
                return e;
        return cudaOccupancyMaxActiveClusters(units, softmax_cluster<Tag, Bwd, false>, &cfg);
    }
    if (checked)
        return cudaLaunchKernelEx(&cfg, softmax_cluster<Tag, Bwd, true>, *a);
    return cudaLaunchKernelEx(&cfg, softmax_cluster<Tag, Bwd, false>, *a);
}

cudaError_t cluster_dispatch(const KernelArgs *a, int dtype, bool bwd, int K, int grid, size_t smem, cudaStream_t st,
                             bool checked, int *units)
{
    if (dtype == BSM_F32)
        return bwd ? cluster_launch<F32, true>(a, K, grid, smem, st, checked, units)
                   : cluster_launch<F32, false>(a, K, grid, smem, st, checked, units);
    return bwd ? cluster_launch<BF16, true>(a, K, grid, smem, st, checked, units)
               : cluster_launch<BF16, false>(a, K, grid, smem, st, checked, units);
}
}  // namespace

int cluster_units(int dtype, bool bwd, int K, int n_sm, int smem, int *units)
{
    *units = 0;
    return static_cast<int>(cluster_dispatch(nullptr, dtype, bwd, K, K * (n_sm / K), static_cast<size_t>(smem), nullptr,
                                             false, units));
}

int launch_softmax(const KernelArgs &a, int dtype, int op, int grid, void *stream, bool checked)
{
    const size_t smem = kSmemHeader + (size_t)a.n_stages * a.stage_bytes;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (op == OP_FORWARD_CLUSTER || op == OP_BACKWARD_CLUSTER) {
        const size_t csmem = cluster_header(a.group_k) + (size_t)a.n_stages * a.stage_bytes;
        const cudaError_t e = cluster_dispatch(&a, dtype, op == OP_BACKWARD_CLUSTER, a.group_k, grid, csmem, st, checked,
                                               nullptr);
        const cudaError_t l = cudaGetLastError();
        return static_cast<int>(e ? e : l);
    }
    if (op == OP_FORWARD_GROUP) {
        if (dtype == BSM_F32)
            launch_group<F32>(a, grid, smem, st, checked);
        else
            launch_group<BF16>(a, grid, smem, st, checked);
    } else if (op == OP_BACKWARD) {
        if (dtype == BSM_F32)
            launch_one<F32, OP_BACKWARD>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_BACKWARD>(a, grid, smem, st, checked);
    } else if (op == OP_BACKWARD_TEAM) {
        if (dtype == BSM_F32)
            launch_one<F32, OP_BACKWARD_TEAM>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_BACKWARD_TEAM>(a, grid, smem, st, checked);
    } else if (op == OP_BACKWARD_LONG) {
        if (dtype == BSM_F32)
            launch_one<F32, OP_BACKWARD_LONG>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_BACKWARD_LONG>(a, grid, smem, st, checked);
    } else if (op == OP_FORWARD_TEAM) {
        if (dtype == BSM_F32)
            launch_one<F32, OP_FORWARD_TEAM>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_FORWARD_TEAM>(a, grid, smem, st, checked);
    } else if (op == OP_FORWARD_LONG) {
        if (dtype == BSM_F32)
            launch_one<F32, OP_FORWARD_LONG>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_FORWARD_LONG>(a, grid, smem, st, checked);
    } else {
        if (dtype == BSM_F32)
            launch_one<F32, OP_FORWARD>(a, grid, smem, st, checked);
        else
            launch_one<BF16, OP_FORWARD>(a, grid, smem, st, checked);
    }
    return static_cast<int>(cudaGetLastError());
}

}  // namespace bsm
