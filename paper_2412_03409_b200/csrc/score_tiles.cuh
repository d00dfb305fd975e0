// Device helpers of the tensor-core scoring kernels (sm_100a): mbarriers with bounded waits, TMA,
// tcgen05 descriptors, MMA issue and tensor-memory loads.  Tiles are 128 x 128 throughout.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace pkv {

constexpr int TT = 128;                    // tile side
constexpr uint32_t kSpin = 1u << 20;       // tries per wait; each may sleep up to kSuspendNs
constexpr uint32_t kSuspendNs = 2000;      // suspend-time hint of one try: a waiting thread leaves the issue slots alone
constexpr float kLog2eT = 1.4426950408889634f;

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count));
}
__device__ __forceinline__ void bar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}
// Bounded wait.  `dead` latches for the calling thread once any wait in the CTA has run out.
__device__ __forceinline__ void bar_wait(uint64_t *bar, uint32_t parity, bool &dead, int *abort_flag,
                                         uint32_t limit = kSpin)
{
    if (dead) return;
    for (uint32_t i = 0; i < limit; ++i) {
        if (bar_try(bar, parity)) return;
        if ((i & 255u) == 255u && *(volatile int *)abort_flag) break;
    }
    dead = true;
    atomicExch(abort_flag, 1);
}

// Bounded wait of a role that has given up for what it has in flight itself.
__device__ __forceinline__ void drain(uint64_t *bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kSpin && !bar_try(bar, parity); ++i) {}
}

// Bounded wait of a whole warp: every lane learns when any lane's wait has run out.
__device__ __forceinline__ void warp_wait(uint64_t *bar, uint32_t parity, bool &dead, int *abort_flag)
{
    bar_wait(bar, parity, dead, abort_flag);
    dead = __any_sync(0xffffffffu, dead);
}

// Bounded wait of a whole warp for a count in shared memory, which another warp raises, to be above `n`; `seen` is what
// was last read of it.  Read often at first, as it is seldom far behind; the limit is about as long as the other waits'.
__device__ __forceinline__ void count_wait(const int *count, int n, int &seen, bool &dead, int *abort_flag, uint32_t limit = kSpin)
{
    for (uint32_t i = 0; seen <= n && !dead; ++i) {
        seen = __shfl_sync(0xffffffffu, *(const volatile int *)count, 0);
        if (seen > n) return;
        if (i >= limit || *(volatile int *)abort_flag) {
            dead = true;
            atomicExch(abort_flag, 1);
        }
        dead = __any_sync(0xffffffffu, dead);
        if (i >= 64) __nanosleep(i < 4096 ? 50 : kSuspendNs);
    }
}

__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1,
                                            int c2, int c3, int c4)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(saddr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(saddr(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
        : "memory");
}

// Shared-memory matrix descriptor, K-major operand with the 128-byte swizzle: rows of 128 bytes,
// eight-row groups 1024 bytes apart, tile base aligned to 1024 bytes.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);  // start address, bits [0,14)
    d |= (uint64_t)1 << 16;                   // leading byte offset (not used by swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset, bits [32,46)
    d |= (uint64_t)1 << 46;                   // descriptor version for sm_100
    d |= (uint64_t)2 << 61;                   // layout type: 128-byte swizzle
    return d;
}

// The descriptor of an operand `bytes` further on (tiles end below 256 KiB, so the address field cannot carry).
__device__ __forceinline__ uint64_t desc_add(uint64_t desc, uint32_t bytes)
{
    return (desc & 0xffffffff00000000ull) | ((uint32_t)desc + (bytes >> 4));
}

// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = N = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TT >> 3) << 17) |
                            ((uint32_t)(TT >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// True in one lane of a converged warp, always the same one.
__device__ __forceinline__ bool elect_one()
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok));
    return ok != 0;
}
__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// Two blocks of 32 columns, both loads on their way at once.
__device__ __forceinline__ void tmem_ld32x2(uint32_t taddr0, uint32_t taddr1, float (&v)[32], float (&w)[32])
{
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, "
        "%8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, "
        "%24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr0));
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, "
        "%8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, "
        "%24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
          "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
          "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
          "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr1));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        v[i] = __uint_as_float(r[i]);
        w[i] = __uint_as_float(r[32 + i]);
    }
}
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64])
{
    uint32_t r[64];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}
// 2^x on the special-function unit, one instruction (inputs here are <= 0 or -inf; flushing
// denormal results to zero is harmless for sums of probabilities).
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("{\n\t.reg .b64 x, y, w;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "add.rn.f32x2 w, x, y;\n\tmov.b64 {%0, %1}, w;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
// acc + 2^x on the FMA and integer pipes, two values at a time.  Rounding to the nearest integer n by
// adding 1.5 * 2^23, a degree-5 polynomial in f = x - n (minimax in relative error on [-1/2, 1/2] with
// p(0) = 1, fitted by Lawson's weighted least squares: 1.1e-7 as rounded, 1.7e-7 with the rounding of Horner's rule;
// ex2.approx is specified to 2^-22 = 2.4e-7), and 2^n put together in the exponent field.  x is held in
// [-127, 128], where 2^n is 0 and infinity; NaN stays NaN.  UPPER: x may be above 128.
template <bool UPPER> __device__ __forceinline__ float2 add_exp2(float2 acc, float2 x)
{
    asm("max.NaN.f32 %0, %0, 0fC2FE0000;" : "+f"(x.x));
    asm("max.NaN.f32 %0, %0, 0fC2FE0000;" : "+f"(x.y));
    if (UPPER) {
        asm("min.NaN.f32 %0, %0, 0f43000000;" : "+f"(x.x));
        asm("min.NaN.f32 %0, %0, 0f43000000;" : "+f"(x.y));
    }
    const float big = 12582912.f;
    const float2 t = add2(x, make_float2(big, big));
    const float2 n = add2(t, make_float2(-big, -big));
    const float2 f = fma2(n, make_float2(-1.f, -1.f), x);
    const float c[5] = {0x1.5bba14p-10f, 0x1.3cea88p-7f, 0x1.c6b752p-5f, 0x1.ebf9bcp-3f, 0x1.62e42ap-1f};
    float2 p = make_float2(c[0], c[0]);
#pragma unroll
    for (int i = 1; i < 5; ++i) p = fma2(p, f, make_float2(c[i], c[i]));
    p = fma2(p, f, make_float2(1.f, 1.f));
    const float2 s = make_float2(__uint_as_float((__float_as_uint(t.x) << 23) + 0x3f800000u),
                                 __uint_as_float((__float_as_uint(t.y) << 23) + 0x3f800000u));
    return fma2(p, s, acc);
}
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

struct Ring2 {
    int idx;
    uint32_t phase;
    __device__ __forceinline__ void next(int n)
    {
        if (++idx == n) {
            idx = 0;
            phase ^= 1u;
        }
    }
};

// Whether pair i of a row goes to the FMA pipe: even pairs, POLY (0 to 4) of every eight, spread evenly.
template <int POLY> __device__ __forceinline__ constexpr bool poly_pair(int i)
{
    return i % 2 == 0 && (i / 2 % 4) * POLY % 4 + POLY > 3;
}

// Pass 1 on NC consecutive logits of one query row: running maximum and sum in the log2
// domain.  Four interleaved chains each for the maximum and the sum: with two reader warps per
// scheduler a long dependent chain would leave it idle.  `fast` (scale > 0, the usual case):
// the extreme of sc * x is sc * max x, so masked logits may stay -inf.
// Of every eight pairs of exponentials POLY are computed on the FMA pipe, the others on the
// special-function unit.
template <int NC, int POLY>
__device__ __forceinline__ void lse_block(float (&v)[NC], float sc, bool fast, float &run_max, float &run_sum)
{
    if (!fast) {
#pragma unroll
        for (int i = 0; i < NC; ++i) v[i] = v[i] == -INFINITY ? -INFINITY : v[i] * sc;
    }
    // (three-input maximum: half the comparisons; the loop takes four values at a time, the last two come at the end)
    float c2[2] = {v[0], v[1]};
#pragma unroll
    for (int i = 2; i + 2 < NC; i += 4) {
        c2[0] = max3(c2[0], v[i], v[i + 1]);
        c2[1] = max3(c2[1], v[i + 2], v[i + 3]);
    }
    const float cmax = max3(c2[0], c2[1], fmaxf(v[NC - 2], v[NC - 1]));
    const float nm = fmaxf(run_max, fast ? cmax * sc : cmax);
    // (the maximum is still -infinity when keys of infinite elements have masked all columns so far: sums of 0)
    const float base = nm == -INFINITY ? 0.f : nm;
    const float mul = fast ? sc : 1.f;  // (the other way v is scaled already)
    float2 p[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int i = 0; i < NC; i += 2) {
        const float2 x = fma2(make_float2(v[i], v[i + 1]), make_float2(mul, mul), make_float2(-base, -base));
        float2 &acc = p[(i >> 1) & 1];
        acc = poly_pair<POLY>(i >> 1) ? add_exp2<false>(acc, x) : add2(acc, make_float2(ex2(x.x), ex2(x.y)));
    }
    run_sum = fmaf(run_sum, ex2(run_max - base), (p[0].x + p[0].y) + (p[1].x + p[1].y));
    run_max = nm;
}

// Pass 2 on the logits of NC consecutive queries against one key: sum of the probabilities,
// lse = the queries' normalisers (shared memory, log2 domain).  On the block the causal boundary
// crosses (`edge`) query i of the block counts only when i >= lane.
template <int NC, int POLY>
__device__ __forceinline__ float colsum_block(const float (&v)[NC], const float *lse, float sc, bool edge, int lane)
{
    const float4 *lp = reinterpret_cast<const float4 *>(lse);
    float2 p[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int i4 = 0; i4 < NC / 4; ++i4) {
        const float4 ls = lp[i4];
        const int i = i4 * 4;
        const float2 x = fma2(make_float2(v[i], v[i + 1]), make_float2(sc, sc), make_float2(-ls.x, -ls.y));
        const float2 y = fma2(make_float2(v[i + 2], v[i + 3]), make_float2(sc, sc), make_float2(-ls.z, -ls.w));
        if (!edge && poly_pair<POLY>(2 * i4)) {
            p[0] = add_exp2<true>(p[0], x);
            p[1] = add2(p[1], make_float2(ex2(y.x), ex2(y.y)));
            continue;
        }
        float e[4] = {ex2(x.x), ex2(x.y), ex2(y.x), ex2(y.y)};
        if (edge) {
#pragma unroll
            for (int u = 0; u < 4; ++u) e[u] = i + u >= lane ? e[u] : 0.f;
        }
        p[0] = add2(p[0], make_float2(e[0], e[1]));
        p[1] = add2(p[1], make_float2(e[2], e[3]));
    }
    return (p[0].x + p[0].y) + (p[1].x + p[1].y);
}

// Work item w -> (segment-head sh, tile t).  CTAs take items in order from a counter.  Heads come in
// groups whose Q and K stay in L2 (head_group), so that every operand byte comes from HBM once per
// pass.  Within a group the longest items of all its heads come first (pass 1: the last query tiles,
// pass 2: the first key tiles), so that what is left for the end of the pass is short.  Pass 2 walks
// the groups backwards: it starts on what pass 1 touched last.
template <int PASS> __device__ __forceinline__ void decode_item(int w, int nsh, int tiles, int group, int &sh, int &t)
{
    const int g = w / (group * tiles), r = w - g * group * tiles;
    const int heads = min(group, nsh - g * group);
    const int step = r / heads, first = g * group;
    t = PASS == 1 ? tiles - 1 - step : step;
    sh = first + (r - step * heads);
    if (PASS == 2) sh = nsh - 1 - sh;
}
// Heads of a group: as many as 64 MB hold, half of the L2, evenly over the groups.
inline int head_group(int nsh, int N, int D, size_t elem)
{
    const size_t fit = ((size_t)64 << 20) / (2 * (size_t)N * D * elem);
    const int most = fit < 1 ? 1 : (fit < (size_t)nsh ? (int)fit : nsh);
    const int groups = (nsh + most - 1) / most;
    return (nsh + groups - 1) / groups;
}

}  // namespace pkv
