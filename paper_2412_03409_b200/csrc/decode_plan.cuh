// What one decode step does to a segment, 16-byte row vectors, and the flags and counts that order the reads of
// the lengths before their writes: shared by the decode kernels.
#pragma once
#include <chrono>

#include "common.cuh"

namespace pkv {

// 16 bytes of a cache row as floats.
template <typename T> struct RowVec;
template <> struct RowVec<float> {
    static constexpr int VE = 4;
    __device__ static void unpack(const uint4 &r, float *x)
    {
        x[0] = __uint_as_float(r.x); x[1] = __uint_as_float(r.y);
        x[2] = __uint_as_float(r.z); x[3] = __uint_as_float(r.w);
    }
    __device__ static uint4 pack(const float *x)
    {
        return make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
    }
};
template <> struct RowVec<__nv_bfloat16> {
    static constexpr int VE = 8;
    __device__ static void unpack(const uint4 &r, float *x)
    {
        x[0] = __uint_as_float(r.x << 16); x[1] = __uint_as_float(r.x & 0xffff0000u);
        x[2] = __uint_as_float(r.y << 16); x[3] = __uint_as_float(r.y & 0xffff0000u);
        x[4] = __uint_as_float(r.z << 16); x[5] = __uint_as_float(r.z & 0xffff0000u);
        x[6] = __uint_as_float(r.w << 16); x[7] = __uint_as_float(r.w & 0xffff0000u);
    }
    __device__ static uint4 pack(const float *x)
    {
        __nv_bfloat162 a = __floats2bfloat162_rn(x[0], x[1]), b = __floats2bfloat162_rn(x[2], x[3]);
        __nv_bfloat162 c = __floats2bfloat162_rn(x[4], x[5]), d = __floats2bfloat162_rn(x[6], x[7]);
        return make_uint4(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b),
                          *reinterpret_cast<uint32_t *>(&c), *reinterpret_cast<uint32_t *>(&d));
    }
};

struct DecodePlanArgs {
    const int64_t *row_offset;
    int32_t *len;
    const int32_t *cap;
    const int32_t *len0;  // [B*L] rows kept by compaction        } only with
    int32_t *gen;         // [B*L] tokens decoded so far          } decode-time
    int32_t *slot_ring;   // [B*L][distance + 1] rows of recent tokens } pruning
    int64_t total_cap_rows;
    int evict_distance, N, L, layer_begin, nl, nact;
    bool append;
};

inline DecodePlanArgs decode_plan_args(const pkv_shape *s, const pkv_cache *c, bool append, int layer_begin, int nl)
{
    DecodePlanArgs a;
    a.row_offset = c->row_offset; a.len = c->len; a.cap = c->cap;
    a.len0 = c->len0; a.gen = c->gen; a.slot_ring = c->slot_ring;
    a.total_cap_rows = c->total_cap_rows;
    a.evict_distance = c->evict_distance;
    a.N = s->prompt_len; a.L = s->layers;
    a.layer_begin = layer_begin; a.nl = nl; a.nact = s->batch * nl;
    a.append = append;
    return a;
}

// What this step does to active segment si: the rows it attends over (the new row included),
// or -1 when the segment cannot take the row (full, never compacted, or outside the cache);
// the row the new token is written to; the length afterwards.  Without decode-time pruning
// the new row is appended.  With it (Sec. 3.1: prune at a fixed distance to the latest token,
// keep the layer's proportion): when generated token g would push the layer past
// floor(len0 * (N + g + 1) / N) rows and token g - distance is still cached, the new row
// takes that token's slot instead and the length stays.
struct SegPlan {
    int rows, dst, len_after;
    bool evict;
    int64_t off;
};
// (Read past the L1 cache: a kernel may ask once while the kernel in front still runs, as a guess, and again after it.)
__device__ __forceinline__ int32_t load_l2(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int64_t load_l2(const int64_t *p)
{
    int64_t v;
    asm volatile("ld.relaxed.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// What decode-time pruning goes by: tokens so far, rows kept by compaction, the place of the token `distance` back.
struct PruneState {
    int g, len0, slot;
};
__device__ __forceinline__ PruneState prune_state(const DecodePlanArgs &a, int seg)
{
    PruneState s{0, 0, -1};
    const int d = a.append ? a.evict_distance : 0;
    if (d > 0) {
        s.g = a.gen[seg];
        s.len0 = a.len0[seg];
        if (s.g >= d) s.slot = a.slot_ring[(size_t)seg * (d + 1) + (s.g - d) % (d + 1)];
    }
    return s;
}
__device__ __forceinline__ SegPlan plan_of(const DecodePlanArgs &a, int ln, int cp, int64_t off, const PruneState &ps)
{
    SegPlan p;
    p.off = off;
    p.evict = false;
    p.dst = ln;
    bool ok = ln >= 1 && p.off >= 0 && p.off <= a.total_cap_rows - cp && ln <= cp;
    if (!a.append) {  // nothing to append: attend over the rows that are there
        p.dst = 0x3fffffff;
        p.rows = ok ? ln : -1;
        p.len_after = p.rows;
        return p;
    }
    const int d = a.evict_distance;
    if (ok && d > 0) {
        const int64_t target = ((int64_t)ps.len0 * ((int64_t)a.N + ps.g + 1)) / a.N;
        if ((int64_t)ln + 1 > target && ps.g >= d && ps.slot >= 0 && ps.slot < ln) {
            p.evict = true;
            p.dst = ps.slot;
        }
    }
    if (!p.evict && ln >= cp) ok = false;  // appending needs head-room
    p.rows = ok ? (p.evict ? ln : ln + 1) : -1;
    p.len_after = p.rows;
    return p;
}
__device__ __forceinline__ SegPlan segment_plan(const DecodePlanArgs &a, int si)
{
    const int seg = (si / a.nl) * a.L + a.layer_begin + si % a.nl;
    return plan_of(a, a.len[seg], a.cap[seg], a.row_offset[seg], prune_state(a, seg));
}
// Writes what the step leaves for the next one: the length and, with pruning, the token's place.
// (Only one thread of the call touches a segment's token count and slot ring.)
__device__ __forceinline__ void segment_write(const DecodePlanArgs &a, int seg, int len_after, int dst, bool evict)
{
    a.len[seg] = len_after;
    const int d = a.append ? a.evict_distance : 0;
    if (d > 0) {
        const int g = a.gen[seg];
        int32_t *ring = a.slot_ring + (size_t)seg * (d + 1);
        if (evict) ring[(g - d) % (d + 1)] = -1;  // the token d steps back gave up its slot
        ring[g % (d + 1)] = dst;
        a.gen[seg] = g + 1;
    }
}
__device__ __forceinline__ void segment_advance(const DecodePlanArgs &a, int si, const SegPlan &sp)
{
    segment_write(a, (si / a.nl) * a.L + a.layer_begin + si % a.nl, sp.len_after, sp.dst, sp.evict);
}

// ---- flags: "this CTA has read the lengths" ----------------------------------------------------------
// One per CTA in the workspace, which may hold anything before; raised with the call's token, an odd number.
// A flag of kGone ^ token belongs to a CTA that is no longer waited for.
constexpr unsigned long long kGone = 2;

// One thread of a CTA: this CTA has read the lengths.  What the flag held goes to unraise_flag when the CTA's work
// is done (and the answer has come): when nobody was waiting any more, it puts the flag to zero; true then.
__device__ __forceinline__ unsigned long long raise_flag(unsigned long long *flag, unsigned long long token)
{
    unsigned long long held;
    asm volatile("atom.release.gpu.exch.b64 %0, [%1], %2;" : "=l"(held) : "l"(flag), "l"(token) : "memory");
    return held;
}
__device__ __forceinline__ void lower_flag(unsigned long long *flag) { *(volatile unsigned long long *)flag = 0ull; }
__device__ __forceinline__ bool unraise_flag(unsigned long long *flag, unsigned long long token, unsigned long long held)
{
    const bool late = held == (token ^ kGone);
    if (late) lower_flag(flag);
    return late;
}

__device__ __forceinline__ unsigned long long load_flag(const unsigned long long *flag)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(v) : "l"(flag) : "memory");
    return v;
}

// A whole CTA: waits for n flags and puts them back to zero.  False when the limit ran out: the flags
// of those that have come are zero then, the others' get zero from their own CTAs when these come.
__device__ __forceinline__ bool settle_flags(unsigned long long *flags, int n, unsigned long long token, uint32_t limit)
{
    constexpr int kBatch = 8;  // flags of a thread asked for at once
    bool all_in = true;
    for (int i0 = threadIdx.x; i0 < n && all_in; i0 += kBatch * blockDim.x) {
        unsigned long long v[kBatch];
#pragma unroll
        for (int e = 0; e < kBatch; ++e) {
            const int i = i0 + e * (int)blockDim.x;
            v[e] = i < n ? load_flag(flags + i) : token;
        }
#pragma unroll
        for (int e = 0; e < kBatch; ++e)
            for (uint32_t t = 0; v[e] != token && t < limit; ++t) v[e] = load_flag(flags + i0 + e * blockDim.x);
#pragma unroll
        for (int e = 0; e < kBatch; ++e) all_in = all_in && v[e] == token;
    }
    // (as raise_flag releases: what follows comes after the reads that the flags stand for)
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    all_in = __syncthreads_and(all_in);
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        if (all_in || atomicExch(flags + i, token ^ kGone) == token) lower_flag(flags + i);
    return all_in;
}

// ---- counts: how many of a segment's CTAs have read its length ----------------------------------------
// One word per segment in the workspace, which may hold anything before: a tag of this process in the upper bits says that the
// lower ones are a count.  Calls leave it at none.
constexpr int kVisitBits = 20;
constexpr int kVisitStride = 16;  // words from one segment's to the next (in one line, 32 segments' counts are made one by one: +0.1 us)

inline unsigned long long visit_tag()
{
    static const unsigned long long tag =
        (0x9e3779b97f4a7c15ull ^ (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count()) << kVisitBits;
    return tag;
}
// One thread of a CTA, after its reads; `seen` is what the word held a moment ago.  Tag and count, itself not included: the first
// to come makes the word a count.  (Whether to count at all hangs on the length, so the count cannot come before its read;
// `others` asks for the same of what else was read.)
__device__ __forceinline__ unsigned long long count_visit(unsigned long long *word, unsigned long long tag, unsigned long long seen, bool others)
{
    unsigned long long before;
    if (others) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    if (seen >> kVisitBits != tag >> kVisitBits) {
        before = atomicCAS(word, seen, tag + 1);
        if (before == seen) return tag;
    }
    asm volatile("atom.relaxed.gpu.global.add.u64 %0, [%1], 1;" : "=l"(before) : "l"(word) : "memory");
    return before;
}
// The thread that found itself to be the last, before it writes what all have read.
__device__ __forceinline__ void settle_visits(unsigned long long *word, unsigned long long tag, bool others)
{
    if (others) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    *(volatile unsigned long long *)word = tag;
}

// ---- parts of an item that CTAs pass on: a flag of the same kind for each, which the CTA that takes the parts puts back ----
// A whole warp: waits for a part; false when the limit ran out.
__device__ __forceinline__ bool await_part(const unsigned long long *flag, unsigned long long token, uint32_t limit)
{
    unsigned long long v = load_flag(flag);
    for (uint32_t i = 0; v != token && i < limit; ++i) v = load_flag(flag);
    const bool came = __all_sync(0xffffffffu, v == token);
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    return came;
}
// One thread, after the part has been read or given up: the flag is zero again, or will be when a late part comes.
__device__ __forceinline__ void retire_part(unsigned long long *flag, unsigned long long token, bool came)
{
    if (came || atomicExch(flag, token ^ kGone) == token) lower_flag(flag);
}

}  // namespace pkv
