// Importance score (Sec. 3.2) of fp32 inputs on the bf16 tensor cores, in fp32 precision.
//
// Every fp32 element of magnitude 2^-110 and above is the exact sum of three bf16 numbers x = x0 + x1 + x2
// (8 significant bits each, rounded to nearest, so |x1| <= 2^-8 |x| and |x2| <= 2^-17 |x|; below that, what
// is lost is less than 2^-133).  A logit is the sum of the six products that matter, smallest first,
//   x0 y2 + x1 y1 + x2 y0 + x0 y1 + x1 y0 + x0 y0
// (the dropped x1 y2 + x2 y1 + x2 y2 are at most 2^-24 of the product), accumulated in fp32 by
// tcgen05.mma.  A single product that outweighs all others thus has an error of up to 2^-24 + 2^-23 (an FMA's
// 2^-24), a sum of many terms less than a chain of FMAs.  The tensor core truncates a sum where an FMA rounds it, so a long chain drifts
// towards zero; the large products of a logit are therefore spread over several accumulators
// (D = 128: one for each 64 elements; D = 64: one for each 16) that are added in registers.
// Measured against fp64 on N(0, 1) operands, D = 128: error of a logit 0.9e-6 rms, against 2.3e-6
// for a chain of fp32 FMAs, which rounds 128 times.
//
// Passes, tiles and work items are those of score_tc.cu.  What differs is how operands get to
// shared memory: eight loader warps read fp32 rows from global memory (a chunk of 128 rows x 64
// elements at a time, the next chunk's loads in flight while the current one is converted), split
// them and write the three bf16 tiles in the 128-byte swizzle that the tensor core reads.  One CTA
// per SM, 13 warps.  A prompt of at most 128 tokens is one tile: both passes then run on it in one
// launch (MODE 0), the second on the transposed product of the operands already in shared memory.
//
// Prompts of a few tiles keep their logits (MODE 3): one pass, one launch and the mean.
//
// Measured, 8 layers x 16 heads of 128, 777 tokens: 161 us for the whole call (1263 us with 64 x 64 tiles on FMA units; 167
// in two passes, 175 before a loader's lane took 32 bytes of a row at a time, with 16-byte stores and half the address
// arithmetic), 92 us with the caller's log-sum-exp.  A tile needs 48 MMAs of 64 clocks = 3072, during which their operands
// take all of shared memory's bandwidth; storing the split ones takes 768 more.  It takes 5250: the issuing warp
// waits 1250 of them for chunks.  Pairs of CTAs (cta_group::2, a streamed row split once for two tiles): 198 us.
// Sixteen loader warps leave 80 registers a thread and spill (211 us).  4 layers x 4 heads of 64, 300 tokens:
// 17.4 us (26.9 in two passes before), 128 tokens (one tile each): 10.2 us for the call (11.3 with the mean in a launch of its
// own, 30.7 with three FMA kernels).
// Reading the logits back: eight rows at a time 168 us, sixteen 161; by three warps of their own 177-187; kept in blocks that
// pass through shared memory 177-206 (memory's latency, not the stores, is what the warps wait for).
#include "score_tiles.cuh"

namespace pkv {

namespace {

constexpr int kReaders = 4;                  // accumulator reader warps (warps 0-3: one TMEM lane quarter each)
constexpr int kLoaders = 8;                  // loader warps (warps 5-12; warp 4 issues the MMAs)
constexpr int kRows = TT / kLoaders / 4;     // rows of a chunk per loader lane, eight elements of each
constexpr int kVecs = 2 * kRows;
constexpr int kSplitThreads = (kReaders + 1 + kLoaders) * 32;
constexpr int kRing = 2;                     // streamed chunks in shared memory
static_assert(kRing == 2, "with two chunks a tile, chunk c of every tile goes through ring slot c");
constexpr uint32_t kPart = TT * 128;         // bytes of one bf16 part of a chunk: 128 rows x 64 elements
constexpr uint32_t kChunk = 3 * kPart;
constexpr uint32_t kBuf = 256;               // tensor-memory columns of one of the two accumulator buffers
constexpr int kMeanHeads = 8;                // CTAs of a portable cluster
constexpr int kKeepTiles = 8, kKeepTilesFew = 16;  // tiles of the longest prompt whose logits are kept (1 MiB a CTA)
constexpr size_t kKeepCtas = 148;            // CTAs of such a call at most
constexpr size_t kPartBytes = 128u << 20;    // and its part sums: more segments than these hold take turns
constexpr int kBack = 16;                    // rows of them a warp reads back at a time
constexpr int kQueue = 4;                    // item numbers in flight between the loaders and the other roles

struct SplitArgs {
    const float *q, *k;
    pkv_strides qs, ks;
    const float *layer_scale;
    const float *lse_in;  // pass 2: [B*L*H][N] log-sum-exp; times lse_mul it is in the log2 domain
    float lse_mul;
    float *lse2;          // pass 1 out, same layout, log2 domain
    float *partial;       // [B*L*H][N] per-head column sums; mode 3: [B*L*H][pairs of a query and a key tile][quarter of the queries][128]
    float *logits;        // mode 3: [CTA][tiles][128 queries][128 keys], of the item at hand
    float *scores;        // mode 0 by clusters (below): [B*L][N], or NULL
    int32_t *abort_word;  // set when a bounded wait runs out: the head mean then writes NaN scores
    int *next_item;       // work counter of this pass, zeroed before it; NULL: a CTA takes item blockIdx.x alone
    int clear_abort;      // this launch is the call's first and nothing has zeroed the abort word
    int L, H, N, tiles, nsh, group;
};

// One float into its three bf16 parts, two elements at a time (packed low, high).  (Above the largest bf16,
// 2^128 - 2^120, the first part is infinite and the logit is formed by FMA, see below.)
__device__ __forceinline__ void split2(float x, float y, uint32_t &p0, uint32_t &p1, uint32_t &p2)
{
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p0) : "f"(y), "f"(x));
    const float2 neg = make_float2(-1.f, -1.f);  // (the remainders are exact, whichever way they are formed)
    const float2 r = fma2(make_float2(__uint_as_float(p0 << 16), __uint_as_float(p0 & 0xffff0000u)), neg, make_float2(x, y));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p1) : "f"(r.y), "f"(r.x));
    const float2 u = fma2(make_float2(__uint_as_float(p1 << 16), __uint_as_float(p1 & 0xffff0000u)), neg, r);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2) : "f"(u.y), "f"(u.x));
}

// An accumulator buffer holds one unit of a tile: UN columns, in NACC partial accumulators.
template <int D> struct Unit {
    static constexpr int UN = D == 128 ? 128 : 64;
    static constexpr int NACC = (int)kBuf / UN;
    static constexpr int PER_TILE = TT / UN;
    static constexpr int BLOCKS = UN / 32;  // 32-column blocks of a unit
};

// Logits of 32 columns: the sum of the partial accumulators.
template <int D> __device__ __forceinline__ void load_logits(uint32_t taddr, float (&v)[32])
{
    float w[32];
    tmem_ld32x2(taddr, taddr + Unit<D>::UN, v, w);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] += w[i];
    if (Unit<D>::NACC == 4) {
        float x[32];
        tmem_ld32x2(taddr + 2 * Unit<D>::UN, taddr + 3 * Unit<D>::UN, w, x);
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] += w[i] + x[i];
    }
}

// What the parts cannot carry -- an element whose first part is infinite, so that its remainder is NaN, and products whose parts pass the
// range where the product itself may not -- comes out as a NaN logit.  The thread that finds its sum turned
// NaN by a tile forms that tile's logits again from the inputs with fp32 FMAs, so that NaN remains only
// where the definition has one.  (A sum that is NaN already stays: nothing can change it.)
template <int D> __device__ __forceinline__ float fma_logit(const float *x, const float *y)
{
    float s = 0.f;
#pragma unroll 4
    for (int d = 0; d < D; d += 4) {
        const float4 u = __ldg(reinterpret_cast<const float4 *>(x + d)), v = __ldg(reinterpret_cast<const float4 *>(y + d));
        s = fmaf(u.w, v.w, fmaf(u.z, v.z, fmaf(u.y, v.y, fmaf(u.x, v.x, s))));
    }
    return s;
}
__device__ __forceinline__ const float *head_rows(const float *p, const pkv_strides &st, const SplitArgs &a, int sh)
{
    const int seg = sh / a.H, h = sh - seg * a.H, b = seg / a.L, l = seg - b * a.L;
    return p + b * st.b + l * st.l + h * st.h;
}
__device__ __forceinline__ void store8(float *p, const float *v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]),
                 "f"(v[6]), "f"(v[7])
                 : "memory");
}

// Running maximum and sum of a query over the keys of the tile from key0 on; `keep` (or NULL) gets the logits.
template <int D>
__device__ __noinline__ float2 redo_lse(const SplitArgs &a, int sh, int query, int key0, float sc, float run_max, float run_sum, float *keep)
{
    const float *q = head_rows(a.q, a.qs, a, sh) + query * a.qs.n, *k = head_rows(a.k, a.ks, a, sh);
    for (int key = key0; key <= min(query, key0 + TT - 1); ++key) {
        const float v = fma_logit<D>(q, k + key * a.ks.n), x = v * sc;
        if (keep) keep[key - key0] = v;
        const float nm = fmaxf(run_max, x), base = nm == -INFINITY ? 0.f : nm;
        run_sum = fmaf(run_sum, ex2(run_max - base), ex2(x - base));
        run_max = nm;
    }
    return make_float2(run_max, run_sum);
}
// Probabilities that a key gets from the queries of the tile from query0 on; lse = their normalisers.
template <int D>
__device__ __noinline__ float redo_colsum(const SplitArgs &a, int sh, int key, int query0, const float *lse, float sc)
{
    const float *q = head_rows(a.q, a.qs, a, sh), *k = head_rows(a.k, a.ks, a, sh) + key * a.ks.n;
    float sum = 0.f;
    for (int m = max(key, query0); m < min(a.N, query0 + TT); ++m)
        sum += ex2(fmaf(fma_logit<D>(q + m * a.qs.n, k), sc, -lse[m - query0]));
    return sum;
}

// MODE 3: as MODE 1, and the item's logits are kept (64 KiB a tile, half of which go no further than the L2); once a query's
// normaliser is known, the reader warp that has its row reads them back and adds up what the warp's queries give to every
// key: the second pass without its products and splits.
// MODE 1: stationary = Q tile t, streamed = K tiles 0..t (log-sum-exp).  MODE 2: stationary = K tile
// t, streamed = Q tiles t..tiles-1 (column sums).  MODE 0: one tile, Q stationary, both results.  With a CTA for every
// head and at most eight heads a segment's CTAs are a cluster, whose first one takes the mean: no second launch.
template <int MODE, int D>
__global__ void __launch_bounds__(kSplitThreads, 1) score_split_kernel(const __grid_constant__ SplitArgs a)
{
    constexpr int KH = D / 64;
    constexpr int PASS = MODE == 2 ? 2 : 1;
    using U = Unit<D>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base;                 // [KH] chunks
    unsigned char *sB = base + KH * kChunk;   // [kRing] chunks
    __shared__ __align__(8) uint64_t a_full[KH], a_empty[KH], b_full[kRing], b_empty[kRing], s_full[2], s_empty[2],
        q_full[kQueue], q_empty[kQueue], lse_full[2], drained;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ int q_item[kQueue];
    __shared__ __align__(16) float s_lse[2][kReaders][TT];
    __shared__ float s_col[MODE == 0 ? TT : 1], s_cols[MODE == 0 ? kMeanHeads : 1][MODE == 0 ? TT : 1];  // column sums; (first CTA) those of all heads
    __shared__ int s_gave_up[MODE == 0 ? kMeanHeads : 1];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int nitems = a.nsh * a.tiles;

    if (tid == 0) {
        s_abort = 0;
        for (int i = 0; i < KH; ++i) {
            bar_init(a_full + i, kLoaders);
            bar_init(a_empty + i, 1);
        }
        for (int i = 0; i < kRing; ++i) {
            bar_init(b_full + i, kLoaders);
            bar_init(b_empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(s_full + i, 1);
            bar_init(s_empty + i, kReaders);
            bar_init(lse_full + i, kReaders);
        }
        for (int i = 0; i < kQueue; ++i) {
            bar_init(q_full + i, 1);
            bar_init(q_empty + i, kReaders + 1 + kLoaders);
        }
        bar_init(&drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kReaders) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(2 * kBuf)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const bool by_cluster = MODE == 0 && a.scores != nullptr;
    // (the first CTA must be running before anyone writes to its shared memory)
    if (by_cluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = tmem_slot;
    dependent_entry();  // the set-up above overlapped the kernel before this one; its results are read from here on
    if (a.clear_abort && blockIdx.x == 0 && tid == 0) *a.abort_word = 0;

    if (warp > kReaders) {
        // ---- loaders: fp32 rows -> three bf16 parts in shared memory --------------------------------
        const int lw = warp - kReaders - 1;
        // Lane: eight neighbouring elements of the rows r0, r0 + 4, ... of a chunk.
        const int r0 = lw * 4 * kRows + (lane >> 3), c8 = lane & 7;
        const uint32_t off0 = r0 * 128 + ((c8 ^ (r0 & 7)) << 4), off1 = (off0 ^ 64u) + 512u;  // rows r0 + 8 i and r0 + 8 i + 4
        bool dead = false;
        Ring2 rb{0, 0u}, rq{0, 0u}, rp{0, 0u};
        uint32_t a_phase = 0;
        // the chunk whose global loads come next: steps of the item done and in all; of either operand the place of this
        // lane's first row in the tile at hand, a row's length, and how many rows from there the prompt still has
        int step = 0, nsteps = 0, a_left = 0, b_left = 0;
        const float *pa = nullptr, *pb = nullptr;
        int64_t an = 0, bn = 0;
        // (only the announcing thread) the next item number, asked for one item ahead
        int ahead = blockIdx.x;
        if (a.next_item && lw == 0 && lane == 0) ahead = atomicAdd(a.next_item, 1);
        auto announce = [&]() {  // publishes one item number, or -1 for the end
            const int v = ahead < nitems ? ahead : -1;
            if (v >= 0) ahead = a.next_item ? atomicAdd(a.next_item, 1) : nitems;
            bar_wait(q_empty + rp.idx, rp.phase ^ 1u, dead, &s_abort);
            if (dead) return;
            q_item[rp.idx] = v;
            bar_arrive(q_full + rp.idx);
            rp.next(kQueue);
        };
        auto next_item = [&]() {
            if (lw == 0 && lane == 0) announce();
            warp_wait(q_full + rq.idx, rq.phase, dead, &s_abort);
            const int w = dead ? -1 : *(volatile int *)(q_item + rq.idx);
            __syncwarp();
            if (lane == 0) bar_arrive(q_empty + rq.idx);
            rq.next(kQueue);
            if (w < 0) {
                nsteps = -1;  // (nothing comes after the end)
                return;
            }
            int sh, t;
            decode_item<PASS>(w, a.nsh, a.tiles, a.group, sh, t);
            const int seg = sh / a.H, h = sh - seg * a.H, b = seg / a.L, l = seg - b * a.L;
            const float *qb = a.q + b * a.qs.b + l * a.qs.l + h * a.qs.h + c8 * 8;
            const float *kb = a.k + b * a.ks.b + l * a.ks.l + h * a.ks.h + c8 * 8;
            const int arow = t * TT + r0, brow = (PASS == 1 ? 0 : t) * TT + r0;
            an = PASS == 1 ? a.qs.n : a.ks.n;
            bn = PASS == 1 ? a.ks.n : a.qs.n;
            pa = (PASS == 1 ? qb : kb) + arow * an;
            pb = (PASS == 1 ? kb : qb) + brow * bn;
            a_left = a.N - arow;
            b_left = a.N - brow;
            step = 0;
            nsteps = KH + KH * (PASS == 1 ? t + 1 : a.tiles - t);
        };
        // Steps of an item: the stationary chunk c and the first streamed tile's chunk c in turn, then
        // the chunks of the other streamed tiles.
        auto fetch = [&](float4 (&x)[kVecs], int &where) {
            if (step == nsteps) next_item();
            if (nsteps < 0) {
                where = -1;
                return;
            }
            const bool head = step < 2 * KH, is_a = head && (step & 1) == 0;
            const int c = KH == 1 ? 0 : head ? step >> 1 : step & 1;
            const int64_t rn = is_a ? an : bn;
            const float *p = (is_a ? pa : pb) + c * 64;
            const int left = is_a ? a_left : b_left;
            if (!is_a && c == KH - 1) {  // the streamed tile's last chunk
                pb += TT * bn;
                b_left -= TT;
            }
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const float4 *v = reinterpret_cast<const float4 *>(p + 4 * i * rn);
                x[2 * i] = 4 * i < left ? __ldg(v) : zero;
                x[2 * i + 1] = 4 * i < left ? __ldg(v + 1) : zero;
            }
            where = is_a ? c : KH;  // which stationary chunk, or KH: the ring
            ++step;
        };
        auto store = [&](const float4 (&x)[kVecs], int where) {
            unsigned char *dst;
            uint64_t *full;
            if (where < KH) {
                warp_wait(a_empty + where, a_phase ^ 1u, dead, &s_abort);
                dst = sA + where * kChunk;
                full = a_full + where;
                if (where == KH - 1) a_phase ^= 1u;
            } else {
                warp_wait(b_empty + rb.idx, rb.phase ^ 1u, dead, &s_abort);
                dst = sB + rb.idx * kChunk;
                full = b_full + rb.idx;
                rb.next(kRing);
            }
            if (dead) return;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                uint4 p0, p1, p2;
                split2(x[2 * i].x, x[2 * i].y, p0.x, p1.x, p2.x);
                split2(x[2 * i].z, x[2 * i].w, p0.y, p1.y, p2.y);
                split2(x[2 * i + 1].x, x[2 * i + 1].y, p0.z, p1.z, p2.z);
                split2(x[2 * i + 1].z, x[2 * i + 1].w, p0.w, p1.w, p2.w);
                unsigned char *d = dst + (i % 2 == 0 ? off0 : off1) + i / 2 * 1024;
                *reinterpret_cast<uint4 *>(d) = p0;
                *reinterpret_cast<uint4 *>(d + kPart) = p1;
                *reinterpret_cast<uint4 *>(d + 2 * kPart) = p2;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) bar_arrive(full);
        };
        float4 x0[kVecs], x1[kVecs];
        int w0, w1;
        fetch(x0, w0);
        while (w0 >= 0 && !dead) {
            fetch(x1, w1);
            store(x0, w0);
            if (w1 < 0 || dead) break;
            fetch(x0, w0);
            store(x1, w1);
        }
    } else if (warp == kReaders) {
        // ---- MMA issuer: the whole warp walks the stream, one elected lane issues.  (Every value that
        // an MMA takes is then the same in all lanes and can be formed in uniform registers ahead of it;
        // with a single lane in the loop each MMA waited for its operands to be moved there, and 128 x
        // 128 x 16 took 94-108 clocks of its 64.) --------------------------------------------------------
        bool dead = false;
        uint32_t a_phase = 0;
        Ring2 rb{0, 0u}, rs{0, 0u}, rq{0, 0u};
        const uint64_t da = smem_desc(saddr(sA)), db = smem_desc(saddr(sB));
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(U::UN >> 3) << 17) |
                                   ((uint32_t)(TT >> 4) << 24);  // as kIdesc, N = UN
        // One chunk's products, smallest first, into its accumulators of buffer d_tmem: D = 128
        // accumulator c; D = 64 (one chunk) accumulator 0 up to the first large product, then one each.
        // x, y describe part 0 of the operands.
        auto issue = [&](uint32_t d_tmem, int c, uint64_t x, uint64_t y) {
            constexpr int px[6] = {0, 1, 2, 0, 1, 0}, py[6] = {2, 1, 0, 1, 0, 0};
#pragma unroll
            for (int m = 0; m < 6; ++m)
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    const int acc = KH == 2 ? c : (m == 5 ? ks : 0);
                    mma_bf16(d_tmem + acc * U::UN, desc_add(x, px[m] * kPart + ks * 32), desc_add(y, py[m] * kPart + ks * 32), idesc,
                             KH == 2 ? ((m | ks) != 0) : (m != 5 ? ((m | ks) != 0) : ks == 0));
                }
        };
        for (;;) {
            warp_wait(q_full + rq.idx, rq.phase, dead, &s_abort);
            if (dead) break;
            const int w = __shfl_sync(0xffffffffu, *(volatile int *)(q_item + rq.idx), 0);
            __syncwarp();
            if (lane == 0) bar_arrive(q_empty + rq.idx);
            rq.next(kQueue);
            if (w < 0) break;
            int sh, t;
            decode_item<PASS>(w, a.nsh, a.tiles, a.group, sh, t);
            const int count = PASS == 1 ? t + 1 : a.tiles - t;
            for (int jj = 0; jj < count; ++jj) {
                if (KH == 2) {  // one unit of 128 columns; its two chunks are the ring's two slots
                    warp_wait(s_empty + rs.idx, rs.phase ^ 1u, dead, &s_abort);
#pragma unroll
                    for (int c = 0; c < KH; ++c) {
                        if (jj == 0) warp_wait(a_full + c, a_phase, dead, &s_abort);
                        warp_wait(b_full + c, rb.phase, dead, &s_abort);
                        if (dead) break;
                        fence_after();
                        if (elect_one()) {
                            issue(tmem_base + rs.idx * kBuf, c, desc_add(da, c * kChunk), desc_add(db, c * kChunk));
                            if (MODE != 0) {
                                mma_commit(b_empty + c);
                                if (jj == count - 1) mma_commit(a_empty + c);
                            }
                            if (c == KH - 1) mma_commit(s_full + rs.idx);
                        }
                    }
                    if (dead) break;
                    rs.next(2);
                    if (MODE == 0) {  // the transposed product: keys on the lanes
                        warp_wait(s_empty + rs.idx, rs.phase ^ 1u, dead, &s_abort);
                        if (dead) break;
                        fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int c = 0; c < KH; ++c) {
                                issue(tmem_base + rs.idx * kBuf, c, desc_add(db, c * kChunk), desc_add(da, c * kChunk));
                                mma_commit(b_empty + c);
                                mma_commit(a_empty + c);
                            }
                            mma_commit(s_full + rs.idx);
                        }
                        rs.next(2);
                    }
                    rb.phase ^= 1u;
                } else {  // two units of 64 columns each
                    if (jj == 0) warp_wait(a_full, a_phase, dead, &s_abort);
                    warp_wait(b_full + rb.idx, rb.phase, dead, &s_abort);
                    const uint64_t dk = desc_add(db, rb.idx * kChunk);
#pragma unroll
                    for (int u = 0; u < (MODE == 0 ? 2 : 1) * U::PER_TILE; ++u) {
                        warp_wait(s_empty + rs.idx, rs.phase ^ 1u, dead, &s_abort);
                        if (dead) break;
                        fence_after();
                        const uint32_t rows = (u % U::PER_TILE) * (U::UN * 128);
                        const bool swap = u >= U::PER_TILE;  // (MODE 0) the transposed product
                        if (elect_one()) {
                            issue(tmem_base + rs.idx * kBuf, 0, swap ? dk : da, desc_add(swap ? da : dk, rows));
                            mma_commit(s_full + rs.idx);
                            if (u == (MODE == 0 ? 2 : 1) * U::PER_TILE - 1) {
                                mma_commit(b_empty + rb.idx);
                                if (jj == count - 1) mma_commit(a_empty);
                            }
                        }
                        rs.next(2);
                    }
                    if (dead) break;
                    rb.next(kRing);
                }
            }
            if (dead) break;
            a_phase ^= 1u;
        }
        if (dead) {  // let the products in flight finish before the CTA can exit (bounded)
            if (elect_one()) mma_commit(&drained);
            drain(&drained, 0u);
        }
    } else {
        // ---- accumulator readers: one TMEM lane (tile row) per thread --------------------------------
        const int row = warp * 32 + lane;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(warp * 32) << 16);
        bool dead = false;
        Ring2 rs{0, 0u}, rq{0, 0u};
        int flip = 0;
        uint32_t lse_phase = 0;
        auto release = [&]() {
            fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(s_empty + rs.idx);
            rs.next(2);
        };
        // Column sums of a tile; on the diagonal tile only the blocks from this warp's keys on count.
        auto sum_tile = [&](const float *lse, int sh, int key, int tile, bool diag, float sc, float &col_sum) {
            const float before = col_sum;
            for (int u = 0; u < U::PER_TILE; ++u) {
                warp_wait(s_full + rs.idx, rs.phase, dead, &s_abort);
                fence_after();
#pragma unroll 1
                for (int cb = max(diag ? warp : 0, u * U::BLOCKS); cb < (u + 1) * U::BLOCKS; ++cb) {
                    float v[32];
                    load_logits<D>(lane_addr + rs.idx * kBuf + (cb - u * U::BLOCKS) * 32, v);
                    col_sum += colsum_block<32, 0>(v, lse + cb * 32, sc, diag && cb == warp, lane);
                }
                release();
            }
            const bool redo = col_sum != col_sum && before == before && key < a.N;
            if (__any_sync(0xffffffffu, redo)) {
                if (redo) col_sum = before + redo_colsum<D>(a, sh, key, tile * TT, lse, sc);
                __syncwarp();
            }
        };
        for (;;) {
            warp_wait(q_full + rq.idx, rq.phase, dead, &s_abort);
            if (dead) break;
            const int w = *(volatile int *)(q_item + rq.idx);
            __syncwarp();
            if (lane == 0) bar_arrive(q_empty + rq.idx);
            rq.next(kQueue);
            if (w < 0) break;
            int sh, t;
            decode_item<PASS>(w, a.nsh, a.tiles, a.group, sh, t);
            const float sc = a.layer_scale[(sh / a.H) % a.L] * kLog2eT;
            const int grow = t * TT + row;  // query (pass 1) or key (pass 2) of this thread
            float *kept = MODE == 3 ? a.logits + ((size_t)blockIdx.x * a.tiles * TT + row) * TT : nullptr;
            float run_max = -INFINITY, run_sum = 0.f, col_sum = 0.f;
            if (PASS == 1) {
                for (int j = 0; j <= t; ++j) {
                    // on the diagonal tile only the 32-column blocks up to this warp's rows count
                    const int c_hi = j == t ? warp : TT / 32 - 1;
                    const float old_max = run_max, old_sum = run_sum;
                    for (int u = 0; u < U::PER_TILE; ++u) {
                        warp_wait(s_full + rs.idx, rs.phase, dead, &s_abort);
                        fence_after();
#pragma unroll 1
                        for (int cb = u * U::BLOCKS; cb < (u + 1) * U::BLOCKS && cb <= c_hi; ++cb) {
                            float v[32];
                            load_logits<D>(lane_addr + rs.idx * kBuf + (cb - u * U::BLOCKS) * 32, v);
                            if (MODE == 3) {
#pragma unroll
                                for (int i = 0; i < 32; i += 8) store8(kept + j * TT * TT + cb * 32 + i, v + i);
                            }
                            if (j == t && cb == warp) {  // the block the causal boundary crosses
#pragma unroll
                                for (int i = 0; i < 32; ++i) v[i] = i <= lane ? v[i] : -INFINITY;
                            }
                            lse_block<32, 0>(v, sc, sc > 0.f, run_max, run_sum);
                        }
                        release();
                    }
                    const bool redo = run_sum != run_sum && old_sum == old_sum && grow < a.N;
                    if (__any_sync(0xffffffffu, redo)) {
                        if (redo) {
                            const float2 r = redo_lse<D>(a, sh, grow, j * TT, sc, old_max, old_sum, MODE == 3 ? kept + j * TT * TT : nullptr);
                            run_max = r.x;
                            run_sum = r.y;
                        }
                        __syncwarp();
                    }
                }
                const float lse = run_max + log2f(run_sum);
                if (MODE == 3) {
                    // What the warp's 32 queries give to every key of a tile, four keys to a lane.
                    __syncwarp();  // (the rows are the warp's own: its lanes' stores are seen from here on)
                    const int rows = min(32, a.N - t * TT - warp * 32);
                    const float *back = kept - lane * TT + lane * 4;
                    float *out = a.partial + ((size_t)sh * (a.tiles * (a.tiles + 1) / 2) + t * (t + 1) / 2) * (4 * TT) + warp * TT + lane * 4;
                    for (int j = 0; j <= t; ++j) {
                        float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
                        const int edge = j == t ? warp * 32 - lane * 4 : TT;  // key e of query i counts when e <= edge + i
#pragma unroll 1
                        for (int i0 = 0; i0 < rows; i0 += kBack) {
                            float4 x[kBack];
#pragma unroll
                            for (int i = 0; i < kBack; ++i)  // (rows past the prompt's end have a place too, and are left out below)
                                x[i] = __ldcg(reinterpret_cast<const float4 *>(back + j * TT * TT + (i0 + i) * TT));
#pragma unroll
                            for (int i = 0; i < kBack; ++i) {
                                const float nl = -__shfl_sync(0xffffffffu, lse, i0 + i);
                                const int last = i0 + i < rows ? edge + i0 + i : -1;
                                s0.x += last >= 0 ? ex2(fmaf(x[i].x, sc, nl)) : 0.f;
                                s0.y += last >= 1 ? ex2(fmaf(x[i].y, sc, nl)) : 0.f;
                                s1.x += last >= 2 ? ex2(fmaf(x[i].z, sc, nl)) : 0.f;
                                s1.y += last >= 3 ? ex2(fmaf(x[i].w, sc, nl)) : 0.f;
                            }
                        }
                        *reinterpret_cast<float4 *>(out + j * (4 * TT)) = make_float4(s0.x, s0.y, s1.x, s1.y);
                    }
                    __syncwarp();  // the next item's logits go to the same place
                } else if (MODE == 1) {
                    if (grow < a.N) a.lse2[(size_t)sh * a.N + grow] = lse;
                } else {
                    // every reader warp needs all 128 normalisers (two buffers in turn, so that
                    // no warp can write a buffer that another still reads)
                    s_lse[flip][0][row] = grow < a.N ? lse : INFINITY;
                    __syncwarp();
                    if (lane == 0) bar_arrive(lse_full + flip);
                    warp_wait(lse_full + flip, lse_phase, dead, &s_abort);
                    sum_tile(s_lse[flip][0], sh, grow, t, true, sc, col_sum);
                    flip ^= 1;
                    if (flip == 0) lse_phase ^= 1u;
                    if (by_cluster) s_col[row] = col_sum;
                    else if (grow < a.N) a.partial[(size_t)sh * a.N + grow] = col_sum;
                }
            } else {
                const float *lrow = a.lse_in + (size_t)sh * a.N;
                // four of the tile's 128 query normalisers per lane, fetched a tile ahead; each warp keeps its own copy
                float4 mine;
                auto get = [&](int j) {
                    const int m = j * TT + lane * 4;
                    mine.x = m < a.N ? __ldg(lrow + m) * a.lse_mul : INFINITY;
                    mine.y = m + 1 < a.N ? __ldg(lrow + m + 1) * a.lse_mul : INFINITY;
                    mine.z = m + 2 < a.N ? __ldg(lrow + m + 2) * a.lse_mul : INFINITY;
                    mine.w = m + 3 < a.N ? __ldg(lrow + m + 3) * a.lse_mul : INFINITY;
                };
                get(t);
                for (int j = t; j < a.tiles; ++j) {
                    __syncwarp();
                    const int buf = j & 1;
                    reinterpret_cast<float4 *>(s_lse[buf][warp])[lane] = mine;
                    if (j + 1 < a.tiles) get(j + 1);
                    __syncwarp();
                    sum_tile(s_lse[buf][warp], sh, grow, j, j == t, sc, col_sum);
                }
                if (grow < a.N) a.partial[(size_t)sh * a.N + grow] = col_sum;
            }
        }
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0 && s_abort && !by_cluster) atomicExch(a.abort_word, (int)PKV_DEV_TIMEOUT);
    if (warp == kReaders) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * kBuf) : "memory");
    }
    if (MODE == 0 && by_cluster) {
        const int seg = blockIdx.x / a.H, h = blockIdx.x - seg * a.H;
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        if (tid < TT) store_in_first_cta(&s_cols[h][tid], s_col[tid]);
        if (tid == 0) store_in_first_cta(reinterpret_cast<float *>(s_gave_up + h), __int_as_float(s_abort));
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (h != 0) return;  // (only the first CTA's memory is written, and it waits for everyone)
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (tid < a.N) {  // (at most a tile)
            float sum = 0.f;
            int gave_up = 0;
            for (int i = 0; i < a.H; ++i) {
                sum += s_cols[i][tid];
                gave_up |= s_gave_up[i];
            }
            a.scores[(size_t)seg * a.N + tid] = gave_up ? __int_as_float(0x7fc00000) : sum / (float)a.H;
        }
    }
}

// Mode 3's part sums: 32 keys of a segment to a block, a warp to the heads w, w + 8, ...; the sums of the warps in order.
__global__ void __launch_bounds__(256) split_mean_kernel(const float *__restrict__ partial, int H, int N, int tiles, float *__restrict__ scores,
                                                         const int32_t *__restrict__ abort_word)
{
    __shared__ float s_sum[8][32];
    const int blocks = (N + 31) / 32, seg = blockIdx.x / blocks, n = (blockIdx.x - seg * blocks) * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
    const int j = n / TT, all = tiles * (tiles + 1) / 2;
    dependent_entry();
    float sum = 0.f;
    for (int h = w; h < H; h += 8) {
        const float *p = partial + (size_t)(seg * H + h) * all * (4 * TT) + n % TT;
        for (int t = j; t < tiles; ++t) {
            const float *q = p + (size_t)(t * (t + 1) / 2 + j) * (4 * TT);
            sum += (__ldcg(q) + __ldcg(q + TT)) + (__ldcg(q + 2 * TT) + __ldcg(q + 3 * TT));
        }
    }
    s_sum[w][threadIdx.x & 31] = sum;
    __syncthreads();
    if (w != 0 || n >= N) return;
    for (int i = 1; i < 8; ++i) sum += s_sum[i][threadIdx.x];
    scores[(size_t)seg * N + n] = *abort_word != 0 ? __int_as_float(0x7fc00000) : sum / (float)H;
}

// (Calls of several turns) every score of a call is NaN when a wait in any of them ran out.
__global__ void __launch_bounds__(256) split_abort_kernel(float *__restrict__ scores, size_t total, const int32_t *__restrict__ abort_word)
{
    dependent_entry();
    if (*abort_word == 0) return;
    for (size_t i = blockIdx.x * 256ull + threadIdx.x; i < total; i += gridDim.x * 256ull) scores[i] = __int_as_float(0x7fc00000);
}

// Whether mode 3 takes a prompt, without the caller's log-sum-exp.  Us a call, tokens x heads:
//   heads of 128    two passes  kept      heads of 64     two passes  kept
//   130 x 192          53.0     37.4      256 x 192          49.3     36.9
//   300 x 1024          333      237      256 x 1536          227      160
//   777 x 128           168      163      777 x 128           146      128
//   1024 x 1024        1575     1540      1024 x 1536        1959     1872
//   1500 x 4           84.1     71.9      1152 x 128          224      231
//   1500 x 16           107      125      2048 x 1536        7086     8370
// With more than eight tiles to an item the logits in use leave the L2, unless a CTA has one item: with heads of 64, 1152 x 16
// 56.6 / 50.6, 1500 x 12 73.2 / 65.1, x 16 (192 items) 92.0 / 98.3, 2048 x 7 89.9 / 79.6, x 9 91.9 / 92.5.
size_t part_bytes(size_t heads, size_t tiles) { return heads * (tiles * (tiles + 1) / 2) * (4 * TT) * sizeof(float); }
bool keeps_logits(const pkv_shape *s)
{
    const size_t heads = (size_t)s->batch * s->layers * s->heads, tiles = ((size_t)s->prompt_len + TT - 1) / TT;
    if (s->dtype != PKV_F32 || tiles < 2 || part_bytes(s->heads, tiles) > kPartBytes) return false;
    return tiles <= kKeepTiles || (s->head_dim == 64 && tiles <= kKeepTilesFew && heads * tiles <= kKeepCtas);
}

template <int MODE, int D> int launch_split(const SplitArgs &a, int sms, cudaStream_t st)
{
    static bool done[64] = {};
    const size_t smem = (size_t)(D / 64 + kRing) * kChunk + 1024;
    int rc = ensure_dynamic_smem((const void *)score_split_kernel<MODE, D>, (int)smem, done);
    if (rc != PKV_OK) return rc;
    const int items = a.nsh * a.tiles;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)a.H;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(items < sms ? items : sms);
    cfg.blockDim = dim3(kSplitThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = a.scores ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, score_split_kernel<MODE, D>, a);
    if (e != cudaSuccess) {
        set_cuda_error(e, "score_split_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

}  // namespace

int launch_head_mean(const float *partial, int H, int N, size_t total, float *scores, const int32_t *abort_word,
                     cudaStream_t st);

// Workspace: partial [rows][N], lse2 [rows][N], then two work counters and the abort word.  Short prompts: part sums of every
// pair of tiles in the place of these, of as many segments at a time as kPartBytes hold, and the logits of a CTA's item, where the
// workspace has room for them: one that was sized for a longer prompt, or for the caller's log-sum-exp, need not, and then
// serves two passes.  (1024 tokens, us at once, in turns of 128 MiB, 64, 16: 6144 heads of 64, 432 MiB, 7386, 7498, 7589, 8182; 1024 heads
// of 128, 72 MiB, 1538, 1538, 1605, 1783.  A turn's first segment as an argument of the kernel instead of whole samples or layers of one:
// 300 tokens x 16 17.2 -> 17.8.)
struct SplitSpace {
    size_t partial, lse2, logits, words, bytes;
    int turn;  // segments of a turn: whole samples, or some of a sample's layers
};
static SplitSpace split_space(const pkv_shape *s, bool keep)
{
    const size_t segs = (size_t)s->batch * s->layers, heads = segs * s->heads, tiles = ((size_t)s->prompt_len + TT - 1) / TT;
    const size_t per = heads * s->prompt_len * sizeof(float);
    SplitSpace w = {0, per, 0, 0, 0, 0};
    size_t end = 2 * per;
    if (keep) {
        const size_t one = part_bytes(s->heads, tiles), most = kPartBytes / one, B = s->batch, L = s->layers;
        auto evenly = [](size_t n, size_t at_once) { const size_t turns = (n + at_once - 1) / at_once; return (n + turns - 1) / turns; };
        const size_t turn = most >= L ? evenly(B, most / L) * L : evenly(L, most);
        const size_t ctas = turn * s->heads * tiles < kKeepCtas ? turn * s->heads * tiles : kKeepCtas;
        w.turn = (int)turn;
        w.logits = round_up(turn * one, kWsAlign);
        const size_t kept = w.logits + ctas * tiles * TT * TT * sizeof(float);
        if (kept > end) end = kept;
    }
    w.words = round_up(end, kWsAlign);
    w.bytes = w.words + kWsAlign;
    return w;
}
size_t score_split_ws_bytes(const pkv_shape *s, bool least) { return split_space(s, !least && keeps_logits(s)).bytes; }

int launch_score_split(const pkv_shape *s, const float *q, pkv_strides qs, const float *k, pkv_strides ks,
                       const float *scale, const float *lse, float *scores, void *ws, size_t ws_bytes, cudaStream_t st)
{
    const int B = s->batch, L = s->layers, H = s->heads, N = s->prompt_len;
    const bool keep = !lse && keeps_logits(s) && ws_bytes >= split_space(s, true).bytes;
    const SplitSpace space = split_space(s, keep);
    unsigned char *mem = (unsigned char *)ws;
    SplitArgs a = {};
    a.q = q; a.k = k; a.qs = qs; a.ks = ks;
    a.layer_scale = scale;
    a.partial = (float *)(mem + space.partial);
    a.lse2 = (float *)(mem + space.lse2);
    a.logits = (float *)(mem + space.logits);
    int *words = (int *)(mem + space.words);
    a.abort_word = words + 2;
    a.L = L; a.H = H; a.N = N;
    a.tiles = (N + TT - 1) / TT;
    a.nsh = B * L * H;
    a.group = head_group(a.nsh, N, s->head_dim, 4);
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    // With an item for every CTA there is nothing to hand out: no counter, and so nothing to zero first.
    const bool counted = a.nsh * a.tiles > (sms < (int)kKeepCtas ? sms : (int)kKeepCtas);
    if (counted) {
        cudaError_t e = cudaMemsetAsync(words, 0, 4 * sizeof(int), st);
        if (e != cudaSuccess) {
            set_cuda_error(e, "cudaMemsetAsync(score work counters)");
            return PKV_ERR_CUDA;
        }
    }
    a.clear_abort = !counted;
    const bool wide = s->head_dim == 128;
    int rc = PKV_OK;
    if (!lse && a.tiles == 1) {
        a.next_item = counted ? words : nullptr;
        // (clusters that run at once: 12 segments of 8 heads 13.7 -> 10.5 us, 6 of 3 12.3 -> 10.7, but 16 of 8, 128 CTAs
        // of 148 SMs, take two waves, 13.9 -> 19.5)
        if (3 * a.nsh <= 2 * sms && H <= kMeanHeads) {
            a.scores = scores;
            return wide ? launch_split<0, 128>(a, sms, st) : launch_split<0, 64>(a, sms, st);
        }
        rc = wide ? launch_split<0, 128>(a, sms, st) : launch_split<0, 64>(a, sms, st);
    } else if (keep) {
        const int ctas = sms < (int)kKeepCtas ? sms : (int)kKeepCtas, segs = B * L;
        a.next_item = counted ? words : nullptr;
        for (int seg0 = 0, now; seg0 < segs; seg0 += now) {
            const int b0 = seg0 / L, l0 = seg0 % L, end = space.turn < L ? (b0 + 1) * L : segs;
            now = end - seg0 < space.turn ? end - seg0 : space.turn;
            a.q = q + b0 * qs.b + l0 * qs.l;
            a.k = k + b0 * ks.b + l0 * ks.l;
            a.layer_scale = scale + l0;
            a.nsh = now * H;
            a.group = head_group(a.nsh, N, s->head_dim, 4);
            cudaError_t e = seg0 > 0 ? cudaMemsetAsync(words, 0, sizeof(int), st) : cudaSuccess;
            if (e != cudaSuccess) {
                set_cuda_error(e, "cudaMemsetAsync(score work counter)");
                return PKV_ERR_CUDA;
            }
            rc = wide ? launch_split<3, 128>(a, ctas, st) : launch_split<3, 64>(a, ctas, st);
            if (rc != PKV_OK) return rc;
            e = launch_dependent(split_mean_kernel, dim3((unsigned)((size_t)now * ((N + 31) / 32))), dim3(256), 0, st, a.partial, H, N, a.tiles,
                                 scores + (size_t)seg0 * N, a.abort_word);
            if (e == cudaSuccess && now < segs && seg0 + now == segs)
                e = launch_dependent(split_abort_kernel, dim3((unsigned)sms), dim3(256), 0, st, scores, (size_t)segs * N, a.abort_word);
            if (e != cudaSuccess) {
                set_cuda_error(e, "split_mean_kernel");
                return PKV_ERR_CUDA;
            }
        }
        return PKV_OK;
    } else {
        if (!lse) {
            a.next_item = counted ? words : nullptr;
            rc = wide ? launch_split<1, 128>(a, sms, st) : launch_split<1, 64>(a, sms, st);
            if (rc != PKV_OK) return rc;
            a.clear_abort = 0;
        }
        a.lse_in = lse ? lse : a.lse2;
        a.lse_mul = lse ? kLog2eT : 1.f;
        a.next_item = counted ? words + 1 : nullptr;
        rc = wide ? launch_split<2, 128>(a, sms, st) : launch_split<2, 64>(a, sms, st);
    }
    if (rc != PKV_OK) return rc;
    return launch_head_mean(a.partial, H, N, (size_t)B * L * N, scores, a.abort_word, st);
}

}  // namespace pkv
