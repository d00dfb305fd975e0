// Importance score (Sec. 3.2) of bf16 prompts of up to five key tiles (640 tokens), both sums in one kernel.
//
// A CTA owns a head: all its keys sit in shared memory and its queries stream through in strips of 64.  The
// exponentials of a strip against every key it attends to fit in tensor memory (at most 5 x 64 of its 512 columns), so
// that each is computed once: it replaces its logit there while the strip's row sums are formed, and is then weighted
// with 1 / row sum into the keys' column sums.  The two-pass kernel of score_tc.cu reads Q and K twice and computes
// every exponential twice.
//
// A tile of logits is 128 keys (lanes of tensor memory) x 64 queries (columns): A = a key tile, B = a query strip.
// Tensor memory is a ring of eight tiles.  Odd and even strips have an MMA warp and a team of eight reader warps each,
// so that one team's exchange and weighing, and one MMA warp's waits, fall into the other's work.  A reader warp takes
// blocks of 32 keys (its lane quarter) x 32 queries: the exponentials in the 16x256b register layout, where a thread has
// 4 keys x 8 queries and a query's sum takes three shuffles and an exchange among four warps, the weighing with a key
// to a lane.
//
// Strips go from the last to the first and a head's last key tile is loaded first: tiles of the five-tile ring become
// free in the order of their loads, and the next head's come in while this one's last strips are still in work.
//
// The exponentials are of the logits themselves, without the maximum: that would be another walk over tensor memory with a
// barrier in it.  A head whose first blocks show logits (log2) above 60, or a query with none above -45, is taken relative to
// the maximum: in the later strips of such a head the four warps that share one exchange their maxima first; in the first strip
// a warp that sees such logits takes its own, as the other three may not see any, and with the sums' exchange all are brought to one
// scale.  A strip whose sum is out of 2^-80 ... 2^100 all the same (or NaN) has its head done again, after the CTA's others.
// 1024 heads of 128, 640 tokens: 125 us; with all heads relative to the maximum 178 (two passes 182 to 207), with one in eight
// 138.  With every such head done twice these took 118, 305 and 171; a look at every block instead of the first 144.
//
// What bounds it: the chain of short steps, not a unit.  A tile of 128 x 64 takes some 1000 clocks (of 385 to 430 in the
// tensor pipe and 512 in the special-function unit); the waits of an MMA warp and of a reader, 200 to 300 clocks each
// although complete, and a strip's exchange are what the second MMA warp and the second team are for.  The readers' code is kept
// short (one loop for both walks, one copy of the weighing): the same steps with the weighing unrolled over five tiles and a loop to
// each walk took 134.  Scores of 32 x 32 heads of 128: 640 tokens 182 us with two passes, 125 here; 300 tokens 87 and 56;
// 64 tokens 25 and 20.  Before the look at the first block 118, and of these without exponentials 109; one MMA warp 163; logits
// of a strip in registers (80 a thread) instead of exponentials put back 160, weighing by eight warps of their own 163; three
// teams 138; halves of a block loaded ahead 145; an eighth, a quarter of the exponentials on the FMA pipe 123, 126; two query
// stages 122; L2 prefetch of the next head 123.
//
// Every wait is bounded: when one runs out the CTA stops waiting, sets the call's abort word (the head mean then
// writes NaN for every score) and still releases its tensor memory.
#include "score_tiles.cuh"

namespace pkv {

bool score_make_map(CUtensorMap *map, const void *ptr, const pkv_shape *s, pkv_strides st, int box_rows);
int launch_head_mean(const float *partial, int H, int N, size_t total, float *scores, const int32_t *abort_word,
                     cudaStream_t st);

namespace {

constexpr int kMaxTiles = 5;       // key tiles of a head
constexpr int QS = 64;             // queries of a strip
constexpr int kSlots = 512 / QS;   // tiles in tensor memory
constexpr int kReadWarps = 16;     // two teams x two halves of a strip x four lane quarters
constexpr int kMmaWarp = 0, kLoadWarp = 2, kFlushWarp = 3, kFirstReader = 4;
constexpr int kFThreads = (kFirstReader + kReadWarps) * 32;
constexpr int kBadWords = 64;      // heads to be done again, a bit to each of the CTA's (modulo the bits there are)
// Sums of exponentials of the logits themselves that are taken: what flushes to zero is below 2^-46 of them, and
// neither they nor their reciprocals are near the ends of the range.
constexpr float kLowSum = 0x1p-80f, kHighSum = 0x1p+100f;
// Logits (log2) of a head's first block within which its maxima are not formed: some way from where the sums go out of range.
constexpr float kHighLogit = 60.f, kLowLogit = -45.f;
constexpr float kLowest = -1e30f;  // scale of a sum of nothing
constexpr uint32_t kIdescStrip = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(QS >> 3) << 17) | ((uint32_t)(TT >> 4) << 24);

struct FusedArgs {
    const float *layer_scale;
    float *partial;       // [B*L*H][N] per-head column sums
    int32_t *abort_word;
    int L, H, N, tiles, strips, heads;
};

template <int D> struct FusedSmem {
    static constexpr uint32_t KTILE = TT * D * 2, QTILE = QS * D * 2;
    static constexpr int kK = 5, kQ = D == 128 ? 3 : 6;  // stages of the two rings
    static constexpr size_t bytes = kK * (size_t)KTILE + kQ * (size_t)QTILE + sizeof(float) *
        (4 * kMaxTiles * TT + 4 * 2 * 4 * 32 + kReadWarps * 32) + 512 + 1024;
};

// As warp_wait, for a phase that is usually complete already.
__device__ __forceinline__ void warp_wait_ready(uint64_t *bar, uint32_t parity, bool &dead, int *abort_flag)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    if (!__all_sync(0xffffffffu, ok != 0)) warp_wait(bar, parity, dead, abort_flag);
}

// A block of 32 keys x 32 queries: a thread has, of 16-key half hf and 8-query group i, queries 2 * (lane % 4) + {0, 1}
// of keys lane / 4 (v[hf][i][0]) and lane / 4 + 8 (v[hf][i][1]).
typedef float2 Block[2][4][2];
#define PKV_HALF(T, v)                                                                                                 \
    T((v)[0][0].x), T((v)[0][0].y), T((v)[0][1].x), T((v)[0][1].y), T((v)[1][0].x), T((v)[1][0].y), T((v)[1][1].x),     \
        T((v)[1][1].y), T((v)[2][0].x), T((v)[2][0].y), T((v)[2][1].x), T((v)[2][1].y), T((v)[3][0].x), T((v)[3][0].y), \
        T((v)[3][1].x), T((v)[3][1].y)
__device__ __forceinline__ void block_load(uint32_t taddr, Block &v)
{
#pragma unroll
    for (int hf = 0; hf < 2; ++hf)
        asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 "
                     "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : PKV_HALF("=f", v[hf])
                     : "r"(taddr + ((uint32_t)hf << 20)));
    // (the values are there from here on)
    asm volatile("tcgen05.wait::ld.sync.aligned;" : PKV_HALF("+f", v[0]), PKV_HALF("+f", v[1])::"memory");
}
__device__ __forceinline__ void block_store(uint32_t taddr, const Block &v)
{
#pragma unroll
    for (int hf = 0; hf < 2; ++hf)
        asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%16], "
                     "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::PKV_HALF("f", v[hf]),
                     "r"(taddr + ((uint32_t)hf << 20))
                     : "memory");
}
#undef PKV_HALF
// The block the causal boundary crosses, `d` = the thread's first query less its first key: what lies beyond becomes `x`.
__device__ __forceinline__ void block_mask(Block &v, int d, float x)
{
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        const int hf = n >> 3, i = (n >> 1) & 3, rr = n & 1, at = d + 8 * i - 16 * hf - 8 * rr;
        v[hf][i][rr].x = at < 0 ? x : v[hf][i][rr].x;
        v[hf][i][rr].y = at + 1 < 0 ? x : v[hf][i][rr].y;
    }
}
// Whether the thread's logits are within the range: every query's largest of the four keys, unless all of these are masked.
__device__ __forceinline__ bool block_in_range(const Block &v, float sc)
{
    float up = 0.f, low = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float x = fmaxf(max3(v[0][i][0].x * sc, v[0][i][1].x * sc, v[1][i][0].x * sc), v[1][i][1].x * sc);
        const float y = fmaxf(max3(v[0][i][0].y * sc, v[0][i][1].y * sc, v[1][i][0].y * sc), v[1][i][1].y * sc);
        up = max3(up, x, y);
        low = fminf(low, fminf(x == -INFINITY ? 0.f : x, y == -INFINITY ? 0.f : y));
    }
    return up <= kHighLogit && low >= kLowLogit;
}
__device__ __forceinline__ float2 shfl_xor2(float2 v, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
// 32 columns of the warp's lanes, a lane to a thread.
__device__ __forceinline__ void tmem_ld_row(uint32_t taddr, float (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
          "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17]),
          "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]), "=f"(v[24]), "=f"(v[25]), "=f"(v[26]),
          "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]),
                   "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]), "+f"(v[16]),
                   "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]),
                   "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29])
                 :
                 : "memory");
    asm volatile("" : "+f"(v[30]), "+f"(v[31]));
}

template <int D>
__global__ void __launch_bounds__(kFThreads, 1)
score_fused_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const FusedArgs a)
{
    using SM = FusedSmem<D>;
    constexpr int KH = D / 64;
    constexpr uint32_t KBOX = TT * 128, QBOX = QS * 128;  // bytes of a box, 64 elements of every row
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sK = base, *sQ = sK + SM::kK * SM::KTILE;
    float *s_col = reinterpret_cast<float *>(sQ + SM::kQ * SM::QTILE);  // [team][half][tiles * 128]: a head's column sums
    float *s_x = s_col + 4 * kMaxTiles * TT;     // [team][half][2][quarter][32]: parts of a strip's sums
    float *s_w = s_x + 4 * 2 * 4 * 32;           // [warp][32]: a strip's weights
    uint64_t *bars = reinterpret_cast<uint64_t *>(s_w + kReadWarps * 32);
    uint64_t *k_full = bars, *k_empty = k_full + SM::kK, *q_full = k_empty + SM::kK, *q_empty = q_full + SM::kQ;
    uint64_t *s_full = q_empty + SM::kQ, *s_empty = s_full + 2 * kSlots, *c_full = s_empty + kSlots, *c_empty = c_full + 1;
    uint64_t *drained = c_empty + 1;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort, s_again;
    __shared__ int s_next[2];  // of either MMA warp: the next tile of its own (all before are issued)
    __shared__ uint32_t s_bad[kBadWords];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (tid < kBadWords) s_bad[tid] = 0;
    if (tid == 0) {
        s_abort = s_again = 0;
        for (int i = 0; i < SM::kK; ++i) {
            bar_init(k_full + i, 1);
            bar_init(k_empty + i, 2);
        }
        for (int i = 0; i < SM::kQ; ++i) {
            bar_init(q_full + i, 1);
            bar_init(q_empty + i, 2);
        }
        for (int i = 0; i < kSlots; ++i) {
            bar_init(s_empty + i, kReadWarps / 2);
        }
        for (int i = 0; i < 2 * kSlots; ++i) bar_init(s_full + i, 1);  // of either team, whose phases only it counts
        s_next[0] = s_next[1] = 0;
        bar_init(c_full, kReadWarps);
        bar_init(c_empty, 1);
        bar_init(drained, 1);
        bar_init(drained + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {  // (one CTA per SM: its shared memory leaves no room for another)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = tmem_slot;
    dependent_entry();
    if (blockIdx.x == 0 && tid == 0) *a.abort_word = 0;
    const int T = a.tiles, S = a.strips;
    const int mine = (a.heads - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;  // heads of this CTA

    // What a role has passed on so far; it goes on from the first round to the second.
    uint32_t n_tile = 0, n_head = 0, k_loads = 0, q_loads = 0;
    Ring2 ring_k{0, 0u}, ring_q{0, 0u};
    bool dead = false;
    auto wanted = [&](int i, bool safe) { return !safe || (s_bad[i / 32 % kBadWords] >> (i & 31) & 1u) != 0; };
    // Between the two rounds: whether there is a second.
    auto another = [&]() {
        __syncwarp();
        __syncthreads();
        return *(volatile int *)&s_again != 0;
    };

    if (warp < kFirstReader) {
#pragma unroll 1
        for (int round = 0; round < 2; ++round) {
        const bool safe = round == 1;
        if (safe && !another()) break;
        if (warp < kLoadWarp) {
            // ---- products: one warp has the odd strips, one the even ones, so that the waits of one fall into the
            // other's products; the whole warp walks the stream, one elected lane issues ----------------------------
            const int odd = warp == kMmaWarp;
            int seen = 0;  // of the other's progress
            const uint64_t dk = smem_desc(saddr(sK)), dq = smem_desc(saddr(sQ));
            for (int i = 0; i < mine && !dead; ++i) {
                if (!wanted(i, safe)) continue;
                for (int s = S - 1; s >= 0 && !dead; --s) {
                    const int top = s >> 1;
                    // (both warps wait for every strip and both give its stage back, whoever multiplies it: the stage's next
                    // phase then cannot end before either has seen this one, which a parity test would miss)
                    warp_wait_ready(q_full + ring_q.idx, ring_q.phase, dead, &s_abort);
                    if ((s & 1) == odd) {
                        const uint64_t db = desc_add(dq, ring_q.idx * SM::QTILE);
                        Ring2 k = ring_k;  // the head's last key tile came first
                        for (int g = T - 1; g > top; --g) k.next(SM::kK);
                        uint32_t n = n_tile;
                        for (int g = top; g >= 0; --g, ++n) {
                            if (s >= S - 2) warp_wait_ready(k_full + k.idx, k.phase, dead, &s_abort);
                            // the slot's last user must have been issued, so that the phase waited for is the next
                            count_wait(s_next + !odd, (int)n - kSlots, seen, dead, &s_abort);
                            warp_wait_ready(s_empty + n % kSlots, (n / kSlots & 1u) ^ 1u, dead, &s_abort);
                            if (dead) break;
                            fence_after();
                            const uint32_t d_tmem = tmem_base + n % kSlots * QS;
                            const uint64_t da = desc_add(dk, k.idx * SM::KTILE);
                            if (elect_one()) {
#pragma unroll
                                for (int kk = 0; kk < D / 16; ++kk)
                                    mma_bf16(d_tmem, desc_add(da, (uint32_t)(kk / 4) * KBOX + (uint32_t)(kk % 4) * 32),
                                             desc_add(db, (uint32_t)(kk / 4) * QBOX + (uint32_t)(kk % 4) * 32), kIdescStrip, kk > 0 ? 1u : 0u);
                                mma_commit(s_full + odd * kSlots + n % kSlots);
                                if (g == top) mma_commit(k_empty + k.idx);  // the warp's last strip that attends to the tile
                                if (g == 0) mma_commit(q_empty + ring_q.idx);
                            }
                            k.next(SM::kK);
                        }
                        // (the next tile of the warp's own lies beyond the other's strip, or is the next head's)
                        const int skip = s > 0 ? ((s - 1) >> 1) + 1 : ((S - 1) & 1) == odd ? 0 : ((S - 1) >> 1) + 1;
                        if (lane == 0) *(volatile int *)(s_next + odd) = (int)n + skip;
                    } else {
                        if (lane == 0) bar_arrive(q_empty + ring_q.idx);
                        if (s == S - 1 && odd) {  // no odd strip attends to the last tile
                            warp_wait_ready(k_full + ring_k.idx, ring_k.phase, dead, &s_abort);
                            if (lane == 0) {
                                bar_arrive(k_empty + ring_k.idx);
                                *(volatile int *)(s_next + odd) = (int)n_tile + top + 1;
                            }
                        }
                    }
                    n_tile += (uint32_t)top + 1;
                    ring_q.next(SM::kQ);
                }
                for (int g = 0; g < T; ++g) ring_k.next(SM::kK);
            }
            if (dead) {  // products in flight finish before tensor memory is given back (bounded)
                if (elect_one()) mma_commit(drained + odd);
                drain(drained + odd, 0u);
            }
        } else if (warp == kLoadWarp) {
            // ---- loads ----------------------------------------------------------------------------------------------
            // A strip and the stage it takes become free together; behind every even strip comes the next head's key
            // tile in the place of the one that no further strip attends to.
            if (lane == 0) {
                struct Place {
                    int i, h, l, b;  // the CTA's head, and its coordinates
                } pk, pq;
                // (worked out once a head: the thread's instructions are what a load's latency consists of)
                auto go_to = [&](Place &p, int i) {
                    while (i < mine && !wanted(i, safe)) ++i;
                    const int head = blockIdx.x + i * gridDim.x, seg = head / a.H;
                    p.i = i;
                    p.h = head - seg * a.H;
                    p.b = seg / a.L;
                    p.l = seg - p.b * a.L;
                };
                auto load_k = [&](int g) {
                    bar_wait(k_empty + ring_k.idx, ring_k.phase ^ 1u, dead, &s_abort);
                    if (dead) return;
                    bar_expect_tx(k_full + ring_k.idx, SM::KTILE);
#pragma unroll
                    for (int kh = 0; kh < KH; ++kh)
                        tma_load_5d(sK + ring_k.idx * SM::KTILE + kh * KBOX, &map_k, k_full + ring_k.idx, kh * 64, g * TT, pk.h, pk.l, pk.b);
                    ring_k.next(SM::kK);
                    ++k_loads;
                };
                go_to(pq, 0);
                int qs = S - 1;  // the strip to be loaded next
                auto next_q = [&]() {
                    if (pq.i >= mine || dead) return;
                    bar_wait(q_empty + ring_q.idx, ring_q.phase ^ 1u, dead, &s_abort);
                    if (dead) return;
                    bar_expect_tx(q_full + ring_q.idx, SM::QTILE);
#pragma unroll
                    for (int kh = 0; kh < KH; ++kh)
                        tma_load_5d(sQ + ring_q.idx * SM::QTILE + kh * QBOX, &map_q, q_full + ring_q.idx, kh * 64, qs * QS, pq.h, pq.l, pq.b);
                    ring_q.next(SM::kQ);
                    ++q_loads;
                    if (--qs < 0) {
                        qs = S - 1;
                        go_to(pq, pq.i + 1);
                    }
                };
                pk = pq;
                if (pk.i < mine) {
                    next_q();
                    for (int g = T - 1; g >= 0; --g) load_k(g);
                    for (int x = 1; x < SM::kQ; ++x) next_q();
                }
                for (int i = pk.i; i < mine && !dead; i = pk.i) {
                    go_to(pk, i + 1);
                    for (int s = S - 1; s >= 0 && !dead; --s) {
                        next_q();
                        if (!(s & 1) && pk.i < mine && !dead) load_k(s >> 1);
                    }
                }
                if (dead) {  // loads on their way land before the CTA can exit (bounded)
                    for (uint32_t n = k_loads > SM::kK ? k_loads - SM::kK : 0; n < k_loads; ++n) drain(k_full + n % SM::kK, n / SM::kK & 1u);
                    for (uint32_t n = q_loads > SM::kQ ? q_loads - SM::kQ : 0; n < q_loads; ++n) drain(q_full + n % SM::kQ, n / SM::kQ & 1u);
                }
            }
        } else if (warp == kFlushWarp) {
            // ---- a head's column sums: the four groups', added in their order ----------------------------------------
            for (int i = 0; i < mine; ++i) {
                if (!wanted(i, safe)) continue;
                const int head = blockIdx.x + i * gridDim.x;
                const float *p = s_col;
                warp_wait(c_full, n_head & 1u, dead, &s_abort);
                for (int n = lane; n < a.N; n += 32)
                    a.partial[(size_t)head * a.N + n] =
                        ((p[n] + p[kMaxTiles * TT + n]) + p[2 * kMaxTiles * TT + n]) + p[3 * kMaxTiles * TT + n];
                __syncwarp();
                if (lane == 0) bar_arrive(c_empty);
                ++n_head;
            }
        }
        }
    } else {
        // ---- readers ------------------------------------------------------------------------------------------------
        const int quarter = warp & 3, part = (warp - kFirstReader) >> 2, half = part & 1, team = part >> 1;
        const int c2 = 2 * (lane & 3), r = lane >> 2;  // the thread's first query of eight, its first key
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)half * 32;
        float *my_w = s_w + (warp - kFirstReader) * 32;
        uint32_t full_phase = 0;  // a bit to each of the team's s_full
        uint32_t turn = 0;  // of the two exchange buffers: whoever writes one again has passed the barrier of the
                            // other, which everybody reaches only after reading this one
#pragma unroll 1
        for (int round = 0; round < 2; ++round) {
            if (round == 1 && !another()) break;
#pragma unroll 1
            for (int i = 0; i < mine; ++i) {
                if (!wanted(i, round == 1)) continue;
                bool safe = round == 1;
                const int head = blockIdx.x + i * gridDim.x;
                float sc = a.layer_scale[head / a.H % a.L] * kLog2eT;
                if (sc == 0.f) sc = 0x1p-149f;  // (what is masked is infinite, and times 0 it would be NaN)
                const float masked = sc > 0.f ? -INFINITY : INFINITY;
                float acc[kMaxTiles] = {};
#pragma unroll 1
                for (int s = S - 1; s >= 0; --s) {
                    const int top = s >> 1;  // the tile the causal boundary crosses
                    if ((s & 1) != team) {
                        n_tile += (uint32_t)top + 1;
                        continue;
                    }
                    const int rel = (s & 1) * 2 + half - quarter;  // its block is full (> 0), crossed (0) or empty
                    const int hi = rel < 0 ? top - 1 : top;        // last tile the warp has work in
                    auto wait_tile = [&](int g) {
                        const uint32_t slot = (n_tile + (uint32_t)(top - g)) % kSlots;
                        warp_wait_ready(s_full + team * kSlots + slot, full_phase >> slot & 1u, dead, &s_abort);
                        fence_after();
                        return taddr + slot * QS;
                    };
                    auto exchange = [&](const float2 (&v)[4]) {
                        float *b = s_x + (part * 2 + (turn++ & 1u)) * 128;
                        if (lane < 4) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) *reinterpret_cast<float2 *>(b + quarter * 32 + 8 * c + c2) = v[c];
                        }
                        asm volatile("bar.sync %0, 128;" ::"r"(1 + part) : "memory");
                        return (const float *)b;
                    };
                    float2 base2[4], sum[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) base2[c] = sum[c] = make_float2(0.f, 0.f);
                    const bool mixed = round == 0 && s >= S - 2;  // the team's first strip of the head
                    bool look = mixed;
                    // Over the blocks: for the maximum of every query, where that is needed, and for the exponentials.
#pragma unroll 1
                    for (int walk = safe ? 0 : 1; walk < 2; ++walk) {
#pragma unroll 1
                        for (int g = hi; g >= 0; --g) {
                            const uint32_t at = wait_tile(g);
                            Block v;
                            block_load(at, v);
                            if (g == top && rel == 0) block_mask(v, c2 - r, masked);
                            if (walk == 0) {
#pragma unroll
                                for (int x = 0; x < 16; ++x) {
                                    const float2 t = v[x >> 3][x & 3][x >> 2 & 1];
                                    float2 &m = base2[x & 3];
                                    m = g == hi && x < 4 ? make_float2(t.x * sc, t.y * sc) : make_float2(fmaxf(m.x, t.x * sc), fmaxf(m.y, t.y * sc));
                                }
                                continue;
                            }
                            if (look) {
                                // The first block shows whether the head's exponentials need a maximum: the warp's own here,
                                // as the others may not need one.
                                look = false;
                                safe = !__all_sync(0xffffffffu, block_in_range(v, sc));
                                if (safe) {
                                    walk = -1;
                                    break;
                                }
                            }
#pragma unroll
                            for (int x = 0; x < 16; ++x) {
                                float2 &t = v[x >> 3][x & 3][x >> 2 & 1];
                                t = fma2(t, make_float2(sc, sc), make_float2(-base2[x & 3].x, -base2[x & 3].y));
                                t = make_float2(ex2(t.x), ex2(t.y));
                            }
                            block_store(at, v);
#pragma unroll
                            for (int x = 0; x < 16; ++x) sum[x & 3] = add2(sum[x & 3], v[x >> 3][x & 3][x >> 2 & 1]);
                        }
                        if (walk != 0) continue;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if (hi < 0) base2[c] = make_float2(-INFINITY, -INFINITY);
#pragma unroll
                            for (int o = 4; o < 32; o <<= 1) {
                                const float2 t = shfl_xor2(base2[c], o);
                                base2[c] = make_float2(fmaxf(base2[c].x, t.x), fmaxf(base2[c].y, t.y));
                            }
                        }
                        if (!mixed) {
                            const float *mx = exchange(base2);
#pragma unroll
                            for (int c = 0; c < 4; ++c)
#pragma unroll
                                for (int p = 0; p < 4; ++p) {
                                    const float2 t = *reinterpret_cast<const float2 *>(mx + p * 32 + 8 * c + c2);
                                    base2[c] = make_float2(fmaxf(base2[c].x, t.x), fmaxf(base2[c].y, t.y));
                                }
                        }
                        // (-infinity when infinite elements mask every key: sums of 0)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            base2[c] = make_float2(base2[c].x == -INFINITY ? 0.f : base2[c].x, base2[c].y == -INFINITY ? 0.f : base2[c].y);
                    }
                    // The lanes' and then the four quarters' parts of a query's sum; its weight goes to a lane.
#pragma unroll
                    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
                        for (int c = 0; c < 4; ++c) sum[c] = add2(sum[c], shfl_xor2(sum[c], o));
                    const float *x;
                    float factor = 1.f;  // from the warp's scale to the strip's, for the lane's query
                    if (!mixed) {
                        x = exchange(sum);
                    } else {
                        float2 y[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) y[c] = safe ? make_float2(-1.f, -1.f) : sum[c];
                        x = exchange(y);  // (a sign shows all four that scales differ)
                        if (__any_sync(0xffffffffu, fminf(fminf(x[lane], x[32 + lane]), fminf(x[64 + lane], x[96 + lane])) < 0.f)) {
                            safe = true;
#pragma unroll
                            for (int c = 0; c < 4; ++c) y[c] = hi < 0 ? make_float2(kLowest, kLowest) : base2[c];
                            x = exchange(y);
                            factor = ex2(x[quarter * 32 + lane] - fmaxf(fmaxf(x[lane], x[32 + lane]), fmaxf(x[64 + lane], x[96 + lane])));
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                float2 n = y[c];
#pragma unroll
                                for (int p = 0; p < 4; ++p) {
                                    const float2 t = *reinterpret_cast<const float2 *>(x + p * 32 + 8 * c + c2);
                                    n = make_float2(fmaxf(n.x, t.x), fmaxf(n.y, t.y));
                                }
                                sum[c] = make_float2(sum[c].x * ex2(y[c].x - n.x), sum[c].y * ex2(y[c].y - n.y));
                            }
                            x = exchange(sum);
                        }
                    }
                    const float z = (x[lane] + x[32 + lane]) + (x[64 + lane] + x[96 + lane]);
                    const bool real = s * QS + half * 32 + lane < a.N;
                    if ((mixed || !safe) && real && !(z >= kLowSum && z <= kHighSum)) {
                        atomicOr(s_bad + i / 32 % kBadWords, 1u << (i & 31));
                        s_again = 1;
                    }
                    my_w[lane] = real ? __frcp_rn(z) * factor : 0.f;
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    __syncwarp();
                    // A key to a lane: the weighted sum of its exponentials.
                    float4 w[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) w[c] = reinterpret_cast<const float4 *>(my_w)[c];
                    __syncwarp();
#pragma unroll 1
                    for (int g = top; g >= 0; --g) {
                        const uint32_t slot = (n_tile + (uint32_t)(top - g)) % kSlots;
                        if (g > hi) {
                            wait_tile(g);  // (so that the release before this one is over)
                            if (lane == 0) bar_arrive(s_empty + slot);
                            continue;
                        }
                        float e[32];
                        tmem_ld_row(taddr + slot * QS, e);
                        fence_before();
                        if (lane == 0) bar_arrive(s_empty + slot);
                        float2 t[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                        if (safe && g == top && rel == 0) {
                            // (a weight that is no finite number must not reach the keys beyond the boundary, 0 times it)
#pragma unroll
                            for (int c = 0; c < 32; ++c)
                                if (c >= lane) t[0].x = fmaf(e[c], (&w[c / 4].x)[c % 4], t[0].x);
                        } else {
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                t[0] = fma2(make_float2(e[4 * c], e[4 * c + 1]), make_float2(w[c].x, w[c].y), t[0]);
                                t[1] = fma2(make_float2(e[4 * c + 2], e[4 * c + 3]), make_float2(w[c].z, w[c].w), t[1]);
                            }
                        }
                        const float add = (t[0].x + t[0].y) + (t[1].x + t[1].y);
#pragma unroll
                        for (int j = 0; j < kMaxTiles; ++j)
                            if (j == g) acc[j] += add;
                    }
                    const uint32_t used = ((2u << top) - 1) << n_tile % kSlots;
                    full_phase ^= (used | used >> kSlots) & ((1u << kSlots) - 1);
                    n_tile += (uint32_t)top + 1;
                }
                warp_wait_ready(c_empty, (n_head & 1u) ^ 1u, dead, &s_abort);
                float *col = s_col + part * kMaxTiles * TT + quarter * 32 + lane;
#pragma unroll
                for (int g = 0; g < kMaxTiles; ++g)
                    if (g < T) col[g * TT] = acc[g];
                __syncwarp();
                if (lane == 0) bar_arrive(c_full);
                ++n_head;
            }
        }
    }
    // Any role whose wait ran out has set s_abort; one thread passes it on.
    fence_before();
    __syncwarp();
    __syncthreads();
    fence_after();
    if (tid == 0 && s_abort) atomicExch(a.abort_word, (int)PKV_DEV_TIMEOUT);
    if (warp == kMmaWarp) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// The wait for a count that nothing raises gives up, latches `dead` and sets the abort word.
__global__ void selftest_count_kernel(int32_t *dev_status, uint32_t limit)
{
    __shared__ int s_abort, s_count;
    if (threadIdx.x == 0) s_abort = s_count = 0;
    __syncthreads();
    bool dead = false, past = false;
    int seen = -1;
    count_wait(&s_count, -1, seen, past, &s_abort, limit);  // (there already)
    count_wait(&s_count, 0, seen, dead, &s_abort, limit);
    __syncwarp();
    if (threadIdx.x == 0 && dead && !past && s_abort) raise_status(dev_status, 0, PKV_DEV_TIMEOUT);
}

template <int D>
int launch_fused(const CUtensorMap &mq, const CUtensorMap &mk, const FusedArgs &a, int sms, cudaStream_t st)
{
    static bool done[64] = {};
    const size_t smem = FusedSmem<D>::bytes;
    int rc = ensure_dynamic_smem((const void *)score_fused_kernel<D>, (int)smem, done);
    if (rc != PKV_OK) return rc;
    cudaError_t e = launch_dependent(score_fused_kernel<D>, dim3(a.heads < sms ? a.heads : sms), dim3(kFThreads), smem, st,
                                     mq, mk, a);
    if (e != cudaSuccess) {
        set_cuda_error(e, "score_fused_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

}  // namespace

int selftest_wait_fused(int32_t *dev_status, cudaStream_t st)
{
    selftest_count_kernel<<<1, 32, 0, st>>>(dev_status, 500u);
    return check_launch("selftest_count_kernel");
}

// Prompts whose keys a CTA holds, where that is the faster way; otherwise two passes that spread heads over the SMs by tiles
// (whole calls, us, here / there; heads of 64, then of 128):
// - From four key tiles on a head takes one CTA 10 us or more, and few heads leave SMs idle: 512 tokens, 8 heads 16.4 / 14.5 and 16.8
//   / 15.3, 32 16.9 / 15.6 and 17.3 / 16.8, 64 17.1 / 18.9 and 17.7 / 21.1; 448 tokens, 8 heads 15.2 / 14.4 and 15.4 / 15.2; of three
//   tiles, 384 tokens, 12.4 / 13.4 and 12.9 / 14.1.  Of 600 tokens or more some heads above the number of SMs cost a second
//   head's time for a few: 149 heads of 640 tokens 37.9 / 36.1 and 39.5 / 38.7, 166 38.4 / 38.6 and 39.9 / 41.5.
// - Of 65 to 128 tokens the second strip has half of its keys masked, while there one tile takes all queries: 128 tokens, 320 heads
//   12.9 / 14.2 and 13.2 / 16.4, 592 16.2 / 16.1 and 16.3 / 19.2, 1600 32.0 / 29.7 and 35.2 / 37.7; 65 tokens, 1024 heads 22.7 / 22.3 and
//   22.9 / 24.3, 1184 25.0 / 22.6 and 25.3 / 25.1; 100 tokens, 4096 72 / 60 and 77.6 / 73.7.
bool score_fused_covers(const pkv_shape *s)
{
    const int64_t heads = (int64_t)s->batch * s->layers * s->heads, sms = sm_count();
    const int N = s->prompt_len;
    if (N <= 64) return true;
    if (N <= TT) return heads <= (s->head_dim == 64 ? 3 : 7) * sms;
    if (N <= 3 * TT) return true;
    if (N >= 600 && heads > sms && heads < sms + sms / 8) return false;
    return N <= kMaxTiles * TT && heads >= 64;
}

// Returns PKV_OK, an error, or -1 when the tensor maps cannot describe the caller's layout.
int launch_score_fused(const pkv_shape *s, const void *q, pkv_strides qs, const void *k, pkv_strides ks, const float *scale,
                       float *scores, float *partial, int32_t *abort_word, cudaStream_t st)
{
    CUtensorMap mq, mk;
    if (!score_make_map(&mq, q, s, qs, QS) || !score_make_map(&mk, k, s, ks, TT)) return -1;
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    const int N = s->prompt_len;
    FusedArgs a;
    a.layer_scale = scale;
    a.partial = partial;
    a.abort_word = abort_word;
    a.L = s->layers; a.H = s->heads; a.N = N;
    a.tiles = (N + TT - 1) / TT;
    a.strips = (N + QS - 1) / QS;
    a.heads = s->batch * s->layers * s->heads;
    const int rc = s->head_dim == 128 ? launch_fused<128>(mq, mk, a, sms, st) : launch_fused<64>(mq, mk, a, sms, st);
    if (rc != PKV_OK) return rc;
    return launch_head_mean(partial, s->heads, N, (size_t)s->batch * s->layers * N, scores, abort_word, st);
}

}  // namespace pkv
