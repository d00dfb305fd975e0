// Importance score (Sec. 3.2), tensor-core path for bf16 inputs (most prompts of up to 640 tokens without the caller's
// log-sum-exp: score_fused.cu, whose score_fused_covers has the line).
//
//   pass 1: per query m, log2-sum-exp of the scaled causal logits over keys j <= m
//   pass 2: per key n, sum over queries m >= n of exp2(logit - lse[m])
//   then the mean over heads in index order (shared with the FP32 path)
//
// Both passes walk 128 x 128 logit tiles of one (sample, layer, head).  The tile is one
// tcgen05.mma chain (M = N = 128, K = 16 x D/16) whose operands TMA stages in shared memory
// with the 128-byte swizzle and whose fp32 accumulator lives in tensor memory.  The operand
// that stays for a whole work item supplies the accumulator's lanes: queries in pass 1, so a
// thread owns one query row and keeps its running max / sum in registers; keys in pass 2, so
// a thread owns one key and its column sum needs no cross-thread reduction or atomics.
//
// Roles per CTA (ten warps): warp 0 lane 0 issues TMA, warp 1 owns tensor memory and issues the MMAs,
// warps 2-9 read the accumulators (tcgen05.ld, one TMEM lane quarter per warp) and do the
// exponentials.  Two accumulators alternate, each read by a set of four warps, so that the MMAs of
// tile j + 1 overlap the exponentials of tile j; the two sets' parts of an item's result meet in shared
// memory.  Two CTAs share an SM.  Work items (one stationary tile and the tiles streamed against it)
// come from a device counter, or by position where that serves as well: the TMA thread takes the
// next number and announces it to the other roles through a four-entry shared-memory queue.  Every
// mbarrier wait is bounded: when one runs out the CTA stops waiting, sets the call's abort word (the
// head mean then writes NaN for every score, which the selection stage reports as
// PKV_DEV_BAD_SCORE) and still releases its tensor memory.
//
// What bounds it: one exponential per logit per pass, 1024 clocks of the special-function unit for a
// tile against 512 of the tensor pipe.  A quarter of them are therefore computed on the FMA pipe (a
// degree-5 polynomial, add_exp2), and the arithmetic around them is packed two to an instruction.
// Clocks a tile at 16384 tokens, 32 heads: 1340 with neither (issue slots 32 % used after packing), 1080
// now (special-function unit 67-77 % busy, issue slots 54-60 %, FMA pipe 50 %).  Time of a pass pair, 64
// heads of 16384 tokens / 1024 of 640: four reader warps and no polynomial 5168 / 191 us, a quarter
// polynomial 4490 / 184; eight reader warps without it 4758 / 191, with an eighth 4465 / 187, a quarter
// 4417 / 185, three eighths 4624 / 187.  A row read from tensor memory in quarters with the next on its
// way 4650 / 191; one CTA per SM with sixteen reader warps, two stationary and four streamed stages
// 4370 / 208.
#include "score_tiles.cuh"

namespace pkv {

namespace {

constexpr int kStagesB = 2;        // streamed-operand stages
constexpr int kPoly1 = 2, kPoly2 = 2;  // pairs of exponentials in eight on the FMA pipe, pass 1 and 2

struct ScoreArgs {
    const float *layer_scale;
    float *lse2;         // pass 1 out: [B*L*H][Npad] log2-sum-exp of scaled logits, +inf beyond N
    const float *lse_in; // pass 2: the caller's [B*L*H][N] natural-log sum-exp, or NULL (lse2 is taken)
    float *partial;  // [B*L*H][N] per-head column sums
    int32_t *abort_word;  // device word set when a bounded wait runs out: the head mean then writes NaN scores
    int *next_item;       // [2] work counters, one per pass; zeroed, with the abort word, before the first pass
    int L, H, N, Npad, tiles, nseg, group;
    bool counted;      // items come from the counters; otherwise they are dealt out by position
    bool clear_abort;  // this launch is the call's first and nothing has zeroed the abort word
};

constexpr int kItemQ = 4;  // item numbers in flight between the loader and the other roles
constexpr int kReaders = 8;  // reader warps: two sets of four
constexpr int kTileThreads = (2 + kReaders) * 32;
// Items whose parts may be waiting for the other set's.  A set that is at item i + kItemQ + 1 knows, from the
// queue's slot being free, that the other has taken item i + 1 and so is done with item i.
constexpr int kPartSlots = kItemQ + 1;

// PASS 1: stationary = Q tile t, streamed = K tiles 0..t.  PASS 2: stationary = K tile t,
// streamed = Q tiles t..tiles-1.
template <int PASS, int D>
__global__ void __launch_bounds__(kTileThreads, 2)
score_tile_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                  const ScoreArgs a)
{
    constexpr int KH = D / 64;                  // 128-byte swizzle atoms along the head dimension
    constexpr uint32_t HALF = TT * 128;         // bytes of one [128 rows x 64 elements] box
    constexpr uint32_t TILE = KH * HALF;        // bytes of one operand tile
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base;
    unsigned char *sB = base + TILE;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + kStagesB * TILE);
    uint64_t *a_full = bars, *a_empty = bars + 1, *b_full = bars + 2, *b_empty = b_full + kStagesB;
    uint64_t *s_full = b_empty + kStagesB, *s_empty = s_full + 2;
    uint64_t *q_full = s_empty + 2, *q_empty = q_full + kItemQ;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(q_empty + kItemQ);
    __shared__ __align__(8) uint64_t drained;
    __shared__ int s_abort;
    __shared__ int q_item[kItemQ];  // the loader's announcements: an item number, or -1 for the end
    __shared__ __align__(16) float s_lse[2][4][TT];  // [reader set][lane quarter][query of the tile]
    __shared__ float2 s_part[kPartSlots][2][4][32];  // an item's two parts: maximum and sum of every row
    __shared__ int s_arrived[kPartSlots][4];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const CUtensorMap *map_stat = PASS == 1 ? &map_q : &map_k;
    const CUtensorMap *map_strm = PASS == 1 ? &map_k : &map_q;
    const int nsh = a.nseg * a.H;
    const int nitems = nsh * a.tiles;

    if (tid == 0) {
        s_abort = 0;
        bar_init(a_full, 1);
        bar_init(a_empty, 1);
        for (int i = 0; i < kStagesB; ++i) {
            bar_init(b_full + i, 1);
            bar_init(b_empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(s_full + i, 1);
            bar_init(s_empty + i, 4);
        }
        for (int i = 0; i < kItemQ; ++i) {
            bar_init(q_full + i, 1);
            bar_init(q_empty + i, 1 + kReaders);  // the MMA warp and the reader warps
        }
        bar_init(&drained, 1);
        for (int i = 0; i < kPartSlots * 4; ++i) s_arrived[i / 4][i % 4] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {  // two 128-column fp32 accumulators
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                     "r"(256u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // Launched as a programmatic dependent: everything above (barriers, tensor memory) was set up
    // while the kernel before it drained; its results (Q, K, the normalisers) are read from here on.
    dependent_entry();
    if (a.clear_abort && blockIdx.x == 0 && tid == 0) *a.abort_word = 0;

    if (warp == 0) {
        // ---- TMA producer ---------------------------------------------------------------------
        if (lane == 0) {
            bool dead = false;
            uint32_t a_phase = 0, a_loads = 0, b_loads = 0;  // loads issued
            Ring2 rb{0, 0u}, rq{0, 0u};
            int *ctr = a.counted ? a.next_item + (PASS - 1) : nullptr;
            int next = ctr ? atomicAdd(ctr, 1) : blockIdx.x;  // asked for one item ahead: the answer takes a microsecond
            for (;;) {
                const int w = next < nitems ? next : -1;
                if (w >= 0) next = ctr ? atomicAdd(ctr, 1) : next + (int)gridDim.x;
                bar_wait(q_empty + rq.idx, rq.phase ^ 1u, dead, &s_abort);
                if (dead) break;
                q_item[rq.idx] = w;
                bar_arrive(q_full + rq.idx);
                rq.next(kItemQ);
                if (w < 0) break;
                int sh, t;
                decode_item<PASS>(w, nsh, a.tiles, a.group, sh, t);
                const int seg = sh / a.H, h = sh - seg * a.H, b = seg / a.L, l = seg - b * a.L;
                bar_wait(a_empty, a_phase ^ 1u, dead, &s_abort);
                if (dead) break;
                bar_expect_tx(a_full, TILE);
#pragma unroll
                for (int kh = 0; kh < KH; ++kh)
                    tma_load_5d(sA + kh * HALF, map_stat, a_full, kh * 64, t * TT, h, l, b);
                a_phase ^= 1u;
                ++a_loads;
                const int j0 = PASS == 1 ? 0 : t, j1 = PASS == 1 ? t : a.tiles - 1;
                for (int j = j0; j <= j1; ++j) {
                    bar_wait(b_empty + rb.idx, rb.phase ^ 1u, dead, &s_abort);
                    if (dead) break;
                    bar_expect_tx(b_full + rb.idx, TILE);
#pragma unroll
                    for (int kh = 0; kh < KH; ++kh)
                        tma_load_5d(sB + rb.idx * TILE + kh * HALF, map_strm, b_full + rb.idx, kh * 64, j * TT, h, l, b);
                    rb.next(kStagesB);
                    ++b_loads;
                }
            }
            if (dead) {  // let the loads on their way land before the CTA can exit (bounded)
                if (a_loads > 0) drain(a_full, (a_loads - 1) & 1u);
                for (uint32_t n = b_loads > kStagesB ? b_loads - kStagesB : 0; n < b_loads; ++n)
                    drain(b_full + n % kStagesB, n / kStagesB & 1u);
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer: the whole warp walks the stream, one elected lane issues, so that the operands'
        // descriptors are formed in uniform registers ahead of each instruction -----------------------------
        bool dead = false;
        uint32_t a_phase = 0;
        Ring2 rb{0, 0u}, rs{0, 0u}, rq{0, 0u};
        const uint64_t da = smem_desc(saddr(sA)), db = smem_desc(saddr(sB));
        for (;;) {
            warp_wait(q_full + rq.idx, rq.phase, dead, &s_abort);
            if (dead) break;
            const int w = __shfl_sync(0xffffffffu, *(volatile int *)(q_item + rq.idx), 0);
            __syncwarp();
            if (lane == 0) bar_arrive(q_empty + rq.idx);
            rq.next(kItemQ);
            if (w < 0) break;
            int sh, t;
            decode_item<PASS>(w, nsh, a.tiles, a.group, sh, t);
            warp_wait(a_full, a_phase, dead, &s_abort);
            a_phase ^= 1u;
            const int count = PASS == 1 ? t + 1 : a.tiles - t;
            for (int jj = 0; jj < count && !dead; ++jj) {
                warp_wait(b_full + rb.idx, rb.phase, dead, &s_abort);
                warp_wait(s_empty + rs.idx, rs.phase ^ 1u, dead, &s_abort);
                if (dead) break;
                fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)rs.idx * TT;
                const uint64_t dk = desc_add(db, rb.idx * TILE);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const uint32_t off = (uint32_t)(k / 4) * HALF + (uint32_t)(k % 4) * 32;
                        mma_bf16(d_tmem, desc_add(da, off), desc_add(dk, off), kIdesc, k > 0 ? 1u : 0u);
                    }
                    mma_commit(b_empty + rb.idx);  // the streamed stage is free once these MMAs retire
                    mma_commit(s_full + rs.idx);   // and the accumulator is ready to be read
                    if (jj == count - 1) mma_commit(a_empty);  // the stationary tile may be replaced
                }
                rb.next(kStagesB);
                rs.next(2);
            }
            if (dead) break;
        }
        if (dead) {  // and the products in flight finish before tensor memory is given back (bounded)
            if (elect_one()) mma_commit(&drained);
            drain(&drained, 0u);
        }
    } else {
        // ---- accumulator readers: one TMEM lane (tile row) per thread.  Tile c of the CTA's stream goes
        // through accumulator c mod 2 to reader set c mod 2 ------------------------------------------------
        const int set = (warp - 2) >> 2, quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)set * TT;
        float *my_lse = s_lse[set][quarter];
        bool dead = false;
        uint32_t phase = 0, seq = 0, tile0 = 0;  // of the accumulator; number of the item; tiles before it
        Ring2 rq{0, 0u};
        for (;; ++seq) {
            warp_wait(q_full + rq.idx, rq.phase, dead, &s_abort);
            if (dead) break;
            const int w = *(volatile int *)(q_item + rq.idx);
            __syncwarp();
            if (lane == 0) bar_arrive(q_empty + rq.idx);
            rq.next(kItemQ);
            if (w < 0) break;
            int sh, t;
            decode_item<PASS>(w, nsh, a.tiles, a.group, sh, t);
            const int seg = sh / a.H, l = seg % a.L;
            const float sc = a.layer_scale[l] * kLog2eT;
            const bool fast = sc > 0.f;     // the usual case: the extreme of sc * x is sc * max x
            const int grow = t * TT + row;  // query (pass 1) or key (pass 2) index of this thread
            const float *lse_row = a.lse2 + (size_t)sh * a.Npad;
            float run_max = -INFINITY, run_sum = 0.f;  // pass 1 (pass 2: run_sum alone)
            const int j0 = PASS == 1 ? 0 : t, count = PASS == 1 ? t + 1 : a.tiles - t;
            const int odd = (set + tile0) & 1;  // this set's tiles of the item: j0 + odd, + 2, ...
            tile0 += count;
            // pass 2: every thread needs the tile's 128 query normalisers.  Each warp keeps its own copy
            // in shared memory (four per lane, fetched a tile ahead so that the load's latency is not
            // in the way), so the reader warps never wait for one another.
            float4 lse_mine = make_float4(0.f, 0.f, 0.f, 0.f);
            auto fetch_lse = [&](int j) {
                if (a.lse_in == nullptr) {
                    lse_mine = __ldg(reinterpret_cast<const float4 *>(lse_row + j * TT) + lane);
                } else {  // (rows of N floats: no alignment to count on)
                    const float *p = a.lse_in + (size_t)sh * a.N;
                    const int m = j * TT + lane * 4;
                    lse_mine.x = m < a.N ? __ldg(p + m) * kLog2eT : INFINITY;
                    lse_mine.y = m + 1 < a.N ? __ldg(p + m + 1) * kLog2eT : INFINITY;
                    lse_mine.z = m + 2 < a.N ? __ldg(p + m + 2) * kLog2eT : INFINITY;
                    lse_mine.w = m + 3 < a.N ? __ldg(p + m + 3) * kLog2eT : INFINITY;
                }
            };
            if (PASS == 2 && odd < count) fetch_lse(j0 + odd);
            for (int jj = odd; jj < count; jj += 2) {
                const int j = j0 + jj;
                if (PASS == 2) {
                    __syncwarp();  // the warp is done with the copy this one replaces
                    reinterpret_cast<float4 *>(my_lse)[lane] = lse_mine;
                    if (jj + 2 < count) fetch_lse(j + 2);
                    __syncwarp();
                }
                warp_wait(s_full + set, phase, dead, &s_abort);
                phase ^= 1u;
                fence_after();
                auto release = [&]() {  // the accumulator's columns are all in registers: back to the MMA warp
                    fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(s_empty + set);
                };
                if (j != t) {
                    // a full tile, half a row at a time
#pragma unroll 1
                    for (int half = 0; half < 2; ++half) {
                        float v[64];
                        tmem_ld64(taddr + half * 64, v);
                        if (half == 1) release();
                        if (PASS == 1) lse_block<64, kPoly1>(v, sc, fast, run_max, run_sum);
                        else run_sum += colsum_block<64, kPoly2>(v, my_lse + half * 64, sc, false, lane);
                    }
                } else {
                    // On the diagonal tile only the 32-column blocks that reach this warp's rows matter:
                    // blocks 0..quarter in pass 1 (keys <= query), quarter..3 in pass 2 (queries >= key).
#pragma unroll 1
                    for (int cblk = PASS == 1 ? 0 : quarter; cblk <= (PASS == 1 ? quarter : TT / 32 - 1); ++cblk) {
                        float v[32];
                        tmem_ld32(taddr + cblk * 32, v);
                        const bool edge = cblk == quarter;  // the block the causal boundary crosses
                        if (PASS == 1) {
                            if (edge) {
#pragma unroll
                                for (int i = 0; i < 32; ++i) v[i] = i <= lane ? v[i] : -INFINITY;
                            }
                            lse_block<32, 0>(v, sc, fast, run_max, run_sum);
                        } else {
                            run_sum += colsum_block<32, 0>(v, my_lse + cblk * 32, sc, edge, lane);
                        }
                    }
                    release();
                }
            }
            // The item's result.  With two tiles or more both sets have a part of it, which they leave in
            // shared memory: whichever warp is the second there adds the two (always the part with the
            // first tile before the other, so that the sum does not depend on which warp it is).
            bool writes = odd < count;
            if (count > 1) {
                float2 (*part)[4][32] = s_part[seq % kPartSlots];
                int *arrived = s_arrived[seq % kPartSlots] + quarter;
                part[odd][quarter][lane] = make_float2(run_max, run_sum);
                __threadfence_block();
                __syncwarp();
                int before = 0;
                if (lane == 0) before = atomicAdd(arrived, 1);
                writes = __shfl_sync(0xffffffffu, before, 0) != 0;
                if (writes) {
                    __threadfence_block();
                    const float2 p0 = part[0][quarter][lane], p1 = part[1][quarter][lane];
                    if (PASS == 1) {
                        run_max = fmaxf(p0.x, p1.x);
                        run_sum = fmaf(p0.y, ex2(p0.x - run_max), p1.y * ex2(p1.x - run_max));
                    } else {
                        run_sum = p0.y + p1.y;
                    }
                    if (lane == 0) *(volatile int *)arrived = 0;
                }
            }
            if (writes) {
                if (PASS == 1) a.lse2[(size_t)sh * a.Npad + grow] = grow < a.N ? run_max + log2f(run_sum) : INFINITY;
                else if (grow < a.N) a.partial[(size_t)sh * a.N + grow] = run_sum;
            }
        }
    }
    // Any role whose wait ran out has set s_abort; one thread passes it on (after the barrier below).

    fence_before();
    __syncthreads();
    fence_after();
    if (tid == 0 && s_abort && a.abort_word) atomicExch(a.abort_word, (int)PKV_DEV_TIMEOUT);
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(256u) : "memory");
    }
}

// One warp waits, with a short limit, on a barrier phase that nothing completes: the wait gives
// up, latches `dead`, and the status word reads PKV_DEV_TIMEOUT.  This is the whole give-up path
// of the kernel above in isolation (its roles then stop waiting, drain and release tensor memory).
__global__ void selftest_wait_kernel(int32_t *dev_status, uint32_t limit)
{
    __shared__ uint64_t bar;
    __shared__ int s_abort;
    if (threadIdx.x == 0) {
        s_abort = 0;
        bar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    bool dead = false;
    if (threadIdx.x == 0) bar_wait(&bar, 0u, dead, &s_abort, limit);
    __syncthreads();
    bar_wait(&bar, 0u, dead, &s_abort, limit);  // the other lanes see the flag and stop at once
    if (threadIdx.x == 0 && dead && s_abort) raise_status(dev_status, 0, PKV_DEV_TIMEOUT);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

}  // namespace

// [B, L, H, N, D] bf16 with element strides -> rank-5 map, box = 64 elements x box_rows rows.
bool score_make_map(CUtensorMap *map, const void *ptr, const pkv_shape *s, pkv_strides st, int box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[5] = {(cuuint64_t)s->head_dim, (cuuint64_t)s->prompt_len, (cuuint64_t)s->heads,
                          (cuuint64_t)s->layers, (cuuint64_t)s->batch};
    int64_t es[4] = {st.n, st.h, st.l, st.b};
    cuuint64_t strides[4];
    for (int i = 0; i < 4; ++i) {
        int64_t v = es[i];
        if (dims[i + 1] == 1 && v == 0) v = s->head_dim;  // a size-1 dimension's stride is never used
        strides[i] = (cuuint64_t)v * 2;
        if (strides[i] % 16 != 0 || strides[i] >= ((cuuint64_t)1 << 40) || strides[i] == 0) return false;
    }
    cuuint32_t box[5] = {64, (cuuint32_t)box_rows, 1, 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

namespace {

template <int PASS, int D>
int launch_pass(const CUtensorMap &mq, const CUtensorMap &mk, const ScoreArgs &a, int sms, cudaStream_t st)
{
    static bool done[64] = {};
    const size_t smem = (size_t)(1 + kStagesB) * (D / 64) * TT * 128 + 1024 + 256;
    int rc = ensure_dynamic_smem((const void *)score_tile_kernel<PASS, D>, (int)smem, done);
    if (rc != PKV_OK) return rc;
    const int items = a.nseg * a.H * a.tiles;
    const int grid = items < 2 * sms ? items : 2 * sms;
    cudaError_t e = launch_dependent(score_tile_kernel<PASS, D>, dim3(grid), dim3(kTileThreads), smem, st, mq, mk, a);
    if (e != cudaSuccess) {
        set_cuda_error(e, PASS == 1 ? "score_tile_kernel<1>" : "score_tile_kernel<2>");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

}  // namespace

int launch_head_mean(const float *partial, int H, int N, size_t total, float *scores, const int32_t *abort_word,
                     cudaStream_t st);
bool score_fused_covers(const pkv_shape *s);
int launch_score_fused(const pkv_shape *s, const void *q, pkv_strides qs, const void *k, pkv_strides ks, const float *scale,
                       float *scores, float *partial, int32_t *abort_word, cudaStream_t st);

int selftest_wait_score(int32_t *dev_status, cudaStream_t st)
{
    selftest_wait_kernel<<<1, 32, 0, st>>>(dev_status, 2000u);  // each try may sleep up to kSuspendNs
    return check_launch("selftest_wait_kernel");
}

bool score_tc_usable(const pkv_shape *s, const void *, pkv_strides, const void *, pkv_strides)
{
    return s->dtype == PKV_BF16 && (s->head_dim == 64 || s->head_dim == 128) && encode_fn() != nullptr;
}

size_t score_tc_ws_bytes(const pkv_shape *s)
{
    const size_t rows = (size_t)s->batch * s->layers * s->heads;
    const size_t npad = ((size_t)s->prompt_len + TT - 1) / TT * TT;
    return round_up(rows * s->prompt_len * sizeof(float), kWsAlign) + round_up(rows * npad * sizeof(float), kWsAlign) +
           kWsAlign;  // the two work counters and the abort word
}

// Returns PKV_OK, an error, or -1 when the tensor maps cannot describe the caller's layout.
int launch_score_tc(const pkv_shape *s, const void *q, pkv_strides qs, const void *k, pkv_strides ks,
                    const float *scale, const float *lse, float *scores, void *ws, cudaStream_t st)
{
    const int B = s->batch, L = s->layers, H = s->heads, N = s->prompt_len;
    const size_t rows = (size_t)B * L * H;
    ScoreArgs a;
    a.layer_scale = scale;
    a.partial = (float *)ws;
    a.lse2 = (float *)((unsigned char *)ws + round_up(rows * N * sizeof(float), kWsAlign));
    a.L = L; a.H = H; a.N = N;
    a.tiles = (N + TT - 1) / TT;
    a.Npad = a.tiles * TT;
    a.next_item = (int *)((unsigned char *)a.lse2 + round_up(rows * a.Npad * sizeof(float), kWsAlign));
    a.abort_word = a.next_item + 2;
    a.nseg = B * L;
    a.group = head_group(B * L * H, N, s->head_dim, 2);
    // (with the caller's log-sum-exp one pass is left, and the tile kernel is at least as fast: 32 x 32 heads of 640
    // tokens 102 us, 101 in a form of the fused kernel for it, of 100 tokens 17 and 25)
    if (!lse && score_fused_covers(s)) return launch_score_fused(s, q, qs, k, ks, scale, scores, a.partial, a.abort_word, st);

    CUtensorMap mq, mk;
    if (!score_make_map(&mq, q, s, qs, TT) || !score_make_map(&mk, k, s, ks, TT)) return -1;
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    // Items of nearly one length (a tile or two), or a few for each CTA: dealt out by position, which needs
    // no counters and so no memset in front (32 x 32 heads of 100 tokens 42 -> 36 us, 2 x 32 of 640 38 ->
    // 33.5, 128 x 32 of 200 193 -> 179).  Otherwise CTAs that run ahead take more (32 x 32 of 640 tokens
    // 185 us, dealt 196; 2 x 32 of 16384 4.6 ms, dealt 5.0).
    a.counted = a.tiles > 2 && rows * a.tiles > 8 * (size_t)sms;
    if (a.counted) {
        cudaError_t e = cudaMemsetAsync(a.next_item, 0, 4 * sizeof(int), st);
        if (e != cudaSuccess) {
            set_cuda_error(e, "cudaMemsetAsync(score work counters)");
            return PKV_ERR_CUDA;
        }
    }
    a.lse_in = lse;
    int rc = PKV_OK;
    a.clear_abort = !a.counted;
    if (!lse) rc = s->head_dim == 128 ? launch_pass<1, 128>(mq, mk, a, sms, st) : launch_pass<1, 64>(mq, mk, a, sms, st);
    if (rc != PKV_OK) return rc;
    a.clear_abort = !a.counted && lse;
    rc = s->head_dim == 128 ? launch_pass<2, 128>(mq, mk, a, sms, st) : launch_pass<2, 64>(mq, mk, a, sms, st);
    if (rc != PKV_OK) return rc;
    return launch_head_mean(a.partial, H, N, (size_t)B * L * N, scores, a.abort_word, st);
}

}  // namespace pkv
