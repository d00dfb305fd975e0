// Decode attention over the ragged cache (Sec. 3.1, Fig. 2a), (segment, head) pair by pair: calls with few pairs (a layer at
// a time, or a few layers, of a small batch) by a cluster of CTAs to a pair, most others by a CTA to a pair
// (decode_cluster_ctas has the lines).
//
// A call of few pairs moves a few megabytes, so what counts is the chain of latencies of one launch and that
// every SM has a share.  A cluster of C CTAs takes one (segment, head); each CTA takes a C-th of its
// rows.  Every warp copies its rows' slices of the head into a ring of its own with 16-byte cp.async
// and reads back what the same lane copied, so that no warp waits for another until the merge.  The
// CTAs' partial softmax states go to the first CTA of the cluster through distributed shared memory,
// which merges them in rank order and writes the head's output: one launch, nothing in global memory
// in between.  The last CTA of a cluster also attends to the new row and appends it.
// Lengths: every CTA reads its segment's length and then counts itself in a word of the workspace; the one that
// completes the count writes the length of the next step.  A call that appends nothing counts nothing.  (Every CTA
// raising a flag in the workspace, and an extra cluster waiting for them: its chain of round trips ended after the rows',
// 4.43 us a call below for 3.96 without.  A count in the upper bits of the length's own word: a word that was no length
// before the call could pass for one that some CTAs had been at.  Plan and count by a thread of the first warp, which
// may have the new row to take: 3.65 us a call for 3.51; the count only after the barrier: 3.82; its answer looked at
// before the rows: 3.80; by the clusters' first CTAs alone, after their merge's first barrier: 3.90.)
// Where the rows are is also read ahead, while the kernel in front still runs: the rows of that guess are
// asked for as soon as it has completed, and the guess is held against the plan made afterwards.  The
// values are not looked at before then, so that a CTA that starts late has both loads on their way at once
// (looked at before: 19.3 us for 17.7 in the case of 8 x 40 x 410 rows; one thread's loads, passed on through
// shared memory: 20.1, and 4.15 for 3.77 in the smallest).
//
// A round's arithmetic is half of what a warp does: dot products and sums two elements to an instruction, whole rounds without a look at
// their ends, rescaling where the maximum moves, pointers instead of products of row numbers: 8 x 40 x 410 17.7 -> 15.9 us, 1024 pairs of
// 136 rows 16.7 -> 15.0.  (Partial sums of four rows reduced together, 12 shuffles for 17: no gain.)
//
// Measured, device time of calls replayed from a graph, one layer, bf16, D = 128, every call on another layer: 1 segment
// x 32 heads x 128 rows 3.64 us (4.44 before all of this), 4 x 32 x 128 rows 5.30 (6.01), 16 x 32 x 128 9.87 (11.55),
// 1 x 40 x 410 4.91 (5.65), 8 x 40 x 410 15.7 (18.8; 10.3 us of bytes); against the row-split kernel and its merge
// kernel, before that: 1 x 32 x 128 rows 4.5 (10.0), 1024 rows 8.0 (26.4); 4 x 32 x 128 rows 6.1 (12.1);
// 8 x 40 x 410 rows 17.4 (25.7); 8 x 64 x 900 rows 50 (51).  A second wave of CTAs costs as much as the
// first's latency, 4-5 us (C = 8 for 4 x 32 x 128 rows: 8.9 us), hence the choice of C below.  Loads to
// registers instead of the rings, eight steps of K and V in flight: the same for one round of rows,
// 20.5 us for 8 x 40 x 410.  Ring shapes (steps, rounds, CTAs per SM): 4, 2, 5 as here; 8, 2, 3 and
// 4, 3, 4 18.9-19.4 us there; 2, 4, 5 18.7.  With a CTA to a pair (1024 of 136 rows / 4096 of 820; 17.4 / 259 us as here): one warp
// with four to eight rounds in flight 23.1-29.2 / 336-396, two 19.5-21 / 300, eight 19.8 / 262; a loop over several pairs with the next
// one's rows under way, 10-18 % slower throughout.  Clusters of 12 or 16: slower throughout.
#include "decode_plan.cuh"

namespace pkv {

bool decode_stream_covers(const pkv_shape *s, int nact);

namespace {

constexpr int kCWarps = 4;             // warps per CTA
constexpr int kPlanner = kCWarps * 32 - 32;  // the thread that reads a CTA's plan and counts: not of the warp that takes the new row
constexpr int kCStages = 2;            // rounds in flight per warp
constexpr int kCPerSm = 5;             // CTAs an SM holds at a time, rounds of four steps (their rings fill its shared memory)
constexpr int kCMaxCluster = 8;        // portable cluster size
constexpr int kCSmShared = 228 * 1024; // an SM's shared memory; a CTA takes 1 KiB more than it asks for
constexpr float kLog2eC = 1.4426950408889634f;
constexpr float kNoLogit = -3.402823466e38f;  // the lowest finite number

struct ClusterArgs {
    DecodePlanArgs p;
    const void *q, *k_new, *v_new;
    void *ck, *cv, *out;
    const float *layer_scale;
    unsigned long long *visits;  // [active segments][kVisitStride] how many CTAs have read the segment's length
    unsigned long long visit_tag;
    int32_t *dev_status;
    int H;
    int guess_more;  // rows that a length read ahead may be short of
    uint32_t row_bytes;
};

__device__ __forceinline__ void copy16(void *dst, const unsigned char *src)
{
    asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// A head's slice of a row is D * sizeof(T) bytes: LPR lanes share a row, a warp reads G = 32 / LPR
// rows per step.
// A round is U steps; an SM holds P CTAs (their rings and registers are cut for that).
template <typename T, int D, int U, int P>
__global__ void __launch_bounds__(kCWarps * 32, P) decode_cluster_kernel(const ClusterArgs a)
{
    constexpr int kCU = U;
    constexpr uint32_t kCRound = U * 512;  // bytes of a round's K (or V) rows: a warp reads 512 bytes per step
    constexpr int VE = RowVec<T>::VE;
    constexpr uint32_t SLICE = D * sizeof(T);
    constexpr int LPR = SLICE / 16, G = 32 / LPR;
    constexpr int STEP = kCU * G;  // rows of one round of a warp
    static_assert(kCWarps * 32 >= D, "a thread per element of the output");
    extern __shared__ __align__(16) unsigned char s_ring[];  // [kCWarps][kCStages][K, V][kCRound]
    __shared__ __align__(8) float s_acc[kCWarps][D];
    __shared__ float s_ml[kCWarps][2];
    __shared__ float c_acc[P == kCPerSm ? kCMaxCluster : 1][D], c_ml[kCMaxCluster][2];  // (first CTA of a cluster) the cluster's partials

    __shared__ SegPlan s_plan;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int item = blockIdx.x / C;    // (the first CTA must be running before anyone writes to its shared memory)
    if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    const int si = item / a.H, h = item - si * a.H;
    const int seg = (si / a.p.nl) * a.p.L + a.p.layer_begin + si % a.p.nl;
    const size_t hoff = ((size_t)seg * a.H + h) * SLICE;
    const int grp = lane / LPR, c = lane % LPR;
    const bool takes_new = a.p.append && rank == C - 1 && warp == 0;
    // What this CTA reads of a segment: the cached rows less the slot that the new row reuses, a C-th of them.
    struct Rows {
        const unsigned char *kb, *vb;
        int r0, r1, skip;
    };
    auto rows_of = [&](const SegPlan &sp) {
        const int cached = sp.rows < 0 ? 0 : (a.p.append ? (sp.evict ? sp.rows : sp.rows - 1) : sp.rows);
        const int per = (cached + C - 1) / C;
        Rows r;
        r.r0 = min(cached, rank * per);
        r.r1 = min(cached, r.r0 + per);
        r.skip = sp.evict ? sp.dst : -1;
        r.kb = static_cast<const unsigned char *>(a.ck) + (size_t)sp.off * a.row_bytes + (size_t)h * SLICE + c * 16;
        r.vb = static_cast<const unsigned char *>(a.cv) + (size_t)sp.off * a.row_bytes + (size_t)h * SLICE + c * 16;
        return r;
    };
    // Every warp runs its own ring: a lane copies, and later reads, the same 16 bytes of a step's rows, so
    // that waiting for its own copies is all that it needs.
    unsigned char *ring = s_ring + (size_t)warp * kCStages * 2 * kCRound + lane * 16;
    auto request = [&](const Rows &rw, int base, int stage) {
        unsigned char *d = ring + stage * 2 * kCRound;
        const size_t first = (size_t)(base + grp) * a.row_bytes;
        const unsigned char *kp = rw.kb + first, *vp = rw.vb + first;
        const uint32_t step = G * a.row_bytes;
#pragma unroll
        for (int j = 0; j < kCU; ++j) {
            const int r = base + j * G + grp;
            if (r < rw.r1 && r != rw.skip) {
                copy16(d + j * 512, kp);
                copy16(d + kCRound + j * 512, vp);
            }
            kp += step;
            vp += step;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // Where the rows are is read before the kernel in front has completed, and the first rounds are asked for as soon
    // as it has, together with the plan that counts.  Should that one be another, they are asked for again.
    const bool guesses = a.p.evict_distance == 0;
    int guess_ln = 0, guess_cp = 0;
    int64_t guess_off = 0;
    if (guesses) {  // (not looked at yet: a CTA that starts late must not wait for these before it asks for the others)
        guess_ln = load_l2(a.p.len + seg);
        guess_cp = load_l2(a.p.cap + seg);
        guess_off = load_l2(a.p.row_offset + seg);
    }
    dependent_entry();
    int ln = 0, cp = 0;
    int64_t off = 0;
    unsigned long long seen = 0, before = 0, *const visits = a.visits + (size_t)si * kVisitStride;
    PruneState ps;
    if (tid == kPlanner) {
        ps = prune_state(a.p, seg);
        ln = load_l2(a.p.len + seg);
        cp = load_l2(a.p.cap + seg);
        off = load_l2(a.p.row_offset + seg);
        if (a.p.append) seen = load_flag(visits);
    }
    // When all of the segment's CTAs have read its length.  The answer comes while the rows are looked at; it is not kept waiting where six
    // and seven CTAs of an SM leave a thread few registers (1024 pairs of 140 rows 15.6 us so, 15.9 after the rows; 2048 pairs, five CTAs
    // an SM: 27.2 and 26.2).
    auto last_one = [&]() {
        if (tid != kPlanner || before != a.visit_tag + (uint32_t)(a.H * C - 1)) return;
        settle_visits(visits, a.visit_tag, a.p.evict_distance > 0);
        segment_advance(a.p, si, s_plan);
    };
    Rows rw{nullptr, nullptr, 0, 0, -1};
    if (guesses) {
        rw = rows_of(plan_of(a.p, guess_ln, guess_cp, guess_off, PruneState{0, 0, -1}));
        if (rw.r1 > 0) rw.r1 += a.guess_more;
#pragma unroll
        for (int i = 0; i < kCStages; ++i) request(rw, rw.r0 + (warp + i * kCWarps) * STEP, i);
    }
    uint4 qraw = *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(a.q) + hoff + c * 16);
    uint4 knew = make_uint4(0u, 0u, 0u, 0u), vnew = knew;
    if (takes_new) {
        knew = *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(a.k_new) + hoff + c * 16);
        vnew = *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(a.v_new) + hoff + c * 16);
    }
    const float sc = a.layer_scale[a.p.layer_begin + si % a.p.nl] * kLog2eC;
    if (tid == kPlanner) {
        const SegPlan sp = plan_of(a.p, ln, cp, off, ps);
        s_plan = sp;
        // (a segment that cannot take the step is counted by nobody; the count's answer is looked at later)
        if (sp.rows < 0) raise_status(a.dev_status, si / a.p.nl, PKV_DEV_CAPACITY);
        else if (a.p.append) before = count_visit(visits, a.visit_tag, seen, a.p.evict_distance > 0);
    }
    __syncthreads();
    const SegPlan sp = s_plan;
    if (P != kCPerSm) last_one();
    const Rows now = rows_of(sp);
    if (now.r1 + a.guess_more >= rw.r1 && now.r1 < rw.r1) rw.r1 = now.r1;
    if (now.r0 != rw.r0 || now.r1 != rw.r1 || now.skip != rw.skip || now.kb != rw.kb) {
        // (a row more or less at the end: the same bytes come to the same places again)
        if (now.r0 != rw.r0 || now.skip != rw.skip || now.kb != rw.kb) asm volatile("cp.async.wait_all;" ::: "memory");
        rw = now;
#pragma unroll
        for (int i = 0; i < kCStages; ++i) request(rw, rw.r0 + (warp + i * kCWarps) * STEP, i);
    }

    // M: the running maximum of the logits, from the lowest finite number on, so that exp2f(s - M) is 0 for a logit
    // of -infinity and NaN for NaN whatever came before it.
    float qf[VE], M = kNoLogit, lsum = 0.f;
    float2 acc[VE / 2];
    RowVec<T>::unpack(qraw, qf);
#pragma unroll
    for (int i = 0; i < VE; ++i) {
        qf[i] *= sc;
        acc[i / 2] = make_float2(0.f, 0.f);
    }
    // One round: logits of the warp's rows, one rescale, accumulation (every lane group keeps the
    // warp-wide running maximum, so that the groups' sums simply add at the end).
    auto dot = [&](const uint4 &raw) {
        float x[VE];
        float2 d = make_float2(0.f, 0.f);
        RowVec<T>::unpack(raw, x);
#pragma unroll
        for (int i = 0; i < VE; i += 2) d = fma2(make_float2(qf[i], qf[i + 1]), make_float2(x[i], x[i + 1]), d);
        return d.x + d.y;
    };
    auto add = [&](float p, const uint4 &raw) {
        float x[VE];
        RowVec<T>::unpack(raw, x);
        lsum += p;
#pragma unroll
        for (int i = 0; i < VE; i += 2) acc[i / 2] = fma2(make_float2(p, p), make_float2(x[i], x[i + 1]), acc[i / 2]);
    };
    auto rescale = [&](float mx) {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (!(mx > M)) return;  // (the same in all lanes)
        const float corr = exp2f(M - mx);
        M = mx;
        lsum *= corr;
#pragma unroll
        for (int i = 0; i < VE / 2; ++i) acc[i] = mul2(acc[i], make_float2(corr, corr));
    };
    int stage = 0;
    for (int base = rw.r0 + warp * STEP; base < rw.r1; base += kCWarps * STEP) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kCStages - 1) : "memory");
        const unsigned char *kt = ring + stage * 2 * kCRound;
        float s[kCU], mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < kCU; ++j) s[j] = dot(*reinterpret_cast<const uint4 *>(kt + j * 512));
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < kCU; ++j) s[j] += __shfl_xor_sync(0xffffffffu, s[j], o);
        if (base + STEP <= rw.r1 && rw.skip < 0) {
#pragma unroll
            for (int j = 0; j < kCU; ++j) mx = fmaxf(mx, s[j]);
            rescale(mx);
#pragma unroll
            for (int j = 0; j < kCU; ++j) add(exp2f(s[j] - M), *reinterpret_cast<const uint4 *>(kt + kCRound + j * 512));
        } else {
#pragma unroll
            for (int j = 0; j < kCU; ++j) {
                const int r = base + j * G + grp;  // (what was not copied may be anything, NaN included)
                if (r >= rw.r1 || r == rw.skip) s[j] = -INFINITY;
                mx = fmaxf(mx, s[j]);
            }
            rescale(mx);
#pragma unroll
            for (int j = 0; j < kCU; ++j) {
                const int r = base + j * G + grp;
                if (r < rw.r1 && r != rw.skip) add(exp2f(s[j] - M), *reinterpret_cast<const uint4 *>(kt + kCRound + j * 512));
            }
        }
        request(rw, base + kCStages * kCWarps * STEP, stage);
        if (++stage == kCStages) stage = 0;
    }
    if (takes_new && sp.rows >= 0) {
        float s = dot(knew);
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        rescale(s);
        if (grp == 0) {
            add(exp2f(s - M), vnew);
            // the append: this head's slice of the new row goes to its place in the cache
            const size_t at = (size_t)(sp.off + sp.dst) * a.row_bytes + (size_t)h * SLICE + c * 16;
            *reinterpret_cast<uint4 *>(static_cast<unsigned char *>(a.ck) + at) = knew;
            *reinterpret_cast<uint4 *>(static_cast<unsigned char *>(a.cv) + at) = vnew;
        }
    }

    if (P == kCPerSm) last_one();

    // ---- merge: lane groups, warps, then the CTAs of the cluster ---------------------------------------
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
#pragma unroll
        for (int i = 0; i < VE / 2; ++i) {
            acc[i].x += __shfl_xor_sync(0xffffffffu, acc[i].x, o);
            acc[i].y += __shfl_xor_sync(0xffffffffu, acc[i].y, o);
        }
    }
    if (grp == 0) {
#pragma unroll
        for (int i = 0; i < VE; i += 2) *reinterpret_cast<float2 *>(&s_acc[warp][c * VE + i]) = acc[i / 2];
    }
    if (lane == 0) {
        s_ml[warp][0] = M;
        s_ml[warp][1] = lsum;
    }
    __syncthreads();
    // (a state without rows has sums of 0; one whose only logits are NaN has sums of NaN, whatever their factor)
    float z = 0.f, o = 0.f, m = kNoLogit;
#pragma unroll
    for (int w = 0; w < kCWarps; ++w) m = fmaxf(m, s_ml[w][0]);
#pragma unroll
    for (int w = 0; w < kCWarps; ++w) {
        const float f = exp2f(s_ml[w][0] - m);
        z = fmaf(f, s_ml[w][1], z);
        if (tid < D) o = fmaf(f, s_acc[w][tid], o);
    }
    if (C > 1) {
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        if (tid < D) store_in_first_cta(&c_acc[rank][tid], o);
        if (tid == 0) {
            store_in_first_cta(&c_ml[rank][0], m);
            store_in_first_cta(&c_ml[rank][1], z);
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (rank != 0) return;  // (only the first CTA's memory is written, and it waits for everyone)
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        m = kNoLogit;
        for (int r = 0; r < C; ++r) m = fmaxf(m, c_ml[r][0]);
        z = 0.f;
        o = 0.f;
        for (int r = 0; r < C; ++r) {
            const float f = exp2f(c_ml[r][0] - m);
            z = fmaf(f, c_ml[r][1], z);
            if (tid < D) o = fmaf(f, c_acc[r][tid], o);
        }
    }
    if (tid < D)  // (the output of a segment that cannot take the step is zero)
        reinterpret_cast<T *>(static_cast<unsigned char *>(a.out) + hoff)[tid] = from_float<T>(sp.rows < 0 ? 0.f : o * (1.f / z));
}

template <typename T, int D, int U, int P> int launch_cluster(const ClusterArgs &a, int C, cudaStream_t st)
{
    // Room for P CTAs and not for one more.  (Clusters have the first shape; the others need no place for partials.)
    constexpr int rings = kCWarps * kCStages * 2 * U * 512;
    // (its static part, rounded up, and what every CTA takes)
    constexpr int fixed = kCWarps * (D + 2) * (int)sizeof(float) + (P == kCPerSm ? kCMaxCluster : 1) * D * (int)sizeof(float) + 1344;
    constexpr int one_more = kCSmShared / (P + 1) - fixed + 512;
    constexpr int smem = rings > one_more ? rings : one_more;
    static_assert(P * (smem + fixed) <= kCSmShared, "P CTAs fit");
    static bool smem_done[64] = {};
    int rc = ensure_dynamic_smem((const void *)decode_cluster_kernel<T, D, U, P>, smem, smem_done);
    if (rc != PKV_OK) return rc;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)C;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.p.nact * a.H * C));
    cfg.blockDim = dim3(kCWarps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, decode_cluster_kernel<T, D, U, P>, a);
    if (e != cudaSuccess) {
        set_cuda_error(e, "decode_cluster_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}
template <int U, int P> int launch_shape(const pkv_shape *s, const ClusterArgs &a, int C, cudaStream_t st)
{
    if (s->dtype == PKV_BF16)
        return s->head_dim == 128 ? launch_cluster<__nv_bfloat16, 128, U, P>(a, C, st) : launch_cluster<__nv_bfloat16, 64, U, P>(a, C, st);
    return s->head_dim == 128 ? launch_cluster<float, 128, U, P>(a, C, st) : launch_cluster<float, 64, U, P>(a, C, st);
}

}  // namespace

// CTAs to a pair for a call of nact segments; 0 when another kernel is to take it.
int decode_cluster_ctas(const pkv_shape *s, const pkv_cache *c, int nact, int sms)
{
    const int H = s->heads, D = s->head_dim;
    const int64_t items = (int64_t)nact * H, seg_rows = c->total_cap_rows / ((int64_t)s->batch * s->layers);
    const int64_t pair_bytes = seg_rows * D * 2 * (int64_t)esize(s);
    const int wave = kCPerSm * sms;
    if (items >= 4 * (int64_t)sms) {
        // A CTA for every pair.  Measured, us a call replayed from a graph, the kernel that takes the call otherwise (per head, or split by rows
        // with more than 256 segments or 1024 rows, or with pruning) / this one; lengths all alike, random (lognormal, sigma 0.5), as a
        // search at a budget of 0.2 leaves them; bf16 heads of 128 (512 bytes a row) where nothing else is said:
        //   pairs x rows          alike           random          searched
        //   one wave, five CTAs an SM and fewer:
        //    640 x 64          10.1 / 7.5       9.7 / 7.5      10.4 / 7.7
        //    640 x 512         34.0 / 30.5     32.4 / 29.1     42.4 / 31.5
        //    640 x 820         48.8 / 44.7     46.3 / 43.6     53.1 / 47.2
        //    640 x 1000        59.4 / 53.4     54.2 / 51.6     58.2 / 56.6
        //   six and seven CTAs an SM, in one wave too:
        //    888 x 64          12.3 / 9.2      11.7 / 10.0     11.6 / 9.4
        //    888 x 480         40.1 / 37.8     40.4 / 44.4     42.1 / 39.8
        //    888 x 640         50.4 / 48.2     50.7 / 57.2     52.1 / 51.6
        //   1024 x 32          10.5 / 7.0      10.3 / 7.7      10.6 / 7.4
        //   1024 x 136         17.3 / 14.9     17.5 / 17.5     20.7 / 15.5
        //   1024 x 256         26.1 / 24.8     27.5 / 29.5     32.8 / 25.4
        //   1024 x 600         52.9 / 52.6     52.4 / 61.7     58.0 / 56.0
        //   1024 x 820         69.3 / 69.6     67.8 / 83.0     73.2 / 73.9
        //   more waves: CTAs that begin cost the first rows' latency, which is little against long rows:
        //   1280 x 32          11.8 / 9.5      12.2 / 10.2     11.9 / 9.9
        //   1280 x 410         47.6 / 44.8     47.3 / 49.7     50.7 / 46.7
        //   1280 x 700         75.0 / 69.7     72.7 / 80.8     76.4 / 76.5
        //   2048 x 64          20.0 / 19.2     18.9 / 19.5     21.5 / 19.0
        //   2048 x 128         27.8 / 27.7     27.3 / 26.5     32.6 / 26.0
        //   2048 x 820          131 / 125       127 / 121       143 / 130
        //   4096 x 16          20.3 / 22.2     20.6 / 21.9     20.1 / 22.0
        //   4096 x 64          35.5 / 33.6     34.3 / 34.0     35.8 / 31.7
        //   4096 x 820          257 / 243       260 / 251       283 / 250
        //   8192 x 128         97.1 / 89.6                      101 / 87.5
        //   heads of 64:
        //   2048 x 100         17.4 / 17.4     17.5 / 17.4
        //   4096 x 32          20.4 / 22.1     20.6 / 22.6     20.3 / 22.3
        //   4096 x 256         50.7 / 47.6     50.5 / 49.5     54.0 / 47.6
        //   fp32:
        //   2048 x 128         46.7 / 45.7     46.6 / 43.3     55.5 / 44.1
        //   4096 x 100, of 64  42.1 / 40.2                     42.7 / 39.8
        //   with pruning:
        //    640 x 64          16.3 / 9.3                      18.5 / 9.5
        //   2048 x 64          22.1 / 22.3                     22.8 / 21.2
        //   2048 x 128         33.1 / 31.2                     33.3 / 28.5
        //   4096 x 64          33.5 / 38.4                     34.8 / 36.1
        //   4096 x 220         82.5 / 79.0                     80.8 / 74.2
        //   8192 x 128         95.7 / 96.7                     95.2 / 92.4
        //   more than 256 segments, 32 heads of 128, 16 of 64, eight of 64:
        //   9216 x 64          60.2 / 65.4                     59.8 / 64.0
        //   9216 x 128          106 / 98.7                      104 / 96.4
        //   30720 x 128         320 / 304                       321 / 308
        //   4608 x 128         42.6 / 34.6                     44.0 / 33.9
        //   2304 x 16          13.4 / 13.0                     15.1 / 12.8
        //   7680 x 64          65.7 / 40.5                     66.8 / 40.3
        // One segment of a multiple of the mean (first or last of the call) sets the time of its CTAs, which the other kernels split up: 1024 x
        // 136 five times the mean 19.6 / 24.2, twenty 33.2 / 75.5; 1024 x 512 ten 50 / 122, twenty 53 / 222; 4096 x 820 five 266 / 289, ten
        // 266 / 345; 6400 x 410 ten 225 / 243.  A search of the repository's workloads leaves 2.7 times the mean at most.
        // By a pair's rows, and their bytes, halfway through the tokens that the cache has room for.
        const int64_t rows = seg_rows - c->decode_cap / 2, kb = rows * D * 2 * (int64_t)esize(s) >> 10;
        int64_t least = 0, most_kb = INT64_MAX;
        if (items <= wave) most_kb = 448;
        else if (items <= 6 * (int64_t)sms) most_kb = 256;
        else if (items < 10 * (int64_t)sms) most_kb = 320;
        else if (c->evict_distance > 0) least = items < 20 * (int64_t)sms ? 80 : 200;
        else if (nact > 256) least = (size_t)H * D * esize(s) <= 1024 ? 0 : 112;
        else least = items < 20 * (int64_t)sms ? 96 : 80;
        if (rows < least || kb > most_kb || items > INT32_MAX / 2) return 0;
    }
    // Few pairs, but the longest, for which the row-split kernel is as fast where it covers the shape, row-split / this one, one layer: 1 head
    // of 128, bf16, 8000 rows 18.1 / 13.4, 15000 31.1 / 21.8, fp32 8000 26.8 / 20.9; 8 heads fp32 8000 40.1 / 31.9, 12000 (12.3 MB a pair) 45.0 / 45.6;
    // 32 pairs of 12000 67.9 / 63.3; 128 pairs of bf16, 6000 72.5 / 65.1, 12000 129 / 121; 320 x 1800 57.6 / 53.4, x 4500 120 / 110; 512 x 1800 79.9 / 77.9,
    // x 2400 103 / 98, heads of 64 47.5 / 48.3; 576 x 1800 88.3 / 85.2.  (Nothing longer measured.)
    if (items < 4 * (int64_t)sms &&
        (pair_bytes > ((int64_t)(items < 24 ? 11 : 13) << 20) ||
         items * seg_rows > (D == 64 ? (items <= 320 ? 1 << 20 : 704 << 10) : 1536 << 10) || items * pair_bytes > ((int64_t)800 << 20)) &&
        decode_stream_covers(s, nact))
        return 0;
    // As many CTAs as the SMs hold at a time, none of them with less than one round of rows (32) unless
    // the call is so small that SMs would be idle; further waves only for CTAs of 256 rows and more,
    // whose bytes outweigh a wave's latency (16 x 32 x 2048 rows: C = 1 111 us, 6 89 us in one run, 99 in another).
    int C = 1;
    while (C < kCMaxCluster && items < 4 * (int64_t)sms) {
        const int n = C + 1;
        const bool one_wave = items * n <= wave &&
                              (seg_rows >= 32 * n || items * n <= 2 * (int64_t)sms);
        if (!one_wave && seg_rows < 256 * (int64_t)n) break;
        C = n;
    }
    return (int64_t)H * C >= (int64_t)1 << kVisitBits ? 0 : C;
}

// Returns PKV_OK, an error, or -1 when this call is outside what the kernel covers.
int launch_decode_cluster(const pkv_shape *s, pkv_cache *c, const void *q, const void *kn, const void *vn,
                          const float *scale, int lb, int le, void *out, int32_t *dev_status, void *ws, cudaStream_t st)
{
    const int H = s->heads, D = s->head_dim, nl = le - lb, nact = s->batch * nl;
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    const int C = decode_cluster_ctas(s, c, nact, sms);
    if (C == 0) return -1;
    const int64_t items = (int64_t)nact * H;
    ClusterArgs a;
    a.p = decode_plan_args(s, c, kn != nullptr, lb, nl);
    a.q = q; a.k_new = kn; a.v_new = vn; a.ck = c->k; a.cv = c->v; a.out = out;
    a.layer_scale = scale;
    a.visits = (unsigned long long *)ws;
    a.visit_tag = visit_tag();
    a.dev_status = dev_status;
    a.H = H;
    // A call of one wave is set up while the one in front, of the same cache maybe, has yet to write the lengths.  (24 x 16 heads of 64, 90
    // rows, call after call: 5.9 us a call, 5.25 so.)  With clusters another length moves most CTAs' rows.
    a.guess_more = kn != nullptr && c->evict_distance == 0 && C == 1 && items <= kCPerSm * (int64_t)sms ? 1 : 0;
    a.row_bytes = (uint32_t)((size_t)H * D * esize(s));
    if (C == 1 && items > kCPerSm * (int64_t)sms && items <= 6 * (int64_t)sms) return launch_shape<4, 6>(s, a, C, st);
    if (C == 1 && items > kCPerSm * (int64_t)sms && items <= 7 * (int64_t)sms) return launch_shape<3, 7>(s, a, C, st);
    return launch_shape<4, kCPerSm>(s, a, C, st);
}

}  // namespace pkv
