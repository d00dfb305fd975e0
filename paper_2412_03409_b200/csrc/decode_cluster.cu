// Decode attention over the ragged cache (Sec. 3.1, Fig. 2a), (segment, head) pair by pair: calls with few pairs (a layer at
// a time, or a few layers, of a small batch) by a cluster of CTAs to a pair, most others by a CTA to a pair
// (launch_decode_cluster has the lines).
//
// A call of few pairs moves a few megabytes, so what counts is the chain of latencies of one launch and that
// every SM has a share.  A cluster of C CTAs takes one (segment, head); each CTA takes a C-th of its
// rows.  Every warp copies its rows' slices of the head into a ring of its own with 16-byte cp.async
// and reads back what the same lane copied, so that no warp waits for another until the merge.  The
// CTAs' partial softmax states go to the first CTA of the cluster through distributed shared memory,
// which merges them in rank order and writes the head's output: one launch, nothing in global memory
// in between.  The last CTA of a cluster also attends to the new row and appends it.
// Lengths: a CTA reads its segment's length by adding one to the upper bits of its word, which so counts
// the CTAs that have been there; the last of them writes the length of the next step over it.  A call
// that appends nothing leaves the word alone.  (Before, every CTA raised a flag in the workspace and an
// extra cluster waited for them: its chain of round trips ended after the rows', 4.43 us a call below for 3.96 without.)
// Where the rows are is also read ahead, while the kernel in front still runs: the rows of that guess are
// asked for as soon as it has completed, and the guess is held against the plan made afterwards.  The
// values are not looked at before then, so that a CTA that starts late has both loads on their way at once
// (looked at before: 19.3 us for 17.7 in the case of 8 x 40 x 410 rows; one thread's loads, passed on through
// shared memory: 20.1, and 4.15 for 3.77 in the smallest).
//
// Measured, device time of calls replayed from a graph, one layer, bf16, D = 128, every call on another layer: 1 segment
// x 32 heads x 128 rows 3.77 us (4.43 with flags and without the guess), 4 x 32 x 128 rows 5.46 (6.00), 16 x 32 x 128 10.98 (11.55),
// 1 x 40 x 410 5.05 (5.63), 8 x 40 x 410 17.7 (18.8; 10.3 us of bytes); against the row-split kernel and its merge
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
    int32_t *dev_status;
    int H, visit_shift;  // a length's word counts its readers from this bit on
    uint32_t guess_mask;  // what a length read ahead is taken from: the word without that count, where CTAs come in waves
    uint32_t row_bytes;
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Store into the first CTA of the cluster, at the place that `p` has in this CTA's shared memory.
__device__ __forceinline__ void store_first_cta(float *p, float v)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}
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
    __shared__ float s_acc[kCWarps][D], s_ml[kCWarps][2];
    __shared__ float c_acc[P == kCPerSm ? kCMaxCluster : 1][D], c_ml[kCMaxCluster][2];  // (first CTA of a cluster) the cluster's partials

    __shared__ SegPlan s_plan[2];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int item = blockIdx.x / C;
    // (the first CTA must be running before anyone writes to its shared memory)
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
#pragma unroll
        for (int j = 0; j < kCU; ++j) {
            const int r = base + j * G + grp;
            if (r < rw.r1 && r != rw.skip) {
                copy16(d + j * 512, rw.kb + (size_t)r * a.row_bytes);
                copy16(d + kCRound + j * 512, rw.vb + (size_t)r * a.row_bytes);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // A length's word: the length, and above it how many of the segment's CTAs have been there.
    const uint32_t ln_mask = a.p.append ? (1u << a.visit_shift) - 1u : 0xffffffffu;
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
    // The length is read by adding to its word's upper bits: whoever finds that all CTAs of the segment but itself have
    // been there writes what the step leaves.  (With pruning what else the plan is made of has been read before that.)
    uint32_t word = 0;
    int cp = 0;
    int64_t off = 0;
    PruneState ps;
    if (tid == 0) {
        ps = prune_state(a.p, seg);
        if (!a.p.append) word = (uint32_t)load_l2(a.p.len + seg);
        else if (a.p.evict_distance == 0) asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], %2;" : "=r"(word) : "l"(a.p.len + seg), "r"(1u << a.visit_shift) : "memory");
        else asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(word) : "l"(a.p.len + seg), "r"(1u << a.visit_shift) : "memory");
        cp = load_l2(a.p.cap + seg);
        off = load_l2(a.p.row_offset + seg);
    }
    Rows rw{nullptr, nullptr, 0, 0, -1};
    if (guesses) {
        rw = rows_of(plan_of(a.p, (int)((uint32_t)guess_ln & a.guess_mask), guess_cp, guess_off, PruneState{0, 0, -1}));
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
    if (tid == 0) {
        const uint32_t before = a.p.append ? word >> a.visit_shift : 0u, all = (uint32_t)(a.H * C);
        SegPlan sp = plan_of(a.p, (int)(word & ln_mask), cp, off, ps);
        if (before >= all) sp.rows = -1;  // (the word was no length)
        if (sp.rows < 0) {  // (every CTA finds the same, and takes back what it added)
            raise_status(a.dev_status, si / a.p.nl, PKV_DEV_CAPACITY);
            if (a.p.append) atomicSub(reinterpret_cast<unsigned int *>(a.p.len + seg), 1u << a.visit_shift);
        } else if (a.p.append && before == all - 1) {
            segment_advance(a.p, si, sp);
        }
        s_plan[1] = sp;
    }
    __syncthreads();
    const SegPlan sp = s_plan[1];
    const Rows now = rows_of(sp);
    if (now.r0 != rw.r0 || now.r1 != rw.r1 || now.skip != rw.skip || now.kb != rw.kb) {
        // (a row more or less at the end: the same bytes come to the same places again)
        if (now.r0 != rw.r0 || now.skip != rw.skip || now.kb != rw.kb) asm volatile("cp.async.wait_all;" ::: "memory");
        rw = now;
#pragma unroll
        for (int i = 0; i < kCStages; ++i) request(rw, rw.r0 + (warp + i * kCWarps) * STEP, i);
    }

    // M: the running maximum of the logits, from the lowest finite number on, so that exp2f(s - M) is 0 for a logit
    // of -infinity and NaN for NaN whatever came before it.
    float qf[VE], acc[VE], M = kNoLogit, lsum = 0.f;
    RowVec<T>::unpack(qraw, qf);
#pragma unroll
    for (int i = 0; i < VE; ++i) {
        qf[i] *= sc;
        acc[i] = 0.f;
    }
    // One round: logits of the warp's rows, one rescale, accumulation (every lane group keeps the
    // warp-wide running maximum, so that the groups' sums simply add at the end).
    auto dot = [&](const uint4 &raw) {
        float x[VE], d0 = 0.f, d1 = 0.f;
        RowVec<T>::unpack(raw, x);
#pragma unroll
        for (int i = 0; i < VE; i += 2) {
            d0 = fmaf(qf[i], x[i], d0);
            d1 = fmaf(qf[i + 1], x[i + 1], d1);
        }
        return d0 + d1;
    };
    auto add = [&](float p, const uint4 &raw) {
        float x[VE];
        RowVec<T>::unpack(raw, x);
        lsum += p;
#pragma unroll
        for (int i = 0; i < VE; ++i) acc[i] = fmaf(p, x[i], acc[i]);
    };
    auto rescale = [&](float mx) {
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float Mn = fmaxf(M, mx);
        const float corr = exp2f(M - Mn);
        M = Mn;
        lsum *= corr;
#pragma unroll
        for (int i = 0; i < VE; ++i) acc[i] *= corr;
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
            if (r < rw.r1 && r != rw.skip)
                add(exp2f(s[j] - M), *reinterpret_cast<const uint4 *>(kt + kCRound + j * 512));
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

    // ---- merge: lane groups, warps, then the CTAs of the cluster ---------------------------------------
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
#pragma unroll
        for (int i = 0; i < VE; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    }
    if (grp == 0) {
#pragma unroll
        for (int i = 0; i < VE; ++i) s_acc[warp][c * VE + i] = acc[i];
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
        if (tid < D) store_first_cta(&c_acc[rank][tid], o);
        if (tid == 0) {
            store_first_cta(&c_ml[rank][0], m);
            store_first_cta(&c_ml[rank][1], z);
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

// Returns PKV_OK, an error, or -1 when this call is outside what the kernel covers.
int launch_decode_cluster(const pkv_shape *s, pkv_cache *c, const void *q, const void *kn, const void *vn,
                          const float *scale, int lb, int le, void *out, int32_t *dev_status, cudaStream_t st)
{
    const int H = s->heads, D = s->head_dim, nl = le - lb, nact = s->batch * nl;
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    const int64_t items = (int64_t)nact * H, seg_rows = c->total_cap_rows / ((int64_t)s->batch * s->layers);
    const int64_t pair_bytes = seg_rows * D * 2 * (int64_t)esize(s);
    const int wave = kCPerSm * sms;
    if (items >= 4 * (int64_t)sms) {
        // A CTA for every pair.  Measured, the per-head (or row-split) kernel / this one, us a call, bf16, heads of 128, lengths alike and
        // from 0.3 to 1.7 of the mean.  One wave: 640 pairs of 30 rows 7.5 / 4.9, 8.4 / 5.4, of 128 12.7 / 10.4, 13.4 / 11.6, of 400
        // 28.3 / 25.6, 28.7 / 28.6, but of 820 48.9 / 48.6, 46.9 / 50.2: the longest pairs end alone.  740 pairs of 128 14.0 / 12.0.
        // Up to seven CTAs an SM, in one wave too: 800 x 64 11.2 / 9.1, x 256 22.7 / 22.3, 26.7 / 24.4, x 400 33.1 / 31.8, 33.8 / 35.2, 1024 x 30 8.9 / 7.1, 10.2 / 7.4, x 128 16.6 / 15.5, 18.0 / 16.5,
        // but x 256 26.1 / 27.1, 31.8 / 30.1, x 400 38.8 / 39.6, 39.8 / 43.5.  More waves: CTAs that begin cost the first rows' latency,
        // which is little against long rows, and is hidden where lengths differ, as they do after a search: 1280 x 256 31.9 / 33.1,
        // 38.4 / 31.9, 1536 x 384 54.5 / 54.2, 55.3 / 52.7, 2048 x 64 20.0 / 21.4, 19.9 / 20.6, x 128 27.6 / 29.5, 28.8 / 28.1, x 256 46.5 / 48.3,
        // 52.1 / 48.1, 1600 x 820 104.4 / 107.4, 107.1 / 110.2, 4096 x 128 50.7 / 51.9, 52.3 / 50.9, x 400 130.7 / 128.1, 143.9 / 129.8, 8192 x 400
        // 257 / 248, 284 / 247; against the row-split kernel 12800 x 410 395 / 377, 16384 x 128 174 / 177, x 256 343 / 313;
        // with pruning 640 x 64 17.0 / 10.3, 4096 x 64 33.9 / 36.7, x 200 75.3 / 74.1.
        // By a pair's bytes halfway through the tokens that the cache has room for.
        const int64_t kb = (seg_rows - c->decode_cap / 2) * D * 2 * (int64_t)esize(s) >> 10;
        bool here;
        if (items <= wave) here = kb <= 256;
        else if (items <= 6 * (int64_t)sms) here = kb <= 176;
        else if (items <= 7 * (int64_t)sms) here = kb <= 96;
        else if (items < 10 * (int64_t)sms) here = kb >= 96 && kb <= 256;
        else here = kb >= (nact > 256 || c->evict_distance > 0 ? 96 : 64) && (items >= 20 * (int64_t)sms || kb <= 320) && items <= INT32_MAX / 2;
        if (!here) return -1;
    }
    // Long segments are the row-split kernel's, where it covers the shape: eight CTAs of a pair keep 256 KiB in
    // flight however long it is, and CTAs that come in waves read the slices of a row at different times.
    // Measured, one layer, this kernel / row-split.  Few pairs, by a pair's bytes: 1 head of 128, bf16, 12000 rows
    // (6.1 MB) 29 / 33 us, 16000 (8.2) 38 / 35, fp32 6000 rows 29 / 30, 8000 38 / 31, 16000 70 / 35; 8 heads
    // fp32 8000 38 / 40, 12000 56 / 45.  From 24 pairs on the row-split kernel's merge costs more: 24 heads fp32
    // 12000 rows (12.3 MB) 64 / 81, 32 pairs of 4 segments 72 / 73, 16000 rows 94 / 92.  Many pairs, by pairs x
    // rows: 128 x 6000 rows 73 / 73, x 12000 137 / 130; 320 x 1800 58 / 59, x 3200 86 / 92; 512 x 1100 55 / 59, x
    // 1800 89 / 83 (heads of 64: 34 / 36, 55 / 49); 576 x 1100 60 / 60, x 1800 96 / 90; and by bytes: 64 pairs of 8000 rows of fp32
    // (524 MB) 90 / 90, 12000 134 / 126.
    if (items < 4 * (int64_t)sms &&
        (pair_bytes > ((int64_t)(items < 24 ? 6 : 12) << 20) || items * seg_rows > (items <= 320 ? 1 << 20 : 704 << 10) ||
         items * pair_bytes > ((int64_t)512 << 20)) &&
        decode_stream_covers(s, nact))
        return -1;
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
    // (the bits of a length's word that its readers are counted in leave room for any length)
    int visit_bits = 1;
    while ((H * C) >> visit_bits) ++visit_bits;
    if (c->total_cap_rows >> (32 - visit_bits)) return -1;

    ClusterArgs a;
    a.p = decode_plan_args(s, c, kn != nullptr, lb, nl);
    a.q = q; a.k_new = kn; a.v_new = vn; a.ck = c->k; a.cv = c->v; a.out = out;
    a.layer_scale = scale;
    a.visit_shift = 32 - visit_bits;
    a.guess_mask = kn != nullptr && items * C > wave ? (1u << a.visit_shift) - 1u : 0xffffffffu;
    a.dev_status = dev_status;
    a.H = H;
    a.row_bytes = (uint32_t)((size_t)H * D * esize(s));
    if (C == 1 && items > wave && items <= 6 * (int64_t)sms) return launch_shape<4, 6>(s, a, C, st);
    if (C == 1 && items > wave && items <= 7 * (int64_t)sms) return launch_shape<3, 7>(s, a, C, st);
    return launch_shape<4, kCPerSm>(s, a, C, st);
}

}  // namespace pkv
