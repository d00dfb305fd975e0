// Decode attention over the ragged cache (Sec. 3.1, Fig. 2a) for calls with few (segment, head)
// pairs: a layer at a time, or a few layers, of a small batch.
//
// Such a call moves a few megabytes, so what counts is the chain of latencies of one launch and that
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
// 4, 3, 4 18.9-19.4 us there; 2, 4, 5 18.7.  Clusters of 12 or 16: slower throughout.
#include "decode_plan.cuh"

namespace pkv {

bool decode_stream_covers(const pkv_shape *s, int nact);

namespace {

constexpr int kCWarps = 4;             // warps per CTA
constexpr int kCU = 4;                 // row steps of a round
constexpr int kCStages = 2;            // rounds in flight per warp
constexpr int kCPerSm = 5;             // CTAs an SM holds at a time (their rings fill its shared memory)
constexpr uint32_t kCRound = kCU * 512;  // bytes of a round's K (or V) rows: a warp reads 512 bytes per step
constexpr int kCMaxCluster = 8;        // portable cluster size
constexpr float kLog2eC = 1.4426950408889634f;
constexpr float kNoLogit = -3.402823466e38f;  // the lowest finite number

struct ClusterArgs {
    DecodePlanArgs p;
    const void *q, *k_new, *v_new;
    void *ck, *cv, *out;
    const float *layer_scale;
    int32_t *dev_status;
    int H, visit_shift;  // a length's word counts its readers from this bit on
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
template <typename T, int D>
__global__ void __launch_bounds__(kCWarps * 32, kCPerSm) decode_cluster_kernel(const ClusterArgs a)
{
    constexpr int VE = RowVec<T>::VE;
    constexpr uint32_t SLICE = D * sizeof(T);
    constexpr int LPR = SLICE / 16, G = 32 / LPR;
    constexpr int STEP = kCU * G;  // rows of one round of a warp
    static_assert(kCWarps * 32 >= D, "a thread per element of the output");
    extern __shared__ __align__(16) unsigned char s_ring[];  // [kCWarps][kCStages][K, V][kCRound]
    __shared__ float s_acc[kCWarps][D], s_ml[kCWarps][2];
    __shared__ float c_acc[kCMaxCluster][D], c_ml[kCMaxCluster][2];  // (first CTA) the cluster's partials

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
        rw = rows_of(plan_of(a.p, guess_ln, guess_cp, guess_off, PruneState{0, 0, -1}));
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
        const int ln = a.p.append ? (int)(word & ((1u << a.visit_shift) - 1u)) : (int)word;
        SegPlan sp = plan_of(a.p, ln, cp, off, ps);
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

template <typename T, int D> int launch_cluster(const ClusterArgs &a, int C, cudaStream_t st)
{
    constexpr int smem = kCWarps * kCStages * 2 * (int)kCRound;
    static bool smem_done[64] = {};
    int rc = ensure_dynamic_smem((const void *)decode_cluster_kernel<T, D>, smem, smem_done);
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
    cudaError_t e = cudaLaunchKernelEx(&cfg, decode_cluster_kernel<T, D>, a);
    if (e != cudaSuccess) {
        set_cuda_error(e, "decode_cluster_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

}  // namespace

// Returns PKV_OK, an error, or -1 when this call is outside what the kernel covers.
int launch_decode_cluster(const pkv_shape *s, pkv_cache *c, const void *q, const void *kn, const void *vn,
                          const float *scale, int lb, int le, void *out, int32_t *dev_status, cudaStream_t st)
{
    const int H = s->heads, D = s->head_dim, nl = le - lb, nact = s->batch * nl;
    const int sms = sm_count();
    if (sms <= 0) return PKV_ERR_CUDA;
    if ((int64_t)nact * H >= 4 * (int64_t)sms) return -1;  // (the per-head kernel's and the row-split kernel's calls)
    const int items = nact * H;
    const int64_t seg_rows = c->total_cap_rows / ((int64_t)s->batch * s->layers);
    // Long segments are the row-split kernel's, where it covers the shape: eight CTAs of a pair keep 256 KiB in
    // flight however long it is, and CTAs that come in waves read the slices of a row at different times.
    // Measured, one layer, this kernel / row-split.  Few pairs, by a pair's bytes: 1 head of 128, bf16, 12000 rows
    // (6.1 MB) 29 / 33 us, 16000 (8.2) 38 / 35, fp32 6000 rows 29 / 30, 8000 38 / 31, 16000 70 / 35; 8 heads
    // fp32 8000 38 / 40, 12000 56 / 45.  From 24 pairs on the row-split kernel's merge costs more: 24 heads fp32
    // 12000 rows (12.3 MB) 64 / 81, 32 pairs of 4 segments 72 / 73, 16000 rows 94 / 92.  Many pairs, by pairs x
    // rows: 128 x 6000 rows 73 / 73, x 12000 137 / 130; 320 x 1800 58 / 59, x 3200 86 / 92; 512 x 1100 55 / 59, x
    // 1800 89 / 83 (heads of 64: 34 / 36, 55 / 49); 576 x 1100 60 / 60, x 1800 96 / 90; and by bytes: 64 pairs of 8000 rows of fp32
    // (524 MB) 90 / 90, 12000 134 / 126.
    const int64_t pair_bytes = seg_rows * D * 2 * (int64_t)esize(s);
    if ((pair_bytes > ((int64_t)(items < 24 ? 6 : 12) << 20) || items * seg_rows > (items <= 320 ? 1 << 20 : 704 << 10) ||
         items * pair_bytes > ((int64_t)512 << 20)) &&
        decode_stream_covers(s, nact))
        return -1;
    // As many CTAs as the SMs hold at a time, none of them with less than one round of rows (32) unless
    // the call is so small that SMs would be idle; further waves only for CTAs of 256 rows and more,
    // whose bytes outweigh a wave's latency (16 x 32 x 2048 rows: C = 1 111 us, 6 89 us in one run, 99 in another).
    int C = 1;
    while (C < kCMaxCluster) {
        const int n = C + 1;
        const bool one_wave = (int64_t)items * n <= (int64_t)kCPerSm * sms &&
                              (seg_rows >= 32 * n || (int64_t)items * n <= 2 * (int64_t)sms);
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
    a.dev_status = dev_status;
    a.H = H;
    a.row_bytes = (uint32_t)((size_t)H * D * esize(s));
    if (s->dtype == PKV_BF16) return D == 128 ? launch_cluster<__nv_bfloat16, 128>(a, C, st) : launch_cluster<__nv_bfloat16, 64>(a, C, st);
    return D == 128 ? launch_cluster<float, 128>(a, C, st) : launch_cluster<float, 64>(a, C, st);
}

}  // namespace pkv
