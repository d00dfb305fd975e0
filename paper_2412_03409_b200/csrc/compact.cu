// Compression after prefilling (Sec. 3.1, Fig. 2a): the len top-ranked rows of
// every segment are copied, in ascending prompt position, into one packed
// ragged cache.  Pure data movement in 16-byte vectors; HBM-bound.
#include <algorithm>

#include "common.cuh"

namespace pkv {

// One CTA per segment: row offset of the segment (exclusive sum of capacities of
// the segments before it), capacity check, and the ascending list of retained
// positions (a bitmap over positions filled from the first len ranks, then a
// scan over word popcounts).
//
// A chain of latencies between the search and the copy: what can be set up is, before the wait for the search, a thread's first rank
// is read along with the lengths, and the offset's sum and the bitmap meet at one barrier (plan and copy, six barriers after the wait /
// so: 640 tokens, 32 layers 23.4 / 23.0 us; 300 tokens, 16 layers of 8 heads of 64 6.0 / 5.5; 16384 tokens, batch 2 275.6 / 275.2).
__global__ void __launch_bounds__(1024)
compact_plan_kernel(const int32_t *__restrict__ order, const int32_t *__restrict__ len_in, int nseg,
                    int L, int N, int decode_cap, int64_t total_cap_rows,
                    int64_t *__restrict__ row_offset, int32_t *__restrict__ len_out,
                    int32_t *__restrict__ cap_out, int32_t *__restrict__ kept, int32_t *dev_status,
                    int32_t *len0, int32_t *gen, int32_t *slot_ring, int ring_size)
{
    __shared__ uint32_t bitmap[kMaxPromptLen / 32];
    __shared__ int64_t red[32];
    __shared__ int wsum[32];
    const int seg = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = seg / L;
    const int nwords = (N + 31) >> 5;  // <= 512 <= blockDim.x
    if (tid < nwords) bitmap[tid] = 0;
    __syncthreads();
    dependent_entry();

    auto clamp_len = [&](int v) { return (v < 1 || v > N) ? 0 : v; };
    const int32_t *ord = order + (size_t)seg * N;
    const int first = tid < N ? ord[tid] : -1;
    const int raw = len_in[seg];

    // offset = sum over earlier segments of (len + decode_cap)
    int64_t part = 0;
    for (int s = tid; s < seg; s += blockDim.x) part += (int64_t)clamp_len(len_in[s]) + decode_cap;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) red[warp] = part;

    int n = clamp_len(raw);
    for (int j = tid; j < n; j += blockDim.x) {
        const int pos = j == tid ? first : ord[j];
        if (pos >= 0 && pos < N) atomicOr(&bitmap[pos >> 5], 1u << (pos & 31));
    }
    if (slot_ring)
        for (int i = tid; i < ring_size; i += blockDim.x) slot_ring[(size_t)seg * ring_size + i] = -1;
    __syncthreads();

    int64_t off = lane < (int)(blockDim.x >> 5) ? red[lane] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
    const int cap = n + decode_cap;
    const bool fits = off + cap <= total_cap_rows;
    if (tid == 0) {
        if (raw != n) raise_status(dev_status, b, PKV_DEV_BAD_LENGTH);
        if (!fits) raise_status(dev_status, b, PKV_DEV_CAPACITY);
        row_offset[seg] = off;
        if (seg == nseg - 1) row_offset[nseg] = off + cap;
        len_out[seg] = fits ? n : 0;
        cap_out[seg] = fits ? cap : 0;
        if (len0) len0[seg] = fits ? n : 0;
        if (gen) gen[seg] = 0;
    }
    if (!fits) n = 0;

    uint32_t word = tid < nwords ? bitmap[tid] : 0;
    int cnt = __popc(word), incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    int dst = incl - cnt;
    if (nwords > 32) {
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        dst += __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0);
    }
    int32_t *out = kept + (size_t)seg * N;
    while (word) {
        int bit = __ffs(word) - 1;
        word &= word - 1;
        if (dst < n) out[dst] = tid * 32 + bit;
        ++dst;
    }
}

// The copy is bound by memory, and by how much of it is in flight: a thread issues all its loads of
// K and V, kGatherHeads of each, before its first store.  A CTA takes kGatherThreads / VEC_PER_HEAD
// rows of kGatherHeads heads at a time, so that a warp's reads follow one head through the rows
// (neighbours where the kept positions are) and its writes stay within one stretch of each row.
// Plan and copy, in us, before (a CTA to a whole row, four loads in flight) and now; the bytes at the
// measured copy rate in brackets.  640-token prompt, 32 layers, 32 heads of 128, budget 0.2: 26.9 ->
// 23.7 (20.5); the same, batch 8: 210 -> 174 (164); in fp32, batch 1: 54.4 -> 48.7 (41.0); 2048
// tokens, 40 layers of 40 heads, batch 2: 269 -> 215 (205); 16384 tokens, 32 layers, batch 2, budget
// 0.1: 337 -> 275 (265); 24 layers of 5 heads, 700 tokens, batch 2: 14.4 -> 9.7 (5.3).  Four loads
// of each instead of eight: 25.0, 180 and 288 at the first, second and fifth; stores with the
// streaming hint: 26.9, 211 and 340; a predicate on each load: 28.6, 179 and 274.
constexpr int kGatherThreads = 128;
constexpr int kGatherHeads = 8;

// grid (segments, row slices, groups of kGatherHeads heads from `group0` on).
template <int VEC_PER_HEAD>
__global__ void __launch_bounds__(kGatherThreads)
gather_rows_kernel(const uint4 *__restrict__ k, const uint4 *__restrict__ v, pkv_strides ks16,
                   pkv_strides vs16, const int32_t *__restrict__ kept,
                   const int32_t *__restrict__ len, const int64_t *__restrict__ row_offset, int L,
                   int N, int H, uint4 *__restrict__ ck, uint4 *__restrict__ cv, int group0)
{
    constexpr int ROWS = kGatherThreads / VEC_PER_HEAD;
    const int seg = blockIdx.x;
    dependent_entry();  // the plan kernel's lists, lengths and offsets are complete
    const int n = len[seg];
    const int b = seg / L, l = seg % L;
    const int64_t off = row_offset[seg];
    const int row_vecs = H * VEC_PER_HEAD;
    const int i = threadIdx.x / VEC_PER_HEAD, c = threadIdx.x % VEC_PER_HEAD;
    const int h0 = (group0 + blockIdx.z) * kGatherHeads, nh = min(H - h0, kGatherHeads);
    const uint4 *kb = k + b * ks16.b + l * ks16.l + h0 * ks16.h + c;
    const uint4 *vb = v + b * vs16.b + l * vs16.l + h0 * vs16.h + c;
    const int32_t *kp = kept + (size_t)seg * N;
    for (int r = blockIdx.y * ROWS + i; r < n; r += gridDim.y * ROWS) {
        const int pos = kp[r];
        const uint4 *kr = kb + pos * ks16.n, *vr = vb + pos * vs16.n;
        const int64_t at = (off + r) * row_vecs + h0 * VEC_PER_HEAD + c;
        if (nh == kGatherHeads) {
            uint4 x[kGatherHeads], y[kGatherHeads];
#pragma unroll
            for (int u = 0; u < kGatherHeads; ++u) {
                x[u] = __ldg(kr + u * ks16.h);
                y[u] = __ldg(vr + u * vs16.h);
            }
#pragma unroll
            for (int u = 0; u < kGatherHeads; ++u) {
                ck[at + u * VEC_PER_HEAD] = x[u];
                cv[at + u * VEC_PER_HEAD] = y[u];
            }
        } else {
#pragma unroll 4
            for (int u = 0; u < nh; ++u) {
                const uint4 x = __ldg(kr + u * ks16.h), y = __ldg(vr + u * vs16.h);
                ck[at + u * VEC_PER_HEAD] = x;
                cv[at + u * VEC_PER_HEAD] = y;
            }
        }
    }
}

cudaError_t launch_compact_plan(const pkv_shape *shape, const int32_t *order, const int32_t *len, pkv_cache *cache,
                                int32_t *kept, int32_t *dev_status, cudaStream_t stream)
{
    const int nseg = shape->batch * shape->layers;
    const bool pruning = cache->evict_distance > 0;
    return launch_dependent(compact_plan_kernel, dim3(nseg), dim3(1024), 0, stream, order, len, nseg, (int)shape->layers,
                            (int)shape->prompt_len, cache->decode_cap, cache->total_cap_rows, cache->row_offset,
                            cache->len, cache->cap, kept, dev_status, pruning ? cache->len0 : nullptr,
                            pruning ? cache->gen : nullptr, pruning ? cache->slot_ring : nullptr,
                            cache->evict_distance + 1);
}

}  // namespace pkv

using namespace pkv;

extern "C" int prefixkv_compact(const pkv_shape *shape, const void *k, pkv_strides ks,
                                const void *v, pkv_strides vs, const int32_t *order,
                                const int32_t *len, pkv_cache *cache, int32_t *kept,
                                int32_t *dev_status, void *ws, size_t ws_bytes, void *cuda_stream)
{
    if (!shape_ok(shape) || !k || !v || !order || !len || !cache || !cache->k || !cache->v ||
        !cache->row_offset || !cache->len || !cache->cap || cache->decode_cap < 0 ||
        cache->total_cap_rows <= 0 || !dev_status)
        return PKV_ERR_INVALID_ARG;
    if (!shape_supported(shape)) return PKV_ERR_UNSUPPORTED;
    const int B = shape->batch, L = shape->layers, N = shape->prompt_len, H = shape->heads;
    const size_t es = esize(shape);
    const int per16 = 16 / (int)es;  // elements per 16-byte vector
    int64_t st[8] = {ks.b, ks.l, ks.h, ks.n, vs.b, vs.l, vs.h, vs.n};
    for (int i = 0; i < 8; ++i)
        if (st[i] < 0 || st[i] % per16 != 0) return PKV_ERR_INVALID_ARG;
    if (!aligned(k, 16) || !aligned(v, 16) || !aligned(cache->k, 16) || !aligned(cache->v, 16))
        return PKV_ERR_INVALID_ARG;
    const int nseg = B * L;
    if (!kept) {
        size_t need = (size_t)nseg * N * sizeof(int32_t);
        if (!ws || !aligned(ws, kWsAlign) || ws_bytes < need) return PKV_ERR_WORKSPACE;
        kept = (int32_t *)ws;
    }
    if (cache->evict_distance < 0) return PKV_ERR_INVALID_ARG;
    const bool pruning = cache->evict_distance > 0;
    if (pruning && (!cache->len0 || !cache->gen || !cache->slot_ring)) return PKV_ERR_INVALID_ARG;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    cudaError_t e = launch_compact_plan(shape, order, len, cache, kept, dev_status, stream);
    if (e != cudaSuccess) {
        set_cuda_error(e, "compact_plan_kernel");
        return PKV_ERR_CUDA;
    }

    pkv_strides k16 = {ks.b / per16, ks.l / per16, ks.h / per16, ks.n / per16};
    pkv_strides v16 = {vs.b / per16, vs.l / per16, vs.h / per16, vs.n / per16};
    const int vph = shape->head_dim / per16;
    // Lengths are known on the device only: up to 128 CTAs per SM, no more than the rows of a whole
    // prompt fill.  A CTA to each tile of rows is slower where most find nothing to copy (4096 tokens,
    // budget 0.1: 105 us against 72), 8 per SM leave the copy idle (16384 tokens: 322 against 275).
    const int groups = (H + kGatherHeads - 1) / kGatherHeads, rows_at_once = kGatherThreads / vph;
    const int slices = std::max(1, std::min((148 * 128 + nseg * groups - 1) / (nseg * groups),
                                            (N + rows_at_once - 1) / rows_at_once));
    constexpr int kMostGroups = 65535;  // of a launch
    for (int group0 = 0; group0 < groups && e == cudaSuccess; group0 += kMostGroups) {
        dim3 grid(nseg, slices, std::min(groups - group0, kMostGroups));
#define PKV_GATHER(V)                                                                                  \
    e = launch_dependent(gather_rows_kernel<V>, grid, dim3(kGatherThreads), 0, stream, (const uint4 *)k, \
                         (const uint4 *)v, k16, v16, (const int32_t *)kept, (const int32_t *)cache->len, \
                         (const int64_t *)cache->row_offset, L, N, H, (uint4 *)cache->k, (uint4 *)cache->v, group0)
        switch (vph) {
        case 8: PKV_GATHER(8); break;
        case 16: PKV_GATHER(16); break;
        case 32: PKV_GATHER(32); break;
        default: return PKV_ERR_UNSUPPORTED;
        }
#undef PKV_GATHER
    }
    if (e != cudaSuccess) {
        set_cuda_error(e, "gather_rows_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}
