// Selection stages: priority sequence + cumulative priority (Sec. 3.2) and the
// binary search for the global ratio p (Sec. 3.3, Eq. 1, Algorithm 1).
//
// All arithmetic that decides an index is integer: the sort key is the fp32 bit
// pattern (monotone for non-negative floats), cumulative sums are 2^-32 fixed
// point in uint64, and only p and the threshold p*total are fp64.
#include <algorithm>

#include "common.cuh"

namespace pkv {

// ---------------------------------------------------------------------------
// One CTA per segment: sort (score desc, position asc) and inclusive scan.
//
// A stable radix sort of the inverted score bits, four passes of eight bits, starting in position
// order: equal scores stay in position order.  Warp w owns 32 * IPT consecutive places (place i * 32 +
// lane of them is item i of a lane), so that going through the items in turn goes through the places in
// order.  A pass ranks an item among its warp's items of the same digit (the warp's count so far comes from
// shared memory), turns the table of the warps' counts into offsets with one scan in the order (digit,
// warp), and moves keys and positions to their places in shared memory.
//
// One item a thread (IPT 1) takes no passes but merges: a warp's 32 by counting, four warps' runs into one, those into the whole.
// An item's place in a merge is its own among its run and the number of each other run's items before it, a binary search.
//
// The passes are bounded by the issue slots of the ranking (some 60 instructions an item and pass) and, after it, by the
// scattered stores; with few items by the barriers of the passes and, as each warp brings a table of 256 counts
// to be scanned, by the number of warps, which is why merging beats them there (the figures are at launch_sort).
// 64 segments of 16384: 204 us with a bitonic network of 64-bit keys, 75 by passes; over clusters of two 57, and 45 with a
// warp's items placed among few keys of the other CTA and the counts in separate banks (128 of 16384 77 / 74, 256 of 8192
// 73 / 65, of 4096 46 / 39, 160 of 3000 34 / 31, 320 of 800 14.7 / 14.2).
// ---------------------------------------------------------------------------
// Fixed-point weight of a sort key (inverted score bits): round-half-even(score * 2^32).  In integers:
// fp64 instructions are few per clock here, and two conversions and a product per key took a good part of
// the scan.
__device__ __forceinline__ uint64_t weight_of_key(uint32_t key, bool &range_bad)
{
    const uint32_t bits = ~key;
    if (bits > 0x7F7FFFFFu) return 0;  // a score already reported as bad
    const int e = (int)(bits >> 23) - 118;  // score * 2^32 = m * 2^e
    const uint32_t m = (bits & 0x7fffffu) | 0x800000u;
    if (e >= 30) {  // 2^53 and above
        range_bad = true;
        return 0;
    }
    if (e >= 0) return (uint64_t)m << e;
    if (e < -24) return 0;  // below one half (subnormal scores, whose m is not this one, too)
    const uint32_t q = m >> -e, rest = m & ((1u << -e) - 1), half = 1u << (-e - 1);
    return q + (rest > half || (rest == half && (q & 1)) ? 1u : 0u);
}

constexpr int kDigits = 256;
constexpr int kSplit = 1024;        // scores of a segment above which a cluster of four may share it; one thread each to there,
constexpr int kMergeCrowded = 768;  // or to here where segments outnumber the SMs

// Shared memory: keys [items], counts [warps][kDigits] (a warp's lanes then meet in a bank by chance only; with
// the warps of a digit side by side they always did), positions [items].
// SPLIT: also the sums [items], and room for the keys of another CTA where the counts are.
static size_t sort_smem_bytes(int threads, int ipt, bool split)
{
    const size_t items = (size_t)threads * ipt;
    return items * (sizeof(uint32_t) + sizeof(uint16_t) + (split ? sizeof(uint64_t) : 0)) +
           std::max((size_t)kDigits * (threads / 32), split ? items : 0) * sizeof(uint32_t);
}

// Loads from another CTA of the cluster (in_cta).
__device__ __forceinline__ uint4 load_there16(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint64_t load_there8(uint32_t a)
{
    uint64_t v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// How many of a sorted run of WIDTH keys come before an item of another run: of equal keys those of an earlier run do.
template <int WIDTH>
__device__ __forceinline__ uint32_t not_after(const uint32_t *run, uint32_t key, bool earlier)
{
    const uint32_t last = earlier ? key : key - 1;
    const uint32_t *at = run;
#pragma unroll
    for (int step = WIDTH / 2; step > 0; step >>= 1) at += at[step - 1] <= last ? step : 0;
    at += *at <= last ? 1 : 0;
    return earlier || key != 0 ? (uint32_t)(at - run) : 0u;
}

// For a warp's sorted items, item i of the lanes after item i - 1: the number of the sorted `keys` that come before each (of equal
// ones EARLIER says).  They are neighbours: a search for the first and the last of them leaves the others few keys to look among
// (searching all 8192 keys for each of eight items a thread: 23400 clocks; so: 6600).
template <int IPT, bool EARLIER>
__device__ __forceinline__ void places_among(const uint32_t *keys, int items, const uint32_t (&key)[IPT], int lane, int (&n)[IPT])
{
    auto before = [](uint32_t x, uint32_t k) { return EARLIER ? x <= k : x < k; };
    const uint32_t first = __shfl_sync(0xffffffffu, key[0], 0), last = __shfl_sync(0xffffffffu, key[IPT - 1], 31);
    const uint32_t end = lane < 16 ? first : last;
    int low = 0;
    for (int width = items; width > 0; width >>= 1) {
        const int half = (width + 1) >> 1;
        low += before(keys[low + half - 1], end) ? half : 0;
    }
    const int high = __shfl_sync(0xffffffffu, low, 31);
    low = __shfl_sync(0xffffffffu, low, 0);
#pragma unroll
    for (int i = 0; i < IPT; ++i) n[i] = low;
    for (int width = high - low; width > 0; width >>= 1) {
        const int half = (width + 1) >> 1;
#pragma unroll
        for (int i = 0; i < IPT; ++i) n[i] += before(keys[n[i] + half - 1], key[i]) ? half : 0;
    }
}

// SPLIT: a cluster takes a segment.  Each of its CTAs sorts and sums a run of consecutive positions; an item's place is then its
// own among them and, for every other CTA, the number of that one's items before it (a binary search over its keys,
// copied next door), and its cumulative sum likewise.
template <int IPT, bool SPLIT>
__global__ void __launch_bounds__(1024)
sort_scan_kernel(const float *__restrict__ scores, int N, int32_t *__restrict__ order,
                 uint64_t *__restrict__ cum, int32_t *__restrict__ seg_flags, int split)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nthr = blockDim.x, nwarp = nthr >> 5;
    uint32_t *skey = reinterpret_cast<uint32_t *>(smem_raw);                 // [nthr * IPT]
    uint32_t *count = skey + nthr * IPT;                                     // [nwarp][kDigits]
    const int items = nthr * IPT;
    uint16_t *spos = reinterpret_cast<uint16_t *>(count + (SPLIT ? max(kDigits * nwarp, items) : kDigits * nwarp));  // [nthr * IPT]
    uint64_t *ssum = reinterpret_cast<uint64_t *>(spos + items);             // (SPLIT) [nthr * IPT]
    __shared__ uint32_t warp_sum[32];
    __shared__ uint64_t warp_tot[32], warp_high[32];
    __shared__ int s_flags;
    __shared__ uint64_t s_total[2];  // (SPLIT) the CTA's sum, and that of high parts

    const int rank = SPLIT ? (int)cluster_rank() : 0, ctas = SPLIT ? split : 1;
    const int seg = SPLIT ? blockIdx.x / split : blockIdx.x, first = SPLIT ? rank * items : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t below = (1u << lane) - 1;
    const int base = warp * 32 * IPT + lane;  // place of the lane's item 0
    const float *src = scores + (size_t)seg * N;
    if (tid == 0) s_flags = 0;
    dependent_entry();  // set up while the kernel before it drained; its results are read from here on

    bool bad = false;
    uint32_t key[IPT];
    uint16_t pos[IPT];
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const int n = first + base + i * 32;
        key[i] = ~0u;  // padding: after every score, those of 0 included (it starts behind them)
        pos[i] = (uint16_t)n;
        if (n < N) {
            uint32_t bits = __float_as_uint(src[n]);
            if (bits == 0x80000000u) bits = 0;   // -0.0 is the same value as +0.0
            if (bits > 0x7F7FFFFFu) bad = true;  // negative, inf or NaN
            key[i] = ~bits;
        }
    }
    if constexpr (IPT == 1) {
        uint32_t place = 0;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            const uint32_t x = __shfl_sync(0xffffffffu, key[0], i);
            place += x < key[0] || (x == key[0] && i < lane);
        }
        skey[warp * 32 + place] = key[0];
        spos[warp * 32 + place] = pos[0];
        __syncthreads();
        if (nwarp > 1) {
            // runs of a warp's items into runs of four warps', these into the whole
            key[0] = skey[tid];
            pos[0] = spos[tid];
            place = lane;
            const int mine = warp & 3, from = warp - mine;
#pragma unroll
            for (int g = 1; g < 4; ++g) {
                const int other = (mine + g) & 3;
                if (from + other < nwarp) place += not_after<32>(skey + (from + other) * 32, key[0], other < mine);
            }
            __syncthreads();
            skey[from * 32 + place] = key[0];
            spos[from * 32 + place] = pos[0];
            __syncthreads();
        }
        if (nwarp > 4) {
            key[0] = skey[tid];
            pos[0] = spos[tid];
            place = tid & 127;
            const int mine = tid >> 7, runs = nwarp >> 2;
#pragma unroll 1
            for (int g = 1; g < runs; ++g) {
                const int other = mine + g < runs ? mine + g : mine + g - runs;
                place += not_after<128>(skey + other * 128, key[0], other < mine);
            }
            __syncthreads();
            skey[place] = key[0];
            spos[place] = pos[0];
            __syncthreads();
        }
        key[0] = skey[tid];
        pos[0] = spos[tid];
    } else {
    // A warp counts a digit at the digit with `turned` turned over.  A thread of the scan goes through four warps' counts of a digit
    // and the next four's; where warps come in eights, all of one digit, the threads of a warp do so in 32 banks (32 warps: four
    // ways into eight without, 2950 clocks a scan, 1800 so).
    const int turn = nwarp & 4 ? 0 : nwarp > 16 ? 8 : 16;
    const uint32_t turned = (warp >> 3) * turn;
    for (int shift = 0; shift < 32; shift += 8) {
        for (int i = tid; i < kDigits * nwarp; i += nthr) count[i] = 0;
        __syncthreads();  // (and every item of the pass before is in registers)
        uint32_t rank[IPT];
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const uint32_t digit = ((key[i] >> shift) & (kDigits - 1)) ^ turned;
            // lanes with this digit: bit by bit, or by match.any where digits are few (sign and exponent); it
            // takes a step per distinct value (16 items a warp: 31000 clocks a pass, 6500 on the last digit;
            // bit by bit 16000 throughout)
            uint32_t same = 0xffffffffu;
            if (shift == 24) {
                same = __match_any_sync(0xffffffffu, digit);
            } else {
#pragma unroll
                for (int bit = 0; bit < 8; ++bit) {
                    const uint32_t ones = __ballot_sync(0xffffffffu, (digit >> bit) & 1);
                    same &= (digit >> bit) & 1 ? ones : ~ones;
                }
            }
            uint32_t *c = count + warp * kDigits + digit;
            const uint32_t before = *c;
            rank[i] = before + __popc(same & below);
            __syncwarp();
            if ((same & below) == 0) *c = before + __popc(same);
            __syncwarp();
        }
        __syncthreads();
        {  // exclusive scan in the order (digit, warp): eight entries a thread (kDigits * nwarp = 8 * nthr)
            const int d0 = tid * 8 / nwarp, w0 = tid * 8 - d0 * nwarp, w1 = w0 + 4 < nwarp ? w0 + 4 : 0;
            uint32_t *four[2] = {count + w0 * kDigits + (d0 ^ (w0 >> 3) * turn),
                                 count + w1 * kDigits + ((w1 ? d0 : d0 + 1) ^ (w1 >> 3) * turn)};
            uint32_t x[8], total = 0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                x[e] = four[e >> 2][(e & 3) * kDigits];
                total += x[e];
            }
            uint32_t incl = total;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += up;
            }
            if (lane == 31) warp_sum[warp] = incl;
            __syncthreads();
            uint32_t run = __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum[lane] : 0u) + incl - total;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                four[e >> 2][(e & 3) * kDigits] = run;
                run += x[e];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const uint32_t at = count[warp * kDigits + (((key[i] >> shift) & (kDigits - 1)) ^ turned)] + rank[i];
            skey[at] = key[i];
            spos[at] = pos[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            key[i] = skey[base + i * 32];
            pos[i] = spos[base + i * 32];
        }
    }
    }

    // Inclusive scan of the fixed-point weights.  Each is below 2^53; sums of their high parts cannot wrap
    // and tell whether the sums themselves did (the values are then unspecified, and reported).
    bool range_bad = false;
    uint64_t local = 0, high = 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const uint64_t w = first + base + i * 32 < N ? weight_of_key(key[i], range_bad) : 0;
        local += w;
        high += w >> 20;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        local += __shfl_xor_sync(0xffffffffu, local, o);
        high += __shfl_xor_sync(0xffffffffu, high, o);
    }
    if (lane == 0) {
        warp_tot[warp] = local;
        warp_high[warp] = high;
    }
    __syncthreads();
    uint64_t run = 0;
    for (int w = 0; w < warp; ++w) run += warp_tot[w];
    if (warp == nwarp - 1) {
        uint64_t h = 0;
        for (int w = 0; w < nwarp; ++w) h += warp_high[w];
        if (SPLIT) {
            s_total[0] = run + local;
            s_total[1] = h;
        }
        if (h >= (1ull << 34) || run + local >= (1ull << 53)) range_bad = true;
    }
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const int j = base + i * 32;
        bool dummy = false;
        uint64_t incl = first + j < N ? weight_of_key(key[i], dummy) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        if (SPLIT) {
            ssum[j] = run + incl;
        } else if (j < N) {
            order[(size_t)seg * N + j] = (int32_t)pos[i];
            if (cum) cum[(size_t)seg * N + j] = run + incl;
        }
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (bad) atomicOr(&s_flags, 1);
    if (range_bad) atomicOr(&s_flags, 2);
    if (SPLIT) {
        cluster_sync();
        int place[IPT];
        uint64_t sum[IPT];
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            place[i] = base + i * 32;
            sum[i] = ssum[place[i]];
        }
        for (int step = 1; step < ctas; ++step) {
            const int other = (rank + step) % ctas;
            const uint32_t there = in_cta(skey, other);
            for (int i = tid; i < items / 4; i += nthr) reinterpret_cast<uint4 *>(count)[i] = load_there16(there + i * 16);
            __syncthreads();
            // (of equal keys those of earlier positions, another CTA's as a whole, come first)
            int n[IPT];
            if (other < rank) places_among<IPT, true>(count, items, key, lane, n);
            else places_among<IPT, false>(count, items, key, lane, n);
            const uint32_t sums = in_cta(ssum, other);
#pragma unroll
            for (int i = 0; i < IPT; ++i) {
                place[i] += n[i];
                if (n[i] > 0) sum[i] += load_there8(sums + (n[i] - 1) * 8);
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < IPT; ++i)
            if (first + base + i * 32 < N) {  // (paddings are a CTA's last)
                order[(size_t)seg * N + place[i]] = (int32_t)pos[i];
                if (cum) cum[(size_t)seg * N + place[i]] = sum[i];
            }
        if (rank == 0 && tid == 0) {
            int flags = 0;
            uint64_t total = 0, high = 0;
            for (int r = 0; r < ctas; ++r) {
                uint32_t f;
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(f) : "r"(in_cta(&s_flags, r)) : "memory");
                flags |= (int)f;
                total += load_there8(in_cta(s_total, r));
                high += load_there8(in_cta(s_total + 1, r));
            }
            if (high >= (1ull << 34) || total >= (1ull << 53)) flags |= 2;
            seg_flags[seg] = flags;
        }
        __syncwarp();
        cluster_sync();  // (the others' shared memory is read no more)
        return;
    }
    __syncthreads();
    // What was found goes to the segment's slot of the length array (bit 0: a bad score, bit 1:
    // the fixed-point range); the kernel that follows turns the flags of a sample's layers into
    // its status word and then writes the lengths over them, so no separate clearing pass runs.
    if (tid == 0) seg_flags[seg] = s_flags;
}

// Status of a sample from the flags the sort kernel left in its layers' length slots.
__device__ __forceinline__ int status_from_flags(int flags)
{
    return (flags & 1) ? (int)PKV_DEV_BAD_SCORE : ((flags & 2) ? (int)PKV_DEV_RANGE : (int)PKV_DEV_OK);
}

// Number of cumulative values below theta, known to lie in [a, b]: a search by quarters, three loads at a time.
__device__ __forceinline__ int count_below(const uint64_t *__restrict__ c, int a, int b, uint64_t theta)
{
    while (a < b) {
        const int i1 = a + ((b - a) >> 2), i2 = a + ((b - a) >> 1), i3 = a + (3 * (b - a) >> 2);
        const uint64_t x1 = c[i1], x2 = c[i2], x3 = c[i3];
        if (x2 < theta) {
            a = x3 < theta ? i3 + 1 : i2 + 1;
            b = x3 < theta ? b : i3;
        } else {
            b = x1 < theta ? i2 : i1;
            a = x1 < theta ? i1 + 1 : a;
        }
    }
    return a;
}
// The same for two rows side by side: the numbers end up in a.
template <int M>
__device__ __forceinline__ void count_below(const uint64_t *__restrict__ c0, const uint64_t *__restrict__ c1, int (&a)[M],
                                            int (&b)[M], const uint64_t (&theta)[M])
{
    while (a[0] < b[0] || a[M - 1] < b[M - 1]) {
        uint64_t x[M][3];
        int i[M][3];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int from = a[m] < b[m] ? a[m] : 0, width = max(b[m] - a[m], 0);  // (a row done: its first value)
            const uint64_t *c = m ? c1 : c0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                i[m][j] = from + ((j + 1) * width >> 2);
                x[m][j] = c[i[m][j]];
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            if (a[m] >= b[m]) continue;
            if (x[m][1] < theta[m]) {
                a[m] = x[m][2] < theta[m] ? i[m][2] + 1 : i[m][1] + 1;
                b[m] = x[m][2] < theta[m] ? b[m] : i[m][2];
            } else {
                b[m] = x[m][0] < theta[m] ? i[m][1] : i[m][0];
                a[m] = x[m][0] < theta[m] ? i[m][0] + 1 : a[m];
            }
        }
    }
}

// Length rule of Sec. 3.3 (a layer keeps one row more than there are cumulative values below p * total, at most N) and the
// bisection on p that makes the lengths meet the budget.  One CTA per sample, warp per layer.
//
// A midpoint by itself is a chain of latencies -- a load or two, the sum over the layers, a barrier -- of some 1000
// clocks.  So the tree of the next five bisections is evaluated at once, a lane to each of its 31 midpoints (the values that the
// same additions and halvings would lead to), and the way through it is found by all lanes at once from bit masks of what each
// midpoint came to: a round costs little more than a midpoint did, the first one apart, whose searches cover whole rows; later
// ones lie between the counts at both ends of the interval.  What a warp's layers need is kept in registers for kHoist of them,
// and they are searched two at a time, so that their loads are in flight together.  kHoist is the least that covers the layers of
// a sample: code for layers that are not there costs as much as a layer's (32 layers of 640 scores with four hoisted: 16.2 us).
// Sort and search of one sample, in us, sorting alone in brackets; five levels walked one by one in fp64, four layers hoisted and
// searched one after the other / as here: 32 layers of 640 scores 19.3 / 13.1 (7.9), of 128 12.2 / 7.0 (3.5), of 4096 39.1 / 32.3
// (23.8); 40 of 640 21.8 / 14.8, eight samples 29.5 / 21.4 (13.6); 64 of 640 24.1 / 17.1; 96 27.5 / 22.8; 128 37.4 / 28.1; 200 of
// 300 46.0 / 32.0 (with four hoisted 42.8); 1000 of 2000 478 / 389 (beyond 256 layers a lane searches whole rows).  A midpoint at
// a time cost some 6 us more than the former at 32 layers of 640.
constexpr int kTreeLevels = 5;
// After so many rounds the ends are multiples of 2^-50: every midpoint until then is a sum without rounding, found at once.
constexpr int kExactRounds = 50 / kTreeLevels;
constexpr int kMaxLayers = 5120;  // of a sample (sums of lengths are 32 bits wide, which would do for 2^17 layers)
template <int kHoist>
__global__ void __launch_bounds__(1024)
search_kernel(const uint64_t *__restrict__ cum, const int64_t *__restrict__ budget_rows, int L,
              int N, double tol, int max_iters, int64_t slack, int64_t slack_over, int32_t *__restrict__ len,
              double *__restrict__ p_out, int32_t *__restrict__ iters_out, int32_t *dev_status)
{
    __shared__ int s_flags;
    __shared__ int s_sum[3][32];  // total length at every midpoint of the tree; buffers in turn
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const uint64_t *cb = cum + (size_t)b * L * N;
    if (threadIdx.x < 96) s_sum[threadIdx.x / 32][lane] = 0;
    if (threadIdx.x == 0) s_flags = 0;
    const int depth = 31 - __clz(lane | 1);  // of the lane's node, whose interval is `part` of the tree's,
    const double part = ldexp(1.0, -depth);  // and its midpoint at `place` of it (lane 0: as lane 1)
    const double place = (2 * (lane & ((1 << depth) - 1)) + 1) * part * 0.5;
    uint32_t above = 0, upper = 0;  // the nodes above the lane's, and those of them in whose upper half it is
    for (int i = 0; i < depth; ++i) {
        above |= 1u << (lane >> (i + 1));
        upper |= (uint32_t)(lane >> i & 1) << (lane >> (i + 1));
    }
    __syncthreads();
    dependent_entry();  // the sort kernel's sums and flags are complete
    // What a layer's searches need, for the first kHoist layers of the warp: its total, the counts at both ends of the interval,
    // and a pivot per lane, c[(lane + 1) * chunk - 1] (or ~0 past the end).
    constexpr int M = kHoist > 1 ? 2 : 1;  // rows searched side by side
    const int chunk = (N + 31) >> 5;
    double tot[kHoist];
    uint64_t pivot[kHoist];
    int lo[kHoist], hi[kHoist], at[kHoist];
#pragma unroll
    for (int k = 0; k < kHoist; ++k) {
        const int l = warp + k * nwarp;
        tot[k] = 0.0;
        pivot[k] = ~0ull;
        lo[k] = at[k] = 0;
        hi[k] = N;
        if (l < L) {
            const uint64_t *c = cb + (size_t)l * N;
            const int idx = (lane + 1) * chunk - 1;
            tot[k] = (double)c[N - 1];
            if (idx < N) pivot[k] = c[idx];
        }
    }
    const int64_t budget = budget_rows[b];
    {
        int flags = 0;
        for (int l = threadIdx.x; l < L; l += blockDim.x) flags |= len[(size_t)b * L + l];
        if (flags) atomicOr(&s_flags, flags);  // (looked at after a round's barrier, as the slots are written after one)
    }

    auto threshold = [](double p, double total) { return __double2ull_ru(__dmul_rn(p, total)); };
    auto length_of = [&](int count) { return count + 1 > N ? N : count + 1; };

    double p_final = 0.0;
    int iters = 0, taken = -1;  // taken: the midpoint, of the last tree, that is p_final
    if (budget < (int64_t)L || (int64_t)L * (int64_t)N <= budget) {
        if (budget >= (int64_t)L) p_final = 1.0;
        __syncthreads();
    } else {
        double p1 = 0.0, p2 = 1.0;
        bool done = false;
        for (int round = 0; !done; ++round) {
            // the lane's midpoint: node `lane` of the tree (root 1; the upper half of a node's interval is its odd child)
            double p;
            bool stop;  // no bisection of the node's interval: its ends are neighbours or within the tolerance
            if (round < kExactRounds) {
                const double width = p2 - p1;
                p = fma(width, place, p1);
                stop = width * part <= tol;
            } else {
                double a1 = p1, a2 = p2;
                p = (p1 + p2) * 0.5;
                for (int bit = depth - 1; bit >= 0; --bit) {
                    if (lane >> bit & 1) a1 = p;
                    else a2 = p;
                    p = (a1 + a2) * 0.5;
                }
                stop = p == a1 || p == a2 || a2 - a1 <= tol;
            }
            const uint32_t stops = __ballot_sync(0xffffffffu, stop || depth >= max_iters - iters);
            int total = 0;
#pragma unroll
            for (int k = 0; k < kHoist; k += M) {
                const int l = warp + k * nwarp;
                if (l >= L) continue;
                uint64_t theta[M];
                int x[M], y[M];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    theta[m] = threshold(p, tot[k + m]);
                    x[m] = lo[k + m];
                    y[m] = hi[k + m];
                    if (m == 1 && l + nwarp >= L) {
                        x[m] = y[m] = 0;
                    } else if (y[m] - x[m] > chunk) {  // (the first round: which 32nd of the row)
                        int n = 0;
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            n += __shfl_sync(0xffffffffu, pivot[k + m], n + step - 1) < theta[m] ? step : 0;
                        n += __shfl_sync(0xffffffffu, pivot[k + m], 31) < theta[m] ? n == 31 : 0;
                        x[m] = max(x[m], n * chunk);
                        y[m] = min(y[m], (n + 1) * chunk - 1);
                    }
                }
                const uint64_t *row = cb + (size_t)l * N;
                if (M == 1 || l + nwarp >= L) {
                    at[k] = p < 1.0 ? count_below(row, x[0], y[0], theta[0]) : N;
                    total += length_of(at[k]);
                } else {
                    count_below(row, row + (size_t)nwarp * N, x, y, theta);
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        at[k + m] = p < 1.0 ? x[m] : N;
                        total += length_of(at[k + m]);
                    }
                }
            }
            for (int l = warp + kHoist * nwarp; M > 1 && l < L; l += M * nwarp) {
                const uint64_t *row[2] = {cb + (size_t)l * N, cb + (size_t)(l + nwarp < L ? l + nwarp : l) * N};
                int x[M], y[M];
                uint64_t theta[M];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    x[m] = 0;
                    y[m] = l + m * nwarp < L ? N : 0;
                    theta[m] = threshold(p, (double)row[m][N - 1]);
                }
                count_below(row[0], row[1], x, y, theta);
#pragma unroll
                for (int m = 0; m < M; ++m)
                    if (l + m * nwarp < L) total += length_of(p < 1.0 ? x[m] : N);
            }
            int *sums = s_sum[round % 3];
            atomicAdd(sums + lane, total);
            if (warp == 0) s_sum[(round + 1) % 3][lane] = 0;  // (read two rounds ago, before the last barrier)
            __syncthreads();
            const int64_t delta = (int64_t)sums[lane] - budget;
            const uint32_t low = __ballot_sync(0xffffffffu, delta < 0);
            const uint32_t met = __ballot_sync(0xffffffffu, delta >= -slack && delta <= slack_over);  // (Sec. 3.3)
            // the nodes that the bisection goes through, the interval's new ends among them, and the one where it ends
            const uint32_t path =
                __ballot_sync(0xffffffffu, lane > 0 && ((low ^ upper) & above) == 0 && ((stops | met) & above) == 0);
            const uint32_t met_at = path & met & ~stops, went = path & ~stops & ~met;
            const int at1 = 31 - __clz(went & low), at2 = 31 - __clz(went & ~low);  // (-1: none)
            iters += __popc(path & ~stops);
            taken = 31 - __clz(met_at);
            done = (path & (stops | met)) != 0;
            const double q1 = __shfl_sync(0xffffffffu, p, at1 & 31), q2 = __shfl_sync(0xffffffffu, p, at2 & 31);
            if (at1 >= 0) p1 = q1;
            if (at2 >= 0) p2 = q2;
            if (done) p_final = taken >= 0 ? __shfl_sync(0xffffffffu, p, taken) : p1;
#pragma unroll
            for (int k = 0; k < kHoist; ++k) {
                const int n1 = __shfl_sync(0xffffffffu, at[k], at1 & 31), n2 = __shfl_sync(0xffffffffu, at[k], at2 & 31);
                if (at1 >= 0) lo[k] = n1;
                if (at2 >= 0) hi[k] = n2;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kHoist; ++k) {
        const int l = warp + k * nwarp;
        const int count = __shfl_sync(0xffffffffu, at[k], taken & 31);
        if (l < L && lane == 0) len[(size_t)b * L + l] = p_final >= 1.0 ? N : length_of(taken >= 0 ? count : lo[k]);
    }
    for (int l = warp + kHoist * nwarp; l < L; l += nwarp) {
        const uint64_t *c = cb + (size_t)l * N;
        const int count = p_final < 1.0 ? count_below(c, 0, N, threshold(p_final, (double)c[N - 1])) : N;
        if (lane == 0) len[(size_t)b * L + l] = length_of(count);
    }
    if (threadIdx.x == 0) {
        dev_status[b] = status_from_flags(s_flags);  // overwrites: this call's status starts here
        if (budget < (int64_t)L) raise_status(dev_status, b, PKV_DEV_BUDGET_TOO_SMALL);
        p_out[b] = p_final;
        iters_out[b] = iters;
    }
}

// One CTA per sample: the caller's lengths, checked, and the sample's status word.
__global__ void __launch_bounds__(256)
take_lengths_kernel(const int32_t *__restrict__ len_in, int per_sample, int L, int N,
                    int32_t *__restrict__ len, int32_t *dev_status)
{
    const int b = blockIdx.x;
    dependent_entry();  // the sort kernel's flags are complete
    int flags = 0, bad = 0;
    for (int l = threadIdx.x; l < L; l += blockDim.x) {
        flags |= len[(size_t)b * L + l];
        int v = per_sample ? len_in[(size_t)b * L + l] : len_in[l];
        if (v < 1 || v > N) {
            bad = 1;
            v = v < 1 ? 1 : N;
        }
        len[(size_t)b * L + l] = v;
    }
    flags = (__syncthreads_or(flags & 1) ? 1 : 0) | (__syncthreads_or(flags & 2) ? 2 : 0);  // predicates: one per bit
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        const int st = status_from_flags(flags);
        dev_status[b] = st != PKV_DEV_OK ? st : (bad ? (int)PKV_DEV_BAD_LENGTH : (int)PKV_DEV_OK);
    }
}

template <int IPT, bool SPLIT = false>
static int launch_sort_items(const pkv_shape *s, const float *scores, int32_t *order, uint64_t *cum,
                             int32_t *seg_flags, cudaStream_t st, int split = 1)
{
    const int N = s->prompt_len, share = (N + split - 1) / split;
    int threads = ((share + IPT - 1) / IPT + 31) / 32 * 32;
    if (threads > 128) threads = (threads + 127) / 128 * 128;  // (whole runs; the passes' scan goes by four warps)
    const size_t smem = sort_smem_bytes(threads, IPT, SPLIT);
    // (for every size: the default limit of 48 KiB is for the kernel's static variables and these together)
    static bool attr_done[64] = {};
    int rc = ensure_dynamic_smem((const void *)sort_scan_kernel<IPT, SPLIT>, (int)sort_smem_bytes(1024, IPT, SPLIT), attr_done);
    if (rc != PKV_OK) return rc;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)split;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(s->batch * s->layers * split));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = SPLIT ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, sort_scan_kernel<IPT, SPLIT>, scores, N, order, cum, seg_flags, split);
    if (e != cudaSuccess) {
        set_cuda_error(e, "sort_scan_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

// Clusters of four of the sort kernel that run at once with an SM to each CTA (a block of 1024 threads fills one).  There
// are fewer than SMs / 4: a cluster's SMs are of one GPC, and most of these have no multiple of four.
static int clusters_of_four()
{
    static int count[64] = {};  // plus one
    static bool attr_done[64] = {};
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (count[dev] > 0) return count[dev] - 1;
    const size_t smem = sort_smem_bytes(1024, 4, true);
    if (ensure_dynamic_smem((const void *)sort_scan_kernel<4, true>, (int)smem, attr_done) != PKV_OK) return 0;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 4;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(4);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, sort_scan_kernel<4, true>, &cfg) != cudaSuccess) {
        cudaGetLastError();  // (it only leaves segments whole)
        n = 0;
    }
    count[dev] = n + 1;
    return n;
}

// One item a thread, merged, or radix passes; whole segments, or clusters of two or four to a segment.  Sort alone and a short
// kernel behind it, in us, one item a thread / radix passes over whole segments, split as taken here in brackets:
//   32 segments of 256 scores 4.2 / 4.7 (places counted against all), 300 4.6 / 6.9, 640 5.6 / 7.9 (one a thread over clusters of
//   two 6.5), 768 6.4 / 8.3, 1024 8.2 / 9.0 (7.6); 512 of 256 6.7 / 9.5, 640 14.6 / 17.8, 768 18.1 / 21.2, 1024 24.9 / 18.7;
//   of 1024 148 8.5 / 9.3, 160 13.7 / 11.9.
// Merging takes the square of the runs, so the line falls to 768 where a block of 1024 threads is more than an SM's first.
//   Clusters of two: 64 of 2048 12.1 with one item a thread (whole 13.0), of 3000 15.6 with four (18.0), 4096 18.2 (24.0), 5000 19.1
//   (24.1), 8192 25.7 (33.5); with eight 25.2 there, 44.5 for 64 of 16384.
//   Clusters of four, while all run at once (33 of them on a B200): 32 of 1536 9.3 (two: 9.5), 2048 10.6 (11.7), 3000 13.1 (15.6),
//   4096 16.4 (18.2), 4500 16.2 (18.8), 8192 20.2 (25.2), 16384 34.7 (44.7); beyond that 40 of 2048 13.9 (11.9), of 16384 65.7 (44.6).
static int launch_sort(const pkv_shape *s, const float *scores, int32_t *order, uint64_t *cum,
                       int32_t *seg_flags, cudaStream_t st)
{
    const int N = s->prompt_len, sms = sm_count();
    const int64_t segments = (int64_t)s->batch * s->layers;
    if (N > kSplit && segments <= clusters_of_four())
        return N <= 4096 ? launch_sort_items<1, true>(s, scores, order, cum, seg_flags, st, 4)
                         : launch_sort_items<4, true>(s, scores, order, cum, seg_flags, st, 4);
    if (N > kMergeCrowded && 2 * segments <= sms)
        return N <= 2048   ? launch_sort_items<1, true>(s, scores, order, cum, seg_flags, st, 2)
               : N <= 8192 ? launch_sort_items<4, true>(s, scores, order, cum, seg_flags, st, 2)
                           : launch_sort_items<8, true>(s, scores, order, cum, seg_flags, st, 2);
    if (N <= (segments <= sms ? kSplit : kMergeCrowded)) return launch_sort_items<1>(s, scores, order, cum, seg_flags, st);
    if (N <= 4096) return launch_sort_items<4>(s, scores, order, cum, seg_flags, st);
    if (N <= 8192) return launch_sort_items<8>(s, scores, order, cum, seg_flags, st);
    return launch_sort_items<16>(s, scores, order, cum, seg_flags, st);
}

}  // namespace pkv

using namespace pkv;

extern "C" int prefixkv_search(const pkv_shape *shape, const float *scores,
                               const int64_t *budget_rows, double tol, int32_t max_iters,
                               int64_t slack_rows, int64_t slack_over_rows, int32_t *order, uint64_t *cum,
                               int32_t *len, double *p_out, int32_t *iters_out, int32_t *dev_status,
                               void *ws, size_t ws_bytes, void *cuda_stream)
{
    (void)ws; (void)ws_bytes;
    if (!shape_ok(shape) || !scores || !budget_rows || !order || !cum || !len || !p_out ||
        !iters_out || !dev_status || !(tol >= 0.0) || max_iters < 0 || slack_rows < 0 || slack_over_rows < 0)
        return PKV_ERR_INVALID_ARG;
    if (!shape_supported(shape)) return PKV_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int B = shape->batch, L = shape->layers, N = shape->prompt_len;
    if (L > kMaxLayers) return PKV_ERR_UNSUPPORTED;
    int rc = launch_sort(shape, scores, order, cum, len, st);
    if (rc != PKV_OK) return rc;
    cudaError_t e = launch_dependent(L <= 32 ? search_kernel<1> : L <= 64 ? search_kernel<2> : L <= 128 ? search_kernel<4> : search_kernel<8>, dim3(B), dim3(1024), 0, st,
                                     (const uint64_t *)cum, budget_rows, L, N, tol, (int)max_iters, slack_rows, slack_over_rows, len,
                                     p_out, iters_out, dev_status);
    if (e != cudaSuccess) {
        set_cuda_error(e, "search_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}

extern "C" int prefixkv_apply_lengths(const pkv_shape *shape, const float *scores,
                                      const int32_t *len_in, int32_t per_sample, int32_t *order,
                                      uint64_t *cum, int32_t *len, int32_t *dev_status, void *ws,
                                      size_t ws_bytes, void *cuda_stream)
{
    (void)ws; (void)ws_bytes;
    if (!shape_ok(shape) || !scores || !len_in || !order || !len || !dev_status)
        return PKV_ERR_INVALID_ARG;
    if (!shape_supported(shape)) return PKV_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int B = shape->batch, L = shape->layers, N = shape->prompt_len;
    if (len_in == len) return PKV_ERR_INVALID_ARG;  // (the output slots carry the sort's flags in between)
    int rc = launch_sort(shape, scores, order, cum, len, st);
    if (rc != PKV_OK) return rc;
    cudaError_t e = launch_dependent(take_lengths_kernel, dim3(B), dim3(256), 0, st, len_in, (int)per_sample, L, N, len,
                                     dev_status);
    if (e != cudaSuccess) {
        set_cuda_error(e, "take_lengths_kernel");
        return PKV_ERR_CUDA;
    }
    return PKV_OK;
}
