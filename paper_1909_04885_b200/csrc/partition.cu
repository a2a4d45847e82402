// Partition of the coordinates into K random blocks, and the per-round visiting orders.
// Integer-only: the result is a pure function of (n, K, seed) and (seed, round, epoch).
//
// Both need an order by a 64-bit hash of the id. The hashes are uniform, so their leading bits already say where an
// element lands: the elements are counted and scattered into buckets of about 512 (by the leading bits of the key), and
// a CTA puts a bucket into full-key order in shared memory, again by counting (sub-buckets of about one element each,
// then a comparison with the few that share it). A radix sort of (key, id) pairs passes over 12 bytes per element five
// times and more; this passes over the 4-byte ids four times (the keys are recomputed: a dozen integer instructions),
// in four launches instead of 27 (a step of 1 M rows, K = 16: 6.49 -> 6.31 ms; its orders 245 -> about 50 us).
#include <cstdio>
#include <mutex>

#include "chicle_internal.cuh"

namespace chicle {

constexpr int kBucketMean = 512; // elements per bucket on average; a CTA's arrays hold twice as many

namespace {

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// How positions in key order map to partitions: ascending offsets, or equal blocks (the first `extra` one longer).
struct Cuts {
    const int64_t *off; // K + 1 offsets on the device, or nullptr: equal blocks
    int32_t K;
    uint32_t base, extra;
};
__device__ __forceinline__ int32_t partition_of(const Cuts &c, uint32_t pos)
{
    if (!c.off) {
        const uint32_t thr = c.extra * (c.base + 1u);
        return (int32_t)(pos < thr ? pos / (c.base + 1u) : c.extra + (pos - thr) / c.base);
    }
    int32_t lo = 0, hi = c.K; // off[lo] <= pos < off[hi]
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (c.off[mid] <= (int64_t)pos) lo = mid;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ uint32_t start_of(const Cuts &c, int32_t k)
{
    if (c.off) return (uint32_t)c.off[k];
    return (uint32_t)k * c.base + ((uint32_t)k < c.extra ? (uint32_t)k : c.extra);
}

// ------------------------------------------------------------------------------------------------ buckets
// Segments that are ordered on their own: the partitions (visiting orders), or all ids as one (the partition itself).
struct Segments {
    const int64_t *off;   // first element of each segment (K + 1), nullptr: one segment of n
    const int64_t *bbase; // first bucket of each segment (K + 1)
    int32_t K;
    int64_t n;
    uint32_t nb;          // buckets of the one segment
    __device__ __forceinline__ int64_t first(int k) const { return off ? off[k] : 0; }
    __device__ __forceinline__ int64_t last(int k) const { return off ? off[k + 1] : n; }
    __device__ __forceinline__ uint32_t bucket0(int k) const { return off ? (uint32_t)bbase[k] : 0u; }
    __device__ __forceinline__ uint32_t buckets(int k) const { return off ? (uint32_t)(bbase[k + 1] - bbase[k]) : nb; }
};

constexpr int kCountThreads = 256;
constexpr int kCountItems = 8;
constexpr int kCountTile = kCountThreads * kCountItems;

// The elements a CTA of the counting and scattering kernels takes: f(segment, first element, step, end). Tile t, t + tiles, .. of
// one segment; or (tiles = 0) an equal share of all segments one after the other, counted in buckets. Segments of about the same
// size take the first way. Where one is much longer than what its tiles' CTAs get through meanwhile, the second (see tiles_for).
template <class F> __device__ __forceinline__ void for_my_elements(const Segments &S, int tiles, F f)
{
    if (tiles > 0) {
        const int k = (int)(blockIdx.x / tiles), t = (int)(blockIdx.x % tiles);
        f(k, S.first(k) + (int64_t)t * kCountTile, (int64_t)tiles * kCountTile, S.last(k));
        return;
    }
    const int64_t all = S.bbase[S.K], end = all * ((int64_t)blockIdx.x + 1) / gridDim.x;
    int64_t at = all * blockIdx.x / gridDim.x;
    int lo = 0, hi = S.K; // bbase[lo] <= at < bbase[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (S.bbase[mid] <= at) lo = mid;
        else hi = mid;
    }
    for (int k = lo; at < end; ++k) {
        const int64_t b0 = S.bbase[k], b1 = S.bbase[k + 1], stop = b1 < end ? b1 : end, first = S.first(k), last = S.last(k);
        const int64_t until = first + (stop - b0) * kBucketMean;
        f(k, first + (at - b0) * kBucketMean, (int64_t)kCountTile, until < last ? until : last);
        at = stop;
    }
}

// cursor[bucket] += its elements (zero on entry). LOCAL: a CTA counts in shared memory first and adds what it has of each
// bucket; for segments of at most kLocalBuckets buckets whose CTAs have several elements of each (see launch_count): 1 M
// coordinates in 16 segments took 31 us, a global atomic per coordinate.
constexpr uint32_t kLocalBuckets = 2048;
template <bool LOCAL>
__global__ void __launch_bounds__(kCountThreads)
k_bucket_count(const Segments S, int tiles, const int32_t *__restrict__ ids, uint64_t ab, uint32_t *__restrict__ cursor)
{
    __shared__ uint32_t mine[LOCAL ? kLocalBuckets : 1];
    for_my_elements(S, tiles, [&](int k, int64_t from, int64_t step, int64_t hi) {
        if (from >= hi) return;
        const uint32_t nb = S.buckets(k);
        uint32_t *cur = cursor + S.bucket0(k);
        if (LOCAL) {
            for (uint32_t b = threadIdx.x; b < nb; b += kCountThreads) mine[b] = 0u;
            __syncthreads();
        }
        for (int64_t i0 = from; i0 < hi; i0 += step) {
            uint32_t b[kCountItems];
#pragma unroll
            for (int u = 0; u < kCountItems; ++u) {
                const int64_t i = i0 + u * kCountThreads + threadIdx.x;
                const uint32_t id = i < hi ? (ids ? (uint32_t)ids[i] : (uint32_t)i) : 0u;
                b[u] = __umulhi((uint32_t)(mix64(ab ^ (uint64_t)id) >> 32), nb);
            }
#pragma unroll
            for (int u = 0; u < kCountItems; ++u)
                if (i0 + u * kCountThreads + threadIdx.x < hi) atomicAdd((LOCAL ? mine : cur) + b[u], 1u);
        }
        if (LOCAL) {
            __syncthreads();
            for (uint32_t b = threadIdx.x; b < nb; b += kCountThreads)
                if (mine[b]) atomicAdd(cur + b, mine[b]);
        }
    });
}

// A CTA per segment. start[bucket] = first position of the bucket, cursor[bucket] the same (the scatter's running place);
// nbm[bucket] = buckets of its segment, or 0 if nobody needs the bucket in order: it begins behind the steps that the
// round takes (`need`: per segment, or need_all for all, less the epochs before), or (cuts given) it lies inside one
// partition, whose number goes to bowner.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 8;
__global__ void __launch_bounds__(kScanThreads)
k_bucket_scan(const Segments S, uint32_t *__restrict__ start, uint32_t *__restrict__ cursor, uint32_t *__restrict__ nbm,
              int32_t *__restrict__ bowner, const Cuts cuts, const int64_t *__restrict__ need, int64_t need_all, int64_t epoch)
{
    __shared__ uint32_t warp_tot[kScanThreads / 32];
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nb = S.buckets(k), b0 = S.bucket0(k);
    const int64_t lo = S.first(k), nk = S.last(k) - lo;
    int64_t want = need ? need[k] : (need_all == 0 ? nk : need_all - epoch * nk);
    want = want < nk ? want : nk;
    uint32_t carry = (uint32_t)lo;
    for (uint32_t base = 0; base < nb; base += kScanThreads * kScanPer) {
        uint32_t x[kScanPer], sum = 0;
        const uint32_t at = base + (uint32_t)tid * kScanPer;
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) {
            x[j] = at + j < nb ? cursor[b0 + at + j] : 0u;
            sum += x[j];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            uint32_t w = warp_tot[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_tot[lane] = w;
        }
        __syncthreads();
        uint32_t pos = carry + (warp ? warp_tot[warp - 1] : 0u) + incl - sum;
        carry += warp_tot[kScanThreads / 32 - 1];
#pragma unroll
        for (int j = 0; j < kScanPer; ++j) {
            if (at + j < nb) {
                const uint32_t b = b0 + at + j;
                start[b] = pos;
                cursor[b] = pos;
                uint32_t m = nb;
                if (bowner) {
                    int32_t own = -1;
                    if (x[j] == 0u) own = 0;
                    else {
                        own = partition_of(cuts, pos);
                        if (pos + x[j] > start_of(cuts, own + 1)) own = -1; // a cut lies inside the bucket
                    }
                    bowner[b] = own;
                    if (own >= 0) m = 0u;
                } else if ((int64_t)pos - lo >= want) m = 0u;
                nbm[b] = m;
            }
            pos += x[j];
        }
        __syncthreads();
    }
    if (k == S.K - 1 && tid == 0) start[b0 + nb] = (uint32_t)(lo + nk);
}

// Elements of the buckets that are needed in order go to out, bucket after bucket (any order inside a bucket). With
// `owner`: the others' partition is their bucket's.
__global__ void __launch_bounds__(kCountThreads)
k_bucket_scatter(const Segments S, int tiles, const int32_t *__restrict__ ids, uint64_t ab, uint32_t *__restrict__ cursor,
                 const uint32_t *__restrict__ nbm, const int32_t *__restrict__ bowner, int32_t *__restrict__ owner,
                 int32_t *__restrict__ out)
{
    for_my_elements(S, tiles, [&](int k, int64_t from, int64_t step, int64_t hi) {
        const uint32_t nb = S.buckets(k), b0 = S.bucket0(k);
        for (int64_t i0 = from; i0 < hi; i0 += step) {
            uint32_t id[kCountItems], b[kCountItems], m[kCountItems];
#pragma unroll
            for (int u = 0; u < kCountItems; ++u) {
                const int64_t i = i0 + u * kCountThreads + threadIdx.x;
                id[u] = i < hi ? (ids ? (uint32_t)ids[i] : (uint32_t)i) : 0u;
                b[u] = b0 + __umulhi((uint32_t)(mix64(ab ^ (uint64_t)id[u]) >> 32), nb);
                m[u] = i < hi ? nbm[b[u]] : 0u;
            }
            if (owner) {
#pragma unroll
                for (int u = 0; u < kCountItems; ++u) {
                    const int64_t i = i0 + u * kCountThreads + threadIdx.x;
                    if (i < hi && m[u] == 0u) owner[i] = bowner[b[u]]; // (one segment of all ids: i is the id)
                }
            }
#pragma unroll
            for (int u = 0; u < kCountItems; ++u)
                if (m[u]) m[u] = atomicAdd(cursor + b[u], 1u) + 1u;
#pragma unroll
            for (int u = 0; u < kCountItems; ++u)
                if (m[u]) out[m[u] - 1u] = (int32_t)id[u];
        }
    });
}

template <int CAP> struct OrderShared {
    unsigned long long key[CAP];
    int32_t id[CAP];
    uint32_t sub[CAP / 2 + 1]; // elements per sub-bucket, then where each starts
    uint32_t warp_tot[32];
};

// A CTA per bucket: its elements (src[start .. next start)) in full-key order to dst, or (owner given) the partition of
// each one's position to owner[id]. Sub-buckets by the key bits behind the bucket's (one element on average at the
// usual fill), then a comparison with those that share the sub-bucket: the order is exact whatever the order of arrival.
// start == nullptr: the segments themselves are the buckets (all of them fit).
template <int CAP, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_bucket_order(const int32_t *__restrict__ src, const uint32_t *__restrict__ start, const uint32_t *__restrict__ nbm,
               const int64_t *__restrict__ seg_off, uint64_t ab, uint32_t *__restrict__ cursor, int32_t *__restrict__ dst,
               const Cuts cuts, int32_t *__restrict__ owner)
{
    extern __shared__ __align__(16) unsigned char order_smem[];
    OrderShared<CAP> &sh = *reinterpret_cast<OrderShared<CAP> *>(order_smem);
    constexpr int SUB = CAP / 2;
    constexpr int PER = CAP / THREADS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = blockIdx.x;
    const uint32_t lo = start ? start[b] : (uint32_t)seg_off[b];
    const uint32_t hi = start ? start[b + 1] : (uint32_t)seg_off[b + 1];
    const uint32_t nb = start ? nbm[b] : 1u;
    if (cursor && tid == 0) cursor[b] = 0u; // ready for the next count
    if (nb == 0u || hi == lo) return;
    const uint32_t m = hi - lo;
    if (m > (uint32_t)CAP) {
        // far more elements than hashes ever put here: ranked by comparison with all of the bucket
        for (uint32_t i = tid; i < m; i += THREADS) {
            const int32_t id = src[lo + i];
            const uint64_t key = mix64(ab ^ (uint64_t)(uint32_t)id);
            uint32_t rank = 0;
            for (uint32_t j = 0; j < m; ++j) rank += mix64(ab ^ (uint64_t)(uint32_t)src[lo + j]) < key ? 1u : 0u;
            if (owner) owner[id] = partition_of(cuts, lo + rank);
            else dst[lo + rank] = id;
        }
        return;
    }
    for (int i = tid; i < SUB; i += THREADS) sh.sub[i] = 0u;
    __syncthreads();
    uint64_t key[PER];
    int32_t id[PER];
    uint32_t sub[PER], arrived[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const uint32_t i = (uint32_t)(u * THREADS + tid);
        id[u] = i < m ? src[lo + i] : 0;
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const uint32_t i = (uint32_t)(u * THREADS + tid);
        key[u] = mix64(ab ^ (uint64_t)(uint32_t)id[u]);
        const uint32_t rest = (uint32_t)(key[u] >> 32) * nb; // the fraction behind the bucket number, monotone in the key
        sub[u] = __umulhi(rest, (uint32_t)SUB);
        arrived[u] = 0u;
        if (i < m) arrived[u] = atomicAdd(&sh.sub[sub[u]], 1u);
    }
    __syncthreads();
    {
        // exclusive scan of the SUB counters, SUB / THREADS (at least one) per thread
        constexpr int CPT = SUB / THREADS > 0 ? SUB / THREADS : 1;
        uint32_t x[CPT], sum = 0;
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int at = tid * CPT + j;
            x[j] = at < SUB ? sh.sub[at] : 0u;
            sum += x[j];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sh.warp_tot[warp] = incl;
        __syncthreads();
        uint32_t pos = incl - sum;
        for (int w = 0; w < warp; ++w) pos += sh.warp_tot[w];
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int at = tid * CPT + j;
            if (at < SUB) sh.sub[at] = pos;
            pos += x[j];
        }
        if (tid == 0) sh.sub[SUB] = m;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        if ((uint32_t)(u * THREADS + tid) < m) {
            sh.key[sh.sub[sub[u]] + arrived[u]] = key[u];
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        if ((uint32_t)(u * THREADS + tid) < m) {
            const uint32_t s0 = sh.sub[sub[u]], s1 = sh.sub[sub[u] + 1];
            uint32_t rank = s0;
            for (uint32_t p = s0; p < s1; ++p) rank += sh.key[p] < key[u] ? 1u : 0u;
            if (owner) owner[id[u]] = partition_of(cuts, lo + rank);
            arrived[u] = rank;
        }
    }
    if (owner) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if ((uint32_t)(u * THREADS + tid) < m) sh.id[arrived[u]] = id[u];
    __syncthreads();
    for (uint32_t i = tid; i < m; i += THREADS) dst[lo + i] = sh.id[i]; // whole lines
}

// ------------------------------------------------------------------------------------------------ members by owner
// Ids grouped by owner, ascending inside a partition: counts per (owner, tile), a scan along the tiles of each owner
// (its first position is known: the partition's offset), a stable scatter. Up to 256 partitions in one pass.
constexpr int kGroupWarps = kSortThreads / 32;

__global__ void __launch_bounds__(kSortThreads)
k_group_count(const int32_t *__restrict__ owner, int64_t n, int32_t K, uint32_t *__restrict__ table, int nblk)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const int64_t i = base + (int64_t)it * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[owner[i]], 1u);
    }
    __syncthreads();
    if (threadIdx.x < K) table[(size_t)threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

__global__ void __launch_bounds__(kScanThreads)
k_group_scan(uint32_t *__restrict__ table, int nblk, const int64_t *__restrict__ part_off)
{
    __shared__ uint32_t warp_tot[kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *row = table + (size_t)blockIdx.x * nblk;
    uint32_t carry = (uint32_t)part_off[blockIdx.x];
    for (int base = 0; base < nblk; base += kScanThreads) {
        const uint32_t x = base + tid < nblk ? row[base + tid] : 0u;
        uint32_t incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        uint32_t before = 0, all = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) {
            before += w < warp ? warp_tot[w] : 0u;
            all += warp_tot[w];
        }
        if (base + tid < nblk) row[base + tid] = carry + before + incl - x;
        carry += all;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kSortThreads)
k_group_scatter(const int32_t *__restrict__ owner, int64_t n, int32_t K, const uint32_t *__restrict__ table, int nblk,
                int32_t *__restrict__ members)
{
    __shared__ uint32_t cnt[kGroupWarps][256];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int j = threadIdx.x; j < kGroupWarps * 256; j += kSortThreads) (&cnt[0][0])[j] = 0;
    __syncthreads();
    const int64_t warp_base = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * (kSortItems * 32);
    uint32_t dig[kSortItems], rank[kSortItems];
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const int64_t i = warp_base + it * 32 + lane;
        dig[it] = i < n ? (uint32_t)owner[i] : 256u;
    }
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const bool valid = dig[it] < 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, dig[it]);
        const uint32_t before = valid ? cnt[warp][dig[it]] : 0u;
        __syncwarp();
        if (valid && (peers & lt_mask) == 0u) cnt[warp][dig[it]] = before + __popc(peers);
        __syncwarp();
        rank[it] = before + __popc(peers & lt_mask);
    }
    __syncthreads();
    if (threadIdx.x < K) { // thread t owns partition t: per-warp counts into places in the output
        uint32_t run = table[(size_t)threadIdx.x * nblk + blockIdx.x];
#pragma unroll
        for (int w = 0; w < kGroupWarps; ++w) {
            const uint32_t c = cnt[w][threadIdx.x];
            cnt[w][threadIdx.x] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortItems; ++it)
        if (dig[it] < 256u) members[cnt[warp][dig[it]] + rank[it]] = (int32_t)(warp_base + it * 32 + lane);
}

__global__ void k_iota(int64_t n, int32_t *__restrict__ ids)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ids[i] = (int32_t)i;
}

cudaError_t group_members(Glm &g, int32_t K)
{
    const int64_t n = g.n_coord;
    if (K <= 256) {
        const int nblk = (int)((n + kSortTile - 1) / kSortTile);
        k_group_count<<<nblk, kSortThreads, 0, g.stream>>>(g.owner, n, K, g.ord.table, nblk);
        k_group_scan<<<K, kScanThreads, 0, g.stream>>>(g.ord.table, nblk, g.part_off);
        k_group_scatter<<<nblk, kSortThreads, 0, g.stream>>>(g.owner, n, K, g.ord.table, nblk, g.members);
        return cudaGetLastError();
    }
    // more partitions than one pass can tell apart: stable passes over the digits of owner[id]. The visiting-order
    // buffer is free between rounds; no pass reads what it writes.
    int passes = 2;
    while (passes < 4 && (int64_t)K > (1LL << (8 * passes))) ++passes;
    k_iota<<<blocks_for(n, 256), 256, 0, g.stream>>>(n, g.perm);
    const int32_t *src = g.perm;
    cudaError_t e = cudaSuccess;
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        int32_t *dst = p == passes - 1 ? g.members : (src == g.perm ? g.ord.tmp : g.perm);
        e = radix_pass(nullptr, src, nullptr, dst, g.owner, n, 8 * p, g.ord.table, g.ord.scan_sums, g.stream);
        src = dst;
    }
    return e;
}

// ------------------------------------------------------------------------------------------------ small partitions
// The whole partition (owner map and member lists) of up to 131 072 ids in one launch: a cluster of 8 CTAs. A launch
// costs about 2 us and the chain of dependent small kernels is what such a call consists of (47 launches: 335 us at
// n = 20 000), so the phases meet at cluster barriers instead. CTA r makes the keys of ids [r * chunk, (r + 1) * chunk)
// and holds, in its shared memory, the r-th eighth of the key range: counts per sub-bucket (about as many as ids, all
// CTAs together) and the ids placed by them. A rank is a sub-bucket's start plus the number of smaller keys in it.
constexpr int kMapC = 8;
constexpr int kMapThreads = 1024;
constexpr int kMapPer = CHICLE_NOALLOC_MAX_COORDS / (kMapC * kMapThreads); // ids per thread
constexpr int kMapChunk = kMapThreads * kMapPer;
constexpr int kMapCap = kMapChunk + 1024; // (the fullest eighth of 131 072 hashes: 16 384 + 8 standard deviations)
constexpr int kMapSub = CHICLE_NOALLOC_MAX_COORDS / kMapC;
constexpr int kMapMaxK = 512;  // more partitions: the member lists are made by comparison inside each partition (see launch_partition)
constexpr int kMapWarps = kMapThreads / 32;

struct MapShared {
    uint32_t sub[kMapSub + 1];         // this eighth's sub-buckets
    int32_t id[kMapCap];               // its ids, by sub-bucket; later: wcnt
    int32_t own[kMapChunk];            // owner of the ids of this CTA's chunk
    uint32_t ctot[kMapMaxK];           // how many of the chunk's ids each partition has
    uint32_t warp_tot[32];
    uint32_t total;
};
static_assert(sizeof(uint16_t) * kMapWarps * kMapMaxK <= sizeof(int32_t) * kMapCap, "the warps' counts reuse the ids' space");
static_assert(sizeof(MapShared) <= 227 * 1024, "shared memory");

__device__ __forceinline__ uint32_t map_addr(const void *p, uint32_t rank)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t map_ld(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void map_st(uint32_t a, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t map_inc(uint32_t a)
{
    uint32_t v;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], 1;" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void map_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// scratch: 2 n words (only read and written where K > kMapMaxK)
__global__ void __cluster_dims__(kMapC, 1, 1) __launch_bounds__(kMapThreads, 1)
k_partition_map(int32_t n, uint64_t s, int log_sub, const Cuts cuts, int32_t *__restrict__ owner, int32_t *__restrict__ members,
                int32_t *__restrict__ scratch)
{
    extern __shared__ __align__(16) unsigned char map_smem[];
    MapShared &sh = *reinterpret_cast<MapShared *>(map_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t r = blockIdx.x; // one cluster
    const uint32_t nsub = 1u << log_sub;
    const int32_t chunk = (((n + kMapC - 1) / kMapC) + 31) & ~31;
    const int32_t c0 = (int32_t)r * chunk, c1 = c0 + chunk < n ? c0 + chunk : n;
    const int per = (chunk + kMapThreads - 1) / kMapThreads;
    for (uint32_t i = tid; i < nsub; i += kMapThreads) sh.sub[i] = 0u;
    if (tid == 0) sh.total = 0u;
    map_sync();
    uint32_t place[kMapPer]; // sub-bucket (over all eighths), then the number of arrivals before this one, packed below
    uint32_t arrived[kMapPer];
#pragma unroll
    for (int u = 0; u < kMapPer; ++u) {
        const int32_t i = c0 + u * kMapThreads + tid;
        place[u] = arrived[u] = 0u;
        if (u < per && i < c1) {
            place[u] = (uint32_t)(mix64(s ^ (uint64_t)(uint32_t)i) >> (64 - 3 - log_sub));
            arrived[u] = map_inc(map_addr(&sh.sub[place[u] & (nsub - 1u)], place[u] >> log_sub));
        }
    }
    map_sync();
    {
        // where each of this eighth's sub-buckets starts
        const int cpt = (int)((nsub + kMapThreads - 1) / kMapThreads);
        uint32_t sum = 0;
        for (int j = 0; j < cpt; ++j) {
            const uint32_t at = (uint32_t)(tid * cpt + j);
            sum += at < nsub ? sh.sub[at] : 0u;
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sh.warp_tot[warp] = incl;
        __syncthreads();
        uint32_t pos = incl - sum, all = 0;
        for (int w = 0; w < kMapWarps; ++w) {
            pos += w < warp ? sh.warp_tot[w] : 0u;
            all += sh.warp_tot[w];
        }
        for (int j = 0; j < cpt; ++j) {
            const uint32_t at = (uint32_t)(tid * cpt + j);
            if (at < nsub) {
                const uint32_t x = sh.sub[at];
                sh.sub[at] = pos;
                pos += x;
            }
        }
        if (tid == 0) {
            sh.sub[nsub] = all;
            sh.total = all;
        }
    }
    map_sync();
    uint32_t first = 0; // elements in the eighths before this one
    bool over = false;
    for (uint32_t c = 0; c < (uint32_t)kMapC; ++c) {
        const uint32_t t = map_ld(map_addr(&sh.total, c));
        first += c < r ? t : 0u;
        over |= t > (uint32_t)kMapCap;
    }
    if (!over) {
#pragma unroll
        for (int u = 0; u < kMapPer; ++u) {
            const int32_t i = c0 + u * kMapThreads + tid;
            if (u < per && i < c1) {
                const uint32_t c = place[u] >> log_sub;
                const uint32_t at = map_ld(map_addr(&sh.sub[place[u] & (nsub - 1u)], c)) + arrived[u];
                map_st(map_addr(&sh.id[at], c), (uint32_t)i);
            }
        }
        map_sync();
        const uint32_t m = sh.total;
        for (uint32_t p = tid; p < m; p += kMapThreads) {
            const uint32_t i = (uint32_t)sh.id[p];
            const uint64_t key = mix64(s ^ (uint64_t)i);
            const uint32_t b = (uint32_t)(key >> (64 - 3 - log_sub)) & (nsub - 1u);
            const uint32_t lo = sh.sub[b], hi = sh.sub[b + 1];
            uint32_t rank = first + lo;
            if (hi - lo > 1u)
                for (uint32_t q = lo; q < hi; ++q) rank += mix64(s ^ (uint64_t)(uint32_t)sh.id[q]) < key ? 1u : 0u;
            const int32_t c = (int32_t)i / chunk;
            map_st(map_addr(&sh.own[(int32_t)i - c * chunk], (uint32_t)c), (uint32_t)partition_of(cuts, rank));
        }
    } else {
        // (no set of hashes is that uneven; ranked by comparison with all)
        map_sync();
        for (int32_t i = c0 + tid; i < c1; i += kMapThreads) {
            const uint64_t key = mix64(s ^ (uint64_t)(uint32_t)i);
            uint32_t rank = 0;
            for (int32_t j = 0; j < n; ++j) rank += mix64(s ^ (uint64_t)(uint32_t)j) < key ? 1u : 0u;
            sh.own[i - c0] = partition_of(cuts, rank);
        }
    }
    map_sync();
    for (int32_t i = c0 + tid; i < c1; i += kMapThreads) owner[i] = sh.own[i - c0];
    const int32_t K = cuts.K;
    if (K <= kMapMaxK) {
        // ---- stable by owner: a warp takes consecutive ids; counts per warp, then per CTA, then over the CTAs before
        uint16_t *wcnt = reinterpret_cast<uint16_t *>(sh.id); // [warp][K]
        for (int j = tid; j < kMapWarps * K; j += kMapThreads) wcnt[j] = 0;
        __syncthreads();
        const int32_t seg = ((chunk / 32 + kMapWarps - 1) / kMapWarps) * 32; // ids of a warp
        const int32_t w0 = c0 + warp * seg, w1 = w0 + seg < c1 ? w0 + seg : c1;
        uint16_t *mine = wcnt + warp * K;
        const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
        for (int u = 0; u < kMapPer; ++u) {
            const int32_t i = w0 + u * 32 + lane;
            if (w0 + u * 32 < w1) { // (whole warps)
                const bool on = i < w1;
                const uint32_t d = on ? (uint32_t)sh.own[i - c0] : 0xffffffffu;
                const uint32_t peers = __match_any_sync(0xffffffffu, d);
                const uint32_t before = on ? mine[d] : 0u;
                __syncwarp();
                if (on && (peers & lt) == 0u) mine[d] = (uint16_t)(before + __popc(peers));
                __syncwarp();
                place[u] = d;
                arrived[u] = before + __popc(peers & lt);
            }
        }
        __syncthreads();
        for (int k = tid; k < K; k += kMapThreads) {
            uint32_t run = 0;
            for (int w = 0; w < kMapWarps; ++w) {
                const uint32_t c = wcnt[w * K + k];
                wcnt[w * K + k] = (uint16_t)run;
                run += c;
            }
            sh.ctot[k] = run;
        }
        map_sync();
        for (int k = tid; k < K; k += kMapThreads) {
            uint32_t at = start_of(cuts, k);
            for (uint32_t c = 0; c < r; ++c) at += map_ld(map_addr(&sh.ctot[k], c));
            sh.sub[k] = at; // (the sub-buckets are done with)
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kMapPer; ++u) {
            const int32_t i = w0 + u * 32 + lane;
            if (w0 + u * 32 < w1 && i < w1) members[sh.sub[place[u]] + mine[place[u]] + arrived[u]] = i;
        }
    } else {
        // ---- many small partitions: ids gathered by partition in any order, then ranked inside it by comparison
        uint32_t *cursor = reinterpret_cast<uint32_t *>(scratch);
        int32_t *tmp = scratch + n;
        for (int32_t k = (int32_t)r * kMapThreads + tid; k < K; k += kMapC * kMapThreads) cursor[k] = 0u;
        __threadfence();
        map_sync();
        for (int32_t i = c0 + tid; i < c1; i += kMapThreads) {
            const int32_t k = sh.own[i - c0];
            tmp[start_of(cuts, k) + atomicAdd(cursor + k, 1u)] = i;
        }
        __threadfence();
        map_sync();
        for (int32_t p = (int32_t)r * kMapThreads + tid; p < n; p += kMapC * kMapThreads) {
            const int32_t k = partition_of(cuts, (uint32_t)p);
            const uint32_t lo = start_of(cuts, k), hi = start_of(cuts, k + 1);
            const int32_t id = __ldcg(tmp + p);
            uint32_t rank = lo;
            for (uint32_t q = lo; q < hi; ++q) rank += __ldcg(tmp + q) < id ? 1u : 0u;
            members[rank] = id;
        }
    }
    map_sync(); // nobody leaves while another CTA may still read its shared memory
}

cudaError_t launch_map(int64_t n, uint64_t seed, const Cuts &cuts, int32_t *owner, int32_t *members, int32_t *scratch, cudaStream_t stream)
{
    int log_sub = 0; // about one id per sub-bucket
    while (log_sub < 14 && ((int64_t)kMapC << log_sub) < n) ++log_sub;
    static_assert(kMapSub == 1 << 14, "sub-buckets of an eighth");
    cudaError_t e = cudaFuncSetAttribute(k_partition_map, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MapShared));
    if (e != cudaSuccess) return e;
    k_partition_map<<<kMapC, kMapThreads, sizeof(MapShared), stream>>>((int32_t)n, mix64(seed), log_sub, cuts, owner, members, scratch);
    return cudaGetLastError();
}

// tiles per segment for the counting and scattering kernels: enough CTAs to fill the GPU, no more than the longest needs; 0
// (see for_my_elements): the longest segment's CTAs would have more than four times what a CTA has on average, and more than
// four tiles (10 M coordinates in 1 200 segments, half of them in one: 6.9 ms with a CTA for each, 0.21 this way)
inline int tiles_for(const Glm &g, int64_t longest, int K)
{
    const int64_t ctas = (int64_t)g.sm_count * 8, want = (ctas + K - 1) / K, have = (longest + kCountTile - 1) / kCountTile;
    const int64_t t = want < have ? want : have, even = g.n_coord / ctas;
    if (K > 1 && longest / t > 4 * (even > kCountTile ? even : kCountTile)) return 0;
    return (int)t;
}
// CTAs of such a launch
inline unsigned ctas_for(const Glm &g, int tiles, int K)
{
    if (tiles > 0) return (unsigned)tiles * (unsigned)K;
    const int64_t most = (int64_t)g.sm_count * 8;
    return (unsigned)(g.n_buckets < most ? g.n_buckets : most);
}

template <int CAP, int THREADS>
cudaError_t launch_order(unsigned grid, const int32_t *src, const uint32_t *start, const uint32_t *nbm, const int64_t *seg_off, uint64_t ab,
                         uint32_t *cursor, int32_t *dst, const Cuts &cuts, int32_t *owner, cudaStream_t stream)
{
    auto kern = k_bucket_order<CAP, THREADS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OrderShared<CAP>));
    if (e != cudaSuccess) return e;
    kern<<<grid, THREADS, sizeof(OrderShared<CAP>), stream>>>(src, start, nbm, seg_off, ab, cursor, dst, cuts, owner);
    return cudaGetLastError();
}

} // namespace

int64_t order_buckets(int64_t nk) { return (nk + kBucketMean - 1) / kBucketMean; }

// most, most_buckets: of the largest segment. A CTA counts by itself if it has four elements and more of a bucket.
static void launch_count(const Glm &g, const Segments &S, int segments, int64_t most, uint32_t most_buckets, int tiles, const int32_t *ids,
                         uint64_t ab, uint32_t *cursor, cudaStream_t stream)
{
    const int64_t per_cta = tiles == 0 ? 0 : (most / tiles < kCountTile ? kCountTile : most / tiles);
    const unsigned ctas = ctas_for(g, tiles, segments);
    if (most_buckets <= kLocalBuckets && per_cta >= 4 * (int64_t)most_buckets) k_bucket_count<true><<<ctas, kCountThreads, 0, stream>>>(S, tiles, ids, ab, cursor);
    else k_bucket_count<false><<<ctas, kCountThreads, 0, stream>>>(S, tiles, ids, ab, cursor);
}

cudaError_t launch_partition(Glm &g, int32_t K, uint64_t seed)
{
    const int64_t n = g.n_coord;
    // (the offsets are on the device already: equal blocks, or the sizes the caller gave)
    const Cuts cuts{g.part_off, K, 0, 0};
    // More partitions than the one-launch kernel counts by: it compares every id with all of its partition, on eight SMs, which
    // pays while there are few ids and no large partition. (20 000 ids, K = 513: 64 us a call against 128 on the path below;
    // 131 072 ids, K = 2 000: 270 against 174; one partition of half of 131 072 ids: 17 ms against 0.15.)
    const bool few = n <= 32768 && n * g.max_nk <= (int64_t)1 << 20;
    if (n <= CHICLE_NOALLOC_MAX_COORDS && (K <= kMapMaxK || few)) return launch_map(n, seed, cuts, g.owner, g.members, g.ord.tmp, g.stream);
    // Which partition an id falls to needs its place in key order only where a cut lies inside its bucket: all other
    // ids get their bucket's partition, those (a K / n * 512 share) are put in order.
    const Segments S{nullptr, nullptr, 1, n, (uint32_t)order_buckets(n)};
    const uint64_t s = mix64(seed);
    const int tiles = tiles_for(g, n, 1);
    OrderWorkspace &w = g.ord;
    launch_count(g, S, 1, n, S.nb, tiles, nullptr, s, w.cursor, g.stream);
    k_bucket_scan<<<1, kScanThreads, 0, g.stream>>>(S, w.start, w.cursor, w.nbm, w.bowner, cuts, nullptr, 0, 0);
    k_bucket_scatter<<<tiles, kCountThreads, 0, g.stream>>>(S, tiles, nullptr, s, w.cursor, w.nbm, w.bowner, g.owner, w.tmp);
    cudaError_t e = launch_order<2 * kBucketMean, 256>(S.nb, w.tmp, w.start, w.nbm, nullptr, s, w.cursor, nullptr, cuts, g.owner, g.stream);
    if (e != cudaSuccess) return e;
    return group_members(g, K);
}

// owner[i] = task of the chunk that holds coordinate i: chunk_off[c] <= i < chunk_off[c + 1]
__global__ void k_owner_from_chunks(int64_t n, int64_t C, const int64_t *__restrict__ chunk_off,
                                    const int32_t *__restrict__ chunk_task, int32_t *__restrict__ owner)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        int64_t lo = 0, hi = C;
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (chunk_off[mid] <= i) lo = mid;
            else hi = mid;
        }
        owner[i] = chunk_task[lo];
    }
}

// entries[t] += stored entries of task t's chunks
__global__ void k_chunk_entries(int64_t C, const int64_t *__restrict__ chunk_off, const int32_t *__restrict__ chunk_task,
                                const int64_t *__restrict__ indptr, unsigned long long *__restrict__ entries)
{
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < C) atomicAdd(entries + chunk_task[c], (unsigned long long)(indptr[chunk_off[c + 1]] - indptr[chunk_off[c]]));
}

cudaError_t launch_chunk_entries(Glm &g, int64_t C, const int64_t *chunk_off, const int32_t *chunk_task, unsigned long long *entries)
{
    k_chunk_entries<<<blocks_for(C, 256), 256, 0, g.stream>>>(C, chunk_off, chunk_task, g.indptr, entries);
    return cudaGetLastError();
}

// far[k] = entries with ids from `first` on in up to kFarSample of partition k's coordinates, evenly spaced (a CTA per partition)
__global__ void k_far_sample(const int32_t *__restrict__ members, const int64_t *__restrict__ part_off, const int64_t *__restrict__ indptr,
                             const int32_t *__restrict__ indices, int64_t first, unsigned long long *__restrict__ far)
{
    __shared__ uint32_t sum;
    if (threadIdx.x == 0) sum = 0u;
    __syncthreads();
    const int64_t off = part_off[blockIdx.x], nk = part_off[blockIdx.x + 1] - off, m = nk < kFarSample ? nk : kFarSample;
    uint32_t n = 0u;
    for (int64_t i = threadIdx.x >> 5; i < m; i += blockDim.x >> 5) {
        const int32_t c = members[off + i * nk / m];
        for (int64_t e = indptr[c] + (threadIdx.x & 31); e < indptr[c + 1]; e += 32) n += indices[e] >= first ? 1u : 0u;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(&sum, n);
    __syncthreads();
    if (threadIdx.x == 0) far[blockIdx.x] = sum;
}

cudaError_t launch_far_sample(Glm &g, int32_t K, int64_t first, unsigned long long *far)
{
    k_far_sample<<<K, 256, 0, g.stream>>>(g.members, g.part_off, g.indptr, g.indices, first, far);
    return cudaGetLastError();
}

cudaError_t launch_partition_chunks(Glm &g, int32_t K, int64_t C, const int64_t *chunk_off, const int32_t *chunk_task)
{
    const int64_t n = g.n_coord;
    const int T = 256;
    k_owner_from_chunks<<<blocks_for(n, T), T, 0, g.stream>>>(n, C, chunk_off, chunk_task, g.owner);
    return group_members(g, K);
}

// The visiting orders of `epochs` local epochs. H and steps as in a round (steps: K budgets on the device): only the
// buckets that the round's steps reach are put in order; H = 0 and steps = nullptr: everything.
cudaError_t launch_permutation(Glm &g, int64_t round, int64_t epochs, int64_t H, const int64_t *steps)
{
    const int64_t n = g.n_coord;
    OrderWorkspace &w = g.ord;
    const uint64_t a = mix64(g.seed ^ kPermStream);
    const Cuts none{nullptr, 1, 1, 0};
    const Segments S{g.part_off, g.bucket_off, g.K, n, 0};
    const int tiles = tiles_for(g, g.max_nk, g.K);
    g.order_launches = 0;
    for (int64_t e = 0; e < epochs; ++e) {
        const uint64_t ab = a ^ mix64(((uint64_t)round << 32) + (uint64_t)e);
        int32_t *out = g.perm + (size_t)e * (size_t)n;
        cudaError_t err;
        // partitions that fit a CTA's arrays are buckets themselves: one launch (10 000 coordinates, K = 4: 8 us
        // against 190 us for the 27 launches of a radix sort)
        if (g.max_nk <= 2 * kBucketMean) {
            err = launch_order<2 * kBucketMean, 256>((unsigned)g.K, g.members, nullptr, nullptr, g.part_off, ab, nullptr, out, none, nullptr, g.stream);
            g.order_launches += 1;
        } else if (g.max_nk <= kOrderOneCta) {
            err = launch_order<(int)kOrderOneCta, 1024>((unsigned)g.K, g.members, nullptr, nullptr, g.part_off, ab, nullptr, out, none, nullptr, g.stream);
            g.order_launches += 1;
        } else {
            launch_count(g, S, g.K, g.max_nk, (uint32_t)order_buckets(g.max_nk), tiles, g.members, ab, w.cursor, g.stream);
            k_bucket_scan<<<g.K, kScanThreads, 0, g.stream>>>(S, w.start, w.cursor, w.nbm, nullptr, none, steps, H, e);
            k_bucket_scatter<<<ctas_for(g, tiles, g.K), kCountThreads, 0, g.stream>>>(S, tiles, g.members, ab, w.cursor, w.nbm, nullptr, nullptr, w.tmp);
            err = launch_order<2 * kBucketMean, 256>((unsigned)g.n_buckets, w.tmp, w.start, w.nbm, nullptr, ab, w.cursor, out, none, nullptr, g.stream);
            g.order_launches += 4;
        }
        if (err != cudaSuccess) return err;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------------------
// Partition without any allocation.
//
// Some callers are not allowed to allocate device memory when they need a partition map: code that runs inside a
// region where the allocator must not be touched (a memory pool that was sized and frozen at start-up, a real-time
// or serving loop with a fixed memory budget, a host thread that holds a lock the allocator also takes), or a
// process whose device memory is handed out entirely by someone else. chicle_partition() cannot serve them: it
// creates the workspaces and the per-partition update buffers on its first call. The entry point below does
// the same integer work (the same kernel, the same result) in shared memory; what more than 512 partitions need beyond
// that is a fixed array that is part of the loaded library image, so no cudaMalloc, cudaFree or framework allocator is
// ever called.
//
// The array below is device memory owned by the CUDA module: every GPU that loads this library carries it until
// the process exits. In host code its name is only a handle for the symbol, not an address a kernel may
// dereference; the device address is fetched once per device with cudaGetSymbolAddress and that pointer is what
// the kernels get.
namespace {

static __device__ __align__(256) int32_t g_noalloc_scratch[2 * CHICLE_NOALLOC_MAX_COORDS];

constexpr int kNaMaxDevices = 64;
std::mutex g_na_mutex;
int32_t *g_na_base[kNaMaxDevices] = {};

void na_message(char *buf, size_t len, const char *msg)
{
    if (buf && len) std::snprintf(buf, len, "%s", msg);
}

} // namespace

} // namespace chicle

extern "C" chicle_status_t chicle_partition_noalloc(int device, void *cuda_stream, int64_t n_coord, int32_t K,
                                                    uint64_t seed, int32_t *dev_owner, int32_t *dev_members,
                                                    char *host_errbuf, size_t errbuf_len)
{
    using namespace chicle;
    if (!dev_owner || !dev_members) {
        na_message(host_errbuf, errbuf_len, "dev_owner and dev_members must be non-NULL device pointers");
        return CHICLE_ERR_INVALID_ARG;
    }
    if (n_coord < 1 || n_coord > CHICLE_NOALLOC_MAX_COORDS) {
        na_message(host_errbuf, errbuf_len,
                   "n_coord outside [1, CHICLE_NOALLOC_MAX_COORDS]: the built-in workspace holds at most 131072 "
                   "coordinates; use chicle_partition for larger problems");
        return CHICLE_ERR_UNSUPPORTED;
    }
    if (K < 1 || (int64_t)K > n_coord) {
        na_message(host_errbuf, errbuf_len, "need 1 <= K <= n_coord");
        return CHICLE_ERR_INVALID_ARG;
    }
    if (device < 0 || device >= kNaMaxDevices) {
        na_message(host_errbuf, errbuf_len, "device index out of range");
        return CHICLE_ERR_INVALID_ARG;
    }
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        na_message(host_errbuf, errbuf_len, cudaGetErrorString(e));
        return CHICLE_ERR_CUDA;
    }
    int32_t *base = nullptr;
    {
        // set-up, once per device, with that device current: turn the symbol into a device address
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_base[device]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p) {
                (void)cudaGetLastError();
                na_message(host_errbuf, errbuf_len, e != cudaSuccess ? cudaGetErrorString(e) : "cudaGetSymbolAddress returned NULL");
                return CHICLE_ERR_CUDA;
            }
            g_na_base[device] = static_cast<int32_t *>(p);
        }
        base = g_na_base[device];
    }
    // Nothing in the workspace has to start at zero: what the kernel reads of it, it has written before.
    const Cuts cuts{nullptr, K, (uint32_t)(n_coord / K), (uint32_t)(n_coord % K)};
    e = launch_map(n_coord, seed, cuts, dev_owner, dev_members, base, static_cast<cudaStream_t>(cuda_stream));
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        na_message(host_errbuf, errbuf_len, cudaGetErrorString(e));
        return CHICLE_ERR_CUDA;
    }
    return CHICLE_OK;
}
