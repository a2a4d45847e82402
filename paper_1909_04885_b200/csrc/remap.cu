// Frequency ranking of the entry ids of a sparse problem (features for the dual losses, rows for ridge), done once
// when the problem is created: id 0 becomes the id that occurs in the most non-zeros, ties by ascending old id.
// The matrix indices are relabelled in place; the shared vector lives in the new id space inside the library and is
// translated at the boundary. The local solver keeps the most frequent ids of U_k in a direct shared-memory array.
#include "chicle_internal.cuh"

namespace chicle {

namespace {

constexpr int kT = 256;
inline unsigned blocks_for(int64_t n) { return (unsigned)((n + kT - 1) / kT); }

__global__ void k_count_ids(const int32_t *__restrict__ indices, int64_t nnz, uint32_t *__restrict__ counts)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(counts + indices[e], 1u);
}

__global__ void k_freq_keys(const uint32_t *__restrict__ counts, int64_t dim, uint64_t *__restrict__ keys,
                            int32_t *__restrict__ vals)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < dim) {
        keys[i] = ((uint64_t)(0xFFFFFFFFu - counts[i]) << 32) | (uint64_t)(uint32_t)i; // descending count, ascending id
        vals[i] = (int32_t)i;
    }
}

__global__ void k_invert(const int32_t *__restrict__ sorted_old, int64_t dim, int32_t *__restrict__ new_of_old,
                         int32_t *__restrict__ old_of_new)
{
    const int64_t pos = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pos < dim) {
        const int32_t old = sorted_old[pos];
        new_of_old[old] = (int32_t)pos;
        old_of_new[pos] = old;
    }
}

__global__ void k_relabel(int32_t *__restrict__ indices, int64_t nnz, const int32_t *__restrict__ new_of_old)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
        indices[e] = new_of_old[indices[e]];
}

__global__ void k_mass_of_first(const uint32_t *__restrict__ counts, const int32_t *__restrict__ old_of_new, int64_t first,
                                unsigned long long *__restrict__ out)
{
    unsigned long long s = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < first; i += (int64_t)gridDim.x * blockDim.x)
        s += counts[old_of_new[i]];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

// What a block of 32 random coordinates is expected to have on the ids of class i = (new id) mod kRankClasses: out[i]
// entries (the whole problem's, exactly), out[kRankClasses + i] ids that at least two of the 32 have and
// out[2 kRankClasses + i] entries with such ids (both in units of 2^-20, so that the sums do not depend on their order); and
// out[3 kRankClasses + k] entries with (new) ids of octave k: 2^k .. 2^(k+1) - 1, and id 0 in octave 0.
__global__ void k_expect_blocks(const uint32_t *__restrict__ counts, const int32_t *__restrict__ old_of_new, int64_t dim, double inv_n,
                                unsigned long long *__restrict__ out)
{
    static_assert(kT % kRankClasses == 0, "a thread's ids are of one class");
    unsigned long long all = 0, ids = 0, ent = 0;
    __shared__ unsigned long long octave[kOctaves];
    if (threadIdx.x < kOctaves) octave[threadIdx.x] = 0;
    __syncthreads();
    int at = 0;
    unsigned long long part = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < dim; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = counts[old_of_new[i]];
        const float p = fminf((float)((double)c * inv_n), 0.9999999f), l = log1pf(-p);
        const float others = -expm1f(31.0f * l);                               // one of the other 31 has it
        const float one = 32.0f * p * (1.0f - others), some = -expm1f(32.0f * l); // exactly one has it, some have it
        all += c;
        const int oct = i >= 2 ? 63 - __clzll(i) : 0; // (a thread's ids ascend: it meets every octave once)
        if (oct != at) {
            if (part) atomicAdd(octave + at, part);
            at = oct;
            part = 0;
        }
        part += c;
        ids += (unsigned long long)(fmaxf(some - one, 0.0f) * 1048576.0f);
        ent += (unsigned long long)(32.0f * p * others * 1048576.0f);
    }
    if (part) atomicAdd(octave + at, part);
#pragma unroll
    for (int o = 16; o >= kRankClasses; o >>= 1) {
        all += __shfl_xor_sync(0xffffffffu, all, o);
        ids += __shfl_xor_sync(0xffffffffu, ids, o);
        ent += __shfl_xor_sync(0xffffffffu, ent, o);
    }
    if ((threadIdx.x & 31) < kRankClasses) {
        unsigned long long *o = out + (threadIdx.x & (kRankClasses - 1));
        if (all) atomicAdd(o, all);
        if (ids) atomicAdd(o + kRankClasses, ids);
        if (ent) atomicAdd(o + 2 * kRankClasses, ent);
    }
    __syncthreads();
    if (threadIdx.x < kOctaves && octave[threadIdx.x]) atomicAdd(out + 3 * kRankClasses + threadIdx.x, octave[threadIdx.x]);
}

// out[1] += number of coordinates with more than `long_len` entries; out[2] += the sum of their squared lengths (each
// counted as 65 536 at most)
__global__ void k_count_long(const int64_t *__restrict__ indptr, int64_t n_coord, int32_t long_len,
                             unsigned long long *__restrict__ out)
{
    unsigned long long s = 0, q = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_coord; c += (int64_t)gridDim.x * blockDim.x) {
        const int64_t len = indptr[c + 1] - indptr[c], m = len < 65536 ? len : 65536;
        s += len > long_len ? 1u : 0u;
        q += (unsigned long long)(m * m);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (s) atomicAdd(out + 1, s);
        if (q) atomicAdd(out + 2, q);
    }
}

// dst[i] = src[map[i]]
__global__ void k_gather_f32(const float *__restrict__ src, const int32_t *__restrict__ map, int64_t n, float *__restrict__ dst)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[map[i]];
}

} // namespace

// counts: dim zeroed uint32; keys/vals: two arrays of dim each; mass: kMassWords zeroed 64-bit words (non-zeros on the first
// hot_ids ids; coordinates longer than long_len; the sum of squared lengths; from word 4 on what k_expect_blocks sums).
cudaError_t launch_frequency_remap(Glm &g, uint32_t *counts, uint64_t *keys[2], int32_t *vals[2], uint32_t *hist,
                                   uint32_t *scan_sums, int64_t hot_ids, int32_t long_len, unsigned long long *mass)
{
    const int64_t dim = g.dim;
    const unsigned wide = (unsigned)g.sm_count * 8;
    k_count_ids<<<wide, kT, 0, g.stream>>>(g.indices, g.nnz, counts);
    k_freq_keys<<<blocks_for(dim), kT, 0, g.stream>>>(counts, dim, keys[0], vals[0]);
    int cur = 0;
    for (int pass = 0; pass < 8; ++pass) {
        cudaError_t e = radix_pass(keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], nullptr, dim, 8 * pass, hist,
                                   scan_sums, g.stream);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    k_invert<<<blocks_for(dim), kT, 0, g.stream>>>(vals[cur], dim, g.new_of_old, g.old_of_new);
    k_relabel<<<wide, kT, 0, g.stream>>>(g.indices, g.nnz, g.new_of_old);
    const int64_t first = hot_ids < dim ? hot_ids : dim;
    k_mass_of_first<<<blocks_for(first), kT, 0, g.stream>>>(counts, g.old_of_new, first, mass);
    k_count_long<<<wide, kT, 0, g.stream>>>(g.indptr, g.n_coord, long_len, mass);
    k_expect_blocks<<<blocks_for(dim) < wide ? blocks_for(dim) : wide, kT, 0, g.stream>>>(counts, g.old_of_new, dim, 1.0 / (double)g.n_coord, mass + 4);
    return cudaGetLastError();
}

cudaError_t launch_gather_f32(Glm &g, const float *src, const int32_t *map, int64_t n, float *dst)
{
    k_gather_f32<<<(unsigned)g.sm_count * 4, kT, 0, g.stream>>>(src, map, n, dst);
    return cudaGetLastError();
}

} // namespace chicle
