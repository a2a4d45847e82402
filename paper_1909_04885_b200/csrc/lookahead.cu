// Local SCD solver with block look-ahead: the same result as walking a partition's visiting order coordinate by
// coordinate (paper Sec. 2.2 worker structure with L = 1; Sec. 5.1: SCD local solver), up to rounding order, with
// everything that does not depend on the step before taken off the sequential chain.
//
// The walk is cut into blocks of 32 consecutive steps. With w the local model some steps back,
//     dot_j = x_j . w + sigma' * sum over the steps l since then of delta_l * (x_j . x_l),
// so once the dot products against an OLDER model and the Gram entries x_j . x_l are known, the steps are a scalar
// recurrence. A block's dot products are taken against the model as it was two blocks earlier (while the block
// before it is still being walked); what the block before contributes comes from the cross Gram matrix of the two
// blocks, what the block's own earlier steps contribute from its Gram triangle. Only the recurrence is sequential:
// one warp runs it block after block without waiting for a model update, while the other warps, and the other CTAs
// of the partition's thread-block cluster, apply block b's update to the model and take block b + 2's dot products.
//
//   k_lookahead_prepare   nothing in it depends on the model; a CTA takes a run of consecutive blocks (k_lookahead_prepare_dense:
//                         a block at a time). Writes each block's records: for
//                         the recurrence warp the per-step constants, the scaled Gram triangle and the scaled cross
//                         Gram matrix with the next block; for each CTA of the cluster the block's non-zeros whose
//                         entry id falls to that CTA (id mod cluster size), packed row after row, and for the ids
//                         that several coordinates of the block share the transposed view (one list per id, in
//                         ascending coordinate order), so that the model update needs no atomics and gives the same
//                         bits every run.
//   k_lookahead_chain     one cluster of C CTAs per partition. Entry ids below C * HOT (ids are frequency-ranked)
//                         live in shared memory for the whole kernel as w = v + sigma' U_k, id i in CTA i mod C;
//                         the others live in row k of the update workspace in global memory, which holds the model
//                         itself between the launches of a round (the first launch turns U_k into w in place, the
//                         last one turns it back): one gather or one reduction per non-zero.
//                         Warp 0 of CTA 0 runs the recurrence. The worker warps of every CTA loop over
//                         "wait for block b's deltas, apply them to my part of the model, take my part of block
//                         b + 2's dot products, send the 32 partial sums to CTA 0". Deltas and partial sums travel
//                         through distributed shared memory by asynchronous stores that complete on the receiver's
//                         mbarrier; no multicast, every wait bounded. Ids that are not in shared memory: where a block has a
//                         few of them per CTA, a warp of its own applies their updates and takes their part of the dot products; where
//                         it has many, the worker warps do, and where dot products wait for deltas in any case their gathers go out before.
//
// Where many partitions leave the prepare kernels few SMs (one CTA per partition on sparse data), the dot products are
// taken one block ahead only, against the model after the block before: no cross Gram matrix (the prepare kernels are
// what bounds such rounds), and the recurrence warp waits for each block's dot products; and where the chains take more
// than half of the SMs, the prepare kernels alternate with the chain launches instead of running beside them.
//
// A block with more non-zeros than the shared-memory buffers hold is flagged by the prepare kernel: the pipeline
// drains, warp 0 of CTA 0 walks the block coordinate by coordinate against the whole model, and the pipeline starts
// again behind it. Rounds that span several local epochs run the pair of kernels once per epoch.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>

#include "solver_common.cuh"

namespace chicle {

namespace {

constexpr int kLB = 32;            // steps per block
constexpr int kMaxC = 8;           // CTAs per cluster at most (the portable limit)
constexpr int kDenseSlice = 384;   // columns of a dense row that one CTA of a cluster can take: four blocks' slices fill its shared memory (an
                                   // update takes the columns beyond kWorkThreads in a second turn)
constexpr int kDenseEasy = 128;    // and what it takes where the cluster may be larger
// Where the model entry of an id is, in kIdBits bits: its place in its CTA's part of the model in shared memory (below hotc),
// or the id itself (never below hotc, see k_lookahead_chain). Problems with more ids take the blocked solver.
constexpr int kIdBits = 26;
constexpr uint32_t kIdMask = (1u << kIdBits) - 1u;
constexpr int kSubSlots = 4;       // worker records in shared memory: blocks b .. b + 3 (three of them where long records leave no room, see lookahead_plan)
// Recurrence records in shared memory: a record is fetched when the block that many before it is done, and takes 1 500 cycles
// or more from memory, so two would set the pace (1 M sparse rows: 3 019 cycles a block, with three 2 600). With tables of the logistic step
// (see tab_map: 32 KB or more each, fetched with the record) a block takes longer and two do.
constexpr int kMaxHeadSlots = 3;
__host__ __device__ constexpr int head_slots(bool tables) { return tables ? 2 : 3; }
// Worker warps: warps 1 .. 10 but for those that share warp 0's scheduler (warp ids 0, 4, 8), which stay out of its way.
// Warps 4 and 11 of CTA 0 take from the recurrence warp all that is not the recurrence (see the kernel).
constexpr int kWorkWarps = 8;
constexpr int kWorkThreads = kWorkWarps * 32;
constexpr int kBarWork = 1;        // named barrier of the worker warps
constexpr int kRecordWarp = 8;     // fetches the workers' records
constexpr int kStartWarp = 4;      // in CTA 0: the states that a block's recurrence starts from
constexpr int kFeedWarp = 11;      // in CTA 0: what follows from a block's recurrence; fetches the recurrence records
constexpr int kFarWarp = 13;       // (kSplit) ids beyond the model's part in shared memory; warp 12 would share warp 0's scheduler and has no role

// Per-step constants for the recurrence warp (see coordinate_step for p0 .. p3).
struct alignas(16) CHdr {
    int32_t coord;
    float p0, p1, p2, p3;
    float A, B; // the recurrence's state starts at A + B * (dot product against the older model) (+ the cross terms)
    float lq;   // logistic: log of p2; with tables: tab_map's `off`
};
static_assert(sizeof(CHdr) == 32, "header size");

// What the recurrence warp reads for one block.
struct alignas(16) ChainHead {
    int32_t cnt;    // steps in the block (32 but for a partition's last block)
    int32_t flags;  // bit 0: walk this block coordinate by coordinate
    int32_t pad[2];
    CHdr hdr[kLB];
    float q0n[kLB];      // what the states of this block's coordinates at round start contribute to the next block
    float G[kLB * kLB];  // G[l * 32 + j]: scaled Gram entry of this block's coordinates l < j, else 0
    float X[kLB * kLB];  // X[l * 32 + j]: scaled Gram entry of this block's l with the NEXT block's j (0: no carry)
};
static_assert(sizeof(ChainHead) % 16 == 0, "bulk copy size");

// What one CTA's workers read for one block. Behind it (sparse): val[n] f32, meta[n] u32 (low bits: where the entry's
// part of the model is, see kIdBits; the coordinate's place in the block above them; the top bit marks an id that several
// coordinates of the block have), both row after row; then the entries of those shared ids once more, one list per id,
// each in ascending coordinate order: ids[T] u32 (the same low bits, list length - 1 above them), lval[nl] f32,
// lst[T] u16 (where each list starts), lrow[nl] u8 (coordinates).
// Dense: val[cnt][slice of the row, dense_stride floats].
struct alignas(16) SubHead {
    int32_t n;     // non-zeros of the block that fall to this CTA
    int32_t T;     // shared ids among them
    int32_t nl;    // entries with a shared id
    int32_t cnt;
    uint16_t roff[kLB + 8]; // where each coordinate's non-zeros start ([32] = n)
};
static_assert(sizeof(SubHead) == 96, "sub-record head");

__host__ __device__ constexpr uint32_t sub_bytes(uint32_t n, uint32_t T, uint32_t nl)
{
    return ((uint32_t)sizeof(SubHead) + 8u * n + 6u * T + 5u * nl + 15u) & ~15u;
}
// Dense rows in a record: 16-byte pieces of consecutive rows lie on different banks.
__host__ __device__ constexpr int dense_stride(int cols) { return (((cols + 3) / 4) | 1) * 4; }
__host__ __device__ constexpr uint32_t sub_bytes_dense(int cnt, int cols) { return ((uint32_t)sizeof(SubHead) + 4u * (uint32_t)(cnt * dense_stride(cols)) + 15u) & ~15u; }

struct alignas(16) BlkDir { // where a record is
    unsigned long long offset; // bytes from the start of the launch's region of the record buffer (a multiple of 16)
    uint32_t bytes;            // a multiple of 16; 0: no record was written
    uint32_t flags;            // bit 0: the block is walked coordinate by coordinate
};

// Kinds of data the chain kernel is instantiated for: sparse with the whole model in shared memory, with its most frequent
// ids there (kCold, kEarly, kSplit: how the others are come by); dense rows.
// kCold: the worker warps gather them behind the block's update. kEarly: before its deltas have come, and again what the update may
// have changed. kSplit: a warp of its own does. Which of them: see lookahead_plan.
constexpr int kHot = 0, kCold = 1, kDense = 2, kSplit = 3, kEarly = 4;
__host__ __device__ constexpr int chain_threads(int kind) { return kind == kSplit ? 448 : 384; }

struct LookParams {
    SolverParams S;
    unsigned char *rec;          // this launch's region of the record buffer
    BlkDir *dirS;                // C per block: the workers' records
    unsigned long long *cursor;  // bytes of the pool handed out so far in this launch
    unsigned long long *timing;  // scratch words of a -DCHICLE_LA_TIMING build
    unsigned long long pool_off; // the pool of worker records starts here (the heads lie before it, one per block)
    unsigned long long pool_cap; // bytes of the pool
    unsigned long long pool_piece; // what a CTA of the sparse prepare kernel takes of it at a time
    const int64_t *blk_base;     // K + 1: the first block of each partition in this launch's numbering of the blocks
    int32_t K, logC;
    int32_t depth;               // 2: a block's dot products are taken two blocks ahead and corrected with the cross
                                 // Gram matrix; 1: one block ahead, no cross Gram matrix (the recurrence waits for them)
    uint32_t sub_room;           // bytes of a worker record's slot in shared memory (sparse; a block that needs more is walked in place)
    int32_t slots;               // and how many slots there are (at least depth + 2)
    int32_t hotc;                // entry ids per CTA kept in shared memory
    int32_t far_cap;             // entries of a worker record that the lists of kSplit have room for (a block with more is walked in place)
    int64_t n_blocks;
    int64_t drop_block;          // test aid: this block's records are left unpublished (-1: none)
    int64_t nnz;                 // entries of the matrix (what a coordinate's extent is checked against in a debug build)
    int32_t tab_bins;            // logistic: bins per coordinate of the tables (0: the root is solved on the chain)
    unsigned long long tab_off;  // the tables start here in the region, one per block
    int32_t model_in;            // the round's first chain launch: row k of the update workspace holds U_k and is turned
                                 // into the local model w = v + sigma' U_k in place
    int32_t model_out;           // the round's last chain launch: the row is turned back into U_k. Between a round's
                                 // launches the row holds w itself: an id beyond the part in shared memory costs one
                                 // gather instead of two, and nothing is rounded from launch to launch
};

#ifdef CHICLE_LA_TIMING
#define LA_T(acc) do { asm volatile("" ::: "memory"); t1 = clock64(); asm volatile("" ::: "memory"); acc += t1 - t0; t0 = t1; } while (0)
#else
#define LA_T(acc) do { } while (0)
#endif

__device__ __forceinline__ int64_t steps_of(const LookParams &P, int64_t k, int64_t nk) { return partition_steps(P.S, k, nk); }
// (debug build) an entry id as loaded from the matrix: id 0 stands in for one outside [0, dim) (the call then ends with
// the bounds status, its arithmetic is of no interest; what matters is that nothing is addressed with the bad id)
__device__ __forceinline__ int32_t checked_id(const LookParams &P, int32_t id)
{
    return CHICLE_IN_BOUNDS(P.S.status, id >= 0 && (int64_t)id < P.S.dim) ? id : 0;
}
// The same search over a copy of blk_base in shared memory (a launch with at most kBaseStaged - 1 partitions; block
// counts fit 32 bits): the dependent loads of the search cost 30 cycles each instead of an L2 round trip.
constexpr int kBaseStaged = 132;
__device__ __forceinline__ void block_to_part_staged(const int32_t *base, int32_t K, int64_t bid, int &k, int64_t &b)
{
    int32_t lo = 0, hi = K;
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if ((int64_t)base[mid] <= bid) lo = mid;
        else hi = mid;
    }
    k = lo;
    b = bid - (int64_t)base[lo];
}
__device__ __forceinline__ void block_to_part(const LookParams &P, int64_t bid, int &k, int64_t &b)
{
    int32_t lo = 0, hi = P.K; // blk_base[lo] <= bid < blk_base[hi] (partitions may differ in size)
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (P.blk_base[mid] <= bid) lo = mid;
        else hi = mid;
    }
    k = lo;
    b = bid - P.blk_base[lo];
}

// The constants of coordinate c's scalar step (see coordinate_step), and the line A + B * dot that the recurrence's
// state starts from (what the block's earlier coordinates contribute at their round-start states is taken off A
// once the Gram triangle is known).
template <int LOSS> __device__ __forceinline__ CHdr make_hdr_of(const SolverParams &P, int32_t c, float s, float al, float y)
{
    CHdr hd;
    hd.coord = c;
    hd.lq = 0.0f;
    if (LOSS == CHICLE_LOSS_RIDGE_PRIMAL) {
        hd.p0 = P.inv_n;
        hd.p1 = al;
        hd.p2 = 1.0f / fmaf(P.sigma * s, P.inv_n, P.lambda);
        hd.p3 = P.lambda;
        hd.A = P.lambda * al;
        hd.B = P.inv_n;
    } else {
        hd.p0 = y / P.lam_n;
        hd.p1 = y * al;
        hd.p3 = y;
        if (LOSS == CHICLE_LOSS_HINGE_DUAL) {
            const bool zero = !(s > 0.0f);
            hd.p2 = zero ? CUDART_INF_F : P.lam_n / (P.sigma * s);
            // a + (1 - y dot / (lambda n)) * p2; a zero row goes to a' = 1 whatever the model is
            hd.A = zero ? 2.0f : hd.p2 + hd.p1;
            hd.B = zero ? 0.0f : -hd.p0 * hd.p2;
        } else {
            hd.p2 = P.sigma * s / P.lam_n;
            hd.lq = hd.p2 > 0.0f ? logf(hd.p2) : -CUDART_INF_F; // log q, for the start of the Newton iteration
            hd.A = hd.p2 * hd.p1;
            hd.B = -hd.p0;
        }
    }
    return hd;
}

template <int LOSS> __device__ __forceinline__ CHdr make_hdr(const SolverParams &P, int32_t c)
{
    return make_hdr_of<LOSS>(P, c, P.sqnorm[c], P.alpha[c], LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 0.0f : P.labels[c]);
}

// Loads that are issued only where `on` holds (0 elsewhere), with nothing waiting on them at the point of issue.
__device__ __forceinline__ float ldcg_if(const float *p, bool on)
{
    float v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@q ld.global.cg.f32 %0, [%1];\n\t}"
                 : "=f"(v) : "l"(p), "r"((uint32_t)on) : "memory");
    return v;
}
// The same from shared memory.
__device__ __forceinline__ float lds_f32_if(uint32_t a, bool on)
{
    float v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@q ld.shared.f32 %0, [%1];\n\t}" : "=f"(v) : "r"(a), "r"((uint32_t)on) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u32_if(uint32_t a, bool on)
{
    uint32_t v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.shared.u32 %0, [%1];\n\t}" : "=r"(v) : "r"(a), "r"((uint32_t)on) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u16_if(uint32_t a, bool on)
{
    uint32_t v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.shared.u16 %0, [%1];\n\t}" : "=r"(v) : "r"(a), "r"((uint32_t)on) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds_u8_if(uint32_t a, bool on)
{
    uint32_t v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.shared.u8 %0, [%1];\n\t}" : "=r"(v) : "r"(a), "r"((uint32_t)on) : "memory");
    return v;
}
// Atomics on shared memory, only where `on` holds (a thread's several are under way together).
__device__ __forceinline__ void red_shared_add_if(uint32_t a, int32_t v, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.shared.add.s32 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((uint32_t)on) : "memory");
}
// Two fused multiply-adds in one instruction, each rounded as usual.
__device__ __forceinline__ void fma2(float2 &acc, float ax, float ay, float bx, float by)
{
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%0, %1};\n\tfma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "+f"(acc.x), "+f"(acc.y) : "f"(ax), "f"(ay), "f"(bx), "f"(by));
}
__device__ __forceinline__ void prefetch_if(const float *p, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q prefetch.global.L2 [%0];\n\t}" ::"l"(p), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void sts_u16_if(uint32_t a, uint32_t v, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.u16 [%0], %1;\n\t}" ::"r"(a), "h"((uint16_t)v), "r"((uint32_t)on) : "memory");
}
// (the value stays where `on` does not hold)
__device__ __forceinline__ void ldcg_again_if(float &v, const float *p, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.cg.f32 %0, [%1];\n\t}" : "+f"(v) : "l"(p), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void red_shared_or_if(uint32_t a, uint32_t v, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.shared.or.b32 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void red_add_if(float *p, float v, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.global.add.f32 [%0], %1;\n\t}" ::"l"(p), "f"(v), "r"((uint32_t)on) : "memory");
}

// The recurrence in the form the chain runs it. Every loss keeps one number s_j per coordinate that is linear in the
// dot product, a scalar map s -> out, and the update s_j += Ghat[l][j] * out_l for the later coordinates j:
//   hinge     s = a + (1 - y dot / (lambda n)) * lambda n / (sigma' |x|^2), out = a' = clip(s, 0, 1)
//   logistic  s = q a - y dot / (lambda n),                                  out = a' = sigmoid(root of z + q sigmoid(z) = s)
//   ridge     s = dot / n + lambda w,                                       out = delta = -s / (sigma' |c|^2 / n + lambda)
// With dot_j = (older dot)_j + sigma' sum_l delta_l G_jl and delta_l = y_l (a'_l - a_l) this gives, for the dual
// losses, Ghat[l][j] = c_j y_l G_jl with c_j = -sigma' p2_j y_j / (lambda n) (hinge; 0 for a zero row) or
// -sigma' y_j / (lambda n) (logistic), and s_j starts sum_l Ghat[l][j] a_l lower, so that the chain adds
// Ghat * a'_l and not Ghat * (a'_l - a_l). Ridge: Ghat[l][j] = sigma' G_jl / n, nothing to take off. The prepare kernel
// stores Ghat (inside a block and from a block to the next) and the sums; a step of the chain is then: the scalar
// map, one shuffle per four coordinates, one fused multiply-add.
template <int LOSS> __device__ __forceinline__ float gram_scale(const CHdr &h, float sigma, float inv_n)
{
    if (LOSS == CHICLE_LOSS_RIDGE_PRIMAL) return sigma * inv_n;
    if (LOSS == CHICLE_LOSS_HINGE_DUAL) return h.p2 < CUDART_INF_F ? -sigma * h.p0 * h.p2 : 0.0f;
    return -sigma * h.p0;
}
template <int LOSS> __device__ __forceinline__ float recurrence_map(float s, float p2, float lq)
{
    if (LOSS == CHICLE_LOSS_RIDGE_PRIMAL) return -s * p2;
    if (LOSS == CHICLE_LOSS_HINGE_DUAL) return __saturatef(s);
    return logistic_root(s, p2, lq);
}

// ---- The logistic step from tables. a(c) = sigmoid(root of z + q sigmoid(z) = c) is a function of the state c alone once
// the coordinate's q is known, and q does not depend on the model: the prepare kernel tabulates a(c) for each of a
// block's coordinates as Taylor polynomials of degree 7, and a step of the chain is a look-up and a polynomial instead of
// a root search (two exponentials, two divisions and two reciprocals one behind the other: 510 cycles, now 119).
// a(c) is analytic but for branch points at c0 +- i pi (where 1 + q a (1 - a) = 0) and their mirror images at q - c0, and
// a(q - c) = 1 - a(c), so u = min(c, q - c) is expanded about nodes whose distance grows like the distance to c0: with
// x = (u - c0) / 3, four bins per octave of 1 + |x| on either side of c0. Below c0 the table holds a e^-u instead, which goes
// to 1, and the chain multiplies with e^u: a small a is as exact, relative to itself, as one near 1/2. Beyond x = -7 the last
// value serves (it is within 1e-9 of 1). x comes from two lines, one for c and one for q - c, so that a state near 0 is not
// rounded to the spacing of the numbers near q. Measured against the exact root, q from 0.001 to 40 000 and states from -40 on:
// the largest error of a is 1.3e-7 (logistic_root: 4.6e-7); relative to a, root mean square, 7.1e-7 below c0 and 8e-8 above
// (8.1e-7 and 2.8e-7). Polynomials of a itself below c0 and x from |c - q / 2| took 24.1 instead of 25.4 ms for a step on
// 11 M rows of 28, and left a small a wrong by up to a thousandth at e^-12, by its own size at e^-20.
constexpr int kTabNeg = 12;                // bins below c0: three octaves
constexpr float kTabScale = 3.0f;
constexpr float kTabInv = 1.0f / kTabScale;
constexpr float kTabXmin = -6.99999f;      // (1 + |x| stays inside the third octave)
__host__ __device__ constexpr uint32_t tab_bytes(int bins) { return (uint32_t)(kLB * bins) * 32u; }
// Largest q whose bins fit (u - c0 <= q / 2 - c0 and -c0 <= log(1 + q) + 1): 32 bins have five octaves above c0, 64 thirteen.
inline float tab_max_q(int bins) { return bins >= 64 ? 40000.0f : (bins >= 32 ? 160.0f : -1.0f); }

__device__ __forceinline__ float tab_center(float q)
{
    const float rt = sqrtf(fmaf(q, q, 4.0f * q));
    const float E = 2.0f / (2.0f + q + rt);
    return logf(E) - (q > 1e-12f ? 2.0f * q / (q + rt) : 0.0f);
}
// The lines: x = min(c / 3 + off, q / 3 + off - c / 3).
__device__ __forceinline__ float tab_offset(float q) { return -tab_center(q) * kTabInv; }
// q as the chain takes it: no more than keeps x inside the table (the lines meet at c = q / 2).
__device__ __forceinline__ float tab_q(float q, float off, int bins)
{
    const float top = (float)(1 << ((bins - kTabNeg) >> 2));
    return fminf(q, 2.0f * kTabScale * (top * 0.999999f - 1.0f - off));
}
// Bin i of a coordinate's table: the coefficients, in |x| - (the bin's centre), of a (x > 0) or a e^-u (x < 0).
__device__ __forceinline__ void tab_bin(float q, float log_q, int bins, int i, float4 &lo, float4 &hi)
{
    const int npos = bins - kTabNeg;
    const bool neg = i >= npos;
    const int n = neg ? i - npos : i;
    const float yc = (float)(1 << (n >> 2)) * (1.0f + ((float)(n & 3) + 0.5f) * 0.25f);
    const float step = neg ? -kTabScale : kTabScale;
    float c = fmaf(step, yc - 1.0f, tab_center(q));
    const bool flip = c > 0.5f * q;
    if (flip) c = q - c;
    // the root as in logistic_root, with a third Halley step (the coefficients inherit its error)
    const float kappa = log_q + c;
    float z = kappa <= 0.0f ? fminf(c, 0.0f) : fminf(c - (kappa - __logf(1.0f + kappa)), 0.0f);
#pragma unroll
    for (int it = 0; it < kRootIters + 1; ++it) {
        const float e = __expf(z);
        const float s = 1.0f + e, qe = q * e;
        const float A = fmaf(z - c, s, qe), B = fmaf(s, s, qe), C = qe * (1.0f - e);
        z = fminf(z - __fdividef(2.0f * A * B * s, fmaf(2.0f * B, B, -A * C)), 0.0f);
    }
    const float e = expf(z);
    // a' = p / (1 + q p) with p = a (1 - a): Taylor coefficients a_k of a, p_k of p, y_k of a' one after the other
    float a[8], p[8], y[7];
    a[0] = e / (1.0f + e);
    p[0] = a[0] * (1.0f - a[0]);
    const float r = 1.0f / fmaf(q, p[0], 1.0f);
    a[0] = fmaf(-p[0] * r, fmaf(q, a[0], z - c), a[0]); // (what rounding z to its spacing left)
    p[0] = a[0] * (1.0f - a[0]);
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        float acc = 0.0f;
#pragma unroll
        for (int m = 1; m <= k; ++m) acc = fmaf(p[m], y[k - m], acc);
        y[k] = fmaf(-q, acc, p[k]) * r;
        a[k + 1] = y[k] * (1.0f / (float)(k + 1));
        float sq = 0.0f;
#pragma unroll
        for (int m = 0; m <= k + 1; ++m) sq = fmaf(a[m], a[k + 1 - m], sq);
        p[k + 1] = a[k + 1] - sq;
    }
    if (flip) { // a(q - c) = 1 - a(c)
        a[0] = 1.0f - a[0];
        a[2] = -a[2];
        a[4] = -a[4];
        a[6] = -a[6];
    }
    if (neg) { // times e^-u: u = log a - log(1 - a) + q a, so a e^-u = (1 - a) e^(-q a); e^-u's own coefficients are (-1)^k / k!
        const float g = (1.0f - a[0]) * expf(-q * a[0]) / a[0];
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            float acc = a[k], f = 1.0f;
#pragma unroll
            for (int m = 1; m <= k; ++m) {
                f *= -1.0f / (float)m;
                acc = fmaf(a[k - m], f, acc);
            }
            a[k] = acc * g;
        }
    }
    float w = step;
#pragma unroll
    for (int k = 1; k < 8; ++k) {
        a[k] *= w;
        w *= step;
    }
    lo = make_float4(a[0], a[1], a[2], a[3]);
    hi = make_float4(a[4], a[5], a[6], a[7]);
}
// A block's table (all threads of the CTA; hdr: its coordinates' constants).
__device__ __forceinline__ void write_table(const LookParams &P, int64_t bid, const CHdr *hdr, int threads)
{
    float4 *out = reinterpret_cast<float4 *>(P.rec + P.tab_off + (size_t)bid * tab_bytes(P.tab_bins));
    const int bins = P.tab_bins, lg = bins >= 64 ? 6 : 5;
    for (int i = threadIdx.x; i < kLB << lg; i += threads) {
        const float q = hdr[i >> lg].p2;
        float4 lo, hi;
        tab_bin(q, q > 0.0f ? __logf(q) : -CUDART_INF_F, bins, i & (bins - 1), lo, hi);
        out[2 * i] = lo;
        out[2 * i + 1] = hi;
    }
}
// a(c) from the table, as sgn * v + bias: the caller multiplies sgn into what a(c) is multiplied with next while the look-up is
// under way (e^u, too, is ready before the polynomial is). q, off, off2 (= q / 3 + off): see tab_q and tab_offset; `row`: where the
// coordinate's table would have a bin of exponent 0; `on`: whether this lane's result is wanted (the other lanes keep off the shared-memory
// pipe).
__device__ __forceinline__ float tab_map(float c, float q, float off, float off2, uint32_t row, uint32_t neg, bool on, float4 &lo, float4 &hi, float &sgn, float &bias)
{
    const float x = fmaxf(fminf(fmaf(c, kTabInv, off), fmaf(c, -kTabInv, off2)), kTabXmin);
    const float t = q - c, u = fminf(c, t);
    const float ax = fabsf(x), y = 1.0f + ax;
    const uint32_t bits = __float_as_uint(y);
    const uint32_t at = ((bits & 0xffe00000u) >> 16) + (x < 0.0f ? row + neg : row); // 32 bytes a bin
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t"
                 "@q ld.shared.v4.f32 {%0, %1, %2, %3}, [%8];\n\t@q ld.shared.v4.f32 {%4, %5, %6, %7}, [%8 + 16];\n\t}"
                 : "+f"(lo.x), "+f"(lo.y), "+f"(lo.z), "+f"(lo.w), "+f"(hi.x), "+f"(hi.y), "+f"(hi.z), "+f"(hi.w)
                 : "r"(at), "r"((uint32_t)on));
    float eu;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(eu) : "f"(u * 1.4426950409f));
    eu = x < 0.0f ? eu : 1.0f;
    sgn = t < c ? -eu : eu;
    // (a state that is not finite gives a result that is not, as the root search would)
    bias = fmaf(0.0f, c, t < c ? 1.0f : 0.0f);
    const float dl = ax - (__uint_as_float((bits & 0xffe00000u) | 0x00100000u) - 1.0f);
    const float d2 = dl * dl, d4 = d2 * d2;
    const float p01 = fmaf(lo.y, dl, lo.x), p23 = fmaf(lo.w, dl, lo.z), p45 = fmaf(hi.y, dl, hi.x), p67 = fmaf(hi.w, dl, hi.z);
    return fmaf(fmaf(p67, d2, p45), d4, fmaf(p23, d2, p01));
}

// The most frequent ids (ids are frequency-ranked) are in most of a block's coordinates. Their part of the Gram
// matrices is taken from dense 32 x kHD tiles; only the other entries are walked through the table.
constexpr int kHD = 32;
constexpr int kHDS = kHD + 4; // row stride of the tiles: 16-byte loads of consecutive rows fall on different banks
// Table slots: the ids below kDir have their own (no key, no tries); HT hashed ones behind them for the others.
// (As many as shared memory leaves: at two CTAs per SM nothing is free.)
constexpr int kDir = 768;
// Hashed slots: HT of them, a power of two; the t-th try lies t places behind the one before, which reaches every one.
template <int HT> __device__ __forceinline__ uint32_t home_place(int32_t id) { return __umulhi((uint32_t)id * 2654435761u, (uint32_t)HT); }
template <int HT> __device__ __forceinline__ uint32_t next_place(uint32_t p, int t) { return (p + (uint32_t)t) & (uint32_t)(HT - 1); }
// entries that a block may have: the arrays', and slots for their ids if none is shared
__host__ __device__ constexpr int pre_room(int nz, int ht) { return nz < ht - kHD ? nz : ht - kHD; }

// ------------------------------------------------------------------------------------------------ prepare
// A CTA takes a run of consecutive blocks, so that a block's rows are fetched once: they serve as the next block of the
// one before (cross Gram matrix) and then as the block itself. All fetches are asynchronous copies into shared memory and
// run ahead of their use: while block b is worked on, the rows of b + 1, the row extents and constants of b + 2 and the
// visiting-order entries of b + 3 are under way. Passes over the block's non-zeros take them as one flat array (32 at a
// time whatever the rows' lengths).
// What bounds it is the number of instructions and shared-memory turns (each at 55 to 60 % of what the SM can do), and the barriers
// between the phases; before (a CTA per block, each fetching its own rows and its successor's in three dependent round trips) a
// block of 1 600 non-zeros took 63 000 cycles at three CTAs per SM. Rows of 50 on 1 M coordinates, a slice of 4 096 blocks on the whole
// GPU: 255 us; with slots without tries for frequent ids, entries' findings kept in registers, one atomic per numbered id and the
// pairs shared out evenly 225 us (instructions a block 40 700 -> 35 200); step 4.01 -> 3.59 ms, ridge 12.5 -> 11.1 (longer blocks
// have more tries to save). Rows fetched two pieces at a time, the dense part in front of the last barrier and without its cross half
// where there is no cross Gram matrix, the next constants beside the records' places: 216 us; 3.60 -> 3.45 ms. A thread's several entries together, all loads first: 46 100 instructions, 272 us. 640, 448, 416
// or 384 threads instead of 512: 254, 241, 244 and 250 us.
constexpr int kDirNew = 4; // (metadata slots: a power of two)

// One block's coordinates as the kernel keeps them: constants of the steps and extents of the rows.
struct PreBlock {
    CHdr hdr[kLB];
    int64_t rs[kLB];
    int32_t nnz[kLB];
    int32_t roff[kLB + 1];            // where each coordinate's entries start in the flat array ([32] = all of them)
    float gsc[kLB], ys[kLB], as[kLB]; // per coordinate: its Gram scale, and what multiplies / enters from the earlier ones
    float scl[kLB], inv[kLB];         // a power of two that brings the values below 2^15 (see pre_pairs), and its inverse
    int32_t k, cnt, total, over;      // partition; over: more non-zeros than the arrays hold (total is 0 then): walked in place
};

// The shared ids of a CTA of the cluster, counted while they are numbered: list entries, ids with up to four of them, ids with
// more. One word holds all three where the arrays are small (one atomic per id); else the short lists have their own.
template <int NZ> struct PreCount {
    static constexpr bool kOne = NZ <= 2048;
    static constexpr int kLongBit = kOne ? 23 : 16;
    static_assert(!kOne || (NZ < 1 << 12 && NZ / 2 < 1 << 11 && NZ / 5 < 1 << 9), "the fields of the one word");
    static_assert(NZ <= 4096, "the fields of two words");
    __device__ static uint32_t entries(uint32_t w) { return kOne ? w & 0xfffu : w & 0xffffu; }
    __device__ static uint32_t longs(uint32_t w) { return w >> kLongBit; }
    __device__ static uint32_t shorts(uint32_t w, uint32_t s) { return kOne ? (w >> 12) & 0x7ffu : s; }
};
// A CTA's record of the block: where its parts are (bytes behind the head), and where its lists start in lval.
struct alignas(16) PreRec {
    unsigned long long at; // from the start of the region
    uint32_t meta, ids;
    uint32_t lval, lst, lrow;
    uint16_t base, longs;
};

template <int NZ, int HT, int THREADS> struct PreShared {
    static constexpr int CH = NZ / 32;  // chunks of 32 entries
    static constexpr int TS = kDir + HT; // table slots
    alignas(16) int32_t key[HT];        // id in a hashed slot, -1 = empty
    alignas(16) uint32_t mask[TS];      // bit j: coordinate j of the block has this id
    uint16_t lists[TS];                   // one coordinate has the id: its entry; several: where the id's list starts among those of its CTA (12 bits), CTA
    alignas(128) int32_t idx[2][NZ];    // the block's entries, and the next block's
    float val[3][NZ];                   // [2]: the scaled values of shared ids, one list per id, each in ascending coordinate order
    uint8_t row[3][NZ];                 // coordinate of each entry
    uint32_t bal[2][CH + 1][kMaxC];     // per chunk and CTA: which of the entries fall to it
    uint16_t pre[2][CH + 1][kMaxC];     // and how many before the chunk
    alignas(128) int32_t G[2][kLB][kLB]; // Gram triangle and cross Gram matrix, fixed point (the low words lie in idx, see pre_pairs)
    uint32_t work[THREADS / 32][3 * 32]; // per warp: entries whose pairs are still to be added; then its sums for A and q0n
    alignas(16) float D[2][kLB][kHDS];  // the entries with the kHD most frequent ids, dense
    PreBlock blk[kDirNew];
    int32_t coord[kDirNew][kLB];        // visiting-order entries
    int64_t ip[2][kLB];                 // fetched for a block: row extents, squared norms, states, labels
    float sq[kLB], al[kLB], lb[kLB];
    uint16_t rc[kLB + 1][kMaxC];        // where coordinate j's entries start in CTA c's record
    uint32_t cnt[kMaxC], cntShort[kMaxC]; // per CTA: its shared ids, see PreCount
    PreRec rec[kMaxC];
    int32_t walk;
    unsigned long long pool_at, pool_end; // what this CTA holds of the pool
    int32_t base[kBaseStaged];          // blk_base, and first step and step count of each partition (see pre_locate)
    int64_t off[kBaseStaged];
    int32_t steps[kBaseStaged];
};

// Where block x of the launch lies: partition, first step in the visiting-order array, steps in the block.
struct PrePlace {
    int32_t k;
    int64_t at;
    int32_t cnt;
};
template <class Shared> __device__ __forceinline__ PrePlace pre_locate(const LookParams &P, const Shared &sh, int64_t x)
{
    PrePlace r;
    int k;
    int64_t b, off, steps;
    if (P.K < kBaseStaged) {
        block_to_part_staged(sh.base, P.K, x, k, b);
        off = sh.off[k];
        steps = sh.steps[k];
    } else {
        block_to_part(P, x, k, b);
        off = P.S.part_off[k] + (P.S.first_k ? P.S.first_k[k] : 0);
        steps = steps_of(P, k, P.S.part_off[k + 1] - P.S.part_off[k]);
    }
    r.k = k;
    r.at = off + b * kLB;
    const int64_t left = steps - b * kLB;
    r.cnt = (int32_t)(left < kLB ? left : kLB);
    return r;
}

__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

// The three stages of a block's fetches (a warp each; the caller waits for the copies and meets the other threads).
template <class Shared> __device__ __forceinline__ void pre_fetch_order(const LookParams &P, Shared &sh, int64_t x)
{
    const int lane = threadIdx.x & 31;
    const PrePlace pl = pre_locate(P, sh, x);
    if (lane < pl.cnt) cp_async4(smem_u32(&sh.coord[x & (kDirNew - 1)][lane]), P.S.perm + pl.at + lane);
    else sh.coord[x & (kDirNew - 1)][lane] = -1;
    if (lane == 0) {
        sh.blk[x & (kDirNew - 1)].cnt = pl.cnt;
        sh.blk[x & (kDirNew - 1)].k = pl.k;
    }
}
template <int LOSS, class Shared> __device__ __forceinline__ void pre_fetch_extents(const LookParams &P, Shared &sh, int64_t x)
{
    const int lane = threadIdx.x & 31;
    int32_t c = sh.coord[x & (kDirNew - 1)][lane];
    if (c >= 0 && !CHICLE_IN_BOUNDS(P.S.status, (int64_t)c < P.S.n_coord)) c = 0;
    if (c < 0) return;
    cp_async8(smem_u32(&sh.ip[0][lane]), P.S.indptr + c);
    cp_async8(smem_u32(&sh.ip[1][lane]), P.S.indptr + c + 1);
    cp_async4(smem_u32(&sh.sq[lane]), P.S.sqnorm + c);
    cp_async4(smem_u32(&sh.al[lane]), P.S.alpha + c);
    if (LOSS != CHICLE_LOSS_RIDGE_PRIMAL) cp_async4(smem_u32(&sh.lb[lane]), P.S.labels + c);
}
// (a warp: what was fetched for block x becomes its PreBlock)
template <int LOSS, int NZ, int HT, class Shared> __device__ __forceinline__ void pre_make_block(const LookParams &P, Shared &sh, int64_t x)
{
    const int lane = threadIdx.x & 31;
    PreBlock &B = sh.blk[x & (kDirNew - 1)];
    int32_t c = sh.coord[x & (kDirNew - 1)][lane];
    if (c >= 0 && !CHICLE_IN_BOUNDS(P.S.status, (int64_t)c < P.S.n_coord)) c = 0;
    CHdr hd{0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int64_t rs = 0;
    int32_t n = 0;
    if (c >= 0) {
        rs = sh.ip[0][lane];
        const int64_t len = sh.ip[1][lane] - rs;
        n = (int32_t)len;
        if (!CHICLE_IN_BOUNDS(P.S.status, rs >= 0 && len >= 0 && len <= 0x7fffffff && rs + len <= P.nnz)) { rs = 0; n = 0; }
        hd = make_hdr_of<LOSS>(P.S, c, sh.sq[lane], sh.al[lane], LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 0.0f : sh.lb[lane]);
        if (LOSS == CHICLE_LOSS_LOGISTIC_DUAL && P.tab_bins) hd.lq = tab_offset(hd.p2);
    }
    B.hdr[lane] = hd;
    B.rs[lane] = rs;
    B.nnz[lane] = n;
    B.gsc[lane] = c >= 0 ? gram_scale<LOSS>(hd, P.S.sigma, P.S.inv_n) : 0.0f;
    B.ys[lane] = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 1.0f : hd.p3;
    B.as[lane] = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 0.0f : hd.p1;
    {
        // |x| < 2^e for e = (exponent of |x|^2 + 2) / 2, rounded down (subnormal squares: the exponent of their first bit)
        const uint32_t bits = c >= 0 ? __float_as_uint(sh.sq[lane]) : 0u;
        const int ex = bits >> 23 ? (int)(bits >> 23) - 127 : -118 - __clz((int)bits), e = (ex + 2) >> 1;
        const bool usable = bits != 0u && ex < 128;
        B.scl[lane] = usable ? __uint_as_float((uint32_t)(127 + 15 - e) << 23) : 0.0f;
        B.inv[lane] = usable ? __uint_as_float((uint32_t)(127 - 15 + e) << 23) : 0.0f;
    }
    constexpr int room = pre_room(NZ, HT);
    // (a low word of the Gram matrices takes as many terms of 2^19 at most, see pre_pairs)
    static_assert((int64_t)room << 19 < (int64_t)1 << 31, "the low words' range");
    const int m = n < room + 1 ? n : room + 1; // (more than the arrays hold is all that matters of a longer one)
    int incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const int tot = __shfl_sync(0xffffffffu, incl, 31);
    const bool over = tot > room;
    B.roff[lane] = over ? 0 : incl - m;
    if (lane == 31) {
        B.roff[kLB] = over ? 0 : incl;
        B.total = over ? 0 : incl;
        B.over = over ? 1 : 0;
    }
}
// (all warps: the rows of a block into buffer `buf`; the caller waits)
template <int NZ, int THREADS, class Shared> __device__ __forceinline__ void pre_fetch_rows(const LookParams &P, Shared &sh, int64_t x, int buf)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const PreBlock &B = sh.blk[x & (kDirNew - 1)];
    if (B.over) return;
    for (int j = warp; j < kLB; j += THREADS / 32) {
        const int n = B.nnz[j], r0 = B.roff[j];
        const int32_t *ix = P.S.indices + B.rs[j] + lane;
        const float *xv = P.S.values + B.rs[j] + lane;
        const uint32_t di = smem_u32(&sh.idx[buf][r0 + lane]), dv = smem_u32(&sh.val[buf][r0 + lane]);
        uint8_t *dr = &sh.row[buf][r0 + lane];
#pragma unroll 1
        for (int e = 0; e < n; e += 64)
#pragma unroll
            for (int u = 0; u < 64; u += 32)
                if (e + u + lane < n) {
                    cp_async4(di + 4u * (uint32_t)(e + u), ix + e + u);
                    cp_async4(dv + 4u * (uint32_t)(e + u), xv + e + u);
                    dr[e + u] = (uint8_t)j;
                }
    }
}
// (a warp: which of 32 consecutive entries fall to which CTA, and their part of the dense tile; id < 0: no entry. flip: per bit of a CTA's
// number, all ones where this lane's number has a 0 there)
template <class Shared> __device__ __forceinline__ void pre_classify(const LookParams &P, Shared &sh, int32_t id, int e, int buf, const uint32_t (&flip)[3])
{
    const int lane = threadIdx.x & 31;
    uint32_t mine = __ballot_sync(0xffffffffu, id >= 0);
#pragma unroll
    for (int bit = 0; bit < 3; ++bit)
        if (bit < P.logC) mine &= __ballot_sync(0xffffffffu, (id & (1 << bit)) != 0) ^ flip[bit];
    if (lane >> P.logC == 0) sh.bal[buf][e >> 5][lane] = mine; // lane c: the entries of CTA c
    if ((uint32_t)id < (uint32_t)kHD) sh.D[buf][sh.row[buf][e]][id] = sh.val[buf][e];
}
// (warp c: how many of the entries before each chunk fall to CTA c)
template <class Shared> __device__ __forceinline__ void pre_prefix(Shared &sh, int total, int buf, int c)
{
    const int lane = threadIdx.x & 31;
    const int nch = (total + 31) >> 5;
    int run = 0;
    for (int b = 0; b <= nch; b += 32) {
        const int ch = b + lane;
        const int x = ch < nch ? __popc(sh.bal[buf][ch][c]) : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (ch <= nch) sh.pre[buf][ch][c] = (uint16_t)(run + incl - x);
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// The Gram matrices' entries come from two sources. The kHD most frequent ids: dense 32 x kHD tiles (pre_rows). All others:
// an id that c coordinates have contributes c (c - 1) / 2 products, about 550 per block inside a block of 1 600 entries and
// 1 300 to the cross Gram matrix: they are added one by one with shared-memory atomics, in fixed point, so that the sum
// does not depend on the order. Values are scaled by a power of two below 2^15 / |x| (exact), a product is below 2^30 and
// so is every partial sum of an entry (|sum| <= |x_l| |x_j|); what rounding a product to a whole number leaves goes to a second
// word, 2^20 times finer: together finer than an fp32 sum is.
// (Walking lists with shuffles in a fixed order took 14 000 of 31 000 cycles a block; a lane per entry, whose loops last as long as the
// longest of 32, 7 500 instructions a block of 1 600 entries, against 1 500 with the pairs shared out.)
// Entry (l, j) of a matrix lies at place l ^ j of row j: the 32 entries whose pairs a warp adds together come from one or two
// coordinates j and have any l, so its atomics fall on different banks.
__device__ __forceinline__ int gram_place(int l, int j) { return j * kLB + (l ^ j); }
// A warp takes 32 entries with pairs at a time and shares their pairs out evenly: pair t of the 32 entries' belongs to the last
// entry whose pairs start at or before t.
template <int NZ, class Shared>
__device__ __forceinline__ void pre_pairs(Shared &sh, uint32_t item, bool on, int cur, const PreBlock &N)
{
    const int lane = threadIdx.x & 31;
    int n = 0;          // pairs of this lane's entry
    uint32_t with = 0u; // where the values and coordinates are that it is paired with (as an index of val[0], row[0])
    uint32_t to = 0u;   // row of G (next, j), and j
    float x = 0.0f;
    if (on) {
        const int e = (int)(item & 4095u), p = (int)((item >> 12) & 8191u), next = (int)(item >> 25);
        const int buf = cur ^ next, j = sh.row[buf][e], off = sh.lists[p];
        uint32_t m = sh.mask[p];
        with = (m & (m - 1u)) == 0u ? (uint32_t)(cur * NZ + off) : (uint32_t)(2 * NZ + sh.rec[off >> 12].base + (off & 4095));
        x = sh.val[buf][e];
        if (next) x *= N.scl[j];
        else m &= (1u << j) - 1u;
        n = __popc(m);
        to = (uint32_t)(next * kLB * kLB + j * kLB + j) * 4u; // (its place for l = 0; the others by the bits of 4 l)
    }
    int start = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, start, o);
        if (lane >= o) start += t;
    }
    const int all = __shfl_sync(0xffffffffu, start, 31);
    start -= n;
    with -= (uint32_t)start; // (of the pair t: with + t)
    const uint32_t hi = smem_u32(&sh.G[0][0][0]), lo = smem_u32(&sh.idx[cur][0]), val0 = smem_u32(&sh.val[0][0]), row0 = smem_u32(&sh.row[0][0]);
    int before = -1;    // entries that start before the 32 pairs, less one
#pragma unroll 1
    for (int t0 = 0; t0 < all; t0 += 32) {
        const uint32_t at = (uint32_t)(start - t0);
        const uint32_t starts = __reduce_or_sync(0xffffffffu, n > 0 && at < 32u ? 1u << at : 0u);
        const int from = before + __popc(starts & (0xffffffffu >> (31 - lane)));
        before += __popc(starts);
        const uint32_t u = __shfl_sync(0xffffffffu, with, from) + (uint32_t)(t0 + lane);
        const uint32_t g = __shfl_sync(0xffffffffu, to, from);
        const float y = __shfl_sync(0xffffffffu, x, from);
        if (t0 + lane < all) {
            const float v = lds_f32(val0 + 4u * u) * y;
            const uint32_t word = g ^ (4u * lds_u8_if(row0 + u, true));
            const int h = __float2int_rn(v), r = __float2int_rn((v - (float)h) * 1048576.0f);
            red_shared_add_if(hi + word, h, true);
            red_shared_add_if(lo + word, r, r != 0);
        }
    }
}

// (a warp: the pairs of `have` listed entries)
template <int NZ, class Shared>
__device__ __forceinline__ void pre_listed(Shared &sh, int have, int cur, const PreBlock &N)
{
    const uint32_t *todo = sh.work[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int at = 0; at < have; at += 32) pre_pairs<NZ>(sh, at + lane < have ? todo[at + lane] : 0u, at + lane < have, cur, N);
    __syncwarp();
}
// (not inlined: a list longer than usual between its parts, 32 at a time from its end; what is left)
template <int NZ, class Shared>
__device__ __noinline__ int pre_listed_early(Shared &sh, int have, int cur, const PreBlock &N)
{
    for (; have > 32; have -= 32) pre_pairs<NZ>(sh, sh.work[threadIdx.x >> 5][have - 32 + (threadIdx.x & 31)], true, cur, N);
    __syncwarp();
    return have;
}

// What the states at round start contribute: the warps' sums (sh.work) together, off A and into q0n; the block's constants
// go out. (A warp; one block behind the loop, so that it needs no barrier of its own.)
template <int NW, class Shared> __device__ __forceinline__ void pre_finish_head(const LookParams &P, Shared &sh, int64_t bid)
{
    const int lane = threadIdx.x & 31;
    ChainHead &out = *reinterpret_cast<ChainHead *>(P.rec + (size_t)bid * sizeof(ChainHead));
    float qg = 0.0f, qx = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        qg += __uint_as_float(sh.work[w][lane]);
        qx += __uint_as_float(sh.work[w][32 + lane]);
    }
    CHdr hd = sh.blk[bid & (kDirNew - 1)].hdr[lane];
    hd.A -= qg;
    out.hdr[lane] = hd;
    out.q0n[lane] = qx;
}

template <int LOSS, int NZ, int HT, int THREADS, int PER_SM>
__global__ void __launch_bounds__(THREADS, PER_SM) k_lookahead_prepare(const LookParams P)
{
    extern __shared__ __align__(128) unsigned char smem_pre[];
    using Shared = PreShared<NZ, HT, THREADS>;
    Shared &sh = *reinterpret_cast<Shared *>(smem_pre);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int NW = THREADS / 32, EPT = NZ / THREADS;
    static_assert(NZ % THREADS == 0 && NW >= 8, "entries per thread; a warp per CTA of the cluster");
    const int C = 1 << P.logC;
    const int64_t hot_all = (int64_t)P.hotc << P.logC;
    const uint32_t hot_total = (uint32_t)(hot_all < P.S.dim ? hot_all : P.S.dim);
    const int64_t lo = P.n_blocks * (int64_t)blockIdx.x / gridDim.x, hi = P.n_blocks * ((int64_t)blockIdx.x + 1) / gridDim.x;
    if (lo >= hi) return;
    if (P.K < kBaseStaged)
        for (int i = tid; i <= P.K; i += THREADS) {
            sh.base[i] = (int32_t)P.blk_base[i];
            if (i < P.K) {
                sh.off[i] = P.S.part_off[i] + (P.S.first_k ? P.S.first_k[i] : 0);
                sh.steps[i] = (int32_t)steps_of(P, i, P.S.part_off[i + 1] - P.S.part_off[i]);
            }
        }
    for (int p = tid; p < HT; p += THREADS) sh.key[p] = -1;
    for (int p = tid; p < Shared::TS; p += THREADS) sh.mask[p] = 0u;
    for (int p = tid; p < 2 * kLB * kHDS; p += THREADS) (&sh.D[0][0][0])[p] = 0.0f;
    if (tid < kMaxC) sh.cnt[tid] = sh.cntShort[tid] = 0u;
    if (tid == 0) sh.pool_at = sh.pool_end = 0ull;
    __syncthreads();
    const uint32_t flip[3] = {lane & 1 ? 0u : ~0u, lane & 2 ? 0u : ~0u, lane & 4 ? 0u : ~0u};
    // blocks that are fetched: the run, and the one behind it where the last block has a cross Gram matrix with it
    int64_t end = hi;
    if (P.depth >= 2 && hi < P.n_blocks && pre_locate(P, sh, hi).k == pre_locate(P, sh, hi - 1).k) end = hi + 1;
    if (warp < 3 && lo + warp < end) pre_fetch_order(P, sh, lo + warp);
    cp_async_wait_all();
    __syncthreads();
    if (warp == 0)
        for (int64_t x = lo; x < end && x < lo + 2; ++x) {
            pre_fetch_extents<LOSS>(P, sh, x);
            cp_async_wait_all();
            __syncwarp();
            pre_make_block<LOSS, NZ, HT>(P, sh, x);
            __syncwarp();
        }
    __syncthreads();
    pre_fetch_rows<NZ, THREADS>(P, sh, lo, (int)(lo & 1));
    cp_async_wait_all();
    __syncthreads();
    for (int e = tid; (e & ~31) < sh.blk[lo & (kDirNew - 1)].total; e += THREADS)
        pre_classify(P, sh, e < sh.blk[lo & (kDirNew - 1)].total ? checked_id(P, sh.idx[lo & 1][e]) : -1, e, (int)(lo & 1), flip);
    __syncthreads();
    if (warp < C) pre_prefix(sh, sh.blk[lo & (kDirNew - 1)].total, (int)(lo & 1), warp);
    __syncthreads();
#ifdef CHICLE_LA_TIMING
    long long pt0 = clock64(), pt1 = 0;
#define PRE_T(i) do { asm volatile("" ::: "memory"); pt1 = clock64(); if (tid == 0) atomicAdd(P.timing + 16 + (i), (unsigned long long)(pt1 - pt0)); pt0 = pt1; asm volatile("" ::: "memory"); } while (0)
#else
#define PRE_T(i) do { } while (0)
#endif

#pragma unroll 1
    for (int64_t bid = lo; bid < hi; ++bid) {
        const int cur = (int)(bid & 1), nxt = cur ^ 1;
        PreBlock &B = sh.blk[bid & (kDirNew - 1)];
        const PreBlock &N = sh.blk[(bid + 1) & (kDirNew - 1)];
        const bool have_next = bid + 1 < end;
        const int total = B.total, cnt = B.cnt;
        ChainHead &out = *reinterpret_cast<ChainHead *>(P.rec + (size_t)bid * sizeof(ChainHead));
        // ---- fetches for the blocks ahead
        if (have_next) pre_fetch_rows<NZ, THREADS>(P, sh, bid + 1, nxt);
        if (warp == NW - 1 && bid + 2 < end) pre_fetch_extents<LOSS>(P, sh, bid + 2);
        if (warp == NW - 2 && bid + 3 < end) pre_fetch_order(P, sh, bid + 3);
        for (int p = tid; p < kLB * kHDS / 4; p += THREADS) reinterpret_cast<float4 *>(&sh.D[nxt][0][0])[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p = tid; p < 2 * kLB * kLB / 4; p += THREADS) reinterpret_cast<int4 *>(&sh.G[0][0][0])[p] = make_int4(0, 0, 0, 0);
        if (warp == NW - 4 && bid > lo) pre_finish_head<NW>(P, sh, bid - 1);
        // ---- every id into the table. What a thread has found out about its entries stays in registers for the whole block:
        //      id, table slot, coordinate, mask of the coordinates that have the id. (32 entries of a warp after the other, and not a
        //      thread's several together: what bounds this kernel is the number of instructions.)
        int32_t id[EPT];
        uint32_t slot[EPT], m[EPT]; // (slot: its coordinate in the high half)
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            const int e = tid + i * THREADS;
            id[i] = e < total ? checked_id(P, sh.idx[cur][e]) : -1;
            slot[i] = m[i] = 0u;
        }
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            if ((tid & ~31) + i * THREADS >= total) break; // (whole warps)
            uint32_t p = (uint32_t)id[i];
            if (id[i] >= kDir) {
                p = home_place<HT>(id[i]);
                for (int t = 1; t <= HT; ++t) {
                    const int32_t seen = atomicCAS(&sh.key[p], -1, id[i]);
                    if (seen == -1 || seen == id[i]) break;
                    p = next_place<HT>(p, t);
                }
                p += kDir;
            }
            const uint32_t j = sh.row[cur][tid + i * THREADS];
            if (id[i] >= 0) atomicOr(&sh.mask[p], 1u << j);
            slot[i] = (p & 0xffffu) | j << 16;
        }
        // where each coordinate's entries start in each CTA's record
        for (int i = tid; i < (kLB + 1) << P.logC; i += THREADS) {
            const int j = i >> P.logC, c = i & (C - 1), at = B.roff[j], ch = at >> 5;
            sh.rc[j][c] = (uint16_t)(sh.pre[cur][ch][c] + __popc(sh.bal[cur][ch][c] & ((1u << (at & 31)) - 1u)));
        }
        __syncthreads();
        PRE_T(0);
        // ---- the first coordinate that has an id numbers it, if others have it too: its place among its CTA's lists. (The order of
        //      the numbers varies from run to run, which moves records' contents about but changes no result: every id's own sum
        //      is taken in coordinate order, in a shape that depends on the list's length alone.)
        using Count = PreCount<NZ>;
        uint32_t tl[EPT]; // of an id numbered here: where its list starts (low half), its number among the long or the short ones; else all ones
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            tl[i] = 0xffffffffu;
            if ((tid & ~31) + i * THREADS >= total) break;
            if (id[i] < 0) continue;
            const uint32_t p = slot[i] & 0xffffu;
            m[i] = sh.mask[p];
            if ((m[i] & ((1u << (slot[i] >> 16)) - 1u)) != 0u) continue;
            uint32_t off = (uint32_t)(tid + i * THREADS);
            if ((m[i] & (m[i] - 1u)) != 0u) {
                const uint32_t c = (uint32_t)id[i] & (uint32_t)(C - 1), n = (uint32_t)__popc(m[i]);
                const uint32_t w = atomicAdd(&sh.cnt[c], n + (n > 4u ? 1u << Count::kLongBit : (Count::kOne ? 1u << 12 : 0u)));
                const uint32_t s = !Count::kOne && n <= 4u ? atomicAdd(&sh.cntShort[c], 1u) : 0u;
                off = Count::entries(w) | c << 12;
                tl[i] = Count::entries(w) | (n > 4u ? Count::longs(w) : Count::shorts(w, s)) << 16;
            }
            sh.lists[p] = (uint16_t)off;
        }
        for (int p = tid; p < NZ / 4; p += THREADS) reinterpret_cast<int4 *>(&sh.idx[cur][0])[p] = make_int4(0, 0, 0, 0); // (from here on: the low words of the Gram matrices)
        cp_async_wait_all(); // the next block's rows, the extents after it, the order after that
        __syncthreads();
        PRE_T(1);
        // ---- the records' places: the head has its own (one per block); the workers' records come from the pool, of which
        //      a CTA takes a piece for several blocks at a time. A block that the pool has no room for is walked in place
        //      like one that is too long. (A warp. Meanwhile another one: the constants of the block after the next; and all: the
        //      next block's entries, which CTA's they are, and their dense tile.)
        if (warp == 0) { // (a lane per CTA of the cluster)
            const bool in = lane < C;
            const uint32_t n_c = in ? sh.rc[kLB][lane] : 0u, w = in ? sh.cnt[lane] : 0u;
            const uint32_t lng = Count::longs(w), T_c = lng + Count::shorts(w, in ? sh.cntShort[lane] : 0u), nl_c = Count::entries(w);
            const uint32_t len = in ? sub_bytes(n_c, T_c, nl_c) : 0u;
            uint32_t incl = len, lists = nl_c;
#pragma unroll
            for (int o = 1; o < kMaxC; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o), z = __shfl_up_sync(0xffffffffu, lists, o);
                if (lane >= o) { incl += y; lists += z; }
            }
            const uint32_t need = __shfl_sync(0xffffffffu, incl, kMaxC - 1);
            // 1: longer than the arrays, or more falls to one CTA than its record holds
            int sl = B.over || __any_sync(0xffffffffu, len > P.sub_room || n_c > (uint32_t)P.far_cap) ? 1 : 0;
            unsigned long long at = sh.pool_at, pool_end = sh.pool_end;
            if (!sl && at + need > pool_end) {
                const unsigned long long take = need > P.pool_piece ? need : P.pool_piece;
                if (lane == 0) at = atomicAdd(P.cursor, take);
                at = __shfl_sync(0xffffffffu, at, 0);
                pool_end = at + take < P.pool_cap ? at + take : P.pool_cap;
                if (at + need > P.pool_cap) { sl = 2; pool_end = 0ull; }
            }
            if (sl && lane == 0) atomicAdd(P.S.status + kStatusWalked, 1u);
            if (in) {
                BlkDir d; // nothing to stage: the workers copy the first bytes of the head instead
                d.offset = sl ? (unsigned long long)bid * sizeof(ChainHead) : P.pool_off + at + (incl - len);
                d.bytes = bid == P.drop_block ? 0u : (sl ? 16u : len);
                d.flags = sl ? 1u : 0u;
                P.dirS[bid * C + lane] = d;
                PreRec r;
                r.at = d.offset;
                r.meta = 4u * n_c;
                r.ids = 8u * n_c;
                r.lval = r.ids + 4u * T_c;
                r.lst = r.lval + 4u * nl_c;
                r.lrow = r.lst + 2u * T_c;
                r.base = (uint16_t)(lists - nl_c);
                r.longs = (uint16_t)lng;
                sh.rec[lane] = r;
                if (!sl) *reinterpret_cast<int4 *>(P.rec + d.offset) = make_int4((int)n_c, (int)T_c, (int)nl_c, cnt);
            }
            __syncwarp();
            if (lane == 0) {
                sh.walk = sl;
                sh.pool_at = sl ? at : at + need;
                sh.pool_end = pool_end;
                *reinterpret_cast<int4 *>(&out) = make_int4(cnt, sl ? 1 : 0, 0, 0);
            }
        }
        if (warp == NW - 1 && bid + 2 < end) pre_make_block<LOSS, NZ, HT>(P, sh, bid + 2);
        const int ntotal = have_next ? N.total : 0;
        int32_t nid[EPT];
#pragma unroll
        for (int i = 0; i < EPT; ++i) {
            const int e = tid + i * THREADS;
            nid[i] = e < ntotal ? checked_id(P, sh.idx[nxt][e]) : -1;
        }
#pragma unroll
        for (int i = 0; i < EPT; ++i)
            if (((tid + i * THREADS) & ~31) < ntotal) pre_classify(P, sh, nid[i], tid + i * THREADS, nxt, flip); // (whole warps)
        __syncthreads();
        PRE_T(2);
        const bool walk = sh.walk != 0;
        const bool carry = have_next && !walk && !N.over && P.depth >= 2 && B.k == N.k;
        if (!walk) {
            if (LOSS == CHICLE_LOSS_LOGISTIC_DUAL && P.tab_bins) write_table(P, bid, B.hdr, THREADS);
            // ---- the workers' records: where each coordinate's entries start, and the entries, row after row: place = entries of that
            //      CTA before this one; a shared id's place in its list is the number of lower coordinates that have the id
            for (int i = tid; i < C * (kLB + 8); i += THREADS) {
                const int c = i / (kLB + 8), j = i - c * (kLB + 8);
                reinterpret_cast<SubHead *>(P.rec + sh.rec[c].at)->roff[j] = sh.rc[j < kLB ? j : kLB][c];
            }
#pragma unroll
            for (int i = 0; i < EPT; ++i) {
                const int e = tid + i * THREADS;
                if ((tid & ~31) + i * THREADS >= total) break;
                if (id[i] < 0) continue;
                const int cls = id[i] & (C - 1), j = (int)(slot[i] >> 16);
                const PreRec R = sh.rec[cls];
                const uint32_t place = sh.pre[cur][e >> 5][cls] + (uint32_t)__popc(sh.bal[cur][e >> 5][cls] & ((1u << lane) - 1u));
                const bool shared_id = (m[i] & (m[i] - 1u)) != 0u;
                const float x = sh.val[cur][e], scaled = x * B.scl[j];
                sh.val[cur][e] = scaled; // (the records have the value itself)
                unsigned char *rec = P.rec + R.at + sizeof(SubHead);
                const uint32_t where = (uint32_t)id[i] < hot_total ? (uint32_t)id[i] >> P.logC : (uint32_t)id[i];
                reinterpret_cast<float *>(rec)[place] = x;
                reinterpret_cast<uint32_t *>(rec + R.meta)[place] = where | ((uint32_t)j << kIdBits) | (shared_id ? 0x80000000u : 0u);
                if (shared_id) {
                    const uint32_t start = sh.lists[slot[i] & 0xffffu] & 4095u, at = start + (uint32_t)__popc(m[i] & ((1u << j) - 1u));
                    sh.val[2][R.base + at] = scaled;
                    sh.row[2][R.base + at] = (uint8_t)j;
                    reinterpret_cast<float *>(rec + R.lval)[at] = x;
                    (rec + R.lrow)[at] = (unsigned char)j;
                    if (tl[i] != 0xffffffffu) {
                        const uint32_t pc = (uint32_t)__popc(m[i]), t = (tl[i] >> 16) + (pc > 4u ? 0u : R.longs); // long lists first
                        reinterpret_cast<uint32_t *>(rec + R.ids)[t] = where | ((pc - 1u) << kIdBits);
                        reinterpret_cast<uint16_t *>(rec + R.lst)[t] = (uint16_t)start;
                    }
                }
            }
        }
        __syncthreads();
        PRE_T(3);
        // ---- the next block's entries: which of this block's coordinates have their ids (table of this block); the pairs of both
        //      Gram matrices, 32 entries with some at a time
        {
            uint32_t *todo = sh.work[warp];
            int have = 0;
            auto push = [&](bool on, uint32_t item) {
                const uint32_t b = __ballot_sync(0xffffffffu, on);
                if (on) todo[have + __popc(b & ((1u << lane) - 1u))] = item;
                have += __popc(b);
            };
#pragma unroll
            for (int i = 0; i < EPT; ++i) {
                const uint32_t e = (uint32_t)(tid + i * THREADS);
                if ((e & ~31u) < (uint32_t)total && !walk)
                    push(id[i] >= kHD && (m[i] & ((1u << (slot[i] >> 16)) - 1u)) != 0u, e | (slot[i] & 0xffffu) << 12);
                if ((e & ~31u) < (uint32_t)ntotal && carry) {
                    uint32_t p = (uint32_t)nid[i];
                    bool hit = nid[i] >= kHD;
                    if (nid[i] >= kDir) {
                        p = home_place<HT>(nid[i]);
                        int32_t seen = sh.key[p];
                        for (int t = 1; seen != nid[i] && seen != -1 && t <= HT; ++t) {
                            p = next_place<HT>(p, t);
                            seen = sh.key[p];
                        }
                        hit = seen == nid[i];
                        p += kDir;
                    } else if (hit) hit = sh.mask[p] != 0u;
                    __syncwarp();
                    push(hit, e | p << 12 | 1u << 25);
                }
                if (i + 1 < EPT && have > 32) { // (the list holds 96)
                    __syncwarp();
                    have = pre_listed_early<NZ>(sh, have, cur, N);
                }
            }
            __syncwarp();
            pre_listed<NZ>(sh, have, cur, N);
        }
        // ---- rows l = warp, warp + NW of both matrices, lane = column: the dense part
        constexpr int R = kLB / NW;
        float2 g2[R], x2[R]; // (the even and the odd columns of the tiles)
        {
#pragma unroll
            for (int r = 0; r < R; ++r) g2[r] = x2[r] = make_float2(0.0f, 0.0f);
            const float4 *dj = reinterpret_cast<const float4 *>(&sh.D[cur][lane][0]), *nj = reinterpret_cast<const float4 *>(&sh.D[nxt][lane][0]);
            auto part = [&](auto both_) {
                constexpr bool both = decltype(both_)::value;
#pragma unroll
                for (int h = 0; h < kHD / 4; ++h) {
                    const float4 a = dj[h], b = both ? nj[h] : a;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 c = *reinterpret_cast<const float4 *>(&sh.D[cur][warp + r * NW][4 * h]);
                        fma2(g2[r], a.x, a.y, c.x, c.y);
                        if (both) fma2(x2[r], b.x, b.y, c.x, c.y);
                        fma2(g2[r], a.z, a.w, c.z, c.w);
                        if (both) fma2(x2[r], b.z, b.w, c.z, c.w);
                    }
                }
            };
            if (carry) part(std::true_type{});
            else part(std::false_type{});
        }
        __syncthreads();
        PRE_T(4);
        // ---- both matrices scaled and written
        if (have_next && warp < C) pre_prefix(sh, N.total, nxt, warp);
        {
            float qg = 0.0f, qx = 0.0f;
            // (the two inverse scales one after the other: their product is no fp32 number for two rows of norms below 1e-18)
            const float gsc = B.gsc[lane], inv = B.inv[lane], ngsc = carry ? N.gsc[lane] : 0.0f, ninv = carry ? N.inv[lane] : 0.0f;
            const int32_t *low = &sh.idx[cur][0];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int l = warp + r * NW;
                const float il = B.inv[l], yl = B.ys[l], al = B.as[l];
                const int at = gram_place(l, lane);
                float v = fmaf(fmaf((float)low[at], 1.0f / 1048576.0f, (float)(&sh.G[0][0][0])[at]) * il, inv, g2[r].x + g2[r].y) * (gsc * yl);
                v = lane > l && !walk ? v : 0.0f;
                out.G[l * kLB + lane] = v;
                qg = fmaf(v, al, qg);
                v = fmaf(fmaf((float)low[kLB * kLB + at], 1.0f / 1048576.0f, (float)(&sh.G[1][0][0])[at]) * il, ninv, x2[r].x + x2[r].y) * (ngsc * yl);
                v = l < cnt && carry ? v : 0.0f;
                out.X[l * kLB + lane] = v;
                qx = fmaf(v, al, qx);
            }
            sh.work[warp][lane] = __float_as_uint(qg);
            sh.work[warp][32 + lane] = __float_as_uint(qx);
        }
        for (int p = tid; p < HT / 4; p += THREADS) reinterpret_cast<int4 *>(sh.key)[p] = make_int4(-1, -1, -1, -1);
        for (int p = tid; p < Shared::TS / 4; p += THREADS) reinterpret_cast<uint4 *>(sh.mask)[p] = make_uint4(0u, 0u, 0u, 0u);
        if (tid < kMaxC) sh.cnt[tid] = sh.cntShort[tid] = 0u;
        __syncthreads();
        PRE_T(5);
    }
    if (warp == 0) pre_finish_head<NW>(P, sh, hi - 1);
}

// Short dense rows: every row has every id, so the lists are implicit: constants, Gram triangle, cross Gram matrix
// and the rows themselves (one worker record: the model lives in one CTA).
// All 64 visiting-order entries first, then all headers (a lane per coordinate) and all rows with every load of a thread
// issued before the first is used: three round trips to memory per block. (A warp per row, headers by its first lane, was
// a chain of 24 of them: 72 000 cycles per block at 28 entries per row, with the tables.)
constexpr int kPreThreads = 256;
constexpr int kPreDensePerSm = 4, kPreDenseLongPerSm = 2;
struct PreDenseShared {
    CHdr hdr[kLB];
    float gsc[2 * kLB], ys[kLB], as[kLB];
    int32_t coord[2 * kLB];
    float T[kLB][2 * kLB + 1];       // scaled Gram entries: row l, this block's columns, then the next block's
    int32_t walk;
    unsigned long long sub_off[kMaxC];
    alignas(16) float row[1];        // 64 rows of row_stride(columns at a time) floats: this block's, then the next block's
};
// Longer rows go through shared memory this many columns at a time.
constexpr int kDenseCols = 128;
// What counts as long: more columns than this (all of a shorter row is in shared memory at once). Up to here the kernel for short
// rows is the faster one, with few blocks and with many: a round on rows of 100, 10 000 over K = 4: 133 us against 139 with
// the other one, 100 000 over 64: 185 against 204, 1 M over 64: 1 571 against 1 933; rows of 128: 133 / 138, 197 / 212, 1 769 / 2 037.
constexpr int kDenseLong = 128;
inline bool dense_long(int64_t dim) { return dim > kDenseLong; }
// 16-byte pieces of consecutive rows lie on different banks
__host__ __device__ constexpr int row_stride(int cols) { return (((cols + 3) / 4) | 1) * 4; }
inline size_t pre_dense_bytes(int dim, bool lng)
{
    return sizeof(PreDenseShared) + (lng ? 2 : 1) * 2 * kLB * (size_t)row_stride(dim < kDenseCols ? dim : kDenseCols) * sizeof(float);
}

// Long rows (see dense_long): they pass through shared memory that many columns at a time, fetched two pieces ahead
// by asynchronous copies. Every warp takes every eighth four columns of a piece, a thread l = lp, lp + 4, .. and j = jq,
// jq + 8, .. (8 x 8 sums; pairs of tiles below the triangle are left out), and the warps' sums are added in a fixed order.
// Shared-memory loads bound it (a 16-byte load of a warp takes four turns whatever it broadcasts): 16 of them per 208
// multiply-adds, against 48 with 2 x 4 sums per thread over all columns; that and loads through registers, a round trip exposed
// for every piece, took 295 us for 100 000 rows of 500.
__device__ __forceinline__ void dense_gram_long(const LookParams &P, PreDenseShared &sh, int cnt, bool walk, int stride)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dim = (int)P.S.dim, slice = P.hotc;
    constexpr int TPR = kDenseCols / 4, RPT = kPreThreads / TPR; // threads per row of a piece, rows per turn
    const int sub = 4 * (tid % TPR), row0 = tid / TPR; // of a piece: this thread's four columns of rows row0, row0 + RPT, ..
    float *const buf0 = sh.row, *const buf1 = sh.row + 2 * kLB * stride;
    auto fetch = [&](int e0, float *to) {
#pragma unroll
        for (int i = 0; i < 2 * kLB / RPT; ++i) {
            float *at = to + (row0 + RPT * i) * stride + sub;
            if (e0 + sub >= dim) continue;
            const int c = sh.coord[row0 + RPT * i];
            const float *src = P.S.values + (int64_t)c * dim + (e0 + sub);
            if (c < 0) *reinterpret_cast<float4 *>(at) = make_float4(0.f, 0.f, 0.f, 0.f);
            else if ((dim & 3) == 0) cp_async16(smem_u32(at), src);
            else
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (e0 + sub + u < dim) cp_async4(smem_u32(at + u), src + u);
                    else at[u] = 0.0f;
                }
        }
        cp_async_commit();
    };
    fetch(0, buf0);
    if (kDenseCols < dim) fetch(kDenseCols, buf1);
    else cp_async_commit();
    // where this thread's columns go in the records: CTA c's, `left` columns from its slice's end
    int c = 0, first = 0;
    const int jq = lane & 7, lp = lane >> 3;
    float acc[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.0f;
#pragma unroll 1
    for (int e0 = 0; e0 < dim; e0 += kDenseCols) {
        const int cols = dim - e0 < kDenseCols ? dim - e0 : kDenseCols;
        float *rows = (e0 / kDenseCols) & 1 ? buf1 : buf0;
        cp_async_wait_but_one();
        __syncthreads();
        if (!walk && sub < cols) {
            while (e0 + sub - first >= slice) { first += slice; ++c; }
            const int st = dense_stride(dim - first < slice ? dim - first : slice);
            float *to = reinterpret_cast<float *>(P.rec + sh.sub_off[c] + sizeof(SubHead)) + (e0 + sub - first); // (padding included)
#pragma unroll
            for (int i = 0; i < kLB / RPT; ++i)
                if (row0 + RPT * i < cnt)
                    *reinterpret_cast<float4 *>(to + (row0 + RPT * i) * st) = *reinterpret_cast<const float4 *>(rows + (row0 + RPT * i) * stride + sub);
        }
        const float *rl = rows + lp * stride, *rj = rows + jq * stride;
#pragma unroll 1
        for (int e = 4 * warp; e < cols; e += 4 * (kPreThreads / 32)) {
            float4 xl[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) xl[a] = *reinterpret_cast<const float4 *>(rl + 4 * a * stride + e);
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const float4 xj = *reinterpret_cast<const float4 *>(rj + 8 * b * stride + e);
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    if (b < 4 && 4 * a >= 8 * (b + 1)) continue; // (every l of the tile lies beyond every j)
                    acc[a][b] = fmaf(xj.x, xl[a].x, acc[a][b]);
                    acc[a][b] = fmaf(xj.y, xl[a].y, acc[a][b]);
                    acc[a][b] = fmaf(xj.z, xl[a].z, acc[a][b]);
                    acc[a][b] = fmaf(xj.w, xl[a].w, acc[a][b]);
                }
            }
        }
        __syncthreads(); // the piece has been read
        if (e0 + 2 * kDenseCols < dim) fetch(e0 + 2 * kDenseCols, rows);
        else cp_async_commit();
    }
    // the warps' sums: 4 .. 7 to 0 .. 3, 2 and 3 to 0 and 1, 1 to 0 (every lane has the same places in every warp)
    float4 *part = reinterpret_cast<float4 *>(sh.row);
    static_assert(4 * 64 * 32 <= 2 * 2 * kLB * row_stride(kDenseCols), "four warps' sums fit the rows' buffers");
#pragma unroll
    for (int half = 4; half > 0; half >>= 1) {
        if (warp >= half && warp < 2 * half) {
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    part[((warp - half) * 16 + 2 * a + b) * 32 + lane] = make_float4(acc[a][4 * b], acc[a][4 * b + 1], acc[a][4 * b + 2], acc[a][4 * b + 3]);
        }
        __syncthreads();
        if (warp < half) {
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float4 t = part[(warp * 16 + 2 * a + b) * 32 + lane];
                    acc[a][4 * b] += t.x; acc[a][4 * b + 1] += t.y; acc[a][4 * b + 2] += t.z; acc[a][4 * b + 3] += t.w;
                }
        }
        if (half > 1) __syncthreads();
    }
    if (warp == 0)
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) sh.T[lp + 4 * a][jq + 8 * b] = acc[a][b];
}

template <int LOSS, bool LONG> __device__ __forceinline__ void prepare_block_dense(const LookParams &P, const int64_t bid, PreDenseShared &sh)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int NW = kPreThreads / 32;
    int k;
    int64_t b;
    block_to_part(P, bid, k, b);
    const int64_t nk = P.S.part_off[k + 1] - P.S.part_off[k];
    const int64_t off = P.S.part_off[k] + (P.S.first_k ? P.S.first_k[k] : 0); // of this launch's first step in the order
    const int64_t steps = steps_of(P, k, nk);
    const int cnt = (int)((steps - b * kLB) < kLB ? (steps - b * kLB) : kLB);
    const int64_t left = steps - (b + 1) * kLB;
    const int ncnt = (left <= 0 || P.depth < 2) ? 0 : (left < kLB ? (int)left : kLB);
    const int dim = (int)P.S.dim, C = 1 << P.logC, slice = P.hotc, stride = row_stride(dim < kDenseCols ? dim : kDenseCols);
    auto cols_of = [&](int c) { return dim - c * slice < slice ? (dim > c * slice ? dim - c * slice : 0) : slice; }; // of a CTA
    ChainHead &out = *reinterpret_cast<ChainHead *>(P.rec + (size_t)bid * sizeof(ChainHead));
    if (tid < 2 * kLB) {
        const bool on = tid < kLB ? tid < cnt : tid - kLB < ncnt;
        int32_t c = on ? P.S.perm[off + b * kLB + tid] : -1; // (the next block's entries follow)
        if (on && !CHICLE_IN_BOUNDS(P.S.status, c >= 0 && (int64_t)c < P.S.n_coord)) c = 0;
        sh.coord[tid] = c;
    } else if (tid == 2 * kLB) {
        unsigned long long need = 0;
        for (int c = 0; c < C; ++c) need += sub_bytes_dense(cnt, cols_of(c));
        unsigned long long at = atomicAdd(P.cursor, need);
        sh.walk = at + need > P.pool_cap ? 1 : 0; // no room: walked in place
        if (sh.walk) atomicAdd(P.S.status + kStatusWalked, 1u);
        for (int c = 0; c < C; ++c) {
            BlkDir d;
            if (sh.walk) {
                d.offset = (unsigned long long)bid * sizeof(ChainHead);
                d.bytes = 16u;
                d.flags = 1u;
            } else {
                d.offset = P.pool_off + at;
                d.bytes = sub_bytes_dense(cnt, cols_of(c));
                d.flags = 0u;
                at += d.bytes;
            }
            sh.sub_off[c] = d.offset;
            if (bid == P.drop_block) d.bytes = 0u;
            P.dirS[bid * C + c] = d;
        }
        out.cnt = cnt;
        out.flags = sh.walk;
        out.pad[0] = out.pad[1] = 0;
    }
    __syncthreads();
    const bool walk = sh.walk != 0;
    if (!walk && tid < C) {
        SubHead &h = *reinterpret_cast<SubHead *>(P.rec + sh.sub_off[tid]);
        h.n = cnt * cols_of(tid); h.T = 0; h.nl = 0; h.cnt = cnt;
    }
    // ---- headers: warp 0 this block's coordinates, warp 1 the next block's
    if (warp < 2) {
        const int32_t c = sh.coord[warp * kLB + lane];
        CHdr hd{0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (c >= 0) {
            hd = make_hdr<LOSS>(P.S, c);
            if (LOSS == CHICLE_LOSS_LOGISTIC_DUAL && P.tab_bins) hd.lq = tab_offset(hd.p2);
        }
        sh.gsc[warp * kLB + lane] = c >= 0 ? gram_scale<LOSS>(hd, P.S.sigma, P.S.inv_n) : 0.0f;
        if (warp == 0) {
            sh.hdr[lane] = hd;
            sh.ys[lane] = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 1.0f : hd.p3;
            sh.as[lane] = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? 0.0f : hd.p1;
        }
    }
    // ---- x_l . x_j for this block's l and the 64 columns j. This block's rows go into the workers' records on the way.
    if (LONG) dense_gram_long(P, sh, cnt, walk, stride);
    else {
        // a thread has l = lp, lp + 16 and j = jq, jq + 16, .. (every sum over the entries in ascending order)
        constexpr int RPW = 2 * kLB / NW; // rows a warp loads
        const int jq = tid & 15, lp = tid >> 4, cols4 = (dim + 3) & ~3;
        float acc[2][4];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][c] = 0.0f;
        float *val_g = reinterpret_cast<float *>(P.rec + (walk ? 0 : sh.sub_off[0]) + sizeof(SubHead)); // (one CTA per partition)
        const int st = dense_stride(dim);
        if ((dim & 3) == 0) { // rows start on 16-byte boundaries
            const int nv = dim >> 2;
            const int lpr = nv <= 8 ? 8 : (nv <= 16 ? 16 : 32); // lanes per row
            const int sub = lane & (lpr - 1), per = 32 / lpr; // rows per turn
            float4 v[RPW];
#pragma unroll
            for (int u = 0; u < RPW; ++u) {
                const int j = warp * RPW + u * per + lane / lpr;
                v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (u * per < RPW && sub < nv && sh.coord[j] >= 0)
                    v[u] = reinterpret_cast<const float4 *>(P.S.values + (int64_t)sh.coord[j] * dim)[sub];
            }
#pragma unroll
            for (int u = 0; u < RPW; ++u) {
                const int j = warp * RPW + u * per + lane / lpr;
                if (u * per < RPW && sub < nv) {
                    reinterpret_cast<float4 *>(sh.row + j * stride)[sub] = v[u];
                    if (j < cnt && !walk) reinterpret_cast<float4 *>(val_g + j * st)[sub] = v[u];
                }
            }
        } else {
            for (int f = lane; f < cols4; f += 32) {
                float v[RPW];
#pragma unroll
                for (int u = 0; u < RPW; ++u) {
                    const int j = warp * RPW + u;
                    v[u] = f < dim && sh.coord[j] >= 0 ? P.S.values[(int64_t)sh.coord[j] * dim + f] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < RPW; ++u) {
                    const int j = warp * RPW + u;
                    sh.row[j * stride + f] = v[u];
                    if (j < cnt && !walk) val_g[j * st + f] = v[u]; // (with the zero padding)
                }
            }
        }
        __syncthreads();
        if (!walk) {
            const float *rl = sh.row + lp * stride, *rj = sh.row + jq * stride;
            for (int e = 0; e < dim; e += 4) {
                float4 xl[2], xj[4];
#pragma unroll
                for (int a = 0; a < 2; ++a) xl[a] = *reinterpret_cast<const float4 *>(rl + 16 * a * stride + e);
#pragma unroll
                for (int c = 0; c < 4; ++c) xj[c] = *reinterpret_cast<const float4 *>(rj + 16 * c * stride + e);
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[a][c] = fmaf(xj[c].x, xl[a].x, acc[a][c]);
                        acc[a][c] = fmaf(xj[c].y, xl[a].y, acc[a][c]);
                        acc[a][c] = fmaf(xj[c].z, xl[a].z, acc[a][c]);
                        acc[a][c] = fmaf(xj[c].w, xl[a].w, acc[a][c]);
                    }
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) sh.T[lp + 16 * a][jq + 16 * c] = acc[a][c];
    }
    if (LOSS == CHICLE_LOSS_LOGISTIC_DUAL && P.tab_bins && !walk) write_table(P, bid, sh.hdr, kPreThreads);
    __syncthreads();
    for (int i = tid; i < 2 * kLB * kLB; i += kPreThreads) { // scaled; inside the block: earlier coordinates only
        const int l = (i >> 5) & 31, j = (i & 31) + (i >= kLB * kLB ? kLB : 0);
        const bool on = j < kLB ? l < j : l < cnt;
        const float v = on && !walk ? sh.T[l][j] * (sh.gsc[j] * sh.ys[l]) : 0.0f;
        sh.T[l][j] = v;
        out.G[i] = v; // (X lies behind G)
    }
    __syncthreads();
    for (int j = warp; j < 2 * kLB; j += NW) { // what the states at round start contribute
        float q0 = sh.T[lane][j] * sh.as[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q0 += __shfl_xor_sync(0xffffffffu, q0, o);
        if (lane == 0) {
            if (j >= kLB) out.q0n[j - kLB] = q0;
            else sh.hdr[j].A -= q0;
        }
    }
    __syncthreads();
    if (tid < kLB) out.hdr[tid] = sh.hdr[tid];
}

// (blocks blockIdx.x, blockIdx.x + gridDim.x, ..)
template <int LOSS, bool LONG> __global__ void __launch_bounds__(kPreThreads, LONG ? kPreDenseLongPerSm : kPreDensePerSm) k_lookahead_prepare_dense(const LookParams P)
{
    extern __shared__ __align__(128) unsigned char smem_pre[];
    PreDenseShared &sh = *reinterpret_cast<PreDenseShared *>(smem_pre);
    for (int64_t bid = blockIdx.x; bid < P.n_blocks; bid += gridDim.x) {
        prepare_block_dense<LOSS, LONG>(P, bid, sh);
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------------ chain
// Cluster plumbing. Addresses in another CTA's shared memory come from mapa; data and the signal that it has landed
// travel together: an asynchronous store completes bytes on the receiver's mbarrier (no multicast anywhere).
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t mapa_u32(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Data and the signal that it has landed travel together: an asynchronous store completes bytes on the receiver's
// mbarrier, straight from registers.
__device__ __forceinline__ void st_async_f32_if(uint32_t remote, float v, uint32_t remote_bar, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];\n\t}" ::"r"(remote), "f"(v),
                 "r"(remote_bar), "r"((uint32_t)on)
                 : "memory");
}
__device__ __forceinline__ void st_async_f32x4_if(uint32_t remote, float a, float b, float c, float d, uint32_t remote_bar, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %6, 0;\n\t"
                 "@q st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];\n\t}" ::"r"(remote),
                 "f"(a), "f"(b), "f"(c), "f"(d), "r"(remote_bar), "r"((uint32_t)on)
                 : "memory");
}
// Operations of a single lane as predicated instructions, not branches: a warp whose lanes part ways before a loop
// of shuffles may run the loop as separate groups of lanes that meet again at every shuffle (measured: 125 cycles per
// shuffle instead of 30 in the recurrence warp).
__device__ __forceinline__ void bulk_g2s_if(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %4, 0;\n\t"
                 "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar), "r"((uint32_t)on)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx_if(uint32_t bar, uint32_t bytes, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar),
                 "r"(bytes), "r"((uint32_t)on)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_if(uint32_t bar, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void sts_f32x4_if(uint32_t a, float x, float y, float z, float w, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t@q st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w),
                 "r"((uint32_t)on)
                 : "memory");
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t remote)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster_f32(uint32_t remote, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote_release(uint32_t remote_bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote_bar) : "memory");
}
__device__ __forceinline__ void fence_cluster() { asm volatile("fence.acq_rel.cluster;" ::: "memory"); }
// One look at an mbarrier; the hardware may suspend the thread for up to `hint_ns` until the phase completes. The data
// that the pipeline's barriers guard is written into this CTA's shared memory by asynchronous stores and copies that
// complete on the barrier itself, so the default scope serves (as for a bulk copy); the two waits of the rare
// walked-in-place path, which order ordinary stores of another CTA, add a cluster-scope fence of their own.
__device__ __forceinline__ uint32_t mbar_try_wait_cluster(uint32_t a, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity), "r"(100000u)
        : "memory");
    return ok;
}
// One look without suspension: 16 cycles with the vote, against 47 for try_wait with a time hint.
__device__ __forceinline__ uint32_t mbar_test(uint32_t a, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok;
}
// (not inlined: one copy keeps the loops of the kernel small)
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t *status)
{
    const long long t_start = clock64();
    for (;;) {
        bool ok = false;
        for (int it = 0; it < 64 && !ok; ++it) ok = __all_sync(0xffffffffu, mbar_try_wait_cluster(bar, parity) != 0u);
        if (ok) return true;
        const bool stop = __any_sync(0xffffffffu, *abort_flag != 0);
        const bool late = __any_sync(0xffffffffu, clock64() - t_start > 2500000000ll); // more than a second at any clock
        if (stop || late) {
            if (!stop && (threadIdx.x & 31) == 0) {
                *abort_flag = 1;
                atomicOr(status, ST_WAIT_TIMEOUT);
            }
            __syncwarp();
            return false;
        }
    }
}
// Bounded wait of one warp on an mbarrier (every lane must call it). No pauses of its own (try_wait suspends the thread
// for a while by itself; the waits of the pipeline are short and on its critical path); gives up after about a second, or
// when the CTA is aborting. The result is the same on all lanes: every lane looks at the barrier (one instruction for the
// warp either way) and the lanes agree by a vote, so that the warp stays together.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint32_t *status)
{
    if (__all_sync(0xffffffffu, mbar_test(bar, parity) != 0u)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, status);
}

// The end of a bulk copy that is on its way, for a role that stops early: a CTA must not leave while one still writes to its
// shared memory. Nothing but the copy itself is waited for (an abort does not end this), with a bound all the same. (Not
// inlined: the block loops stay as small as they were.)
__device__ __noinline__ void mbar_drain(uint32_t bar, uint32_t parity)
{
    for (int it = 0; it < (1 << 14) && !__all_sync(0xffffffffu, mbar_try_wait_cluster(bar, parity) != 0u); ++it) { }
}

// The worker warps' barrier: 35 cycles when all are there (with a vote 78, by arrivals on an mbarrier 181).
__device__ __forceinline__ void work_bar() { asm volatile("bar.sync %0, %1;" ::"n"(kBarWork), "n"(kWorkThreads) : "memory"); }

// (kSplit) the worker warps and the far warp, once, behind their last block
__device__ __forceinline__ void far_bar() { asm volatile("bar.sync %0, %1;" ::"n"(kBarWork + 1), "n"(kWorkThreads + 32) : "memory"); }

struct alignas(16) ChainCtl {
    uint64_t subfull[kSubSlots];   // count the bytes of the bulk copies into the workers' record slots
    uint64_t headfull[kMaxHeadSlots]; // the same for the recurrence warp's records (CTA 0)
    uint64_t pbar[2];              // CTA 0: the partial dot products of a block have arrived from all CTAs
    uint64_t dbar[2];              // a block's deltas have arrived from CTA 0
    uint64_t subfree[kSubSlots];   // the worker warps are through with the slot's record
    uint64_t ackbar;               // CTA 0: every worker warp of every CTA is through with all blocks before the one that is walked in place
    alignas(16) float pbuf[2][kMaxC][kLB];
    alignas(16) float dbuf[2][kLB];
    uint64_t ready[2];             // CTA 0: the states that a block's recurrence starts from are in `start`
    uint64_t out[2];               // CTA 0: the recurrence's results are in `res`
    uint64_t farfull[kSubSlots];   // kSplit: the slot's list of entries beyond shared memory is there
    alignas(16) float start[2][3][kLB]; // states; the scalar map's constants (p2 and lq; with tables tab_q and tab_offset)
    alignas(16) float res[2][kLB];
    float sink[32]; // where a lane's stores go that have no target
    int walk[kSubSlots]; // whether the slot's block is walked in place
    int abort_flag;
    int done; // the CTA's workers are through (the warps with no role sleep until then)
};

// Shared-memory layout of the chain kernel (sizes fixed at launch): control, recurrence records, logistic tables,
// worker records, the CTA's part of the model.
struct ChainLayout {
    uint32_t heads, tabs, subs, sub_stride, filter, far, w, total;
};
// kSplit: partial sums of all CTAs (used in CTA 0), products of a block's entries, and per slot a list of the entries: where each
// coordinate's start (kLB + 1 of them, and padding), and their numbers in the record.
constexpr uint32_t kFarSums = 2u * kMaxC * kLB * 4u, kFarHead = 80u;
__host__ __device__ constexpr uint32_t far_list_bytes(int cap) { return kFarHead + 2u * (uint32_t)cap; }
__host__ __device__ constexpr uint32_t far_bytes(int kind, int cap, int slots) { return kind == kSplit ? kFarSums + 4u * (uint32_t)cap + (uint32_t)slots * far_list_bytes(cap) : 0u; }
// kEarly: the model entries of ids beyond the part in shared memory are gathered from L2 before the
// block's deltas have come, and those that the block's update then changes once more. Which may have changed is kept in a bit
// per hashed id, one set of them for even and one for odd blocks: this many bytes a set (a bit that two ids share costs a
// second gather, nothing else).
__host__ __device__ constexpr uint32_t filter_bytes(int kind) { return kind == kEarly ? 4096u : 0u; }
__host__ __device__ inline ChainLayout chain_layout(uint32_t sub_room, int slots, int hotc, bool dense, int tab_bins, int kind, int far_cap = 0)
{
    ChainLayout L;
    L.heads = (uint32_t)((sizeof(ChainCtl) + 127) & ~(size_t)127);
    const uint32_t hs = (uint32_t)head_slots(tab_bins > 0);
    L.tabs = L.heads + hs * (uint32_t)sizeof(ChainHead);
    L.subs = L.tabs + hs * tab_bytes(tab_bins);
    L.sub_stride = dense ? sub_bytes_dense(kLB, hotc) : sub_room;
    L.filter = L.subs + (uint32_t)slots * L.sub_stride;
    L.far = L.filter + 2u * filter_bytes(kind);
    L.w = L.far + far_bytes(kind, far_cap, slots);
    L.total = L.w + 4u * (uint32_t)(hotc > 0 ? hotc : 4);
    return L;
}

template <int LOSS, int KIND, bool TAB>
__global__ void __launch_bounds__(chain_threads(KIND), 1) k_lookahead_chain(const LookParams P)
{
    constexpr bool DENSE = KIND == kDense, SPLIT = KIND == kSplit;
    constexpr int kChainThreads = chain_threads(KIND);
    constexpr uint32_t kRows = SPLIT ? 2u : 1u; // rows of partial sums from each CTA
    extern __shared__ __align__(128) unsigned char smem_chain[];
    const SolverParams &S = P.S;
    const int logC = P.logC, C = 1 << logC;
    const uint32_t crank = cluster_ctarank();
    const int k = (int)(blockIdx.x >> logC);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const ChainLayout L = chain_layout(P.sub_room, P.slots, P.hotc, DENSE, TAB ? P.tab_bins : 0, KIND, P.far_cap);
    ChainCtl &ctl = *reinterpret_cast<ChainCtl *>(smem_chain);
    float *W = reinterpret_cast<float *>(smem_chain + L.w);
    volatile int *abort_flag = &ctl.abort_flag;

    const int64_t nk = S.part_off[k + 1] - S.part_off[k];
    const int64_t steps = steps_of(P, k, nk);
    const int nb = (int)((steps + kLB - 1) / kLB); // (32-bit counters: 64-bit ones cost the chain hundreds of cycles a block)
    const int64_t bid0 = P.blk_base[k];
    float *Uk = S.U + (size_t)k * (size_t)S.dim;
    const float sigma = S.sigma;
    // entry ids below hot_total live in shared memory: id g in CTA g mod C at place g / C
    const int64_t hot_all = (int64_t)P.hotc << logC;
    const uint32_t hot_total = (uint32_t)(hot_all < S.dim ? hot_all : S.dim);
    // (dense rows: consecutive columns to a CTA, hotc of them, a multiple of four)
    const int slice0 = DENSE ? (int)crank * P.hotc : 0;
    const int hot_mine = DENSE ? ((int)S.dim - slice0 < P.hotc ? ((int)S.dim > slice0 ? (int)S.dim - slice0 : 0) : P.hotc)
                               : (hot_total > crank ? (int)((hot_total - crank + C - 1) >> logC) : 0);

    const uint32_t d_bytes = (uint32_t)kLB * 4u; // what a block's deltas bring
    if (tid == 0) {
        ctl.abort_flag = 0;
        ctl.done = 0;
        for (int i = 0; i < kSubSlots; ++i) {
            mbar_init(smem_u32(&ctl.subfull[i]), 1);
            mbar_init(smem_u32(&ctl.subfree[i]), kRows); // (the worker warps, and the far warp)
            mbar_init(smem_u32(&ctl.farfull[i]), 1);
        }
        for (int i = 0; i < kMaxHeadSlots; ++i) mbar_init(smem_u32(&ctl.headfull[i]), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&ctl.pbar[i]), 1);
            mbar_init(smem_u32(&ctl.dbar[i]), 1);
            mbar_init(smem_u32(&ctl.ready[i]), 1);
            mbar_init(smem_u32(&ctl.out[i]), 1);
        }
        mbar_init(smem_u32(&ctl.ackbar), (uint32_t)(C * (kWorkWarps + (SPLIT ? 1 : 0))));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // armed for the first two blocks before anybody can send
        for (int i = 0; i < 2; ++i) {
            mbar_arrive_expect_tx(smem_u32(&ctl.pbar[i]), kRows * (uint32_t)(C * kLB * 4));
            mbar_arrive_expect_tx(smem_u32(&ctl.dbar[i]), d_bytes);
        }
    }
    // (eight words per thread and turn, all loads first: a launch must not spend a memory round trip on every 384 words)
    for (int l0 = tid; l0 < hot_mine; l0 += 8 * kChainThreads) {
        float u[8], v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int l = l0 + i * kChainThreads;
            const bool in = l < hot_mine;
            const size_t g = !in ? 0 : (DENSE ? (size_t)(slice0 + l) : ((size_t)l << logC) + crank);
            u[i] = ldcg_if(Uk + g, in);
            v[i] = ldcg_if(S.vbase + g, in && P.model_in);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (l0 + i * kChainThreads < hot_mine) W[l0 + i * kChainThreads] = P.model_in ? fmaf(sigma, u[i], v[i]) : u[i];
    }
    constexpr bool EARLY = KIND == kEarly, FAR = KIND == kCold || EARLY;
    if constexpr (EARLY)
        for (uint32_t i = (uint32_t)tid; i < 2u * filter_bytes(KIND) / 4u; i += kChainThreads) reinterpret_cast<uint32_t *>(smem_chain + L.filter)[i] = 0u;
    if (DENSE && tid < 4 && hot_mine + tid < P.hotc) W[hot_mine + tid] = 0.0f; // (the padding of the last slice)
    // the ids beyond the part in shared memory that fall to this CTA (id mod C): the model in place
    const size_t cold0 = (size_t)hot_total + (((size_t)crank - (size_t)hot_total) & (size_t)(C - 1));
    if (P.model_in)
        for (size_t g0 = cold0 + ((size_t)tid << logC); g0 < (size_t)S.dim; g0 += (size_t)(8 * kChainThreads) << logC) {
            float u[8], v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const size_t g = g0 + ((size_t)(i * kChainThreads) << logC);
                const bool in = g < (size_t)S.dim;
                u[i] = ldcg_if(Uk + (in ? g : 0), in);
                v[i] = ldcg_if(S.vbase + (in ? g : 0), in);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const size_t g = g0 + ((size_t)(i * kChainThreads) << logC);
                if (g < (size_t)S.dim) Uk[g] = fmaf(sigma, u[i], v[i]);
            }
        }
    __syncthreads();
    cluster_arrive();
    cluster_wait();

    constexpr int HS = head_slots(TAB);
    const bool is_chain = crank == 0 && warp == 0;
    const bool is_worker = (warp & 3) != 0 && warp < kFeedWarp; // warps 1 2 3 5 6 7 9 10
    bool aborted = false;

    if (is_chain && nb > 0) {
        // ============================== the recurrence warp =====================================================
        const int q = lane & 7;
        const uint32_t tab_neg = TAB ? (uint32_t)(P.tab_bins - kTabNeg) * 32u : 0u;
        float xs[4] = {0.f, 0.f, 0.f, 0.f}; // what the block before contributes to this block's states
        int sc = 0;                        // walked blocks so far
        int slot = 0;                      // b mod the head slots
#ifdef CHICLE_LA_TIMING
        long long tw = 0, tr = 0, te = 0, t0 = clock64(), t1 = 0;
#endif
#pragma unroll 1
        for (int b = 0; b < nb; ++b) {
            const uint32_t par = (uint32_t)(b & 1);
            if (!mbar_wait_cluster(smem_u32(&ctl.ready[0]) + 8u * par, (uint32_t)(b >> 1) & 1u, abort_flag, S.status)) { aborted = true; break; }
            const ChainHead &H = *reinterpret_cast<const ChainHead *>(smem_chain + L.heads + (size_t)slot * sizeof(ChainHead));
            if (H.flags & 1) {
                const int cnt = H.cnt;
                // ---- walked in place: wait until every CTA has applied all earlier updates, then coordinate by
                //      coordinate against the whole model (the other CTAs' parts through the cluster's shared memory)
                if (!mbar_wait_cluster(smem_u32(&ctl.ackbar), (uint32_t)sc & 1u, abort_flag, S.status)) { aborted = true; break; }
                fence_cluster(); // the other CTAs' updates of their parts of the model, made by ordinary stores
                ++sc;
                const uint32_t w_base = smem_u32(W);
                auto w_at = [&](uint32_t g) { // where a model entry in shared memory lies
                    const uint32_t c = DENSE ? g / (uint32_t)P.hotc : g & (uint32_t)(C - 1);
                    return mapa_u32(w_base + 4u * (DENSE ? g - c * (uint32_t)P.hotc : g >> logC), c);
                };
                for (int j = 0; j < cnt; ++j) {
                    const CHdr h = H.hdr[j];
                    if (!CHICLE_IN_BOUNDS(S.status, h.coord >= 0 && (int64_t)h.coord < S.n_coord)) continue;
                    const int64_t rs = DENSE ? (int64_t)h.coord * S.dim : S.indptr[h.coord];
                    int n = DENSE ? (int)S.dim : (int)(S.indptr[h.coord + 1] - rs);
                    if (!CHICLE_IN_BOUNDS(S.status, DENSE || (rs >= 0 && n >= 0 && rs + n <= P.nnz))) n = 0;
                    const int32_t *ix = S.indices + rs;
                    const float *xv = S.values + rs;
                    float acc = 0.0f, delta, new_state;
                    for (int e = lane; e < n; e += 32) {
                        uint32_t g = DENSE ? (uint32_t)e : (uint32_t)ix[e];
                        if (!CHICLE_IN_BOUNDS(S.status, (int64_t)g < S.dim)) g = 0u;
                        const float ww = g < hot_total ? ld_cluster_f32(w_at(g))
                                                       : __ldcg(Uk + g);
                        acc = fmaf(xv[e], ww, acc);
                    }
                    acc = warp_sum(acc);
                    coordinate_step<LOSS>(acc, h, delta, new_state);
                    if (!(fabsf(delta) <= CUDART_MAX_NORMAL_F)) {
                        if (lane == 0) atomicOr(S.status, ST_NONFINITE_STEP);
                        delta = 0.0f;
                        new_state = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? h.p1 : h.p3 * h.p1;
                    }
                    if (delta != 0.0f)
                        for (int e = lane; e < n; e += 32) {
                            uint32_t g = DENSE ? (uint32_t)e : (uint32_t)ix[e];
                            if (!CHICLE_IN_BOUNDS(S.status, (int64_t)g < S.dim)) continue;
                            if (g < hot_total) {
                                const uint32_t a = w_at(g);
                                st_cluster_f32(a, fmaf(sigma * delta, xv[e], ld_cluster_f32(a)));
                            } else Uk[g] = fmaf(sigma * delta, xv[e], __ldcg(Uk + g));
                        }
                    if (lane == 0) S.alpha[h.coord] = new_state;
                    __syncwarp();
                }
                // the walk's writes before the signal (the feeder sends a block of zero deltas)
                __threadfence();
                fence_cluster();
                xs[0] = xs[1] = xs[2] = xs[3] = 0.0f;
            } else {
                // ---- four coordinates at a time. Lane q (and its copies q + 8, q + 16, q + 24, which compute the
                //      same) keeps the states of coordinates 4q .. 4q + 3. Group g: its lane walks its four coordinates
                //      by itself, the four results are handed round, and every lane adds what they mean for its own
                //      four, in this block and in the next.
                const uint32_t st0 = smem_u32(&ctl.start[0][0][0]) + par * (uint32_t)sizeof(ctl.start[0]) + 16u * (uint32_t)q;
                const uint32_t res = smem_u32(&ctl.res[0][0]) + par * (uint32_t)(kLB * 4);
                const float4 s0 = lds_f32x4(st0);
                float4 k2 = make_float4(0.f, 0.f, 0.f, 0.f), k3 = k2;
                if (LOSS != CHICLE_LOSS_HINGE_DUAL) k2 = lds_f32x4(st0 + 128u);
                if (LOSS == CHICLE_LOSS_LOGISTIC_DUAL) k3 = lds_f32x4(st0 + 256u);
                const float4 q0n = *reinterpret_cast<const float4 *>(&H.q0n[4 * q]);
                const float hp2[4] = {k2.x, k2.y, k2.z, k2.w}, hlq[4] = {k3.x, k3.y, k3.z, k3.w};
                float s[4] = {s0.x + xs[0], s0.y + xs[1], s0.z + xs[2], s0.w + xs[3]};
                xs[0] = -q0n.x; xs[1] = -q0n.y; xs[2] = -q0n.z; xs[3] = -q0n.w;
                // with tables: where each coordinate's table would have exponent 0
                uint32_t row[4];
                float off2[4];
                if (TAB) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) off2[i] = fmaf(hp2[i], kTabInv, hlq[i]);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        row[i] = smem_u32(smem_chain + L.tabs) + (uint32_t)slot * tab_bytes(P.tab_bins) + (uint32_t)((4 * q + i) * P.tab_bins) * 32u - (127u << 2) * 32u;
                }
                float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo; // (the lanes whose result nobody wants keep what is there)
                // a state's result is sgn * v + bias (sgn = 1, bias = 0 without tables)
                auto step_map = [&](float st, int i, bool on, float &sgn, float &bias) {
                    if (TAB) return tab_map(st, hp2[i], hlq[i], off2[i], row[i], tab_neg, on, lo, hi, sgn, bias);
                    sgn = 1.0f;
                    bias = 0.0f;
                    return recurrence_map<LOSS>(st, hp2[i], hlq[i]);
                };
                LA_T(tw);
                const float4 *G4 = reinterpret_cast<const float4 *>(H.G); // G4[l * 8 + q]: row l, columns 4q .. 4q + 3
                const float4 *X4 = reinterpret_cast<const float4 *>(H.X);
                // (how far this is unrolled was measured: the code of the block loop has to stay near the instruction cache's
                // size, or fetches set the pace of all roles. With tables not at all: 147 -> 119 cycles a step; sparse
                // hinge twice: the recurrence 1 066 -> 1 290 cycles a block, the workers, who are the bound there, 4 610 -> 4 410)
#pragma unroll (TAB ? 1 : (DENSE ? kLB / 4 : 2))
                for (int g = 0; g < kLB / 4; ++g) {
                    float4 blk[4], nxt[4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        blk[kk] = G4[(4 * g + kk) * 8 + q];
                        nxt[kk] = X4[(4 * g + kk) * 8 + q];
                    }
                    // inside the group (the numbers matter on the lanes with q == g, where blk holds the group's own
                    // triangle; the others run the same instructions on copies)
                    float o[4], v, sg, bi;
                    v = step_map(s[0], 0, q == g, sg, bi);
                    o[0] = TAB ? fmaf(v, sg, bi) : v;
                    const float t1 = TAB ? fmaf(v, sg * blk[0].y, fmaf(bi, blk[0].y, s[1])) : fmaf(v, blk[0].y, s[1]);
                    v = step_map(t1, 1, q == g, sg, bi);
                    o[1] = TAB ? fmaf(v, sg, bi) : v;
                    const float u2 = fmaf(o[0], blk[0].z, s[2]);
                    const float t2 = TAB ? fmaf(v, sg * blk[1].z, fmaf(bi, blk[1].z, u2)) : fmaf(v, blk[1].z, u2);
                    v = step_map(t2, 2, q == g, sg, bi);
                    o[2] = TAB ? fmaf(v, sg, bi) : v;
                    const float u3 = fmaf(o[1], blk[1].w, fmaf(o[0], blk[0].w, s[3]));
                    const float t3 = TAB ? fmaf(v, sg * blk[2].w, fmaf(bi, blk[2].w, u3)) : fmaf(v, blk[2].w, u3);
                    v = step_map(t3, 3, q == g, sg, bi);
                    o[3] = TAB ? fmaf(v, sg, bi) : v;
                    sts_f32x4_if(res + 16u * (uint32_t)g, o[0], o[1], o[2], o[3], lane == g);
                    float og[4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) og[kk] = __shfl_sync(0xffffffffu, o[kk], g);
                    // (zero entries of the triangle make this a no-op for the groups at or before g, whose states are final)
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        s[0] = fmaf(og[kk], blk[kk].x, s[0]);
                        s[1] = fmaf(og[kk], blk[kk].y, s[1]);
                        s[2] = fmaf(og[kk], blk[kk].z, s[2]);
                        s[3] = fmaf(og[kk], blk[kk].w, s[3]);
                        xs[0] = fmaf(og[kk], nxt[kk].x, xs[0]);
                        xs[1] = fmaf(og[kk], nxt[kk].y, xs[1]);
                        xs[2] = fmaf(og[kk], nxt[kk].z, xs[2]);
                        xs[3] = fmaf(og[kk], nxt[kk].w, xs[3]);
                    }
                }
                LA_T(tr);
            }
            __syncwarp();
            mbar_arrive_if(smem_u32(&ctl.out[0]) + 8u * par, lane == 0);
            LA_T(te);
            slot = slot + 1 == HS ? 0 : slot + 1;
        }
#ifdef CHICLE_LA_TIMING
        if (blockIdx.x == 0 && lane == 0) {
            unsigned long long *d = P.timing;
            d[0] = tw; d[1] = tr; d[2] = te; d[3] = nb;
        }
#endif
    }
    if (crank == 0 && warp == kStartWarp && nb > 0) {
        // ============================== what a block's recurrence starts from =======================================
        // A lane per coordinate: once the block's dot products are here. In the
        // recurrence warp itself, which keeps four coordinates per lane, this and what the feeder does took 1 090 cycles a
        // block, most of them instruction fetches of code that runs once.
        int fp = 0, slot = 0; // staged blocks so far; blk mod the head slots
        uint32_t turn = 0;    // parity of blk / the head slots
#pragma unroll 1
        for (int blk = 0; blk < nb; ++blk) {
            const uint32_t par = (uint32_t)(blk & 1);
            // (a block walked in place waits for no dot products: not before the recurrence is through with `start`)
            if (blk >= 2 && !mbar_wait_cluster(smem_u32(&ctl.out[0]) + 8u * par, (uint32_t)((blk >> 1) - 1) & 1u, abort_flag, S.status)) break;
            if (!mbar_wait_cluster(smem_u32(&ctl.headfull[slot]), turn, abort_flag, S.status)) break;
            const ChainHead &H = *reinterpret_cast<const ChainHead *>(smem_chain + L.heads + (size_t)slot * sizeof(ChainHead));
            if (!(H.flags & 1)) {
                const CHdr h = H.hdr[lane];
                if (!mbar_wait_cluster(smem_u32(&ctl.pbar[fp & 1]), (uint32_t)(fp >> 1) & 1u, abort_flag, S.status)) break;
                float m0 = 0.0f;
                for (int c = 0; c < C; ++c) m0 += ctl.pbuf[fp & 1][c][lane]; // the CTAs' partial sums in a fixed order
                if (SPLIT)
                    for (int c = 0; c < C; ++c) m0 += reinterpret_cast<const float *>(smem_chain + L.far)[((fp & 1) * kMaxC + c) * kLB + lane];
                ++fp;
                const float s0 = fmaf(h.B, m0, h.A);
                ctl.start[par][0][lane] = s0;
                ctl.start[par][1][lane] = TAB ? tab_q(h.p2, h.lq, P.tab_bins) : h.p2;
                ctl.start[par][2][lane] = h.lq;
            }
            __syncwarp();
            mbar_arrive_if(smem_u32(&ctl.ready[0]) + 8u * par, lane == 0);
            if (++slot == HS) {
                slot = 0;
                turn ^= 1u;
            }
        }
    }
    if (crank == 0 && warp == kFeedWarp && nb > 0) {
        // ============================== the feeder: what follows from a block's recurrence ===========================
        // Deltas to all CTAs' workers, the new states to global memory, and the head (and table) HS blocks on into the slot.
        const int q = lane & 7, rep = lane >> 3;
        // the copy `rep` of lane q sends four values to CTAs rep and rep + 4
        uint32_t d_dst[2], d_bar[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t c = (uint32_t)(rep + 4 * i) & (uint32_t)(C - 1);
            d_dst[i] = mapa_u32(smem_u32(&ctl.dbuf[0][4 * q]), c);
            d_bar[i] = mapa_u32(smem_u32(&ctl.dbar[0]), c);
        }
        const uint32_t tab_len = TAB ? tab_bytes(P.tab_bins) : 0u;
        const uint32_t heads0 = smem_u32(smem_chain + L.heads), tabs0 = smem_u32(smem_chain + L.tabs);
        auto issue_head = [&](int blk, int slot) {
            const bool on = blk < nb && lane == 0;
            const uint32_t bar = smem_u32(&ctl.headfull[slot]);
            const size_t at = (size_t)(bid0 + (blk < nb ? blk : nb - 1));
            mbar_arrive_expect_tx_if(bar, (uint32_t)sizeof(ChainHead) + tab_len, on);
            bulk_g2s_if(heads0 + (uint32_t)slot * (uint32_t)sizeof(ChainHead), P.rec + at * sizeof(ChainHead), (uint32_t)sizeof(ChainHead), bar, on);
            if (TAB) bulk_g2s_if(tabs0 + (uint32_t)slot * tab_len, P.rec + P.tab_off + at * tab_len, tab_len, bar, on);
        };
        for (int i = 0; i < HS; ++i) issue_head(i, i);
        int fp = 0, slot = 0, done = 0;
#pragma unroll 1
        for (int b = 0; b < nb; ++b) {
            const uint32_t par = (uint32_t)(b & 1);
            if (!mbar_wait_cluster(smem_u32(&ctl.out[0]) + 8u * par, (uint32_t)(b >> 1) & 1u, abort_flag, S.status)) break;
            const ChainHead &H = *reinterpret_cast<const ChainHead *>(smem_chain + L.heads + (size_t)slot * sizeof(ChainHead));
            const bool walked = (H.flags & 1) != 0;
            float dl = 0.0f, st = 0.0f;
            bool odd = false; // a step that is not finite
            int32_t coord = -1;
            if (!walked) {
                const CHdr h = H.hdr[lane];
                const float o = ctl.res[par][lane];
                const bool in = lane < H.cnt;
                if (LOSS == CHICLE_LOSS_RIDGE_PRIMAL) {
                    dl = o;
                    st = h.p1 + o;
                } else {
                    dl = h.p3 * (o - h.p1);
                    st = h.p3 * o;
                }
                const bool fine = fabsf(dl) <= CUDART_MAX_NORMAL_F;
                odd = in && !fine;
                if (!fine) st = LOSS == CHICLE_LOSS_RIDGE_PRIMAL ? h.p1 : h.p3 * h.p1;
                if (!in || !fine) dl = 0.0f;
                coord = in ? h.coord : -1;
                // armed for block fp + 2 before the deltas go out (its dot products are sent only after they arrive)
                mbar_arrive_expect_tx_if(smem_u32(&ctl.pbar[fp & 1]), kRows * (uint32_t)(C * kLB * 4), lane == 0);
                ++fp;
            } else fence_cluster(); // (the walk's ordinary stores go before the signal)
            float d4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d4[i] = __shfl_sync(0xffffffffu, dl, 4 * q + i);
#pragma unroll
            for (int i = 0; i < 2; ++i)
                st_async_f32x4_if(d_dst[i] + par * (uint32_t)(kLB * 4), d4[0], d4[1], d4[2], d4[3], d_bar[i] + par * 8u, rep + 4 * i < C);
            if (coord >= 0 && CHICLE_IN_BOUNDS(S.status, (int64_t)coord < S.n_coord)) S.alpha[coord] = st;
            if (__any_sync(0xffffffffu, odd) && lane == 0) atomicOr(S.status, ST_NONFINITE_STEP);
            __syncwarp();
            issue_head(b + HS, slot);
            slot = slot + 1 == HS ? 0 : slot + 1;
            done = b + 1;
        }
        for (int i = done; i < done + HS && i < nb; ++i) mbar_drain(smem_u32(&ctl.headfull[i % HS]), (uint32_t)(i / HS) & 1u);
    }
    if (warp == kRecordWarp && nb > 0) {
        // ============================== the workers' records, four blocks ahead =======================================
        // (directory entries are loaded a block ahead of their use; walk[slot] is written before the arrival that, with the
        // record's bytes, completes the slot's barrier)
        auto load_dir = [&](int blk, uint32_t (&d)[4]) {
            const int at = blk < nb ? blk : nb - 1;
            asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                         : "l"(P.dirS + (((bid0 + at) << logC) + crank))
                         : "memory");
        };
        const int slots = P.slots;
        uint32_t d[4];
        load_dir(0, d);
        int slot = 0, before = 0;     // of this block and of the one before
        int fetched = 0;
        // The slot's block has arrived: its entries beyond the part of the model in shared memory are brought into L2 (the records
        // that stream through it push them out) and, for the far warp, listed row after row.
        auto list_far = [&](int at) {
            const uint32_t rec = smem_u32(smem_chain + L.subs) + (uint32_t)at * L.sub_stride;
            int n = ctl.walk[at] ? 0 : lds_s32(rec);
            if (SPLIT && n > P.far_cap) n = P.far_cap; // (the prepare kernel sees to it)
            const uint32_t meta = rec + (uint32_t)sizeof(SubHead) + 4u * (uint32_t)n;
            const uint32_t list = smem_u32(smem_chain + L.far) + kFarSums + 4u * (uint32_t)P.far_cap + (uint32_t)at * far_list_bytes(P.far_cap);
            const int mine = SPLIT && n > 0 ? (int)lds_u16(rec + (uint32_t)offsetof(SubHead, roff) + 2u * (uint32_t)lane) : 0;
            int count = 0, start = 0;
            const uint32_t hotc = (uint32_t)P.hotc, dim = (uint32_t)(S.dim <= (int64_t)kIdMask ? S.dim : (int64_t)kIdMask + 1), below = (1u << lane) - 1u;
            uint32_t v[4];
            for (int e0 = 0; e0 < n; e0 += 128) { // (four loads under way together: one after the other a list of 312 took 3 000 cycles)
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = lds_u32_if(meta + 4u * (uint32_t)(e0 + 32 * u + lane), e0 + 32 * u + lane < n) & kIdMask; // (0: none)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool far = v[u] >= hotc && v[u] < dim && e0 + 32 * u + lane < n;
                    prefetch_if(Uk + (far ? v[u] : 0u), far);
                    if (!SPLIT) continue;
                    const uint32_t all = __ballot_sync(0xffffffffu, far);
                    const int first = mine - (e0 + 32 * u); // this lane's coordinate's first entry, from here on
                    sts_u16_if(list + kFarHead + 2u * (uint32_t)(count + __popc(all & below)), (uint32_t)(e0 + 32 * u + lane), far);
                    if (first >= 0) start = count + __popc(first < 32 ? all & ((1u << first) - 1u) : all);
                    count += __popc(all);
                }
            }
            if (SPLIT) {
                asm volatile("st.shared.u16 [%0], %1;" ::"r"(list + 2u * (uint32_t)lane), "h"((uint16_t)start) : "memory");
                if (lane == 0) asm volatile("st.shared.u16 [%0], %1;" ::"r"(list + 2u * (uint32_t)kLB), "h"((uint16_t)count) : "memory");
                __syncwarp();
                mbar_arrive_if(smem_u32(&ctl.farfull[at]), lane == 0);
            }
            __syncwarp();
        };
        uint32_t turn = 0, tbefore = 0; // parity of how often the slots have been filled
#ifdef CHICLE_LA_TIMING
        long long ra = 0, rl = 0, rs = 0, t0 = clock64(), t1 = 0;
#endif
#pragma unroll 1
        for (int blk = 0; blk < nb; ++blk) {
            if (__any_sync(0xffffffffu, *abort_flag != 0)) break; // (no slot is refilled for workers that no longer wait for it)
            // (the block before this one arrives while its predecessor's slot is still in use)
            if ((EARLY || SPLIT) && blk > 0) {
                if (!mbar_wait_cluster(smem_u32(&ctl.subfull[before]), tbefore, abort_flag, S.status)) break;
                LA_T(ra);
                list_far(before);
                LA_T(rl);
            }
            if (blk >= slots && !mbar_wait_cluster(smem_u32(&ctl.subfree[slot]), turn ^ 1u, abort_flag, S.status)) break;
            const unsigned long long offset = ((unsigned long long)d[1] << 32) | d[0];
            uint32_t bytes = d[2] <= L.sub_stride ? d[2] : 0u;
            if (!CHICLE_IN_BOUNDS(S.status, (offset & 15ull) == 0ull && offset + bytes <= P.pool_off + P.pool_cap))
                bytes = 0u; // (an entry that points outside the region: as if no record had been written)
            if (bytes == 0u) { // no record: nothing will arrive, say so now
                if (lane == 0) {
                    atomicOr(S.status, ST_WAIT_TIMEOUT);
                    *abort_flag = 1;
                }
                break;
            }
            if (lane == 0) ctl.walk[slot] = (int)(d[3] & 1u);
            __syncwarp();
            const uint32_t bar = smem_u32(&ctl.subfull[slot]);
            mbar_arrive_expect_tx_if(bar, bytes, lane == 0);
            bulk_g2s_if(smem_u32(smem_chain + L.subs) + (uint32_t)slot * L.sub_stride, P.rec + offset, bytes, bar, lane == 0);
            fetched = blk + 1;
            load_dir(blk + 1, d);
            // (kCold: this block's copy goes out first. As above, the round on 0.6 M uniform rows of 39, d = 1 M, K = 9: 4.10 ms instead of
            // 4.06, on 1 M over K = 16 4.24 instead of 4.18. And in few instructions: this warp shares warp 0's scheduler. Logistic rows of 39
            // with tables, 50 000 over K = 2, four loads together as above: 2.31 ms instead of 2.25.)
            if (KIND == kCold && blk > 0) {
                if (!mbar_wait_cluster(smem_u32(&ctl.subfull[before]), tbefore, abort_flag, S.status)) break;
                const uint32_t rec = smem_u32(smem_chain + L.subs) + (uint32_t)before * L.sub_stride;
                const int n = ctl.walk[before] ? 0 : lds_s32(rec);
                const uint32_t meta = rec + (uint32_t)sizeof(SubHead) + 4u * (uint32_t)n;
                for (int e = lane; e < n; e += 32) {
                    const uint32_t v = lds_u32_if(meta + 4u * (uint32_t)e, true) & kIdMask;
                    if (v >= (uint32_t)P.hotc && (int64_t)v < S.dim) asm volatile("prefetch.global.L2 [%0];" ::"l"(Uk + v));
                }
                __syncwarp();
            }
            before = slot;
            tbefore = turn;
            if (++slot == slots) {
                slot = 0;
                turn ^= 1u;
            }
            LA_T(rs);
        }
#ifdef CHICLE_LA_TIMING
        if (blockIdx.x == 0 && lane == 0) {
            unsigned long long *d = P.timing + 24;
            d[0] = ra; d[1] = rl; d[2] = rs;
        }
#endif
        if (SPLIT && fetched == nb && mbar_wait_cluster(smem_u32(&ctl.subfull[before]), tbefore, abort_flag, S.status)) list_far(before);
        for (int i = fetched > slots ? fetched - slots : 0; i < fetched; ++i) mbar_drain(smem_u32(&ctl.subfull[i % slots]), (uint32_t)(i / slots) & 1u);
    }
    if (SPLIT && warp == kFarWarp) {
        // ============================== the far warp ==============================================================
        // What the worker warps do for the ids in shared memory, for the others, whose model entries lie in row k of the update
        // workspace: a block's update by reductions at L2, then the gathers for the dot products that follow, in this warp's own
        // order, beside the workers. A round trip to L2 and the reductions stood in the workers' way otherwise, block after block
        // (45 M hashed rows, K = 16: 3 400 -> 3 060 cycles a block, step 155 -> 145 ms; with the workers' gathers in front of the
        // deltas, as the other kinds have them, 163).
        const uint32_t sums = smem_u32(smem_chain + L.far), prod = sums + kFarSums, lists0 = prod + 4u * (uint32_t)P.far_cap, lstride = far_list_bytes(P.far_cap);
        const uint32_t subs0 = smem_u32(smem_chain + L.subs);
        const uint32_t p_buf0 = mapa_u32(sums + crank * (uint32_t)(kLB * 4), 0u), p_bar0 = mapa_u32(smem_u32(&ctl.pbar[0]), 0u), ack_bar = mapa_u32(smem_u32(&ctl.ackbar), 0u);
        const uint32_t hotc = (uint32_t)P.hotc;
        const int depth = P.depth, slots = P.slots;
        int fg = 0, s_upd = 0, s_dot = 0;
        uint32_t dot_turn = 0;
        bool ok = true, sl0 = false, sl1 = false;
        auto in_dim = [&](uint32_t v) { return CHICLE_IN_BOUNDS(S.status, v >= hotc && (int64_t)v < S.dim); };
        // What bounds this warp is its instructions (code that runs once a block comes from beyond the instruction caches: about four
        // cycles each) and one round trip to L2. The first 64 entries of a block's list stay in registers from its dot products to its
        // update; longer lists' others are looked up each time.
        struct Entries {
            int n;
            float x[2];
            uint32_t m[2]; // (0: no entry)
        };
        auto entry = [&](int s, int e, bool in, float &x, uint32_t &m) {
            const uint32_t rec = subs0 + (uint32_t)s * L.sub_stride, val = rec + (uint32_t)sizeof(SubHead);
            const uint32_t i = 4u * lds_u16_if(lists0 + (uint32_t)s * lstride + kFarHead + 2u * (uint32_t)e, in);
            x = lds_f32_if(val + i, in);
            m = lds_u32_if(val + 4u * (uint32_t)lds_s32(rec) + i, in);
        };
        auto load = [&](int s, Entries &E) {
            E.n = (int)lds_u16(lists0 + (uint32_t)s * lstride + 2u * (uint32_t)kLB);
#pragma unroll
            for (int u = 0; u < 2; ++u) entry(s, lane + 32 * u, lane + 32 * u < E.n, E.x[u], E.m[u]);
        };
        auto gather = [&](uint32_t m) {
            const bool far = m != 0u && in_dim(m & kIdMask);
            return ldcg_if(Uk + (far ? m & kIdMask : 0u), far);
        };
        auto send = [&](int s, const Entries &E, float w0, float w1) {
            if (lane < E.n) sts_f32(prod + 4u * (uint32_t)lane, E.x[0] * w0);
            if (lane + 32 < E.n) sts_f32(prod + 4u * (uint32_t)(lane + 32), E.x[1] * w1);
#pragma unroll 1
            for (int e = lane + 64; e < E.n; e += 32) {
                float x;
                uint32_t m;
                entry(s, e, true, x, m);
                sts_f32(prod + 4u * (uint32_t)e, x * gather(m));
            }
            __syncwarp();
            float acc = 0.0f; // (a lane per coordinate)
            const uint32_t at = lists0 + (uint32_t)s * lstride + 2u * (uint32_t)lane;
            const int end = (int)lds_u16(at + 2u);
#pragma unroll 1
            for (int e = (int)lds_u16(at); e < end; ++e) acc += lds_f32(prod + 4u * (uint32_t)e);
            __syncwarp();
            const uint32_t slot = (uint32_t)(fg & 1);
            ++fg;
            st_async_f32_if(p_buf0 + (slot * (uint32_t)(kMaxC * kLB) + (uint32_t)lane) * 4u, acc, p_bar0 + slot * 8u, true);
        };
        Entries E0 = {0, {0.f, 0.f}, {0u, 0u}}, E1 = E0, E2 = E0; // of blocks b, b + 1, b + depth
        // a list of block b: its id, length (0: none, or one of the worker warps'), where its values and coordinates are, the first four
        uint32_t id = 0u, a_val = 0u, a_row = 0u, rl[4];
        float xl[4];
        int T = 0, len = 0; // (T: how many lists the block has)
        auto list_of = [&](int s, int t) {
            const uint32_t rec = subs0 + (uint32_t)s * L.sub_stride;
            const int4 head = lds_s32x4(rec); // n, T, nl, cnt
            const uint32_t ids = rec + (uint32_t)sizeof(SubHead) + 8u * (uint32_t)head.x, lval = ids + 4u * (uint32_t)head.y, lst = lval + 4u * (uint32_t)head.z;
            T = head.y;
            const uint32_t word = lds_u32_if(ids + 4u * (uint32_t)t, t < T), first = lds_u16_if(lst + 2u * (uint32_t)t, t < T);
            id = word & kIdMask;
            len = t < T && id >= hotc && in_dim(id) ? (int)((word >> kIdBits) & 31u) + 1 : 0;
            if (!CHICLE_IN_BOUNDS(S.status, len == 0 || (int)first + len <= head.z)) len = 0;
            a_val = lval + 4u * first;
            a_row = lst + 2u * (uint32_t)head.y + first;
        };
#ifdef CHICLE_LA_TIMING
        long long fe = 0, fd = 0, fu = 0, fl = 0, fs = 0, t0 = clock64(), t1 = 0;
#endif
#pragma unroll 1
        for (int b = nb > 0 ? -depth : 0; b < nb; ++b) {
            bool sl2 = false, due = b + depth < nb, late = false;
            if (due) {
                ok = ok && mbar_wait_cluster(smem_u32(&ctl.farfull[s_dot]), dot_turn, abort_flag, S.status);
                sl2 = lds_s32(smem_u32(&ctl.walk[0]) + 4u * s_dot) != 0;
                due = !sl2;
            }
            if (sl0 || sl1) {
                late = depth == 2 && sl0 && !sl1 && b + 1 < nb;
                due = due && (depth == 1 || !sl1);
            }
            due = due && ok;
            if (b + depth < nb && ok) load(s_dot, E2); // (nothing where the block is walked in place)
            LA_T(fe);
            if (b >= 0) {
                const uint32_t par = (uint32_t)(b & 1), dl = smem_u32(&ctl.dbuf[0][0]) + par * (uint32_t)(kLB * 4);
                if (sl0) { // (as the worker warps)
                    __syncwarp();
                    if (lane == 0 && ok) mbar_arrive_remote_release(ack_bar);
                }
                ok = ok && mbar_wait_cluster(smem_u32(&ctl.dbar[0]) + 8u * par, (uint32_t)(b >> 1) & 1u, abort_flag, S.status);
                if (sl0) fence_cluster();
                LA_T(fd);
                if (!sl0 && ok) {
                    auto add = [&](float x, uint32_t m) { // an id that no other coordinate of the block has
                        const float p = sigma * (x * lds_f32(dl + ((m >> (kIdBits - 2)) & 124u)));
                        const bool on = m != 0u && (m >> 31) == 0u && p != 0.0f && in_dim(m & kIdMask);
                        red_add_if(Uk + (on ? m & kIdMask : 0u), p, on);
                    };
#pragma unroll
                    for (int u = 0; u < 2; ++u) add(E0.x[u], E0.m[u]);
#pragma unroll 1
                    for (int e = lane + 64; e < E0.n; e += 32) {
                        float x;
                        uint32_t m;
                        entry(s_upd, e, true, x, m);
                        add(x, m);
                    }
                    // ids that several have: a lane per list
                    float sum = 0.0f;
#pragma unroll
                    for (int u = 0; u < 4; ++u) sum = fmaf(xl[u], lds_f32(dl + 4u * (rl[u] & 31u)), sum);
#pragma unroll 1
                    for (int e = 4; e < len; ++e) sum = fmaf(lds_f32(a_val + 4u * (uint32_t)e), lds_f32(dl + 4u * (lds_u8_if(a_row + (uint32_t)e, true) & 31u)), sum);
                    red_add_if(Uk + (len > 0 ? id : 0u), sigma * sum, len > 0 && sum != 0.0f);
#pragma unroll 1
                    for (int t0 = 32; t0 < T; t0 += 32) {
                        list_of(s_upd, t0 + lane);
                        sum = 0.0f;
#pragma unroll 1
                        for (int e = 0; e < len; ++e) sum = fmaf(lds_f32(a_val + 4u * (uint32_t)e), lds_f32(dl + 4u * (lds_u8_if(a_row + (uint32_t)e, true) & 31u)), sum);
                        red_add_if(Uk + (len > 0 ? id : 0u), sigma * sum, len > 0 && sum != 0.0f);
                    }
                }
                __syncwarp();
                mbar_arrive_if(smem_u32(&ctl.subfree[s_upd]), lane == 0 && ok); // (through with the slot's record and list)
                s_upd = s_upd + 1 == slots ? 0 : s_upd + 1;
                LA_T(fu);
            }
            if (ok && late) send(s_dot == 0 ? slots - 1 : s_dot - 1, E1, gather(E1.m[0]), gather(E1.m[1]));
            due = due && ok;
            const float w0 = gather(due ? E2.m[0] : 0u), w1 = gather(due ? E2.m[1] : 0u);
            // (while they are under way) the next block's lists
            const bool next_walked = depth == 1 ? sl2 : sl1;
            if (b + 1 >= 0 && b + 1 < nb && !next_walked && ok) {
                list_of(s_upd, lane);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    xl[u] = lds_f32_if(a_val + 4u * (uint32_t)u, u < len);
                    rl[u] = lds_u8_if(a_row + (uint32_t)u, u < len);
                }
            }
            LA_T(fl);
            if (due) send(s_dot, E2, w0, w1);
            LA_T(fs);
            E0 = depth == 1 ? E2 : E1;
            E1 = E2;
            if (++s_dot == slots) {
                s_dot = 0;
                dot_turn ^= 1u;
            }
            sl0 = next_walked;
            sl1 = sl2;
        }
#ifdef CHICLE_LA_TIMING
        if (blockIdx.x == 0 && lane == 0) {
            unsigned long long *d = P.timing + 28;
            d[0] = fe; d[1] = fd; d[2] = fu; d[3] = fl; d[4] = fs;
        }
#endif
        if (!ok && lane == 0) *abort_flag = 1;
        far_bar();
    }
    if (is_worker) {
        // ============================== the worker warps ========================================================
        // Two barriers per block, whatever the block is: in front of its update (no dot product reads the model any more) and
        // behind it. Every warp waits for deltas and records by itself; one whose wait runs out does no more work but goes on
        // meeting the others at the barriers (its abort flag ends their waits too). Nothing that it reads from then on decides
        // how often: a slot's walk flag may be rewritten under it, and a barrier that one warp leaves out never ends.
        // What these warps are bound by is the number of instructions they issue, most of them the same in every warp
        // (addresses, waits, loop ends): hence eight warps and not twelve, 32-bit shared-memory addresses and one instance
        // of the kernel per kind of data.
        const int wt = (warp - 1 - (warp >> 2)) * 32 + lane; // 0 .. kWorkThreads - 1
        const uint32_t p_bar0 = mapa_u32(smem_u32(&ctl.pbar[0]), 0u);
        const uint32_t p_buf0 = mapa_u32(smem_u32(&ctl.pbuf[0][crank][0]), 0u);
        const uint32_t ack_bar = mapa_u32(smem_u32(&ctl.ackbar), 0u);
        const uint32_t a_w = smem_u32(W), a_sink = smem_u32(&ctl.sink[lane]), stride = L.sub_stride;
        const uint32_t subs0 = smem_u32(smem_chain + L.subs), subs_end = subs0 + (uint32_t)P.slots * stride;
        const uint32_t hotc = (uint32_t)P.hotc;
        const int dstride = dense_stride(hot_mine);                // dense: floats per row of a record
        const int depth = P.depth;
        const int jd = wt >> 3, qd = wt & 7;                       // dot products: eight threads per coordinate
        uint32_t r_upd = subs0, r_dot = subs0;                     // records of blocks b and b + depth
        int fg = 0; // staged blocks whose dot products have been sent
        const int slots = P.slots;
        int s_upd = 0, s_dot = 0;  // and these records' slots (the first turns take the dot products of blocks 0, ..)
        uint32_t dot_turn = 0;     // parity of how often slot s_dot has been filled
        bool ok = true;
#ifdef CHICLE_LA_TIMING
        long long wd = 0, ws1 = 0, wg0 = 0, wg1 = 0, t0 = clock64(), t1 = 0;
#endif
        // (kEarly) where the bit of a model entry in L2 is
        const uint32_t filter0 = smem_u32(smem_chain + L.filter);
        auto bit_of = [&](uint32_t v, uint32_t &word, uint32_t &bit) {
            const uint32_t h = v >> logC;
            word = (h >> 3) & (filter_bytes(KIND) - 4u);
            bit = 1u << (h & 31u);
        };
        // a thread's entries of the dot products at hand: values, places, model entries
        float x[8], w[8];
        uint32_t m[8];
        int left = 0;
        uint32_t a_val = 0u, a_meta = 0u;
        bool more = false;
        auto entry = [&](int u) {
            x[u] = lds_f32_if(a_val + 32u * u, left > 8 * u);
            m[u] = lds_u32_if(a_meta + 32u * u, left > 8 * u) & kIdMask;
        };
        auto entries = [&]() {
            more = __any_sync(0xffffffffu, left > 32);
#pragma unroll
            for (int u = 0; u < 4; ++u) entry(u);
            if (more) {
#pragma unroll
                for (int u = 4; u < 8; ++u) entry(u);
            }
        };
        auto first_entries = [&](uint32_t rec, uint32_t n) {
            const uint32_t roff = rec + (uint32_t)offsetof(SubHead, roff) + 2u * (uint32_t)jd;
            const int first = (int)lds_u16(roff) + qd;
            left = (int)lds_u16(roff + 2u) - first; // entries of this coordinate from this thread's next one on
            a_val = rec + (uint32_t)sizeof(SubHead) + 4u * (uint32_t)first;
            a_meta = a_val + 4u * n;
            entries();
        };
        auto far_id = [&](int u) { return m[u] >= hotc && CHICLE_IN_BOUNDS(S.status, (int64_t)m[u] < S.dim); };
        auto model = [&](int u) {
            if (SPLIT) return;
            if (KIND == kHot) w[u] = lds_f32(a_w + 4u * (CHICLE_IN_BOUNDS(S.status, m[u] < hotc) ? m[u] : 0u));
            else {
                const bool far = far_id(u);
                w[u] = ldcg_if(Uk + (far ? m[u] : 0u), far);
            }
        };
        auto near = [&](int u) { // (once all gathers are on their way)
            if (FAR) {
                const float h = lds_f32(a_w + (m[u] < hotc ? 4u * m[u] : 0u));
                w[u] = m[u] < hotc ? h : w[u];
            }
            if (SPLIT) { // (the others are the far warp's)
                const float h = lds_f32(a_w + (m[u] < hotc ? 4u * m[u] : 0u));
                w[u] = m[u] < hotc ? h : 0.0f;
            }
        };
        auto model_all = [&]() {
#pragma unroll
            for (int u = 0; u < 4; ++u) model(u);
            if (more) {
#pragma unroll
                for (int u = 4; u < 8; ++u) model(u);
            }
        };
        // (debug build) a record whose sizes do not fit its slot is not read: as if its wait had run out
        auto record_fits = [&](const int4 &head) {
            if (CHICLE_IN_BOUNDS(S.status, head.w >= 0 && head.w <= kLB && (DENSE || (head.x >= 0 && head.y >= 0 && head.z >= 0 &&
                                               sub_bytes((uint32_t)head.x, (uint32_t)head.y, (uint32_t)head.z) <= stride)))) return true;
            ok = false;
            *abort_flag = 1;
            return false;
        };
        // The loop starts `depth` blocks early: those turns only take the first blocks' dot products.
        bool sl0 = false, sl1 = false; // whether blocks b and b + 1 are walked in place
#pragma unroll 1
        for (int b = nb > 0 ? -depth : 0; b < nb; ++b) {
            bool sl2 = false, due = b + depth < nb, late = false;
            // the record of the block whose dot products are next: whether it is walked in place
            auto dot_record = [&]() {
                if (!due) return;
                ok = ok && mbar_wait_cluster(smem_u32(&ctl.subfull[0]) + 8u * s_dot, dot_turn, abort_flag, S.status);
                sl2 = lds_s32(smem_u32(&ctl.walk[0]) + 4u * s_dot) != 0;
                due = !sl2;
            };
            // Dense rows: a thread's part of both records is fetched before the deltas are waited for, so that these loads, the
            // waits and the barrier are under way together (11 M logistic rows of 28: 25.5 -> 24.1 ms).
            float xu[DENSE ? kLB : 1];
            float4 xd[4];
            if (DENSE) {
                dot_record();
                const uint32_t row = r_dot + (uint32_t)sizeof(SubHead) + 4u * (uint32_t)(jd * dstride), at = r_upd + (uint32_t)sizeof(SubHead) + 4u * (uint32_t)wt;
                const bool up = b >= 0 && !sl0 && ok && wt < hot_mine && lds_s32(r_upd + 12u) == kLB, dot = ok && due && jd < lds_s32(r_dot + 12u);
                if (up) // (few warps have columns)
#pragma unroll
                    for (int j = 0; j < kLB; ++j) xu[DENSE ? j : 0] = lds_f32(at + 4u * (uint32_t)(j * dstride));
                if (dot)
#pragma unroll
                    for (int i = 0; i < 4; ++i) // (the row's first piece stands in for those it does not have)
                        xd[i] = lds_f32x4(row + (qd + 8 * i < (hot_mine + 3) >> 2 ? 16u * (uint32_t)(qd + 8 * i) : 0u));
            }
            // Ids in L2: the next dot products' gathers go out before the deltas are waited for, against the model as it is (what this
            // block's update changes is gathered again). Not in front of a block that is walked in place.
            // (2 M ridge columns over K = 128: 11.1 -> 10.6 ms a step; 5.6 M hashed rows, whose K = 64 round is of this kind, 29.1 -> 28.4.)
            bool early = false;
            if (EARLY) {
                dot_record();
                if (ok && due && !sl0 && (depth == 1 || !sl1)) {
                    const int4 head = lds_s32x4(r_dot);
                    if (record_fits(head)) {
                        first_entries(r_dot, (uint32_t)head.x);
                        model_all();
                        early = true;
                    }
                }
            }
            if (b >= 0) {
                const uint32_t par = (uint32_t)(b & 1), dbar = smem_u32(&ctl.dbar[0]) + 8u * par;
                if (sl0) {
                    // (walked in place by CTA 0: this warp's part of every update before it has been applied, and its dot
                    // products no longer read the model; say so, and wait for the walk to end)
                    __syncwarp();
                    if (lane == 0 && ok) mbar_arrive_remote_release(ack_bar);
                }
                ok = ok && mbar_wait_cluster(dbar, (uint32_t)(b >> 1) & 1u, abort_flag, S.status);
                if (sl0) fence_cluster(); // the walk's ordinary stores into this CTA's part of the model
                mbar_arrive_expect_tx_if(dbar, d_bytes, wt == 0 && ok); // for block b + 2
                work_bar();
                LA_T(wd);
                const uint32_t filter = filter0 + par * filter_bytes(KIND);
                if constexpr (EARLY) // (the other set: the dot products that looked at it are through)
#pragma unroll
                    for (uint32_t i = 0; i < filter_bytes(KIND) / (16u * kWorkThreads); ++i)
                        sts_f32x4_if(filter0 + (par ^ 1u) * filter_bytes(KIND) + 16u * ((uint32_t)wt + i * kWorkThreads), 0.0f, 0.0f, 0.0f, 0.0f, true);
                if (!sl0 && ok) {
                    // ---- block b's update of this CTA's part of the model
                    const uint32_t dl = smem_u32(&ctl.dbuf[0][0]) + par * (uint32_t)(kLB * 4);
                    const int4 head = lds_s32x4(r_upd); // n, T, nl, cnt
                    const uint32_t val = r_upd + (uint32_t)sizeof(SubHead);
                    if (DENSE) {
                        for (int col = wt; col < hot_mine; col += kWorkThreads) {
                            float s0 = 0.0f, s1 = 0.0f;
                            const uint32_t at = val + 4u * (uint32_t)col, row = 4u * (uint32_t)dstride;
                            if (head.w == kLB) { // all loads first
                                float x[kLB];
#pragma unroll
                                for (int j = 0; j < kLB; ++j) x[j] = xu[DENSE ? j : 0];
                                if (col != wt)
#pragma unroll
                                    for (int j = 0; j < kLB; ++j) x[j] = lds_f32(at + (uint32_t)j * row);
#pragma unroll
                                for (int j = 0; j < kLB; j += 4) {
                                    const float4 d = lds_f32x4(dl + 4u * j);
                                    s0 = fmaf(d.x, x[j], s0);
                                    s1 = fmaf(d.y, x[j + 1], s1);
                                    s0 = fmaf(d.z, x[j + 2], s0);
                                    s1 = fmaf(d.w, x[j + 3], s1);
                                }
                            } else
                                for (int j = 0; j < head.w; ++j) s0 = fmaf(lds_f32(dl + 4u * j), lds_f32(at + (uint32_t)j * row), s0);
                            W[col] = fmaf(sigma, s0 + s1, W[col]);
                        }
                    } else {
                        const int n = head.x, T = head.y, nl = head.z;
                        const uint32_t meta = val + 4u * (uint32_t)n, ids = meta + 4u * (uint32_t)n, lval = ids + 4u * (uint32_t)T,
                                       lst = lval + 4u * (uint32_t)nl, lrow = lst + 2u * (uint32_t)T;
                        // Four threads per shared id: each adds every fourth entry of the list (lists of up to four entries come
                        // last, so that few warps meet a longer one), then the partial sums are added in a fixed order.
                        const int q = wt & 3;
                        for (int t = wt >> 2; (t & ~7) < T; t += kWorkThreads / 4) { // (whole warps)
                            const bool on = t < T;
                            const uint32_t id = lds_u32_if(ids + 4u * (uint32_t)t, on), v = id & kIdMask;
                            const int len = on ? (int)((id >> kIdBits) & 31u) + 1 : 0;
                            const int first = (int)lds_u16_if(lst + 2u * (uint32_t)t, on) + q;
                            const uint32_t a_val = lval + 4u * (uint32_t)first, a_row = lrow + (uint32_t)first;
                            const bool near = KIND == kHot || v < hotc;
                            const float w = lds_f32(a_w + (near ? 4u * v : 0u));
                            float x[8];
                            uint32_t r[8];
                            auto take = [&](int u) {
                                const bool in = q + 4 * u < len && CHICLE_IN_BOUNDS(S.status, first + 4 * u < nl);
                                x[u] = lds_f32_if(a_val + 16u * u, in);
                                r[u] = lds_u8_if(a_row + 4u * u, in);
                            };
                            take(0);
                            float sum;
                            if (__any_sync(0xffffffffu, len > 4)) {
#pragma unroll
                                for (int u = 1; u < 8; ++u) take(u);
                                sum = x[0] * lds_f32(dl + 4u * (r[0] & 31u));
#pragma unroll
                                for (int u = 1; u < 8; ++u) sum = fmaf(x[u], lds_f32(dl + 4u * (r[u] & 31u)), sum);
                            } else sum = x[0] * lds_f32(dl + 4u * (r[0] & 31u));
                            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                            const bool mine = on && q == 0;
                            sts_f32(mine && near ? a_w + 4u * v : a_sink, fmaf(sigma, sum, w));
                            if (FAR) {
                                const bool far = mine && !near && sum != 0.0f && CHICLE_IN_BOUNDS(S.status, (int64_t)v < S.dim);
                                red_add_if(Uk + (far ? v : 0u), sigma * sum, far);
                                if (EARLY) {
                                    uint32_t word, bit;
                                    bit_of(v, word, bit);
                                    red_shared_or_if(filter + word, bit, far);
                                }
                            }
                        }
                        // A thread per entry: one whose id no other coordinate of the block has is applied (no two threads
                        // touch the same word). One store per entry, its address chosen without a branch: the model word, or
                        // a word that nobody reads; ids beyond the part in shared memory are added to at L2, nothing waits.
                        constexpr int U = 2;
                        for (int e0 = wt; (e0 & ~31) < n; e0 += U * kWorkThreads) {
                            uint32_t m[U];
                            float p[U], w[U];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const bool in = e0 + u * kWorkThreads < n;
                                const uint32_t at = 4u * (uint32_t)(e0 + u * kWorkThreads);
                                m[u] = lds_u32_if(meta + at, in);
                                p[u] = lds_f32_if(val + at, in);
                                if (!in) m[u] = 0x80000000u;
                            }
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const uint32_t v = m[u] & kIdMask;
                                p[u] = sigma * (p[u] * lds_f32(dl + ((m[u] >> (kIdBits - 2)) & 124u)));
                                if (KIND == kHot) w[u] = lds_f32(a_w + 4u * (CHICLE_IN_BOUNDS(S.status, v < hotc) ? v : 0u));
                                else w[u] = lds_f32(a_w + (v < hotc ? 4u * v : 0u));
                            }
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const uint32_t v = m[u] & kIdMask;
                                const bool mine = (m[u] >> 31) == 0u, near = KIND == kHot ? CHICLE_IN_BOUNDS(S.status, v < hotc) : v < hotc;
                                sts_f32(mine && near ? a_w + 4u * v : a_sink, p[u] + w[u]);
                                if (FAR) {
                                    const bool far = mine && !near && p[u] != 0.0f && CHICLE_IN_BOUNDS(S.status, (int64_t)v < S.dim);
                                    red_add_if(Uk + (far ? v : 0u), p[u], far);
                                    if (EARLY) {
                                        uint32_t word, bit;
                                        bit_of(v, word, bit);
                                        red_shared_or_if(filter + word, bit, far);
                                    }
                                }
                            }
                        }
                    }
                }
                r_upd = r_upd + stride == subs_end ? subs0 : r_upd + stride;
                LA_T(ws1);
            }
            // ---- dot products: of block b + depth against the model as it is now. A block right behind a walked one starts
            //      from the model as the walk left it: with depth 2 its products wait for that.
            if (!DENSE && !EARLY) dot_record();
            if (sl0 || sl1) {
                late = depth == 2 && sl0 && !sl1 && b + 1 < nb;
                due = due && (depth == 1 || !sl1);
            }
            LA_T(wg0);
            bool met = b < 0; // the barrier behind the update
            auto meet = [&]() {
                if (!met) work_bar();
                if (!met && wt == 0 && ok) mbar_arrive(smem_u32(&ctl.subfree[0]) + 8u * s_upd); // block b's slot is free
                met = true;
            };
#pragma unroll 1
            while (ok && (late || due)) {
                // (block b + 1's record lies in the slot before block b + 2's)
                const uint32_t rec = !late ? r_dot : (r_dot == subs0 ? subs_end : r_dot) - stride, val = rec + (uint32_t)sizeof(SubHead);
                const bool fetched = !late;
                if (late) late = false;
                else due = false;
                const int4 head = lds_s32x4(rec); // n, T, nl, cnt
                if (!record_fits(head)) break;
                const uint32_t slot = (uint32_t)(fg & 1);
                ++fg;
                float acc = 0.0f;
                if (DENSE) {
                    meet();
                    if (jd < head.w) {
                        const uint32_t row = val + 4u * (uint32_t)(jd * dstride);
                        float acc1 = 0.0f;
                        const int pieces = (hot_mine + 3) >> 2;
                        int e = qd;
                        if (fetched) {
                            float4 w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) w[i] = lds_f32x4(a_w + (qd + 8 * i < pieces ? 16u * (uint32_t)(qd + 8 * i) : 0u));
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (qd + 8 * i >= pieces) break;
                                acc = fmaf(xd[i].x, w[i].x, acc); acc1 = fmaf(xd[i].y, w[i].y, acc1); acc = fmaf(xd[i].z, w[i].z, acc); acc1 = fmaf(xd[i].w, w[i].w, acc1);
                            }
                            e = qd + 32;
                        }
#pragma unroll 4
                        for (; e < pieces; e += 8) {
                            const float4 a = lds_f32x4(row + 16u * e), w = lds_f32x4(a_w + 16u * e);
                            acc = fmaf(a.x, w.x, acc); acc1 = fmaf(a.y, w.y, acc1); acc = fmaf(a.z, w.z, acc); acc1 = fmaf(a.w, w.w, acc1);
                        }
                        acc += acc1;
                    }
                } else {
                    // eight entries per thread and turn, all loads of a turn issued before anything is used: an id beyond the
                    // part of the model in shared memory costs a round trip to L2 (the updates are made there by reductions)
                    if (!early) first_entries(rec, (uint32_t)head.x);
                    meet();
                    if (early && b >= 0) { // what this block's update has changed, or may have
                        const uint32_t filter = filter0 + (uint32_t)(b & 1) * filter_bytes(KIND);
                        auto again = [&](int u) {
                            const bool far = far_id(u);
                            uint32_t word, bit;
                            bit_of(m[u], word, bit);
                            ldcg_again_if(w[u], Uk + (far ? m[u] : 0u), (lds_u32_if(filter + word, far) & bit) != 0u);
                        };
#pragma unroll
                        for (int u = 0; u < 4; ++u) again(u);
                        if (more) {
#pragma unroll
                            for (int u = 4; u < 8; ++u) again(u);
                        }
                    }
#pragma unroll 1
                    for (;;) { // (whole warps)
                        if (!early) model_all();
                        early = false;
#pragma unroll
                        for (int u = 0; u < 4; ++u) near(u);
                        if (more) {
#pragma unroll
                            for (int u = 4; u < 8; ++u) near(u);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc = fmaf(x[u], w[u], acc);
                        if (!more) break;
#pragma unroll
                        for (int u = 4; u < 8; ++u) acc = fmaf(x[u], w[u], acc);
                        left -= 64;
                        if (!__any_sync(0xffffffffu, left > 0)) break;
                        a_val += 256u;
                        a_meta += 256u;
                        entries();
                    }
                }
                acc += __shfl_xor_sync(0xffffffffu, acc, 1);
                acc += __shfl_xor_sync(0xffffffffu, acc, 2);
                acc += __shfl_xor_sync(0xffffffffu, acc, 4);
                st_async_f32_if(p_buf0 + (slot * (uint32_t)(kMaxC * kLB) + (uint32_t)jd) * 4u, acc, p_bar0 + slot * 8u, qd == 0);
            }
            meet();
            r_dot = r_dot + stride == subs_end ? subs0 : r_dot + stride;
            if (++s_dot == slots) {
                s_dot = 0;
                dot_turn ^= 1u;
            }
            if (b >= 0) s_upd = s_upd + 1 == slots ? 0 : s_upd + 1;
            LA_T(wg1);
            sl0 = depth == 1 ? sl2 : sl1;
            sl1 = sl2;
        }
        if (!ok && lane == 0) *abort_flag = 1;
        if (SPLIT) far_bar(); // (the far warp's updates have been made)
        aborted = !ok; // (otherwise: every update has been applied, the last barrier says so)
#ifdef CHICLE_LA_TIMING
        if (blockIdx.x == 0 && wt == 0) {
            unsigned long long *d = P.timing + 4;
            d[0] = wd; d[3] = ws1; d[4] = wg0; d[5] = wg1;
        }
#endif
        if (!aborted) {
            // the model goes back to row k: as it is, or after the round's last launch as the update U_k = (w - v) / sigma'
            const float inv_sigma = 1.0f / sigma;
            for (int l0 = wt; l0 < hot_mine; l0 += 8 * kWorkThreads) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int l = l0 + i * kWorkThreads;
                    const bool in = l < hot_mine && P.model_out;
                    v[i] = ldcg_if(S.vbase + (!in ? 0 : (DENSE ? (size_t)(slice0 + l) : ((size_t)l << logC) + crank)), in);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int l = l0 + i * kWorkThreads;
                    if (l < hot_mine) Uk[DENSE ? (size_t)(slice0 + l) : ((size_t)l << logC) + crank] = P.model_out ? (W[l] - v[i]) * inv_sigma : W[l];
                }
            }
            if (P.model_out)
                for (size_t g0 = cold0 + ((size_t)wt << logC); g0 < (size_t)S.dim; g0 += (size_t)(8 * kWorkThreads) << logC) {
                    float u[8], v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const size_t g = g0 + ((size_t)(i * kWorkThreads) << logC);
                        const bool in = g < (size_t)S.dim;
                        u[i] = ldcg_if(Uk + (in ? g : 0), in);
                        v[i] = ldcg_if(S.vbase + (in ? g : 0), in);
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const size_t g = g0 + ((size_t)(i * kWorkThreads) << logC);
                        if (g < (size_t)S.dim) Uk[g] = (u[i] - v[i]) * inv_sigma;
                    }
                }
        }
    }
    if (is_worker || nb == 0) {
        if ((tid & 31) == 0) *reinterpret_cast<volatile int *>(&ctl.done) = 1;
    } else if (!is_chain) {
        // a warp with no role sleeps until the workers are through: waiting at the cluster barrier from the start
        // would take issue slots from the recurrence warp, which shares its scheduler with these warps
        const volatile int *done = &ctl.done;
        for (uint32_t it = 0; it < (1u << 24) && !*done; ++it) __nanosleep(2000);
    }
    // nobody leaves while another CTA of the cluster may still write to, or read from, its shared memory (after an abort
    // asynchronous stores may be on their way that no role waits for any more: a millisecond for them)
    __syncwarp();
    if (*abort_flag)
        for (int i = 0; i < 16; ++i) __nanosleep(64000);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}

template <int LOSS, int KIND, bool TAB> cudaError_t launch_chain_kind(Glm &g, const LookParams &P, cudaEvent_t begun)
{
    auto kern = k_lookahead_chain<LOSS, KIND, TAB>;
    if (chain_layout(P.sub_room, P.slots, P.hotc, KIND == kDense, TAB ? P.tab_bins : 0, KIND, P.far_cap).total > g.la_smem) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.la_smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.K << g.la_logC, 1, 1);
    cfg.blockDim = dim3(chain_threads(KIND), 1, 1);
    cfg.dynamicSmemBytes = g.la_smem;
    cfg.stream = g.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << g.la_logC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (begun) {
        attr[1].id = cudaLaunchAttributeLaunchCompletionEvent;
        attr[1].val.launchCompletionEvent.event = begun;
        attr[1].val.launchCompletionEvent.flags = 0;
        cfg.numAttrs = 2;
    }
    e = cudaLaunchKernelEx(&cfg, kern, P);
#ifdef CHICLE_LA_TIMING
    if (e == cudaSuccess) {
        unsigned long long t[33] = {0};
        (void)cudaStreamSynchronize(g.stream);
        (void)cudaMemcpy(t, P.timing, sizeof(t), cudaMemcpyDeviceToHost);
        const double nb = t[3] ? (double)t[3] : 1.0;
        fprintf(stderr, "lookahead chain, cycles per block (partition 0): waiting for dot products %.0f, recurrence %.0f, deltas %.0f; "
                "workers of CTA 0: waiting for deltas %.0f, update %.0f, record wait %.0f, products %.0f (%llu blocks)\n",
                t[0] / nb, t[1] / nb, t[2] / nb, t[4] / nb, t[7] / nb, t[8] / nb, t[9] / nb, t[3]);
        if (KIND == kEarly || KIND == kSplit) fprintf(stderr, "  record warp of CTA 0: waiting for the record %.0f, entries beyond shared memory %.0f, slot and copy %.0f\n", t[24] / nb, t[25] / nb, t[26] / nb);
        if (KIND == kSplit) fprintf(stderr, "  far warp of CTA 0: entries %.0f, waiting for deltas %.0f, update %.0f, gathers out and next lists %.0f, gathers back and sums %.0f\n",
                                    t[28] / nb, t[29] / nb, t[30] / nb, t[31] / nb, t[32] / nb);
    }
#endif
    return e;
}

template <int LOSS, int NZ, int HT, int THREADS, int PER_SM> cudaError_t launch_prepare(const LookParams &P, unsigned sms, cudaStream_t stream)
{
    using Shared = PreShared<NZ, HT, THREADS>;
    static_assert(PER_SM * (sizeof(Shared) + 1024) <= 228 * 1024, "CTAs per SM");
    auto pre = k_lookahead_prepare<LOSS, NZ, HT, THREADS, PER_SM>;
    cudaError_t e = cudaFuncSetAttribute(pre, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)P.n_blocks;
    const unsigned grid = nb < sms * PER_SM ? nb : sms * PER_SM;
    pre<<<grid, THREADS, sizeof(Shared), stream>>>(P);
    return cudaGetLastError();
}

// Not for the logistic loss: its recurrence is what a block takes, and the record warp, which lists the far warp's entries, shares its
// scheduler. Rows of 39 with tables, 6 to 30 entries a block, local solvers with the far warp and without, ms: 50 000, K = 2: 2.36, 2.25;
// 200 000, K = 9: 2.18, 2.13; 400 000, K = 16: 2.24, 2.18; 500 000, K = 30: 1.95, 1.93; 750 000, K = 64: 2.43, 2.44 (early gathers).
constexpr int kSplitLeast = 4096;    // ids per CTA in shared memory that the far warp's lists must leave
// Entries beyond them that a block may be expected to have in a CTA's record: few blocks then have more than the 64 that the far warp
// keeps in registers; with more of those it is the slowest of all roles. Local solvers, ms, with the far warp and without:
//   two ahead: 47 entries, K = 2, C = 8 (rows of 39): 4.10, 4.37; 58: 4.36, 4.38; 50, K = 4: 4.38, 4.56; 57 (rows of 60): 4.73, 4.70; 62 (rows of
//   39): 4.87, 4.55; 59, K = 9 (rows of 60): 4.63, 4.46; 54, K = 16, C = 4 (rows of 39): 3.76, 3.85; 61 (rows of 15): 4.01, 3.63; 85: 4.96, 3.84;
//   50, K = 30, C = 2 (rows of 15): 2.96, 3.07; 67: 3.58, 3.08; 10 to 40 (rows of 39): 3.96, 3.85
//   one ahead: 36, K = 64, C = 1 (rows of 39): 4.61, 4.72; 77: 4.70, 4.73; 47 (rows of 15): 3.44, 3.38; 62: 3.60, 3.38; 55, K = 100: 4.65, 4.92;
//   several hundred, ridge over K = 128: 17.1, 10.6 (the step)
constexpr double kSplitMost = 56.0;
// Two blocks ahead, a gather has a block's time as it is, and the record warp, which must look at every entry, sets the pace where records
// are long: the far warp only up to this many entries a record. Local solvers, ms, with the far warp and without, 10 to 30 entries beyond shared
// memory: 800 (rows of 50, K = 20, C = 2): 2.55, 1.99; 1 024: 2.87, 2.38; 624 (K = 30): 3.96, 3.85; 240: 2.83, 3.03; 360 (K = 16, C = 4): 2.62, 2.75;
// 400: 2.81, 2.80; 480: 3.11, 3.08; 320 (K = 9, C = 8): 2.75, 2.85; 400: 3.32, 3.32; 480: 3.98, 3.96. (One ahead, K = 64, 1 920: 1.91, 1.92; 2 560: 2.31, 2.31.)
constexpr double kSplitLongest = 380.0;
// Gathers early and behind the update, ms (rows of 39 but where noted).
// Two ahead, going out early costs more than it saves unless most of a record's entries, and at least this many, lie beyond shared memory:
//   72 of 156 entries, K = 2, C = 8: 4.49, 4.16; 84, K = 9: 4.13, 4.05; 133: 5.23, 5.20; 85 of 480, K = 16, C = 4 (rows of 60): 4.26, 4.20; 214: 4.22, 4.18;
//   109 of 120 (rows of 15): 5.07, 4.97; 215 of 240 (rows of 30): 4.71, 4.83; 240 of 312: 4.10, 4.19; 185 of 240, K = 30, C = 2 (rows of 15): 3.15, 3.16;
//   300 of 320 (rows of 20): 3.52, 3.59; 590 of 1 024 (rows of 64): 4.03, 3.94; 919 of 960 (rows of 60): 5.29, 5.63
// One ahead it pays while records are not longer than that:
//   27 of 1 248, K = 64, C = 1: 4.71, 4.71; 77: 4.73, 4.76; 157: 4.73, 4.84; 298: 4.77, 4.95; 60 of 480 (rows of 15): 3.38, 3.51; 110 of 1 248, K = 100:
//   4.94, 5.04; 1 161 of 1 280, C = 2 (rows of 80): 5.31, 5.55; 871 of 1 920 (rows of 60): 3.02, 3.00; 158 of 2 560 (rows of 80): 3.74, 3.67; 7 of 3 520 (rows
//   of 110): 3.14, 3.08; 229 of 1 600, logistic with tables (rows of 50): 2.99, 2.90
constexpr double kEarlyShare = 0.7, kEarlyLongest = 1400.0;
constexpr double kEarlyLeast = 180.0;
// Entries that a block of 32 random coordinates is expected to have with ids from `first` on.
double entries_beyond(const Glm &g, int64_t first)
{
    double e = 0.0;
    for (int k = 0; k < kOctaves; ++k) {
        const double lo = k == 0 ? 0.0 : (double)((int64_t)1 << k), hi = fmin((double)((int64_t)2 << k), (double)g.dim);
        if (hi > (double)first && hi > lo) e += g.blk_octave[k] * (lo >= (double)first ? 1.0 : (hi - (double)first) / (hi - lo));
    }
    return e;
}
constexpr int kPreSmallNz = 2048, kPreSmallHt = 2048;
constexpr int kPreMidNz = 3072, kPreMidHt = 4096;
constexpr int kPreLargeNz = 4096, kPreLargeHt = 4096;

// Whether the prepare kernel with arrays for `nz` non-zeros and `ht` ids per block serves: blocks of average rows `spare` times
// over; partitions by chunks, whose rows may be the long ones, blocks of the longest partition's average rows and three standard
// deviations more. (400 000 rows of 45 on average, sorted by length, K = 64: 3.3 ms a round with the arrays for 2 048, 1.9 with the
// larger ones; the same rows over K = 8 and 16, whose partitions differ less, 2.5 -> 2.2 and 2.2 -> 1.9 with the smaller ones.)
bool arrays_serve(const Glm &g, bool by_chunks, double chunk_mean, int nz, int ht, double spare)
{
    const double mean = (double)g.nnz / (double)g.n_coord;
    return kLB * mean * spare <= (double)nz && (!by_chunks || kLB * chunk_mean + 3.0 * sqrt(kLB * g.row_variance) <= (double)pre_room(nz, ht));
}
// The prepare kernel that serves: 0 small (32 coordinates of 50 on average, with room), 1, 2 the longest blocks
int arrays_of(const Glm &g, bool by_chunks, double chunk_mean)
{
    return arrays_serve(g, by_chunks, chunk_mean, kPreSmallNz, kPreSmallHt, 1.25) ? 0 : (arrays_serve(g, by_chunks, chunk_mean, kPreMidNz, kPreMidHt, 1.1) ? 1 : 2);
}
int arrays_of(const Glm &g) { return arrays_of(g, g.by_chunks, g.chunk_mean); }
// entries of a block that it has room for
int prepare_room(const Glm &g)
{
    const int a = arrays_of(g);
    return a == 0 ? pre_room(kPreSmallNz, kPreSmallHt) : (a == 1 ? pre_room(kPreMidNz, kPreMidHt) : pre_room(kPreLargeNz, kPreLargeHt));
}

// The prepare kernel of one launch's blocks on `stream`.
template <int LOSS> cudaError_t launch_prepare_on(Glm &g, const LookParams &P, cudaStream_t stream)
{
    const unsigned nb = (unsigned)P.n_blocks;
    if (nb == 0) return cudaSuccess;
    // beside the chain kernels: no more CTAs than fit the SMs the chains leave (see k_lookahead_prepare)
    const int chain_sms = g.K << g.la_logC;
    const unsigned free_sms = (unsigned)(g.sm_count > chain_sms ? g.sm_count - chain_sms : 1);
    if (g.fmt == CHICLE_FMT_DENSE_ROWMAJOR) {
        const bool lng = dense_long(g.dim);
        const unsigned per_sm = lng ? kPreDenseLongPerSm : kPreDensePerSm;
        const size_t smem = pre_dense_bytes((int)g.dim, lng);
        const unsigned grid = stream == g.stream || nb < free_sms * per_sm ? nb : free_sms * per_sm;
        auto pre = lng ? k_lookahead_prepare_dense<LOSS, true> : k_lookahead_prepare_dense<LOSS, false>;
        cudaError_t e = cudaFuncSetAttribute(pre, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        pre<<<grid, kPreThreads, smem, stream>>>(P);
        return cudaGetLastError();
    }
    cudaError_t e;
    const unsigned sms = stream == g.stream ? (unsigned)g.sm_count : free_sms;
    const int arrays = arrays_of(g);
    if (arrays == 0) e = launch_prepare<LOSS, kPreSmallNz, kPreSmallHt, 512, 2>(P, sms, stream);
    else if (arrays == 1) e = launch_prepare<LOSS, kPreMidNz, kPreMidHt, 1024, 1>(P, sms, stream);
    else e = launch_prepare<LOSS, kPreLargeNz, kPreLargeHt, 1024, 1>(P, sms, stream);
#ifdef CHICLE_LA_TIMING
    if (e == cudaSuccess) {
        unsigned long long t[8] = {0};
        (void)cudaStreamSynchronize(stream);
        (void)cudaMemcpy(t, P.timing + 16, sizeof(t), cudaMemcpyDeviceToHost);
        (void)cudaMemset(P.timing + 16, 0, sizeof(t));
        const double n = (double)nb;
        fprintf(stderr, "lookahead prepare, cycles per block: insert %.0f, number %.0f, place and next entries %.0f, entries %.0f, pairs and dense part %.0f, write %.0f\n", t[0] / n, t[1] / n, t[2] / n, t[3] / n, t[4] / n, t[5] / n);
    }
#endif
    return e;
}

template <int LOSS, int KIND, bool TABLES> cudaError_t launch_chain(Glm &g, const LookParams &P, cudaEvent_t begun)
{
    return TABLES && P.tab_bins ? launch_chain_kind<LOSS, KIND, TABLES>(g, P, begun) : launch_chain_kind<LOSS, KIND, false>(g, P, begun);
}

int chain_kind(const Glm &g)
{
    if (g.fmt == CHICLE_FMT_DENSE_ROWMAJOR) return kDense;
    if (((int64_t)g.la_hotc << g.la_logC) >= g.dim) return kHot;
    // (Partitions by chunks may be sorted: one with all the rare ids has many where the average over random blocks has few, and its far
    // warp would set the pace. 1 M rows of 39 over K = 16 by chunks, 45 entries a block on average and up to 220: 9.17 against 4.10 ms,
    // 4.18 before there was a far warp; as many everywhere, 8: 3.60 against 3.81.)
    if (g.la_far_cap > 0) return g.la_far_worst <= kSplitMost ? kSplit : kCold;
    return g.la_early ? kEarly : kCold;
}
template <int LOSS> cudaError_t launch_chain_on(Glm &g, const LookParams &P, cudaEvent_t begun = nullptr)
{
    constexpr bool tables = LOSS == CHICLE_LOSS_LOGISTIC_DUAL;
    switch (chain_kind(g)) {
    case kDense: return launch_chain<LOSS, kDense, tables>(g, P, begun);
    case kHot: return launch_chain<LOSS, kHot, tables>(g, P, begun);
    case kSplit:
        if constexpr (LOSS != CHICLE_LOSS_LOGISTIC_DUAL) return launch_chain<LOSS, kSplit, tables>(g, P, begun);
        else return cudaErrorInvalidConfiguration; // (never planned)
    case kEarly: return launch_chain<LOSS, kEarly, tables>(g, P, begun);
    default: return launch_chain<LOSS, kCold, tables>(g, P, begun);
    }
}

constexpr size_t kWordsPerLaunch = 480;
struct WordArgs { int64_t w[kWordsPerLaunch]; };
__global__ void k_words(const __grid_constant__ WordArgs a, int n, int64_t *dst)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = a.w[i];
}

// A round's launches, slice after slice (consecutive pieces of every partition's walk). The first slice's prepare
// kernel runs on the handle's stream; the later ones on the side stream, where they fill the SMs the chain kernels
// leave idle; every chain launch waits for its slice's prepare kernel. The records of slice s lie in region s mod R
// of the record buffer, so the prepare kernel of slice s also waits for the chain launch of slice s - R.
// A chain launch needs whole SMs (whole clusters of them), a prepare kernel spreads over whatever is free: one that gets
// in between two chain launches holds the second up until it is through (1 M sparse rows, K = 16: 0.7 of 5.4 ms). So
// slice s + 1's prepare kernel is let go once the CTAs of slice s's chain launch have begun. (Order of starts only:
// what is read and overwritten is ordered by the other events.)
template <int LOSS> cudaError_t launch_slices(Glm &g, std::vector<LookParams> &P)
{
    const int S = (int)P.size(), R = g.la_regions;
    cudaError_t e = cudaSuccess;
    if (!g.la_overlap) {
        // the chains take most of the SMs: the prepare kernels get the whole GPU between the chain launches instead of
        // the few SMs beside them
        for (int s = 0; s < S && e == cudaSuccess; ++s) {
            e = launch_prepare_on<LOSS>(g, P[s], g.stream);
            if (s == 0 && g.time_prepare) (void)cudaEventRecord(g.ev[4], g.stream);
            if (e == cudaSuccess) e = launch_chain_on<LOSS>(g, P[s]);
        }
        return e;
    }
    e = launch_prepare_on<LOSS>(g, P[0], g.stream);
    if (e != cudaSuccess) return e;
    if (g.time_prepare) (void)cudaEventRecord(g.ev[4], g.stream);
    if (S > 1) {
        e = cudaEventRecord(g.la_ev_prep[0], g.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(g.la_stream, g.la_ev_prep[0], 0); // behind all of the caller's stream so far
    }
    for (int s = 0; s < S && e == cudaSuccess; ++s) {
        if (s > 0) e = cudaStreamWaitEvent(g.stream, g.la_ev_prep[s], 0);
        if (e == cudaSuccess) e = launch_chain_on<LOSS>(g, P[s], s + 1 < S ? g.la_ev_begun[s] : nullptr);
        if (s + 1 == S || e != cudaSuccess) break;
        e = cudaEventRecord(g.la_ev_done[s], g.stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(g.la_stream, g.la_ev_begun[s], 0);
        // (its region is free once the chain launch of slice s + 1 - R is done)
        if (e == cudaSuccess && s + 1 >= R) e = cudaStreamWaitEvent(g.la_stream, g.la_ev_done[s + 1 - R], 0);
        if (e == cudaSuccess) e = launch_prepare_on<LOSS>(g, P[s + 1], g.la_stream);
        if (e == cudaSuccess) e = cudaEventRecord(g.la_ev_prep[s + 1], g.la_stream);
    }
    return e;
}

} // namespace

// A few words of host memory to the device: as arguments of a kernel (a copy from pageable memory costs the host 15 us, and
// the stream waits for it); many of them as a copy from pageable memory, which the runtime has read when the call returns (the
// caller's array may be pinned, and is then read when the stream gets there).
cudaError_t launch_words(Glm &g, int64_t *dst, const int64_t *src, size_t n)
{
    if (n > 8 * kWordsPerLaunch) {
        const std::vector<int64_t> own(src, src + n);
        return cudaMemcpyAsync(dst, own.data(), n * sizeof(int64_t), cudaMemcpyHostToDevice, g.stream);
    }
    for (size_t at = 0; at < n; at += kWordsPerLaunch) {
        WordArgs a;
        const size_t m = n - at < kWordsPerLaunch ? n - at : kWordsPerLaunch;
        std::memcpy(a.w, src + at, m * sizeof(int64_t));
        k_words<<<1, 256, 0, g.stream>>>(a, (int)m, dst + at);
    }
    return cudaGetLastError();
}

// (for the log: which instance of the chain kernel a round takes decides what a test of it has tested)
LookChain lookahead_chain(const Glm &g)
{
    static const char *const names[] = {"whole", "cold", "dense", "far-warp", "early"}; // by kind
    const int64_t hot = std::min((int64_t)g.la_hotc << g.la_logC, g.dim);
    const bool dense = g.fmt == CHICLE_FMT_DENSE_ROWMAJOR;
    return {names[chain_kind(g)], dense ? g.dim : hot, dense ? 0.0 : entries_beyond(g, hot) / (1 << g.la_logC)};
}
int lookahead_arrays(const Glm &g, bool by_chunks, double chunk_mean) { return arrays_of(g, by_chunks, chunk_mean); }
int lookahead_max_dense_dim() { return kMaxC * kDenseSlice; }
int lookahead_max_slices() { return 64; }
int64_t lookahead_max_dim() { return (int64_t)1 << kIdBits; }

// Sizes the look-ahead solver for a partition into K: CTAs per cluster, what stays in shared memory, and the record
// buffer: `regions` regions that each hold one slice of a round (the recurrence records of its blocks, then a pool
// for the workers' records).
void lookahead_plan(Glm &g, int32_t K, bool want_tables)
{
    const bool dense = g.fmt == CHICLE_FMT_DENSE_ROWMAJOR;
    int logC = 0;
    if (!dense) {
        // a cluster per partition, on at most half of the SMs: the prepare kernels need the rest
        while (logC < 3 && ((int64_t)K << (logC + 1)) * 2 <= g.sm_count) ++logC;
        // Many partitions on a long vector with flat ids: all their models together (less what 32 000 words of shared memory each keep) are
        // more than L2 holds, and gathers go to memory. With two CTAs per partition half of the partitions run at a time, each
        // with twice the shared memory (ridge, 2 M columns over 350 000 rows, K = 128: 10 400 cycles a block instead of 26 400;
        // step 14.3 -> 12.6 ms. Four: 6 170, but a quarter of the partitions at a time: 14.8 ms).
        if (logC == 0 && !g.hot_variant && g.l2_bytes > 0 && g.dim > 32000 && (double)K * (double)(g.dim - 32000) * 4.0 > (double)g.l2_bytes) logC = 1;
        const char *env = getenv("CHICLE_LA_CLUSTER");
        if (env && env[0] >= '1' && env[0] <= '8' && env[1] == 0) {
            const int want = env[0] - '0';
            logC = want >= 8 ? 3 : (want >= 4 ? 2 : (want >= 2 ? 1 : 0));
        }
    }
    int slice = (int)((g.dim + 3) & ~(int64_t)3); // dense: columns per CTA
    if (dense) {
        // Long rows are shared out over a cluster: slices of about 128 columns where the SMs allow it for all partitions at
        // once, else as few CTAs as slices of 384 columns need (the most that
        // four blocks' slices leave room for); the clusters then take turns.
        auto cut = [&](int lg) { return (int)((((g.dim + (1 << lg) - 1) >> lg) + 3) & ~(int64_t)3); };
        while (logC < 3 && cut(logC) > kDenseSlice) ++logC;
        while (logC < 3 && cut(logC) > kDenseEasy && ((int64_t)K << (logC + 1)) <= g.sm_count) ++logC;
        slice = cut(logC);
    }
    g.la_logC = logC;
    // Beside chains on at most half of the SMs the prepare kernels run on the side stream; otherwise they alternate with
    // the chain launches and have the whole GPU meanwhile (2 M ridge columns over K = 128: 12.5 against 584 ms a step).
    g.la_overlap = ((int64_t)K << logC) * 2 <= g.sm_count;
    // Two blocks ahead pays where the chains bound the round: dense rows (10 000 of 100, K = 4: 186 against 247 us a step) and
    // sparse data with a cluster per partition (1 M rows of 50, K = 16, before the prepare kernel became shorter: 4.0 against 5.2 ms; 45 M of 39: 156 against 278). One CTA
    // per partition on sparse data means many partitions: there the prepare kernels bound the round, and are shorter without
    // the cross Gram matrices (5.6 M hashed rows, a round with K = 64 and one with K = 16: 28.4 against 29.3 ms).
    g.la_depth = (dense || logC >= 1) && g.la_overlap ? 2 : 1;
    {
        const char *env = getenv("CHICLE_LA_DEPTH");
        if (env && (env[0] == '1' || env[0] == '2') && env[1] == 0) g.la_depth = env[0] - '0';
        env = getenv("CHICLE_LA_OVERLAP");
        if (env && (env[0] == '0' || env[0] == '1') && env[1] == 0) g.la_overlap = env[0] == '1';
    }
    const size_t budget = (size_t)(g.max_smem_optin > 0 ? g.max_smem_optin : 227 * 1024);
    // logistic tables: as many bins as the largest q = sigma' |x|^2 / (lambda n) at sigma' = K needs (a round with a larger
    // sigma' solves the roots on the chain), if two blocks' tables fit beside the rest
    g.la_tab_bins = 0;
    if (g.loss == CHICLE_LOSS_LOGISTIC_DUAL && want_tables) {
        const float q_max = (float)K * g.max_sqnorm / (g.lambda * (float)g.n_examples);
        for (int bins = 64; bins >= 32; bins >>= 1)
            if (q_max <= tab_max_q(bins)) g.la_tab_bins = bins;
        if (dense && chain_layout(0, kSubSlots, slice, true, g.la_tab_bins, kDense).total > budget) g.la_tab_bins = 0;
        const char *env = getenv("CHICLE_LA_TABLES"); // 0: none (tests)
        if (env && env[0] == '0') g.la_tab_bins = 0;
    }
    g.la_slots = kSubSlots;
    g.la_sub_room = 0;
    g.la_hotc = slice;
    g.la_far_cap = 0;
    g.la_far_worst = 0.0; // (of the partition before; what follows sizes the shared memory for the instance that the plan allows)
    g.la_early = false;
    if (!dense) {
        // A slot holds the record that a block of 32 random coordinates is expected to make for a CTA (how many entries, and how
        // many of them with ids that several of the 32 have: from the ids' frequencies, see launch_frequency_remap) and five
        // standard deviations more (`room`). Partitions by chunks may be sorted by class, time or length: the record of a block as
        // long as the prepare kernel takes, whatever its rows share (`most`). (400 000 rows of 50, sorted by topic, K = 8: 82 ms a
        // round with the first, 2.3 with the second.) What is left keeps the model's most frequent ids. Where that leaves the
        // model little, three slots do if dot products are taken one block ahead, and the root search on the chain instead of
        // tables: a block without room is walked in place, 20 times slower. (`most` for random partitions too: 2 M ridge columns
        // over K = 128 12.5 -> 12.8 ms, logistic rows of 80 over K = 64, which lose their tables, 2.8 -> 3.8.)
        const int C = 1 << logC;
        uint32_t room = 256, most = 256;
        double n_max = 0.0, n_mean = 0.0; // entries of a CTA's record: at most, on average
        const double cap = (double)prepare_room(g); // (a block with more entries is walked in place anyway)
        for (int c = 0; c < C; ++c) {
            double n = 0.0, T = 0.0, nl = 0.0;
            for (int i = c; i < kRankClasses; i += C) { n += g.blk_entries[i]; T += g.blk_shared_ids[i]; nl += g.blk_shared[i]; }
            const double all = (double)kLB * (double)g.nnz / (double)g.n_coord, part = all > 0.0 ? n / all : 0.0;
            double n_hi = n + 5.0 * sqrt(n + part * part * kLB * g.row_variance);
            if (g.by_chunks) n_hi = fmax(n_hi, part * cap + 5.0 * sqrt(part * cap));
            n_hi = fmin(n_hi, cap);
            const double f = n > 0.0 ? fmax(1.0, n_hi / n) : 1.0;
            const double nl_hi = fmin(n_hi, f * nl + 5.0 * sqrt(nl)), T_hi = fmin(0.5 * nl_hi, f * T + 5.0 * sqrt(T));
            const uint32_t r = sub_bytes((uint32_t)n_hi + 1u, (uint32_t)T_hi + 1u, (uint32_t)nl_hi + 1u) + 64u;
            const uint32_t m = sub_bytes((uint32_t)n_hi + 1u, (uint32_t)(0.5 * n_hi) + 1u, (uint32_t)n_hi + 1u) + 64u;
            n_max = fmax(n_max, n_hi);
            n_mean = fmax(n_mean, n);
            room = r > room ? r : room;
            most = m > most ? m : most;
        }
        if (g.by_chunks) room = most;
        for (;;) {
            // (The filters of early gathers are set aside where there are no tables, which they must not cost: 89 000 logistic rows of 80 over K = 32
            // by chunks 0.72 ms with tables, 1.05 without.)
            const double left = (double)budget - (double)chain_layout(0, 0, 0, false, g.la_tab_bins, g.la_tab_bins > 0 ? kCold : kEarly).total - 64.0;
            g.la_slots = g.la_depth == 1 && 4.0 * room > 0.6 * left ? 3 : kSubSlots;
            if (g.la_tab_bins == 0 || (double)g.la_slots * room <= 0.8 * left) {
                const uint32_t limit = (uint32_t)(0.8 * left / g.la_slots) & ~15u;
                g.la_sub_room = room < limit ? room : limit;
                break;
            }
            g.la_tab_bins = 0;
        }
        const ChainLayout L0 = chain_layout(g.la_sub_room, g.la_slots, 0, false, g.la_tab_bins, kHot);
        int64_t hotc = ((int64_t)budget - (int64_t)L0.total - 64) / 4;
        const int64_t need = (g.dim + ((int64_t)1 << logC) - 1) >> logC; // per CTA for the whole model
        if (hotc < need) {
            // the rest lies in L2: lists for the far warp, where they leave the model something; two filters for early gathers; or nothing
            const int cap = ((int)n_max + 32) & ~31;
            const int64_t split = hotc - (int64_t)far_bytes(kSplit, cap, g.la_slots) / 4;
            const bool far_warp = split >= kSplitLeast && g.loss != CHICLE_LOSS_LOGISTIC_DUAL && (g.la_depth == 1 || n_mean <= kSplitLongest);
            const double beyond = far_warp ? entries_beyond(g, split << logC) / C : 1e30;
            if (beyond <= kSplitMost) {
                hotc = split;
                g.la_far_cap = cap;
            } else if (hotc > (int64_t)filter_bytes(kEarly) &&
                       (g.la_depth == 1 ? n_mean <= kEarlyLongest : entries_beyond(g, hotc << logC) / C > fmax(kEarlyLeast, kEarlyShare * n_mean))) {
                hotc -= (int64_t)filter_bytes(kEarly) / 2;
                g.la_early = true;
            }
        }
        hotc = (hotc / 32) * 32;
        // (what the whole model leaves goes to the slots: rows may be more alike than their ids' frequencies say)
        const int64_t spare = (4 * (hotc - (need + 31) / 32 * 32) / g.la_slots) & ~(int64_t)15;
        if (spare > 0 && g.la_sub_room < most) g.la_sub_room += (uint32_t)((int64_t)(most - g.la_sub_room) < spare ? most - g.la_sub_room : spare);
        g.la_hotc = (int32_t)(hotc < need ? hotc : (need + 31) / 32 * 32);
    }
    g.la_smem = chain_layout(g.la_sub_room, g.la_slots, g.la_hotc, dense, g.la_tab_bins, chain_kind(g), g.la_far_cap).total;

    // slices: at most a sixteenth of the walk, but at least 256 blocks per partition; two regions
    const int64_t n = g.n_coord;
    const int64_t max_nk = (n + K - 1) / K + 1;
    const int64_t max_nb = (max_nk + kLB - 1) / kLB;
    int64_t per_part = (max_nb + 15) / 16;
    per_part = per_part < 256 ? 256 : per_part;
    per_part = per_part > max_nb ? max_nb : per_part;
    const bool whole = per_part >= max_nb; // a round is one slice
    // (partitions of unequal sizes: the largest may hold almost everything; a region then holds what a sixteenth of
    // the whole walk needs, and the launch cuts finer if a slice does not fit)
    int64_t region_blocks = whole ? n / kLB + K + 1 : per_part * K + K;
    if (region_blocks > n / kLB + K + 1) region_blocks = n / kLB + K + 1;
    g.la_region_blocks = region_blocks;
    g.la_regions = whole ? 1 : 2;
    {
        const char *env = getenv("CHICLE_LA_SLICES"); // forced slicing (tests): the ring as large problems have it
        if (env && atoi(env) > 1) g.la_regions = 2;
    }
    const double frac = whole ? 1.0 : (double)region_blocks / (double)(n / kLB + 1);
    const size_t C = (size_t)1 << logC;
    size_t pool;
    if (dense) pool = (size_t)region_blocks * C * sub_bytes_dense(kLB, slice);
    else {
        const double all = 16.0 * (double)g.nnz;
        double part = whole ? all : 1.2 * frac * all + (double)(1 << 20);
        if (part > all) part = all;
        // (what the prepare kernel's CTAs hold in advance: a piece of about four blocks each)
        g.la_pool_piece = ((size_t)(4.0 * 12.0 * 32.0 * (double)g.nnz / (double)g.n_coord) + 4096) & ~(size_t)255; // (records start on 16-byte boundaries)
        part += (double)g.la_pool_piece * (double)(region_blocks < 2 * (int64_t)g.sm_count ? region_blocks : 2 * (int64_t)g.sm_count);
        // (what is left of a piece when the next block's records are longer: up to a quarter where rows share most ids. Without this,
        // rows of 50 over 100 ids, 1 M of them over K = 128, had no room for 610 of 32 000 blocks: 4.7 instead of 3.4 ms a round)
        pool = (size_t)part + (size_t)region_blocks * (C * 128 + 1408) + 4096;
    }
    const size_t heads = ((size_t)region_blocks * sizeof(ChainHead) + 255) & ~(size_t)255;
    const size_t tabs = (size_t)region_blocks * tab_bytes(g.la_tab_bins);
    g.la_tab_off = heads;
    g.la_pool_off = heads + tabs;
    g.la_region_bytes = (heads + tabs + pool + 255) & ~(size_t)255;
    g.la_dir_bytes = (size_t)g.la_regions * (size_t)region_blocks * C * sizeof(BlkDir);
}

cudaError_t launch_lookahead_solver(Glm &g, const SolverParams &S)
{
    const int32_t K = g.K;
    std::vector<int64_t> steps((size_t)K), nb((size_t)K);
    int64_t total = 0, max_nb = 0;
    for (int32_t k = 0; k < K; ++k) {
        const int64_t nk = g.h_part_off[k + 1] - g.h_part_off[k];
        steps[(size_t)k] = g.round_steps ? g.round_steps[k] : (S.H == 0 ? nk : (nk > 0 ? S.H : 0));
        nb[(size_t)k] = (steps[(size_t)k] + kLB - 1) / kLB;
        total += nb[(size_t)k];
        if (nb[(size_t)k] > max_nb) max_nb = nb[(size_t)k];
    }
    if (total <= 0 || total > 0x7fffffff) return cudaErrorInvalidConfiguration;
    // Slices: fractions 0 = F_0 < F_1 < ... < F_S = 1 of every partition's walk. The first slice is small (its
    // prepare kernel is the one nothing hides), the next ones are 1.3 times as long as the one before (a slice is
    // prepared on the SMs beside the chains while the one before is walked: when both take about as long per block,
    // doubling makes every chain launch of the ramp wait), up to a sixteenth of the walk or 256 blocks of the longest
    // partition, whichever is more; a slice must fit a region of the record buffer.
    // CHICLE_LA_SLICES=1 keeps every round in one piece (to time the prepare kernel alone), CHICLE_LA_SLICES=n cuts
    // into n equal slices whatever the length (to test the slicing on small problems).
    const int max_slices = lookahead_max_slices();
    std::vector<double> F;
    const char *env = getenv("CHICLE_LA_SLICES");
    const int forced = env ? atoi(env) : 0;
    auto build = [&](double first, double cap) {
        F.assign(1, 0.0);
        double at = 0.0, len = first;
        while (at < 1.0 && (int)F.size() < max_slices) {
            at += len;
            F.push_back(at < 1.0 ? at : 1.0);
            len = len * 1.3 < cap ? len * 1.3 : cap;
        }
        F.back() = 1.0;
    };
    double cap = 1.0;
    if (forced >= 1 && (forced == 1 || g.la_stream)) {
        const int n = forced > max_slices ? max_slices : forced;
        F.assign(1, 0.0);
        for (int s = 1; s <= n; ++s) F.push_back((double)s / n);
    } else if ((g.la_overlap && !g.la_stream) || g.la_regions == 1 || max_nb < 512) {
        F = {0.0, 1.0};
    } else {
        cap = 1.0 / 16;
        if (cap * (double)max_nb < 256.0) cap = 256.0 / (double)max_nb;
        build(cap / 8, cap);
    }
    std::vector<int64_t> h;
    std::vector<int64_t> blocks;
    for (int attempt = 0; attempt < 24; ++attempt) {
        const int Sn = (int)F.size() - 1;
        h.assign((size_t)Sn * (3 * (size_t)K + 2), 0); // per slice: step counts, first steps, first blocks (K + 1), 0 for the cursor
        const size_t per = 3 * (size_t)K + 2;
        blocks.assign((size_t)Sn, 0);
        int64_t worst = 0;
        for (int32_t k = 0; k < K; ++k) {
            const int64_t nbk = nb[(size_t)k];
            int64_t prev = 0;
            for (int s = 0; s < Sn; ++s) {
                int64_t cut = s + 1 == Sn ? nbk : (int64_t)((double)nbk * F[(size_t)s + 1]);
                cut = cut < prev ? prev : (cut > nbk ? nbk : cut);
                const int64_t first = prev * kLB;
                const int64_t last = s + 1 == Sn ? steps[(size_t)k] : cut * kLB;
                int64_t *hs = h.data() + (size_t)s * per;
                hs[k] = last - first;
                hs[K + k] = first;
                blocks[(size_t)s] += (last - first + kLB - 1) / kLB;
                hs[2 * K + k + 1] = blocks[(size_t)s];
                prev = cut;
            }
        }
        for (int s = 0; s < Sn; ++s) worst = blocks[(size_t)s] > worst ? blocks[(size_t)s] : worst;
        if (worst <= g.la_region_blocks) break;
        // finer: equal slices, twice as many as would just fit
        int n = (int)((total + g.la_region_blocks - 1) / g.la_region_blocks) * (attempt + 2);
        if (n > max_slices) n = max_slices;
        if (!g.la_stream || g.la_regions < 2 || attempt == 23) return cudaErrorInvalidConfiguration;
        F.assign(1, 0.0);
        for (int s = 1; s <= n; ++s) F.push_back((double)s / n);
    }
    const int Sn = (int)F.size() - 1;
    cudaError_t e = launch_words(g, g.la_slice, h.data(), h.size());
    if (e != cudaSuccess) return e;
    const char *drop = getenv("CHICLE_TEST_DROP_RECORD"); // test aid: leave one block's records unpublished
    const size_t C = (size_t)1 << g.la_logC;
    const bool tables = g.la_tab_bins > 0 && S.sigma * g.max_sqnorm <= tab_max_q(g.la_tab_bins) * S.lam_n;
    std::vector<LookParams> P((size_t)Sn);
    for (int s = 0; s < Sn; ++s) {
        const int r = s % g.la_regions;
        LookParams &p = P[(size_t)s];
        p = LookParams{};
        p.S = S;
        p.S.H = 0;
        int64_t *hs = g.la_slice + (size_t)s * (3 * (size_t)K + 2);
        p.S.steps_k = hs;
        p.S.first_k = hs + K;
        p.rec = static_cast<unsigned char *>(g.la_rec) + (size_t)r * g.la_region_bytes;
        p.dirS = static_cast<BlkDir *>(g.la_dir) + (size_t)r * (size_t)g.la_region_blocks * C;
        p.cursor = reinterpret_cast<unsigned long long *>(hs + 3 * K + 1);
        p.timing = g.la_timing;
        p.pool_off = g.la_pool_off;
        p.pool_cap = g.la_region_bytes - g.la_pool_off;
        p.pool_piece = g.la_pool_piece;
        p.blk_base = hs + 2 * K;
        p.K = K;
        p.logC = g.la_logC;
        p.depth = g.la_depth;
        p.sub_room = g.la_sub_room;
        p.slots = g.la_slots;
        p.hotc = g.la_hotc;
        p.far_cap = chain_kind(g) == kSplit ? g.la_far_cap : INT32_MAX;
        p.n_blocks = blocks[(size_t)s];
        p.drop_block = (drop && s == 0) ? atoll(drop) : -1;
        p.nnz = g.nnz;
        p.tab_bins = tables ? g.la_tab_bins : 0;
        p.tab_off = g.la_tab_off;
        p.model_in = s == 0 ? 1 : 0;
        p.model_out = s == Sn - 1 ? 1 : 0;
    }
    g.la_last_slices = Sn;
    g.solver_launches += 2 * Sn; // a prepare and a chain launch per slice
    switch (g.loss) {
    case CHICLE_LOSS_HINGE_DUAL: return launch_slices<CHICLE_LOSS_HINGE_DUAL>(g, P);
    case CHICLE_LOSS_LOGISTIC_DUAL: return launch_slices<CHICLE_LOSS_LOGISTIC_DUAL>(g, P);
    default: return launch_slices<CHICLE_LOSS_RIDGE_PRIMAL>(g, P);
    }
}

} // namespace chicle
